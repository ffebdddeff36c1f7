"""Performance cases of the early-exit decode library, through its public entry points.

Each case is one call (or one request's calls) as a program that serves a model makes them:

  kind       what a user does
  request    one request: reset, prompt, then n tokens decoded on the device (`decode_n`), exits
             imposed at a rate (the gate still runs); the headline use
  steps      the caller's own loop: `decode_step` once per token, each waited for (latency)
  calibrate  teacher-forced full-depth steps over a token stream (`calibrate`): every readout and
             the LM head at every step
  prefill    a prompt alone, the time to the first token
  repass     a short prompt, a run of early exits, then the full-depth re-pass of all of them
  attention  `attention_decode` on a caller's paged cache
  vocab      `vocab_signals` on a caller's row-major unembedding, logits kept
  tau        `select_tau` over a calibration run's confidences

Model cases keep what a server keeps: an Engine with its weights, readouts and debug logits on (the
logits come back beside the tokens).  Shapes are the repository's workloads (tiny, 0.5b, 1.5b, 3b),
at their own depth where a case stands for the whole call and with fewer layers elsewhere (a layer's
time does not depend on how many there are; making the weights does).  Layers alternate between two
sets of random weights: every layer still has its own copy in device memory.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2609_14144_gb300 as ee

# d_model, query heads, kv heads, head_dim, ffn_dim, layers of the whole model
SHAPES = {
    "tiny": (256, 4, 2, 64, 688, 4),
    "0.5b": (896, 14, 2, 64, 4864, 24),
    "1.5b": (1536, 12, 2, 128, 8960, 28),
    "3b": (2048, 16, 2, 128, 11008, 36),
}
VOCAB = 151936
PAGE = 64


def listed():
    return [
        # the smallest call: one token at a time on the tiny shape, a ragged prompt; launches and latency
        {"name": "steps_tiny", "kind": "steps", "shape": "tiny", "layers": 4, "vocab": 4096, "readouts": 1, "prompt": 19,
         "n": 8, "exits": 0.5, "bias": False},
        # the whole 0.5B-shaped model, a caller that waits for each token
        {"name": "steps_0p5b", "kind": "steps", "shape": "0.5b", "layers": 24, "vocab": VOCAB, "readouts": 1,
         "prompt": 515, "n": 32, "exits": 0.5, "bias": False},
        # the headline: the whole 1.5B-shaped model, 512-token prompt, half of the tokens exit at half depth
        {"name": "request_1p5b", "kind": "request", "shape": "1.5b", "layers": 28, "vocab": VOCAB, "readouts": 1,
         "prompt": 512, "n": 32, "exits": 0.5, "bias": False},
        # long context: three readouts, an odd prompt of thousands of tokens, then decode far into it
        {"name": "request_long", "kind": "request", "shape": "1.5b", "layers": 8, "vocab": VOCAB, "readouts": 3,
         "prompt": 6001, "n": 32, "exits": 0.5, "bias": False},
        # full depth with every readout and the LM head at each step, the largest weights, biases on
        {"name": "calibrate_3b", "kind": "calibrate", "shape": "3b", "layers": 8, "vocab": VOCAB, "readouts": 1,
         "prompt": 520, "n": 40, "exits": 0.0, "bias": True},
        # time to the first token: a short chat turn, the headline's prompt, a long document
        {"name": "prefill_33", "kind": "prefill", "shape": "0.5b", "layers": 24, "vocab": VOCAB, "readouts": 0,
         "prompt": 33, "n": 0, "exits": 0.0, "bias": False},
        {"name": "prefill_512", "kind": "prefill", "shape": "1.5b", "layers": 12, "vocab": VOCAB, "readouts": 0,
         "prompt": 512, "n": 0, "exits": 0.0, "bias": False},
        {"name": "prefill_4099", "kind": "prefill", "shape": "3b", "layers": 6, "vocab": 32000, "readouts": 0,
         "prompt": 4099, "n": 0, "exits": 0.0, "bias": True},
        # the periodic full-depth pass over early exits
        {"name": "repass_1p5b", "kind": "repass", "shape": "1.5b", "layers": 12, "vocab": 32000, "readouts": 1,
         "prompt": 40, "n": 24, "exits": 1.0, "bias": False},
        # the standalone ops of a program that keeps its own cache, unembedding or confidences
        {"name": "attention_16k", "kind": "attention", "shape": "1.5b", "T": 16411, "page": 64},
        {"name": "vocab_1p5b", "kind": "vocab", "shape": "1.5b", "vocab": VOCAB},
        {"name": "tau_2047", "kind": "tau", "n": 2047, "readouts": 3, "target": 0.9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["request", "request", "steps", "calibrate", "prefill", "prefill", "repass", "attention", "vocab",
                       "tau"])
    shape = rng.choice(list(SHAPES))
    if kind == "attention":
        return {"kind": kind, "shape": shape, "T": _log_int(rng, 17, 32768), "page": rng.choice([16, 64, 256])}
    if kind == "vocab":
        return {"kind": kind, "shape": shape, "vocab": _log_int(rng, 4000, VOCAB)}
    if kind == "tau":
        return {"kind": kind, "n": _log_int(rng, 100, 20000), "readouts": rng.randint(1, 4),
                "target": rng.choice([0.5, 0.9, 0.95])}
    # depths and vocabularies that are quick to make; prompts and tokens over the listed range
    layers = rng.randint(3, 8 if shape != "3b" else 6)
    c = {"kind": kind, "shape": shape, "layers": layers, "vocab": rng.choice([4096, 32000, 50257]),
         "readouts": rng.randint(1, 3 if layers > 3 else 1), "prompt": _log_int(rng, 5, 1500), "n": _log_int(rng, 4, 64),
         "exits": rng.choice([0.0, 0.08, 0.5, 0.96]), "bias": rng.random() < 0.5}
    if kind == "prefill":
        c.update(readouts=0, n=0, exits=0.0, prompt=_log_int(rng, 3, 5000))
    if kind == "calibrate":
        c.update(exits=0.0)
    if kind == "repass":
        c.update(readouts=1, exits=1.0, prompt=_log_int(rng, 5, 700))
    return c


# ------------------------------------------------------------------ inputs


def _shape(c):
    d, A, K, D, F, _ = SHAPES[c["shape"]]
    return SimpleNamespace(n_layers=c["layers"], d_model=d, n_heads=A, n_kv_heads=K, head_dim=D, ffn_dim=F,
                           vocab=c["vocab"], rms_eps=1e-6, rope_base=10000.0, qkv_bias=c["bias"],
                           max_ctx=c["prompt"] + max(c["n"], 1))


def _readout_layers(c):
    """Evenly spaced: half depth for one readout, quarters for three."""
    L, R = c["layers"], c["readouts"]
    return [max(1, L * (r + 1) // (R + 1)) for r in range(R)]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape, std=0.02):
    """bf16 N(0, std^2) on the GPU."""
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(std).to(torch.bfloat16)


def _weights(c, seed):
    """The model's bf16 tensors on the GPU: two sets of layer weights, embedding, untied LM head,
    gains, readouts at I + N(0, 0.02^2).  The final gain spreads the logits so that top-1
    probabilities lie all over (0, 1)."""
    d, A, K, D, F, _ = SHAPES[c["shape"]]
    V, g = c["vocab"], _gen(seed)
    sets = []
    for _ in range(min(2, c["layers"])):
        w = {"wq": _normal(g, A * D, d), "wk": _normal(g, K * D, d), "wv": _normal(g, K * D, d),
             "wo": _normal(g, d, A * D), "wg": _normal(g, F, d), "wu": _normal(g, F, d), "wd": _normal(g, d, F),
             "attn_norm": 1 + _normal(g, d, std=0.1), "mlp_norm": 1 + _normal(g, d, std=0.1)}
        if c["bias"]:
            w.update(bq=_normal(g, A * D), bk=_normal(g, K * D), bv=_normal(g, K * D))
        sets.append(w)
    gain = 1.5 * math.sqrt(2 * math.log(V)) / (0.02 * math.sqrt(d))
    eye = torch.eye(d, device="cuda")
    return {"sets": sets, "embed": _normal(g, V, d), "lm_head": _normal(g, V, d),
            "final_norm": torch.full((d,), gain, device="cuda").to(torch.bfloat16),
            "readouts": [(k, (eye + _normal(g, d, d).float()).to(torch.bfloat16), _normal(g, d))
                         for k in _readout_layers(c)]}


def _host(t):
    return t.cpu().view(torch.int16).numpy().view(np.uint16)


def _tokens(c, seed):
    """Prompt ids, the decoded stream's ids (for teacher forcing) and the imposed exits."""
    r = np.random.RandomState(seed % (1 << 31))
    prompt = r.randint(0, c["vocab"], c["prompt"]).astype(np.int32)
    ids = r.randint(0, c["vocab"], max(c["n"], 1)).astype(np.int32)
    force = np.full(max(c["n"], 1), ee.FORCE_FULL, np.int8)
    if c["exits"] > 0:
        # c["exits"] of the steps, spread by the seed, each at one of the readouts
        out = r.permutation(c["n"])[: int(round(c["exits"] * c["n"]))]
        force[out] = [ee.FORCE_EXIT_AT(int(x)) for x in r.randint(0, c["readouts"], len(out))]
        if c["exits"] < 1:
            force[-1] = ee.FORCE_FULL  # the last token's logits are the LM head's
    return prompt, ids, force


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "attention":
        d, A, K, D, F, _ = SHAPES[c["shape"]]
        g, P = _gen(seed), c["page"]
        pages = (c["T"] + P - 1) // P
        return {"case": c, "q": torch.randn(A * D, generator=g, device="cuda"),
                "k": _normal(g, pages, K, P, D, std=1.0), "v": _normal(g, pages, K, P, D, std=1.0),
                "table": torch.randperm(pages, generator=g, device="cuda").to(torch.int32)}
    if kind == "vocab":
        d, V, g = SHAPES[c["shape"]][0], c["vocab"], _gen(seed)
        gain = 1.5 * math.sqrt(2 * math.log(V)) / (0.02 * math.sqrt(d))
        return {"case": c, "x": torch.randn(d, generator=g, device="cuda") * 3, "U": _normal(g, V, d),
                "gain": torch.full((d,), gain, device="cuda").to(torch.bfloat16),
                "logits": torch.empty(V, device="cuda")}
    if kind == "tau":
        g, n = _gen(seed), c["n"]
        conf = torch.rand(n, c["readouts"], generator=g, device="cuda")
        # more confident answers are acceptable more often
        ok = torch.rand(n, generator=g, device="cuda") < 0.4 + 0.58 * conf[:, 0]
        return {"case": c, "conf": conf, "member": ok.to(torch.int32)}
    w = _weights(c, seed)
    hosts = [{k: _host(v) for k, v in s.items()} for s in w["sets"]]
    model = {"embed": _host(w["embed"]), "lm_head": _host(w["lm_head"]), "final_norm": _host(w["final_norm"]),
             "layers": [hosts[j % len(hosts)] for j in range(c["layers"])],
             "readouts": [(k, _host(W), _host(b)) for k, W, b in w["readouts"]]}
    del w
    eng = ee.Engine(_shape(c), model, page_size=PAGE)
    eng.set_option(ee.OPT_DEBUG_LOGITS, 1)
    prompt, ids, force = _tokens(c, seed)
    return {"case": c, "engine": eng, "prompt": prompt, "ids": ids, "force": force}


# ------------------------------------------------------------------ one pass


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "attention":
        d, A, K, D, F, _ = SHAPES[c["shape"]]
        return ee.attention_decode(state["q"], state["k"], state["v"], state["table"], c["T"], A, K, D, c["page"])
    if kind == "vocab":
        token, signals = ee.vocab_signals(state["x"], state["gain"], state["U"], 1e-6, logits=state["logits"])
        return {"token": token, "signals": signals, "logits": state["logits"]}
    if kind == "tau":
        return ee.select_tau(state["conf"][:, 0], state["member"], c["target"])
    eng, taus = state["engine"], [0.5] * c["readouts"]
    eng.reset()
    first = eng.prefill(state["prompt"])
    if kind == "prefill":
        return {"first": first, "logits": eng.final_logits(), "hidden": eng.hidden_final()}
    if kind == "request":
        tokens, exits, conf = eng.decode_n(c["n"], taus, schedule=state["force"])
        return {"first": first, "tokens": tokens, "exits": exits, "confidence": conf, "logits": eng.final_logits()}
    if kind == "calibrate":
        # (the membership flags are mass < share: the mass says more)
        conf, _, mass = eng.calibrate(state["ids"], 0.9)
        return {"first": first, "confidence": conf, "mass": mass, "logits": eng.final_logits()}
    if kind == "steps":
        conf = []
        for i in range(c["n"]):
            conf.append(eng.decode_step(int(state["ids"][i]), taus, int(state["force"][i]))["confidence"][-1])
        return {"first": first, "confidence": np.array(conf, np.float32), "logits": eng.final_logits()}
    # repass
    tokens, exits, conf = eng.decode_n(c["n"], taus, schedule=state["force"])
    n = eng.repass(c["prompt"], c["prompt"] + c["n"])
    return {"first": first, "tokens": tokens, "confidence": conf, "n": n, "hidden": eng.hidden_final()}


# ------------------------------------------------------------------ what a pass cannot do without


def _layer_params(c):
    d, A, K, D, F, _ = SHAPES[c["shape"]]
    return (A + 2 * K) * D * d + A * D * d + 3 * F * d


def work(case):
    c, kind = case, case["kind"]
    if kind == "attention":
        d, A, K, D, F, _ = SHAPES[c["shape"]]
        return {"bytes": 4 * K * D * c["T"] + 8 * A * D, "flops": 4 * A * D * c["T"]}
    if kind == "vocab":
        d = SHAPES[c["shape"]][0]
        return {"bytes": 2 * c["vocab"] * d + 6 * d + 4 * c["vocab"], "flops": 2 * c["vocab"] * d}
    if kind == "tau":
        return {"bytes": 8 * c["n"] + 4, "flops": 2 * c["n"] * math.log2(c["n"] + 1)}
    d, A, K, D, F, _ = SHAPES[c["shape"]]
    L, V, n0, P = c["layers"], c["vocab"], c["prompt"], _layer_params(c)
    kv = 4 * K * D  # bytes of one position's keys and values in one layer
    # the prompt: every weight once, its cache written, the LM head on its last position
    nbytes = L * (2 * P + kv * n0) + 2 * V * d + 2 * n0 * d
    flops = L * (2 * P * n0 + 2 * A * D * n0 * n0) + 2 * V * d
    marks = _readout_layers(c)
    force = _tokens(c, 0)[2] if c["n"] else []
    for i in range(c["n"]):
        T = n0 + i + 1
        at = int(force[i]) - 2  # the readout this step leaves at; -1: none
        layers, heads = (marks[at], at + 1) if at >= 0 else (L, c["readouts"] + 1)
        ros = at + 1 if at >= 0 else c["readouts"]
        nbytes += layers * (2 * P + kv * T) + ros * 2 * d * d + heads * 2 * V * d
        nbytes += (L - layers) * (2 * 2 * K * D * d + kv)
        flops += layers * (2 * P + 4 * A * D * T) + heads * 2 * V * d + ros * 2 * d * d + (L - layers) * 4 * K * D * d
    if kind == "repass":  # the layers above the exit once more, all positions together
        up = L - marks[0]
        nbytes += up * (2 * P + kv * (n0 + 2 * c["n"]))
        flops += up * c["n"] * (2 * P + 4 * A * D * (n0 + c["n"] / 2))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what two builds of the same precision differ by (the tcgen05 prompt against
    one position at a time, the persistent layers against five launches a layer; 60 runs over these
    ranges); for the ops in 32 bits, their distance from 64 bits.  The bf16 cache amplifies a
    difference of summation order of 1e-7 to these sizes: see `exact`."""
    if case["kind"] == "attention":  # seen against 64 bits: 3.4e-7
        return {"rel": 2e-6, "max": 4e-5}
    if case["kind"] == "vocab":  # 1.4e-7 in the logits, 1.3e-6 in the signals
        return {"rel": 5e-6, "max": 4e-5}
    if case["kind"] == "tau":
        return "exact"
    if case["kind"] == "prefill":  # seen: 2.2e-4, 9.4e-4
        return {"rel": 1e-3, "max": 4e-3}
    return {"rel": 4e-3, "max": 2.2e-2}  # seen: 1.0e-3, 5.6e-3 (calibration masses)


# ------------------------------------------------------------------ the same in 64 bits


def _bf16(x):
    return x.to(torch.bfloat16).double()


class _Exact:
    """The decoder in float64: bf16 weights, the key/value cache rounded to bf16 (that is what the
    cache holds), everything else in 64 bits."""

    def __init__(self, c, seed):
        self.c, self.w = c, _weights(c, seed)
        d, self.A, self.K, self.D, F, _ = SHAPES[c["shape"]]
        n = c["prompt"] + max(c["n"], 1)
        self.k = torch.zeros(c["layers"], n, self.K, self.D, dtype=torch.float64, device="cuda")
        self.v = torch.zeros_like(self.k)
        half = self.D // 2
        ang = torch.arange(n, dtype=torch.float64)[:, None] * 10000.0 ** (-torch.arange(half, dtype=torch.float64) / half)
        self.cos, self.sin = (f(ang).float().double().cuda() for f in (torch.cos, torch.sin))  # a 32-bit table

    def norm(self, x, g):
        return x / torch.sqrt((x * x).mean(-1, keepdim=True) + 1e-6) * g.double()

    def rope(self, x, p0):
        n, half = x.shape[0], self.D // 2
        c, s = self.cos[p0 : p0 + n, None], self.sin[p0 : p0 + n, None]
        a, b = x[..., :half], x[..., half:]
        return torch.cat([a * c - b * s, a * s + b * c], -1)

    def lin(self, w, name, x, heads=None):
        y = x @ w["w" + name].double().T
        if heads and self.c["bias"]:
            y = y + w["b" + name].double()
        return y.view(x.shape[0], heads, self.D) if heads else y

    def fill(self, x, p0, j):
        """Keys and values of layer j at positions p0.. from the residual x; the normalised input."""
        w = self.w["sets"][j % len(self.w["sets"])]
        z, n = self.norm(x, w["attn_norm"]), x.shape[0]
        self.k[j, p0 : p0 + n] = _bf16(self.rope(self.lin(w, "k", z, self.K), p0))
        self.v[j, p0 : p0 + n] = _bf16(self.lin(w, "v", z, self.K))
        return w, z

    def layers(self, x, p0, j0, j1):
        n = x.shape[0]
        for j in range(j0, j1):
            w, z = self.fill(x, p0, j)
            q = self.rope(self.lin(w, "q", z, self.A), p0) / math.sqrt(self.D)
            o = torch.empty(n, self.A, self.D, dtype=torch.float64, device="cuda")
            for h in range(self.A):
                g = h * self.K // self.A
                for r in range(0, n, 1024):
                    m = min(n, r + 1024)
                    s = q[r:m, h] @ self.k[j, : p0 + m, g].T
                    s.masked_fill_(torch.arange(p0 + m, device="cuda")[None] > torch.arange(p0 + r, p0 + m, device="cuda")[:, None],
                                   -math.inf)
                    o[r:m, h] = torch.softmax(s, -1) @ self.v[j, : p0 + m, g]
            x = x + self.lin(w, "o", o.view(n, -1))
            z = self.norm(x, w["mlp_norm"])
            x = x + self.lin(w, "d", torch.nn.functional.silu(self.lin(w, "g", z)) * self.lin(w, "u", z))
        return x

    def embed(self, ids):
        return self.w["embed"][torch.as_tensor(np.atleast_1d(ids).astype(np.int64), device="cuda")].double()

    def logits(self, x):
        z, U = self.norm(x, self.w["final_norm"]), self.w["lm_head"]
        return torch.cat([z @ u.double().T for u in U.split(16384)], -1)

    def readout(self, r, x):
        _, W, b = self.w["readouts"][r]
        return self.logits(x @ W.double().T + b.double())


# Cached positions from which the distance to 64 bits says something about a build.  A cache entry
# whose value lies near the middle of two bf16 numbers is rounded one way or the other by luck, and the
# rounding step (4e-3) outweighs all 32-bit error.  Over a short cache a handful of such entries decide:
# on a single layer one of two builds of the same precision was 5 times closer to 64 bits with one seed
# and 5 times further with the next.  From about 500 positions the many entries even out.  The nucleus
# masses (few steps have one that is not near 1) differed by up to 5 times either way at every length.
EXACT_FROM = 500


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind not in ("tau", "vocab", "attention") and c["prompt"] + c["n"] < EXACT_FROM:
        return None
    if kind == "tau":
        s = prepare(c, seed)
        conf, ok = s["conf"][:, 0].cpu().numpy(), s["member"].cpu().numpy() != 0
        best = np.inf
        for t in np.concatenate([[-np.inf], conf]):
            early = conf > t
            if early.any() and ok[early].sum() >= float(np.float32(c["target"])) * early.sum():
                best = min(best, t)
        return np.array([best], np.float32)
    if kind == "vocab":
        s = prepare(c, seed)
        x = s["x"].double()
        z = x / torch.sqrt((x * x).mean() + float(np.float32(1e-6))) * s["gain"].double()
        logits = torch.cat([u.double() @ z for u in s["U"].split(16384)])
        p = torch.softmax(logits, 0)
        top = torch.topk(p, 2).values
        sig = torch.stack([top[0], top[0] - top[1], (p * torch.log_softmax(logits, 0)).sum()])
        return {"token": None, "signals": sig, "logits": logits}
    if kind == "attention":
        s = prepare(c, seed)
        d, A, K, D, F, _ = SHAPES[c["shape"]]
        k, v = (t[s["table"].long()].double().permute(1, 0, 2, 3).reshape(K, -1, D)[:, : c["T"]] for t in (s["k"], s["v"]))
        q = s["q"].double().view(K, A // K, D)
        return (torch.softmax(q @ k.transpose(1, 2) / math.sqrt(D), -1) @ v).reshape(-1)
    m, (prompt, ids, force) = _Exact(c, seed), _tokens(c, seed)
    L, n0, n = c["layers"], c["prompt"], c["n"]
    if kind == "prefill" or kind == "calibrate":
        stream = prompt if kind == "prefill" else np.concatenate([prompt, ids])
        marks = _readout_layers(c)
        x, conf, j = m.embed(stream), [], 0
        for r, k in enumerate(marks):
            x = m.layers(x, 0, j, k)
            conf.append(torch.softmax(m.readout(r, x[n0:]), -1))
            j = k
        x = m.layers(x, 0, j, L)
        if kind == "prefill":
            return {"first": None, "logits": m.logits(x[-1:])[0], "hidden": x[-1]}
        return {"first": None, "confidence": torch.stack([v.max(-1).values for v in conf], 1), "mass": None,
                "logits": m.logits(x[-1:])[0]}
    x = m.layers(m.embed(prompt), 0, 0, L)
    logits, conf, left, marks = m.logits(x[-1:])[0], [], [], _readout_layers(c)
    tok = int(logits.argmax())
    for i in range(n):
        x = m.embed(ids[i] if kind == "steps" else tok)
        p, j, out = n0 + i, 0, int(force[i]) - 2
        for r, k in enumerate(marks):
            x = m.layers(x, p, j, k)
            j = k
            if r <= out or out < 0:
                y = m.readout(r, x)[0]
                top = torch.softmax(y, -1).max()
            if r == out:
                break
        if out >= 0:
            left.append((p, x))
            tok = int(y.argmax())
            for jj in range(j, L):
                m.fill(x, p, jj)
        else:
            x = m.layers(x, p, j, L)
            logits = m.logits(x)[0]
            tok = int(logits.argmax())
        conf.append(float(top))
    if kind == "repass":
        for p, x in left:
            x = m.layers(x, p, marks[0], L)
        return {"first": None, "tokens": None, "confidence": np.array(conf), "n": None, "hidden": x[0]}
    res = {"first": None, "confidence": np.array(conf), "logits": logits}
    return dict(res, tokens=None, exits=None) if kind == "request" else res
