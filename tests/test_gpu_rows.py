"""The multi-position layer pass on the GPU (needs a GB300).

With EE_OPT_ROWS = 1 the prompt and the re-pass run each layer over batches
of up to ROWS_MAX positions, the projections on the tcgen05 tensor cores (2: the
same batches with warp-level mma products).  Checked against the oracle (first token exact outside
the 1e-3 top-2 band, final hidden state and logits and every cache entry
within 1e-2 relative, which (layer, position) entries were computed bit for
bit) and against the same engine one position at a time (EE_OPT_ROWS = 0,
the default): both keep activations at fp32 precision (the batched products
through three bf16 parts of each activation), so fp32 results agree within
1e-3 relative; cache entries are bf16, where one rounding step is 4e-3."""
import math
import os
import re

import numpy as np
import pytest

import oracle
import synth
from helpers import EXCLUDE_EPS, REL_TOL, bf16_bits_to_f32, check_kv, rel_err, to_bf16_bits

pytestmark = pytest.mark.gpu

TINY = synth.CONFIGS["tiny"]
_HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_14144_gb300", "csrc",
                       "ee_internal.h")
ROWS_MAX = int(re.search(r"kRowsMax = (\d+);", open(_HEADER).read()).group(1))  # positions per batch
PATH_TOL = 1e-3  # fp32 results of the batched and the one-position paths


@pytest.fixture(scope="module")
def tiny_model():
    return synth.make_model(TINY)


def _top2_gap(logits) -> float:
    z = np.asarray(logits, np.float64)
    p = np.exp(z - z.max())
    p /= p.sum()
    a = np.sort(p)
    return float(a[-1] - a[-2])


def _engine(shape, model, max_ctx, rows=True, pages=None):
    from paper_2609_14144_gb300 import OPT_DEBUG_LOGITS, OPT_ROWS, Engine

    eng = Engine(shape, model, max_ctx=max_ctx)
    eng.set_option(OPT_ROWS, int(rows))
    eng.set_option(OPT_DEBUG_LOGITS, 1)
    if pages is not None:
        eng.set_page_table(pages)
    return eng


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("n", [1, 7, 16, 17, 255, 256, 257, 600, ROWS_MAX - 1, ROWS_MAX, ROWS_MAX + 1, 2 * ROWS_MAX + 88])
def test_tiny_prompt_batches_match_oracle(tiny_model, n, mode):
    """Prompts of one position, a partial first group of 16 rows (the
    tcgen05 products' N step), one full group, a full group and one row, one
    short of a full row block (256), one full block, two blocks, three; and one
    short of a full batch, one full batch, two batches, and three with a ragged
    tail, on the tcgen05 and the warp-level products (F = 688: a ragged last K
    stage)."""
    prompt = synth.token_ids(TINY.seed, 901, n, TINY.vocab)
    orc = oracle.Oracle(TINY, tiny_model, max_ctx=n + 1)
    tok_o, cap = orc.prefill(prompt, capture=True)
    eng = _engine(TINY, tiny_model, n + 1, rows=mode)
    tok_g = eng.prefill(prompt)
    if _top2_gap(cap["final_logits"]) >= EXCLUDE_EPS:
        assert tok_g == tok_o
    assert eng.position == n
    assert rel_err(eng.hidden_final(), cap["h_final"]) <= REL_TOL
    assert rel_err(eng.final_logits(), cap["final_logits"]) <= REL_TOL
    check_kv(orc, eng, TINY, n)


def test_tiny_prompt_permuted_pages_and_bias():
    shape = TINY.replace(qkv_bias=True)
    model = synth.make_model(shape)
    n = 260
    pages = np.random.default_rng(3).permutation((n + 1 + 63) // 64).astype(np.int32)
    prompt = synth.token_ids(shape.seed, 902, n, shape.vocab)
    orc = oracle.Oracle(shape, model, max_ctx=n + 1)
    tok_o, cap = orc.prefill(prompt, capture=True)
    eng = _engine(shape, model, n + 1, pages=pages)
    tok_g = eng.prefill(prompt)
    if _top2_gap(cap["final_logits"]) >= EXCLUDE_EPS:
        assert tok_g == tok_o
    check_kv(orc, eng, shape, n)


def test_tiny_prompt_paths_agree(tiny_model):
    """The batched prompt and the one-position path: same first token, fp32
    states within 1e-3, and the same continuation."""
    n = 300
    prompt = synth.token_ids(TINY.seed, 903, n, TINY.vocab)
    a = _engine(TINY, tiny_model, n + 9, rows=True)
    b = _engine(TINY, tiny_model, n + 9, rows=False)
    ta, tb = a.prefill(prompt), b.prefill(prompt)
    if _top2_gap(b.final_logits()) >= EXCLUDE_EPS:
        assert ta == tb
    assert rel_err(a.hidden_final(), b.hidden_final()) <= PATH_TOL
    assert rel_err(a.final_logits(), b.final_logits()) <= PATH_TOL
    for j in range(TINY.n_layers):
        for t in range(n):
            assert a.kv_src(j, t) == b.kv_src(j, t) == 1
            ka, va = a.kv(j, t)
            kb, vb = b.kv(j, t)
            assert rel_err(ka, kb) <= REL_TOL and rel_err(va, vb) <= REL_TOL, (j, t)
    tok = tb
    for _ in range(8):  # the same inputs to both
        ra = a.decode_step(tok, [2.0], oracle.FORCE_FULL)
        rb = b.decode_step(tok, [2.0], oracle.FORCE_FULL)
        if _top2_gap(b.final_logits()) >= EXCLUDE_EPS:
            assert ra["token"] == rb["token"]
        assert abs(ra["confidence"][0] - rb["confidence"][0]) <= 5e-4
        tok = rb["token"]


def _cut(x, parts):
    """x as the sum of its first bf16 parts (each the rounding of what is left)."""
    out, rest = np.zeros_like(x), x.astype(np.float32)
    for _ in range(parts):
        p = bf16_bits_to_f32(to_bf16_bits(rest))
        out, rest = out + p, rest - p
    return out


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("n", [70, 129, 700, 1300])
@pytest.mark.parametrize("spread,tol", [(1, 6e-7), (150, 3e-6)])
def test_tcgen05_attention_parts_and_growing_scores(n, D, spread, tol):
    """The last row's attention of the first layer (16 heads, up to 21 blocks of
    64 keys) against 64 bits over the engine's own cache.  spread 1: flat
    probabilities; the third bf16 part of each is 2^-18 of it, 2.2e-6 of the
    output in the mean.  spread 150: scores tens apart, so that the largest so
    far comes in early, middle and late blocks, rows of a tile grow their
    references in different blocks and within chains; the third part of the
    queries moves a score by 1e-4.  What the fp32 sums, the products of Q and O
    and the exponentials leave is 4e-7 and 1.5e-6; a reference whose queries or
    probabilities lack their third part misses the result by more than the
    bound."""
    shape = TINY.replace(n_heads=16, head_dim=D, n_layers=2, readout_layers=(1,))
    model = synth.make_model(shape)
    for lw in model["layers"]:
        lw["wd"] = np.zeros_like(lw["wd"])
    lw = model["layers"][0]
    lw["wo"] = to_bf16_bits(bf16_bits_to_f32(lw["wo"]) * 50)  # large beside the residual
    lw["wq"] = to_bf16_bits(bf16_bits_to_f32(lw["wq"]) * spread)
    model["layers"][1]["wo"] = np.zeros_like(lw["wo"])
    prompt = synth.token_ids(shape.seed, 960 + n, n, shape.vocab)
    eng = _engine(shape, model, n + 1)
    eng.prefill(prompt)
    A, K = shape.n_heads, shape.n_kv_heads
    kv = [eng.kv(0, t) for t in range(n)]
    k, v = (np.stack(x).astype(np.float64).reshape(n, K, D).repeat(A // K, axis=1) for x in zip(*kv))
    w = {name: synth.bf16_to_f32(lw[name]).astype(np.float64) for name in ("wq", "wo", "attn_norm")}
    x = synth.bf16_to_f32(model["embed"])[prompt[-1]].astype(np.float64)
    z = x / np.sqrt((x * x).mean() + np.float32(shape.rms_eps)) * w["attn_norm"]
    ang = (n - 1) * shape.rope_base ** (-2.0 * np.arange(D // 2) / D)
    c, s = (f(ang).astype(np.float32).astype(np.float64) for f in (np.cos, np.sin))
    a, b = (w["wq"] @ z).reshape(A, 2, D // 2).transpose(1, 0, 2)
    q = np.concatenate([a * c - b * s, a * s + b * c], 1) / math.sqrt(D)

    def attend(q, parts=None):
        sc = np.einsum("hd,thd->ht", q, k)
        p = np.exp(sc - sc.max(1, keepdims=True))
        o = np.einsum("ht,thd->hd", _cut(p, parts) if parts else p, v) / p.sum(1, keepdims=True)
        return w["wo"] @ o.reshape(-1), sc

    ref, sc = attend(q)
    off = lambda y: np.linalg.norm(y - ref) / np.linalg.norm(ref)
    if spread == 1:
        assert off(attend(q, 2)[0]) > tol
    else:
        assert off(attend(_cut(q, 2))[0]) > tol
        grows = [(h, t) for h in range(A) for t in range(64, n) if sc[h, t] > sc[h, :t // 64 * 64].max() + 8]
        assert grows or n < 700
    assert off(eng.hidden_final() - x) <= tol, off(eng.hidden_final() - x)


@pytest.mark.parametrize("D,page", [(64, 16), (64, 256), (128, 64), (128, 32)])
@pytest.mark.parametrize("n", [64, 65, 127, 129, 193, 513, 1025])
def test_tcgen05_attention_row_and_key_edges(n, D, page):
    """The batched attention at the edges of its row tile (128 rows, from 65
    on), of a block of 64 keys and of a key split, with pages shorter and
    longer than a block in any order, seven query heads to a key-value head;
    the batch at the edges of the products' row blocks (256 rows; 513 makes
    three of 176) and of its own size (1025 makes two batches): against the
    same prompt one position at a time (fp32 path)."""
    from paper_2609_14144_gb300 import OPT_DEBUG_LOGITS, OPT_ROWS, Engine

    shape = TINY.replace(n_heads=14, head_dim=D, n_layers=2, readout_layers=(1,))
    model = synth.make_model(shape)
    pages = np.random.default_rng(n).permutation((n + 1 + page - 1) // page).astype(np.int32)
    prompt = synth.token_ids(shape.seed, 905, n, shape.vocab)
    got = []
    for rows in (1, 0):
        eng = Engine(shape, model, max_ctx=n + 1, page_size=page)
        eng.set_option(OPT_ROWS, rows)
        eng.set_option(OPT_DEBUG_LOGITS, 1)
        eng.set_page_table(pages)
        eng.prefill(prompt)
        got.append(eng)
    a, b = got
    assert rel_err(a.hidden_final(), b.hidden_final()) <= PATH_TOL
    assert rel_err(a.final_logits(), b.final_logits()) <= PATH_TOL
    for t in sorted({0, 1, 62, 63, n // 2, n - 66, n - 2, n - 1}):
        if 0 <= t < n:  # layer 1's entries carry layer 0's attention of that row
            for x, y in zip(a.kv(1, t), b.kv(1, t)):
                assert rel_err(x, y) <= REL_TOL, t


@pytest.mark.parametrize("n", [33, 65, 300, 700, 1000])
@pytest.mark.parametrize("d", [256, 512, 1024, 1536])
def test_products_in_chains_of_every_length(d, n):
    """1280 inputs of the O projection: with 256, 512, 1024 and 1536 outputs a
    full block's chains hold one, two, three and four stages, and the splits of
    one, two, three and four blocks end in partial chains; a small batch's
    chains have accumulators of their own.  Against one position at a time."""
    shape = TINY.replace(d_model=d, n_heads=20, n_kv_heads=4, n_layers=2, readout_layers=(1,))
    model = synth.make_model(shape)
    prompt = synth.token_ids(shape.seed, 910 + n, n, shape.vocab)
    a, b = (_engine(shape, model, n + 1, rows=r) for r in (1, 0))
    a.prefill(prompt), b.prefill(prompt)
    assert rel_err(a.hidden_final(), b.hidden_final()) <= PATH_TOL
    assert rel_err(a.final_logits(), b.final_logits()) <= PATH_TOL
    for t in sorted({0, n // 2, n - 2, n - 1}):  # layer 1's entries carry layer 0's products of that row
        for x, y in zip(a.kv(1, t), b.kv(1, t)):
            assert rel_err(x, y) <= REL_TOL, t


@pytest.mark.parametrize("n", [48, 64, 400, 1000])
def test_batched_products_round_like_short_chains(n):
    """The feed-forward of one layer (width 256: 8 and 22 stages of 32 columns
    in all) for a prompt's last row, against 64 bits.  The tensor core drops
    what an addition shifts out: half a unit in the last place on average, and
    always towards zero, so it adds up over a chain of additions.  With chains
    of one stage (two additions) the three products come to about 1.6e-7, with
    two or more stages to 2.5e-7 and 3.4e-7; 16 rows scatter by a tenth."""
    shape = TINY.replace(n_layers=2, readout_layers=(1,))
    model = synth.make_model(shape)
    for j, lw in enumerate(model["layers"]):  # layer 0 is its feed-forward alone, layer 1 adds nothing
        lw["wo"] = np.zeros_like(lw["wo"])
        lw["wd"] = to_bf16_bits(bf16_bits_to_f32(lw["wd"]) * (20 if j == 0 else 0))
    w = {k: synth.bf16_to_f32(v).astype(np.float64) for k, v in model["layers"][0].items()}
    embed = synth.bf16_to_f32(model["embed"]).astype(np.float64)
    eng = _engine(shape, model, n + 1)
    off = []
    for i in range(16):
        prompt = synth.token_ids(shape.seed, 920 + i, n, shape.vocab)
        eng.reset()
        eng.prefill(prompt)
        x = embed[prompt[-1]]
        z = x / np.sqrt((x * x).mean() + np.float32(shape.rms_eps)) * w["mlp_norm"]
        g = w["wg"] @ z
        ref = w["wd"] @ (g / (1 + np.exp(-g)) * (w["wu"] @ z))
        off.append(np.linalg.norm(eng.hidden_final() - x - ref) / np.linalg.norm(ref))
    assert np.exp(np.mean(np.log(off))) <= 2.1e-7, off


def _exit_decode(shape, model, n, force_of, rows=True):
    P = shape.prompt_len
    orc = oracle.Oracle(shape, model, max_ctx=P + n + 1)
    eng = _engine(shape, model, P + n + 1, rows=rows)
    tok = orc.prefill(synth.prompt(shape))
    eng.prefill(synth.prompt(shape))
    taus = [2.0] * len(shape.readout_layers)
    for i in range(n):
        o = orc.decode_step(tok, taus, force_of(i))
        eng.decode_step(tok, taus, force_of(i))
        tok = o["token"]
    return orc, eng


@pytest.mark.parametrize("mode", [1, 2])
def test_tiny_repass_in_several_batches(mode):
    """More exited positions than a batch holds (two of three of 1.6 ROWS_MAX:
    a full batch and a partial one), left at three layers in turn: a later batch
    reads an earlier one's entries, and the last position, which left first, is
    not the last of its batch's rows."""
    shape = TINY.replace(readout_layers=(1, 2, 3))
    model = synth.make_model(shape)
    n, P = int(1.6 * ROWS_MAX) // 6 * 6 + 2, shape.prompt_len
    force = lambda i: oracle.FORCE_FULL if i % 3 == 0 else oracle.FORCE_EXIT_AT((n - 1 - i) % 5 % 3)
    assert force(n - 1) == oracle.FORCE_EXIT_AT(0)
    orc, eng = _exit_decode(shape, model, n, force, rows=mode)
    todo = n - (n + 2) // 3
    assert ROWS_MAX < todo < 2 * ROWS_MAX
    assert eng.repass(P, P + n) == orc.repass(P, P + n) == todo
    check_kv(orc, eng, shape, P + n)
    _, one = _exit_decode(shape, model, n, force, rows=0)
    assert one.repass(P, P + n) == todo
    assert rel_err(eng.hidden_final(), one.hidden_final()) <= PATH_TOL  # the last re-passed position's
    assert eng.repass(P, P + n) == 0


@pytest.mark.parametrize("n", [40, 200])
def test_tiny_repass_rows_starting_at_different_layers(n):
    """Three readouts: exits at layers 1, 2 and 3 in one batch, so rows join
    the batch at different layers, their positions in no order (200: up to 146
    rows, on the tcgen05 attention from the second layer on)."""
    shape = TINY.replace(readout_layers=(1, 2, 3))
    model = synth.make_model(shape)
    P = shape.prompt_len
    force = lambda i: oracle.FORCE_FULL if i % 4 == 3 else oracle.FORCE_EXIT_AT(i % 4)
    orc, eng = _exit_decode(shape, model, n, force)
    assert eng.repass(P + 5, P + n) == orc.repass(P + 5, P + n)
    check_kv(orc, eng, shape, P + n)


def test_tiny_repass_paths_agree(tiny_model):
    n, P = 30, TINY.prompt_len
    force = lambda i: oracle.FORCE_FULL if i % 3 == 0 else oracle.FORCE_EXIT_AT(0)
    _, a = _exit_decode(TINY, tiny_model, n, force, rows=True)
    _, b = _exit_decode(TINY, tiny_model, n, force, rows=False)
    assert a.repass(P, P + n) == b.repass(P, P + n) == 20
    for j in range(TINY.n_layers):
        for t in range(P + n):
            assert a.kv_src(j, t) == b.kv_src(j, t) == 1
            ka, va = a.kv(j, t)
            kb, vb = b.kv(j, t)
            assert rel_err(ka, kb) <= REL_TOL and rel_err(va, vb) <= REL_TOL, (j, t)
    assert rel_err(a.hidden_final(), b.hidden_final()) <= PATH_TOL  # the last re-passed position's


def test_1p5b_prompt_batches_sampled():
    """The 1.5B shape with a 300-position prompt (two row blocks): first token,
    final state and sampled cache entries."""
    shape = synth.CONFIGS["1.5b"].replace(prompt_len=300)
    model = synth.make_model(shape)
    n = 300
    prompt = synth.prompt(shape)
    orc = oracle.Oracle(shape, model, max_ctx=n + 1)
    tok_o, cap = orc.prefill(prompt, capture=True)
    eng = _engine(shape, model, n + 1)
    tok_g = eng.prefill(prompt)
    if _top2_gap(cap["final_logits"]) >= EXCLUDE_EPS:
        assert tok_g == tok_o
    assert rel_err(eng.hidden_final(), cap["h_final"]) <= REL_TOL
    for j in (0, 13, 27):
        for t in (0, 127, 128, 255, 256, 299):
            ko, vo, so = orc.kv(j, t)
            kg, vg = eng.kv(j, t)
            assert eng.kv_src(j, t) == so == 1
            assert rel_err(kg, ko) <= REL_TOL and rel_err(vg, vo) <= REL_TOL, (j, t)


@pytest.mark.parametrize("name", ["0.5b", "1.5b"])
def test_tensor_core_paths_agree(name):
    """The tcgen05 products (EE_OPT_ROWS = 1) against the warp-level ones
    (2) on a 300-position batch (two row blocks): same first token, fp32 states within 1e-3, cache entries within 1e-2 (bf16 rounding)."""
    shape = synth.CONFIGS[name].replace(prompt_len=300)
    model = synth.make_model(shape)
    prompt = synth.prompt(shape)
    a = _engine(shape, model, 301, rows=1)
    b = _engine(shape, model, 301, rows=2)
    ta, tb = a.prefill(prompt), b.prefill(prompt)
    if _top2_gap(b.final_logits()) >= EXCLUDE_EPS:
        assert ta == tb
    assert rel_err(a.hidden_final(), b.hidden_final()) <= PATH_TOL
    assert rel_err(a.final_logits(), b.final_logits()) <= PATH_TOL
    for j in (0, shape.n_layers // 2, shape.n_layers - 1):
        for t in (0, 31, 127, 255, 256, 299):
            ka, va = a.kv(j, t)
            kb, vb = b.kv(j, t)
            assert rel_err(ka, kb) <= REL_TOL and rel_err(va, vb) <= REL_TOL, (j, t)
