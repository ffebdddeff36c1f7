"""Standalone kernels through the C ABI vs the oracle's ops (needs a GB300).

Split-K paged attention over T in {1, 2, 15, 16, 17, 63, 64, 65, 1000, 8192}
and several head groupings; the vocabulary pass with ragged vocabularies."""
import math

import numpy as np
import pytest

import oracle
import synth
from helpers import rel_err, to_bf16_bits

pytestmark = pytest.mark.gpu


def _dev(a, dtype=None):
    """numpy -> CUDA tensor; 16-bit bit patterns travel as int16."""
    import torch
    a = np.ascontiguousarray(a)
    if a.dtype == np.uint16:
        a = a.view(np.int16)
    return torch.from_numpy(a).cuda()


@pytest.mark.parametrize("T", [1, 2, 15, 16, 17, 63, 64, 65, 1000, 8192])
@pytest.mark.parametrize("A,KH,D", [(12, 2, 128), (14, 2, 64), (4, 2, 64), (16, 2, 128), (8, 8, 64)])
def test_attention_decode(T, A, KH, D):
    import torch

    from paper_2609_14144_gb300 import attention_decode

    rng = np.random.default_rng(T * 31 + A)
    P = 64
    n_pages = (T + P - 1) // P
    perm = rng.permutation(n_pages).astype(np.int32)
    q = rng.standard_normal(A * D).astype(np.float32)
    K = to_bf16_bits(rng.standard_normal((T, KH, D)).astype(np.float32))
    V = to_bf16_bits(rng.standard_normal((T, KH, D)).astype(np.float32))
    kp = np.zeros((n_pages, KH, P, D), np.uint16)
    vp = np.zeros((n_pages, KH, P, D), np.uint16)
    for t in range(T):
        kp[perm[t // P], :, t % P] = K[t]
        vp[perm[t // P], :, t % P] = V[t]
    out = attention_decode(_dev(q), _dev(kp), _dev(vp), _dev(perm), T, A, KH, D, P)
    torch.cuda.synchronize()
    got = out.cpu().numpy().reshape(A, D)
    Kf, Vf = synth.bf16_to_f32(K), synth.bf16_to_f32(V)
    for h in range(A):
        g = h // (A // KH)
        ref = oracle.attention(q[h * D:(h + 1) * D], Kf[:, g], Vf[:, g])
        assert rel_err(got[h], ref) <= 1e-4, (h, rel_err(got[h], ref))


@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("T,P,D", [(127, 64, 128), (129, 1, 64), (2065, 24, 128), (16384, 256, 64), (16401, 100, 128)])
def test_attention_decode_groups_tiles_and_pages(T, P, D, G):
    """Every group size at the edges of a warp's 16-position tile, of a
    128-position split and of the split count (128 splits hold 16384), with
    pages of any length.  The bound: products and sums in fp32, n terms of a
    convex combination of values up to 4.5 in size, sqrt(T) rounding steps."""
    import torch

    from paper_2609_14144_gb300 import attention_decode

    KH = 2
    g = torch.Generator(device="cuda").manual_seed(T + G)
    n_pages = (T + P - 1) // P
    q = torch.randn(G * KH * D, generator=g, device="cuda")
    kp = torch.randn(n_pages, KH, P, D, generator=g, device="cuda").to(torch.bfloat16)
    vp = torch.randn(n_pages, KH, P, D, generator=g, device="cuda").to(torch.bfloat16)
    table = torch.randperm(n_pages, generator=g, device="cuda").to(torch.int32)
    k, v = (t[table.long()].permute(1, 0, 2, 3).reshape(KH, -1, D)[:, :T].clone() for t in (kp, vp))
    for t in (kp, vp):  # rows past T of the last page are never read
        used = (T - 1) % P + 1
        t[table[-1].long(), :, used:] = float("nan")
    got = attention_decode(q, kp, vp, table, T, G * KH, KH, D, P).view(KH, G, D)
    ref = torch.softmax(q.double().view(KH, G, D) @ k.double().transpose(1, 2) / math.sqrt(D), -1) @ v.double()
    err = (got.double() - ref).abs().max().item()
    assert err <= 4.5 * math.sqrt(T) * 2.0 ** -24 * 8, err


@pytest.mark.parametrize("T,most", [(17, 1.31e-7), (100, 1.63e-7)])
def test_attention_decode_rounds_like_short_chains(T, most):
    """The mean error of short calls against 64 bits.  A rounding to nearest of
    x errs by 0.18 (2^-24 x)^2 in the mean square; counted over the partial sums
    of a score of 128 dimensions (chunks of 8, four chunks, four lanes) that is
    7.5e-8, which each probability and so the output takes over; the rest
    (queries scaled, exponentials, sums over positions) is 9.2e-8 at 17
    positions and 1.2e-7 at 100.  Together 1.19e-7 and 1.47e-7; with one chain
    of 32 dimensions a lane 1.45e-7 and 1.8e-7."""
    import torch

    from paper_2609_14144_gb300 import attention_decode

    A, KH, D, P = 16, 2, 128, 64
    off = []
    for seed in range(32):
        g = torch.Generator(device="cuda").manual_seed(seed)
        n_pages = (T + P - 1) // P
        q = torch.randn(A * D, generator=g, device="cuda")
        kp = torch.randn(n_pages, KH, P, D, generator=g, device="cuda").to(torch.bfloat16)
        vp = torch.randn(n_pages, KH, P, D, generator=g, device="cuda").to(torch.bfloat16)
        table = torch.arange(n_pages, device="cuda", dtype=torch.int32)
        k, v = (t.double().permute(1, 0, 2, 3).reshape(KH, -1, D)[:, :T] for t in (kp, vp))
        ref = torch.softmax(q.double().view(KH, A // KH, D) @ k.transpose(1, 2) / math.sqrt(D), -1) @ v
        got = attention_decode(q, kp, vp, table, T, A, KH, D, P).view_as(ref)
        off.append(((got - ref).norm() / ref.norm()).item())
    assert np.exp(np.mean(np.log(off))) <= most, off


@pytest.mark.parametrize("V,d", [(4096, 256), (4093, 256), (151936, 896), (151937, 1536), (1000, 2048)])
def test_vocab_confidence(V, d):
    import torch

    from paper_2609_14144_gb300 import vocab_confidence

    rng = np.random.default_rng(V + d)
    x = rng.standard_normal(d).astype(np.float32)
    gain = synth.const_bf16(d, 7.0 / (0.02 * math.sqrt(d)))
    U = synth.normal_bf16(5, 0x777, (V, d))
    logits = torch.empty(V, dtype=torch.float32, device="cuda")
    tok, p = vocab_confidence(_dev(x), _dev(gain), _dev(U), 1e-6, logits=logits)
    torch.cuda.synchronize()
    z = oracle.rmsnorm(x, gain, 1e-6)
    ref_l = oracle.matvec(U, z)
    c = oracle.confidence(ref_l)
    assert rel_err(logits.cpu().numpy(), ref_l) <= 1e-4
    assert abs(float(p.item()) - c["p1"]) <= 1e-4
    if c["gap"] >= 1e-3:
        assert int(tok.item()) == c["argmax"]


@pytest.mark.parametrize("V", [2, 151, 2433, 9999, 10001, 13999, 14001, 20011, 20481])
@pytest.mark.parametrize("d", [256, 264, 512, 520, 1024, 1032, 1536, 1544, 2040, 2048, 2056])
def test_vocab_rows_widths(V, d):
    """Row widths at the edges of the columns a lane keeps in registers and of
    the rows a warp takes at once, ragged last column chunks, partly filled
    stages, fewer rows than CTAs, and on both sides of the row counts and
    widths from which the ring takes over from the streaming kernel.  Logits within the fp32 summation bound, the
    token the highest logit's lowest index."""
    import torch

    from paper_2609_14144_gb300 import vocab_signals

    g = torch.Generator(device="cuda").manual_seed(V * 7 + d)
    x = torch.randn(d, generator=g, device="cuda")
    gain = torch.randn(d, generator=g, device="cuda").to(torch.bfloat16)
    U = torch.randn(V, d, generator=g, device="cuda").to(torch.bfloat16)
    logits = torch.full((V,), float("nan"), device="cuda")
    tok, sig = vocab_signals(x, gain, U, 1e-6, logits=logits)
    z = x.double() / torch.sqrt((x.double() ** 2).mean() + 1e-6) * gain.double()
    ref = U.double() @ z
    bound = (U.double().abs() @ z.abs()) * 2.0 ** -24 * (d / 64 + 8)
    assert ((logits.double() - ref).abs() <= bound).all()
    assert tok.item() == logits.argmax().item()
    p = torch.softmax(logits.double(), 0)
    top = torch.topk(p, 2).values
    want = torch.stack([top[0], top[0] - top[1], (p * torch.log_softmax(logits.double(), 0)).sum()])
    assert (sig.double() - want).abs().max().item() <= 1e-5 * max(1.0, want.abs().max().item())


@pytest.mark.parametrize("V,d", [(4096, 256), (151936, 1536), (1000, 2048)])
def test_vocab_signals(V, d):
    """Section 10's three signals from one pass, against the oracle's
    definitions on the same logits."""
    import torch

    from paper_2609_14144_gb300 import vocab_signals

    rng = np.random.default_rng(V * 3 + d)
    x = rng.standard_normal(d).astype(np.float32)
    gain = synth.const_bf16(d, 4.0 / (0.02 * math.sqrt(d)))
    U = synth.normal_bf16(6, 0x778, (V, d))
    tok, sig = vocab_signals(_dev(x), _dev(gain), _dev(U), 1e-6)
    torch.cuda.synchronize()
    c = oracle.confidence(oracle.matvec(U, oracle.rmsnorm(x, gain, 1e-6)))
    got = sig.cpu().numpy()
    assert abs(got[0] - c["p1"]) <= 1e-4
    assert abs(got[1] - c["gap"]) <= 1e-4
    assert abs(got[2] - c["neg_entropy"]) <= 1e-4 * max(1.0, abs(c["neg_entropy"]))
    if c["gap"] >= 1e-3:
        assert int(tok.item()) == c["argmax"]


@pytest.mark.parametrize("n", [31, 2431, 2432, 4864, 9728, 19456, 38912, 77824])
def test_select_tau_slices(n):
    """Each number of lanes a candidate is shared by, at and past its largest
    n, against the counts of every candidate taken from a sort."""
    import torch

    from paper_2609_14144_gb300 import select_tau

    rng = np.random.default_rng(n)
    conf = (np.floor(rng.random(n) * 3 * n) / (3 * n)).astype(np.float32)
    member = (rng.random(n) < 0.4 + 0.6 * conf).astype(np.int32)
    cs, good = np.sort(conf), None
    order = np.argsort(conf, kind="stable")
    good = np.concatenate([np.cumsum(member[order][::-1])[::-1], [0]])
    cands = np.concatenate([[-np.inf], np.unique(cs)])
    at = np.searchsorted(cs, cands, side="right")
    for target in (0.5, 0.9):
        ok = (n - at > 0) & (good[at] >= np.float64(np.float32(target)) * (n - at))
        want = cands[ok].min() if ok.any() else np.inf
        assert select_tau(_dev(conf), _dev(member), target).item() == np.float32(want)


def test_vocab_signals_tie_and_uniform():
    import torch

    from paper_2609_14144_gb300 import vocab_signals

    V, d = 50000, 256
    U = np.zeros((V, d), np.uint16)
    row = to_bf16_bits(np.linspace(-1, 1, d).astype(np.float32))
    for v in (40000, 12345, 49999):
        U[v] = row
    x = np.linspace(-1, 1, d).astype(np.float32)
    gain = synth.const_bf16(d, 1.0)
    tok, sig = vocab_signals(_dev(x), _dev(gain), _dev(U), 1e-6)
    torch.cuda.synchronize()
    c = oracle.confidence(oracle.matvec(U, oracle.rmsnorm(x, gain, 1e-6)))
    assert int(tok.item()) == 12345 and float(sig[1].item()) == 0.0
    assert abs(float(sig[2].item()) - c["neg_entropy"]) <= 1e-4 * abs(c["neg_entropy"])
    # all-zero matrix: uniform distribution, p1 = 1/V, margin 0, -log V
    tok, sig = vocab_signals(_dev(x), _dev(gain), _dev(np.zeros((V, d), np.uint16)), 1e-6)
    torch.cuda.synchronize()
    got = sig.cpu().numpy()
    assert int(tok.item()) == 0 and got[1] == 0.0
    assert abs(got[0] - 1.0 / V) <= 1e-9 and abs(got[2] + math.log(V)) <= 1e-4


@pytest.mark.parametrize("d", [896, 2048])
def test_vocab_rows_wait_that_runs_out_poisons_the_result(d):
    """With the bound of its waits lowered to one SM cycle the row-major pass
    cannot read all of its rows: no token, no signals, no stale logits.  The
    next call on the same scratch is right again."""
    import ctypes

    import torch

    from paper_2609_14144_gb300 import _lib, vocab_signals

    V = 40000
    g = torch.Generator(device="cuda").manual_seed(d)
    x = torch.randn(d, generator=g, device="cuda")
    gain = torch.ones(d, device="cuda").to(torch.bfloat16)
    U = torch.randn(V, d, generator=g, device="cuda").to(torch.bfloat16)
    ref = U.double() @ (x.double() / torch.sqrt((x.double() ** 2).mean() + 1e-6))
    scratch = torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
    token = torch.zeros(1, dtype=torch.int32, device="cuda")
    sig = torch.zeros(3, device="cuda")
    logits = torch.full((V,), 1e9, device="cuda")
    bounded = _lib.load().ee_vocab_signals_bounded
    p = ctypes.c_void_p
    bounded.argtypes = [p, p, p, ctypes.c_int, ctypes.c_int, ctypes.c_float, p, ctypes.c_size_t, p, p, p, p,
                        ctypes.c_longlong]
    args = (x.data_ptr(), gain.data_ptr(), U.data_ptr(), V, d, 1e-6, scratch.data_ptr(), scratch.numel(),
            token.data_ptr(), sig.data_ptr(), logits.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert bounded(*args, 0) == _lib.EE_EINVAL
    assert bounded(*args, 1) == 0
    torch.cuda.synchronize()
    assert token.item() == -1 and torch.isnan(sig).all()
    lost = torch.isnan(logits)
    assert lost.any() and ((logits - ref).abs()[~lost] <= 1e-3 * ref.abs().max()).all()
    tok, s2 = vocab_signals(x, gain, U, 1e-6, logits=logits, scratch=scratch)
    assert tok.item() == ref.argmax().item() and torch.isfinite(s2).all()
    assert ((logits - ref).abs() <= 1e-5 * ref.abs().max()).all()


def test_vocab_confidence_ties_lowest_index():
    import torch

    from paper_2609_14144_gb300 import vocab_confidence

    V, d = 50000, 256
    U = np.zeros((V, d), np.uint16)
    row = to_bf16_bits(np.linspace(-1, 1, d).astype(np.float32))
    for v in (40000, 12345, 49999):
        U[v] = row
    x = np.linspace(-1, 1, d).astype(np.float32)
    gain = synth.const_bf16(d, 1.0)
    tok, p = vocab_confidence(_dev(x), _dev(gain), _dev(U), 1e-6)
    torch.cuda.synchronize()
    assert int(tok.item()) == 12345
