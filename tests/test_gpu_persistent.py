"""The persistent layer-segment kernel (EE_OPT_PERSISTENT, the default) against
the CPU oracle under teacher forcing with small pages and other shapes, and
against the five-launch path (needs a GB300).  Same parity rules as
test_gpu_parity."""
import numpy as np
import pytest

import oracle
import synth
from helpers import check_kv, check_records, gpu_replay, oracle_steps, rel_err, teacher_forced

pytestmark = pytest.mark.gpu

TINY = synth.CONFIGS["tiny"]


@pytest.fixture(scope="module")
def tiny_model():
    return synth.make_model(TINY)


@pytest.mark.parametrize("tau", [0.5, 0.0, 1.01])
def test_tiny_persistent_teacher_forced(tiny_model, tau):
    n = TINY.new_tokens
    fo, fg, recs, orc, eng = teacher_forced(TINY, tiny_model, n, [tau], persistent=True)
    assert fo == fg
    excluded = check_records(recs, [tau])
    assert excluded <= n // 8
    check_kv(orc, eng, TINY, TINY.prompt_len + n)
    assert eng.stats()["exits"] == orc.stats()["exits"]


def test_tiny_persistent_permuted_small_pages(tiny_model):
    n = TINY.new_tokens
    pages = (TINY.max_ctx + 15) // 16
    perm = np.random.default_rng(1).permutation(pages).astype(np.int32)
    fo, fg, recs, orc, eng = teacher_forced(TINY, tiny_model, n, [0.5], page_perm=perm, page_size=16,
                                            persistent=True)
    assert fo == fg
    check_records(recs, [0.5])
    check_kv(orc, eng, TINY, TINY.max_ctx)


def test_tiny_persistent_eager_matches_graphs(tiny_model):
    _, _, a, _, _ = teacher_forced(TINY, tiny_model, 24, [0.5], capture=False, persistent=True)
    _, _, b, _, _ = teacher_forced(TINY, tiny_model, 24, [0.5], capture=False, graphs=False, persistent=True)
    for x, y in zip(a, b):
        assert x["g"] == y["g"]


def test_half_b_persistent_teacher_forced():
    """0.5B: d 896 (a ragged last 256-column chunk), 14/2 heads of 64."""
    shape = synth.CONFIGS["0.5b"].replace(prompt_len=48, new_tokens=12)
    model = synth.make_model(shape)
    fo, fg, recs, orc, eng = teacher_forced(shape, model, shape.new_tokens, [0.5], persistent=True)
    assert fo == fg
    check_records(recs, [0.5])
    check_kv(orc, eng, shape, shape.max_ctx)


def test_1p5b_persistent_teacher_forced():
    shape = synth.CONFIGS["1.5b"].replace(new_tokens=6)
    model = synth.make_model(shape)
    fo, fg, recs, orc, eng = teacher_forced(shape, model, shape.new_tokens, [0.5], persistent=True)
    assert fo == fg
    check_records(recs, [0.5])
    for j in (0, 13, 14, 27):
        for t in (0, 511, 512, shape.max_ctx - 1):
            assert eng.kv_src(j, t) == orc.kv(j, t)[2]


def test_1p5b_long_persistent_three_readouts():
    shape = synth.CONFIGS["1.5b-long"].replace(prompt_len=1024, new_tokens=6)
    model = synth.make_model(shape)
    taus = [0.6, 0.5, 0.4]
    fo, fg, recs, orc, eng = teacher_forced(shape, model, shape.new_tokens, taus, capture=False, persistent=True)
    assert fo == fg
    check_records(recs, taus, capture=False)


def test_1p5b_persistent_agrees_with_five_launch_path():
    """Free-running 1.5B decode: same tokens and gate verdicts on both GPU
    paths; confidences within the parity tolerance."""
    from paper_2609_14144_gb300 import OPT_PERSISTENT, Engine

    shape = synth.CONFIGS["1.5b"].replace(prompt_len=128, new_tokens=32)
    model = synth.make_model(shape)
    outs = []
    for pers in (0, 1):
        eng = Engine(shape, model, max_ctx=shape.prompt_len + shape.new_tokens)
        eng.set_option(OPT_PERSISTENT, pers)
        first = eng.prefill(synth.prompt(shape, shape.prompt_len))
        tok, ex, cf = eng.decode_n(shape.new_tokens, [0.5], input_token=first)
        outs.append((first, tok, ex, cf))
        eng.close()
    (f0, t0, e0, c0), (f1, t1, e1, c1) = outs
    assert f0 == f1
    near = np.abs(c0 - 0.5) < 1e-3
    agree = (t0 == t1) & (e0 == e1)
    # a near-threshold step may go either way; after it the streams may differ
    first_diff = np.argmax(~agree) if not agree.all() else len(agree)
    assert first_diff == len(agree) or near[first_diff]
    assert np.max(np.abs(c0[:first_diff] - c1[:first_diff]), initial=0) < 1e-3


@pytest.mark.parametrize("G,max_ctx", [(1, 200000), (1, 440000), (2, 150000), (3, 100000), (5, 60000), (5, 80000),
                                       (6, 60000), (6, 65000), (7, 50000), (7, 54000)])
def test_long_contexts_keep_the_persistent_layers(G, max_ctx):
    """Contexts whose attention scores fit beside the ring only in rows of the
    group's own heads (groups that are not a multiple of 4), or with half the
    partial-sum slots besides (the second length of a group): eight key-value
    heads of 64, several pages to a split.  The layers stay persistent and agree
    with the five-launch path."""
    from paper_2609_14144_gb300 import OPT_DEBUG_LOGITS, OPT_PERSISTENT, Engine

    shape = TINY.replace(n_heads=8 * G, n_kv_heads=8, n_layers=2, readout_layers=(1,))
    model = synth.make_model(shape)
    prompt = synth.token_ids(shape.seed, 940, 1500, shape.vocab)
    got = []
    for pers in (1, 0):
        eng = Engine(shape, model, max_ctx=max_ctx)
        assert eng.persistent
        eng.set_option(OPT_PERSISTENT, pers)
        eng.set_option(OPT_DEBUG_LOGITS, 1)
        eng.prefill(prompt)
        out = []
        for tok in (5, 6, 7):
            eng.decode_step(tok, [2.0], oracle.FORCE_FULL)
            out.append((eng.hidden_final(), eng.final_logits()))
        got.append(out)
        eng.close()
    for a, b in zip(*got):
        assert rel_err(a[0], b[0]) <= 1e-3 and rel_err(a[1], b[1]) <= 1e-3


def test_ring_products_round_like_short_chains():
    """Rounding of the ring-fed products (LM head of a 2048-wide model) against
    64 bits, the scale that all logits share taken out.  A rounding to nearest
    of x errs by 0.18 (2^-24 x)^2 in the mean square; counted over the partial
    sums of random terms, a row of 2048 summed stage by stage (8 terms, 4
    stages, 2 halves, 4 column groups, 8 warps) comes to 1.70 2^-24 of the
    logits, the input's two roundings included, and one chain of 32 terms per
    half to 2.15 2^-24.  4096 logits scatter by 2%."""
    from paper_2609_14144_gb300 import OPT_DEBUG_LOGITS, Engine

    shape = TINY.replace(d_model=2048, n_layers=1, readout_layers=(1,))
    model = synth.make_model(shape)
    eng = Engine(shape, model)
    assert eng.persistent
    eng.set_option(OPT_DEBUG_LOGITS, 1)
    eng.prefill(synth.prompt(shape, 3))
    off = []
    for tok in range(4):
        eng.decode_step(tok, [2.0], oracle.FORCE_FULL)
        h = eng.hidden_final().astype(np.float64)
        z = h / np.sqrt((h * h).mean() + np.float32(shape.rms_eps)) * synth.bf16_to_f32(model["final_norm"])
        ref = synth.bf16_to_f32(model["lm_head"]).astype(np.float64) @ z
        e = eng.final_logits() - ref
        e -= ref * (e @ ref) / (ref @ ref)
        off.append(np.sqrt((e @ e) / (ref @ ref)) * 2.0 ** 24)
    assert np.mean(off) <= 1.9, off


def test_waits_that_run_out_report_a_stall_and_reset_recovers():
    """Failure detection of the persistent layer kernel's bounded waits: with
    the wait bound lowered to 400 SM cycles, ordinary waits (ring stages,
    values from other CTAs) run out.  The launch ends by itself with the
    device error word set, the call reports EE_EDEVICE, and after ee_reset
    with the normal bound the engine decodes like the oracle again."""
    from paper_2609_14144_gb300 import OPT_WAIT_LIMIT, EEError, Engine

    tiny = synth.CONFIGS["tiny"]
    model = synth.make_model(tiny)
    prompt = synth.prompt(tiny)
    eng = Engine(tiny, model)
    assert eng.persistent
    eng.prefill(prompt)
    eng.set_option(OPT_WAIT_LIMIT, 400)
    with pytest.raises(EEError) as e:
        eng.decode_step(int(prompt[-1]), [0.5])
    assert e.value.code == -5 and "timed out" in str(e.value)
    eng.set_option(OPT_WAIT_LIMIT, 0)
    eng.reset()
    orc = oracle.Oracle(tiny, model)
    first = orc.prefill(prompt)
    assert eng.prefill(prompt) == first
    recs = gpu_replay(eng, oracle_steps(orc, first, 12, [0.5]), [0.5], capture=False)
    check_records(recs, [0.5], capture=False)
    eng.close()
