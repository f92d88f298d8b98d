"""The persistent per-iteration kernel (one launch per Jacobi iteration, grid
barriers between phases) against the one-kernel-per-phase path: same work
split, reductions and epilogues, so predictions, gaps, accepted counts,
committed lengths and decoded tokens must be bit-identical."""
import ctypes
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_00835_gb300 import synthetic as syn
from paper_2403_00835_gb300.cllm import load
from tests.parity_util import engine_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny_bf16():
    cfg = syn.TINY_BF16
    w = syn.make_weights(cfg, seed=0, device="cuda")
    eng = engine_for(cfg, w, max_batch=4, max_seq=160, max_block=16)
    yield cfg, eng
    eng.close()


def _steps(eng, prompts, guesses_list, persistent):
    eng.set_persistent(persistent)
    eng.prefill(prompts)
    outs = []
    for g in guesses_list:
        r = eng.jacobi_step(g, want_gap=True)
        outs.append((r["next"].copy(), r["accepted"].copy(), r["gap"].copy()))
    return outs, eng.committed_lengths().copy()


@pytest.mark.parametrize("n", [1, 8, 16])
def test_persistent_steps_bit_identical(tiny_bf16, n):
    cfg, eng = tiny_bf16
    prompts = syn.make_prompts(cfg.vocab, [32, 17, 45], seed=1)
    gl = [syn.make_guesses(cfg.vocab, 3, n, seed=s) for s in (2, 3, 4)]
    eng.set_persistent(True)
    eng.prefill(prompts)
    assert eng.uses_persistent(n)
    a, la = _steps(eng, prompts, gl, True)
    b, lb = _steps(eng, prompts, gl, False)
    for (n1, a1, g1), (n2, a2, g2) in zip(a, b):
        np.testing.assert_array_equal(n1, n2)
        np.testing.assert_array_equal(a1, a2)
        np.testing.assert_array_equal(g1, g2)
    np.testing.assert_array_equal(la, lb)
    eng.set_persistent(True)


@pytest.mark.parametrize("n", [8, 16])
def test_persistent_logits_bit_identical(tiny_bf16, n):
    """A step asked for its logits runs the persistent kernel (the one the
    decode loop runs) and stores them from its LM-head phase; they equal the
    per-GEMM path's logits bit for bit."""
    cfg, eng = tiny_bf16
    prompts = syn.make_prompts(cfg.vocab, [32, 17, 45], seed=1)
    g = syn.make_guesses(cfg.vocab, 3, n, seed=2)
    out = []
    for persistent in (True, False):
        eng.set_persistent(persistent)
        eng.prefill(prompts)
        assert eng.uses_persistent(n) == persistent
        out.append(eng.jacobi_step(g, want_gap=True, want_logits=True))
    eng.set_persistent(True)
    a, b = out
    assert np.isfinite(a["logits"]).all()
    np.testing.assert_array_equal(a["logits"], b["logits"])
    np.testing.assert_array_equal(a["next"], b["next"])
    np.testing.assert_array_equal(a["gap"], b["gap"])
    np.testing.assert_array_equal(a["accepted"], b["accepted"])


def test_persistent_decode_bit_identical(tiny_bf16):
    cfg, eng = tiny_bf16
    prompts = syn.make_prompts(cfg.vocab, [32, 17, 45, 8], seed=5)
    eng.set_persistent(True)
    pa, ia = eng.jacobi_decode(prompts, 8, 64, seed=3)
    eng.set_persistent(False)
    pb, ib = eng.jacobi_decode(prompts, 8, 64, seed=3)
    eng.set_persistent(True)
    np.testing.assert_array_equal(pa, pb)
    np.testing.assert_array_equal(ia, ib)
    ar = eng.ar_decode(prompts, 64)
    np.testing.assert_array_equal(pa, ar)


def test_persistent_7b_decode_bit_identical():
    cfg = syn.LLAMA7B
    w = syn.make_weights(cfg, seed=0, device="cuda")
    eng = engine_for(cfg, w, max_batch=2, max_seq=128 + 64 + 64, max_block=64)
    prompts = syn.make_prompts(cfg.vocab, [128, 100], seed=1)
    try:
        for n in (16, 64):
            eng.set_persistent(True)
            eng.prefill(prompts)
            assert eng.uses_persistent(n)
            pa, ia = eng.jacobi_decode(prompts, n, 48, seed=2)
            eng.set_persistent(False)
            pb, ib = eng.jacobi_decode(prompts, n, 48, seed=2)
            np.testing.assert_array_equal(pa, pb)
            np.testing.assert_array_equal(ia, ib)
    finally:
        eng.close()


@pytest.mark.parametrize("n", [1, 16])
def test_persistent_dataflow_flags_bit_identical(tiny_bf16, n):
    """Attention and the O projection opened by completion flags (the
    default) or by grid barriers compute the same logits bit for bit."""
    cfg, eng = tiny_bf16
    prompts = syn.make_prompts(cfg.vocab, [32, 17, 45], seed=11)
    g = syn.make_guesses(cfg.vocab, 3, n, seed=12)
    out = []
    try:
        for flags in (True, False):
            eng.set_dataflow(flags)
            eng.prefill(prompts)
            assert eng.uses_persistent(n)
            out.append(eng.jacobi_step(g, want_gap=True, want_logits=True))
    finally:
        eng.set_dataflow(True)
    a, b = out
    np.testing.assert_array_equal(a["logits"], b["logits"])
    np.testing.assert_array_equal(a["next"], b["next"])
    np.testing.assert_array_equal(a["accepted"], b["accepted"])


def test_path_rule_follows_the_committed_lengths():
    """The library's own choice goes by the lengths a decode has reached, not by
    the prompt's: 16 rows of 32 heads run persistent (on 152 SMs) up to 2176
    keys.  A decode that crosses the line gives the same tokens as one that stays
    on either path."""
    cfg = replace(syn.TINY_BF16, n_heads=32, n_kv_heads=4)
    w = syn.make_weights(cfg, seed=21, device="cuda")
    n, max_new = 16, 24
    prompts = syn.make_prompts(cfg.vocab, [2152], seed=22)
    guesses = syn.make_guesses(cfg.vocab, 1, n, seed=23)
    runs = []
    for choice in (None, True, False):
        eng = engine_for(cfg, w, max_batch=1, max_seq=2152 + max_new + 2 * n, max_block=n)
        try:
            if choice is not None:
                eng.set_persistent(choice)
            eng.prefill(prompts)
            eng.decode_begin(n, max_new, seed=24)
            if choice is None:
                assert eng.uses_persistent(n)
            done, _ = eng.decode_run(1)
            while done < max_new and eng.committed_lengths()[0] <= 2176 - n:
                done += eng.decode_run(1)[0]
            if choice is None:
                assert not eng.uses_persistent(n)
            eng.decode_run(max_new + 1)
            tokens, iters = eng.decode_read()
            step = eng.jacobi_step(guesses, want_logits=True)
            runs.append((tokens, iters, step["logits"]))
        finally:
            eng.close()
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            np.testing.assert_array_equal(a, b)


def test_path_choice_can_be_given_back_to_the_library(tiny_bf16):
    cfg, eng = tiny_bf16
    eng.set_persistent_auto()
    eng.prefill(syn.make_prompts(cfg.vocab, [32, 17, 45, 20], seed=13))
    try:
        default = {n: eng.uses_persistent(n) for n in (1, 12, 13)}
        assert default[12] and not default[13]  # 48 and 52 rows
        for on in (True, False):
            eng.set_persistent(on)
            assert all(eng.uses_persistent(n) == on for n in default)
            eng.set_persistent_auto()
            assert {n: eng.uses_persistent(n) for n in default} == default
    finally:
        eng.set_persistent_auto()


def test_pair_launches_are_split_over_resident_pairs(tiny_bf16):
    """Shared tiles' first contributors wait for the others: the split must not
    be made for more CTAs than can be resident as pairs."""
    _, eng = tiny_bf16
    f = load().cllm_test_split_sms
    f.argtypes, f.restype = [ctypes.c_void_p], ctypes.c_int
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = f(eng._h)
    assert 4 <= n <= sms and n % 2 == 0
    assert f(None) == -1


@pytest.mark.parametrize("B,n", [(5, 10), (1, 64), (4, 16), (1, 65), (2, 50), (1, 128), (8, 16)])
def test_wider_blocks_have_the_same_logits_on_both_paths(B, n):
    """50 to 128 rows, the widths at which the library's own choice is the pair
    kernels: every logit bit for bit against the persistent kernel's."""
    cfg = syn.TINY_BF16
    w = syn.make_weights(cfg, seed=0, device="cuda")
    prompts = syn.make_prompts(cfg.vocab, [11 + 9 * b for b in range(B)], seed=31)
    guesses = syn.make_guesses(cfg.vocab, B, n, seed=32)
    eng = engine_for(cfg, w, max_batch=B, max_seq=300, max_block=n)
    try:
        out = []
        for on in (True, False):
            eng.set_persistent(on)
            eng.prefill(prompts)
            assert eng.uses_persistent(n) == on
            out.append(eng.jacobi_step(guesses, want_gap=True, want_logits=True))
        for key in out[0]:
            np.testing.assert_array_equal(out[0][key], out[1][key])
    finally:
        eng.close()


@pytest.mark.parametrize("B,n,keys,persistent", [
    (1, 16, 128, True), (1, 16, 2000, True), (1, 1, 4096, False), (15, 1, 47, True), (15, 1, 250, False),
    (8, 1, 500, True), (8, 1, 1000, False), (1, 32, 500, True), (1, 32, 1000, False), (1, 48, 250, True),
    (6, 7, 30, True), (1, 48, 500, False), (1, 49, 30, False), (24, 1, 30, False)])
def test_path_rule_at_its_lines(B, n, keys, persistent):
    """The library's own choice with 32 heads on 152 SMs, on both sides of its
    lines: rows, waves of attention items and keys per item."""
    cfg = replace(syn.TINY_BF16, n_heads=32, n_kv_heads=4, n_layers=1)
    w = syn.make_weights(cfg, seed=41, device="cuda")
    eng = engine_for(cfg, w, max_batch=B, max_seq=keys + n + 1, max_block=n)
    try:
        eng.prefill(syn.make_prompts(cfg.vocab, [keys] * B, seed=42))
        assert eng.uses_persistent(n) == persistent
    finally:
        eng.close()
