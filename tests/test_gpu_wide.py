"""Launches of more than 256 token rows: the CTA-pair GEMM (512 weight rows x
up to 128 tokens per pair) and its fused epilogues, at the edges of its tiles
and of its work split.

The GEMM alone against fp64 (whole units, units cut between clusters, a unit
shared by several clusters, row units past the matrix, token tiles past the
launch); and the engine against the oracle: prefill of more than 256 rows with
both head sizes, grouped heads and a ragged feature tile, and a block step of
300 rows whose LM head has a ragged vocabulary tile."""
import ctypes
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2403_00835_gb300 import cllm
from paper_2403_00835_gb300 import synthetic as syn
from tests.parity_util import FLAG_GAP, engine_for, logits_ok, oracle_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,T", [
    (128, 64, 257), (512, 64, 512), (640, 72, 300), (256, 4096, 520), (4096, 688, 513),
    (4096, 4096, 1025), (19456, 128, 385), (128, 8192, 2048)])
@pytest.mark.parametrize("noalloc", [False, True])
def test_wide_gemm_matches_fp64(M, K, T, noalloc):
    lib = cllm.load()
    lib.cllm_test_gemm_bf16.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 4
    g = torch.Generator(device="cuda").manual_seed(M + K + T)
    W = (torch.randn(M, K, device="cuda", generator=g) * 0.02).bfloat16()
    rows = (T + 15) // 16 * 16
    x = torch.randn(rows, K, device="cuda", generator=g)
    hi = x.bfloat16()
    X2 = torch.stack([hi, (x - hi.float()).bfloat16()]).contiguous()
    Y0 = torch.randn(T, M, device="cuda", generator=g)
    Y = Y0.clone()
    if noalloc:
        rc = lib.cllm_gemm_bf16_noalloc(W.data_ptr(), X2.data_ptr(), Y.data_ptr(), M, K, T, rows,
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc == -4:
            pytest.skip("beyond the call's scratch")
    else:
        rc = lib.cllm_test_gemm_bf16(W.data_ptr(), X2.data_ptr(), Y.data_ptr(), M, K, T, rows)
    assert rc == 0, cllm.STATUS.get(rc, rc)
    Xd = X2[0, :T].double() + X2[1, :T].double()
    ref = Y0.double() + Xd @ W.double().T
    # fp32 accumulation of K terms: the bound of the narrow kernel's test
    bound = 1e-5 * (Xd.abs() @ W.double().abs().T + Y0.double().abs()) + 1e-7
    assert bool(((Y.double() - ref).abs() <= bound).all())


@pytest.mark.parametrize("M,K,T", [(4096, 4096, 300), (1024, 11008, 257), (512, 688, 400), (12288, 4096, 500)])
def test_wide_gemm_bits_do_not_depend_on_the_order_of_arrival(M, K, T):
    """Units cut over several pairs are finished by the last contributor; the
    sums are added in range order whoever that is.  Products of another stream
    hold SMs meanwhile, so that pairs start late and finish out of order."""
    lib = cllm.load()
    lib.cllm_test_gemm_bf16.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 4
    g = torch.Generator(device="cuda").manual_seed(M + K + T)
    W = (torch.randn(M, K, device="cuda", generator=g) * 0.02).bfloat16()
    rows = (T + 15) // 16 * 16
    x = torch.randn(rows, K, device="cuda", generator=g)
    hi = x.bfloat16()
    X2 = torch.stack([hi, (x - hi.float()).bfloat16()]).contiguous()
    noise = torch.randn(2048, 2048, device="cuda", generator=g).bfloat16()
    other = torch.cuda.Stream()
    outs = []
    for busy in (False, True, True, True, False):
        Y = torch.zeros(T, M, device="cuda")
        torch.cuda.synchronize()
        if busy:
            with torch.cuda.stream(other):
                for _ in range(200):
                    noise @ noise
        assert lib.cllm_test_gemm_bf16(W.data_ptr(), X2.data_ptr(), Y.data_ptr(), M, K, T, rows) == 0
        torch.cuda.synchronize()
        outs.append(Y)
    for Y in outs[1:]:
        assert torch.equal(Y, outs[0])


@pytest.mark.parametrize("hd,kv,ffn,lens", [
    (64, 4, 688, [300]), (64, 2, 264, [150, 200, 7]), (128, 1, 688, [257]), (128, 2, 520, [100, 420])])
def test_wide_prefill_matches_oracle(hd, kv, ffn, lens):
    cfg = replace(syn.TINY_BF16, n_heads=256 // hd, n_kv_heads=kv, head_dim=hd, ffn=ffn)
    w_cpu = syn.make_weights(cfg, seed=1, device="cpu")
    om = oracle_for(cfg, w_cpu)
    prompts = syn.make_prompts(cfg.vocab, lens, seed=2)
    n = 4
    guesses = syn.make_guesses(cfg.vocab, len(lens), n, seed=3)
    eng = engine_for(cfg, syn.weights_to(w_cpu, "cuda"), max_batch=len(lens), max_seq=max(lens) + 2 * n, max_block=n)
    try:
        heads = eng.prefill(prompts)
        r = eng.jacobi_step(guesses, want_logits=True)
    finally:
        eng.close()
    for b, p in enumerate(prompts):
        s = om.session(len(p) + n + 1)
        head, gap, _ = orc.prefill(s, p)
        if gap >= FLAG_GAP:
            assert heads[b] == head
        st = orc.jacobi_step(s, [int(heads[b])] + list(guesses[b][1:]), len(p), keep_logits=True)
        ok, worst = logits_ok(r["logits"][b], st.logits, "bf16")
        assert ok, (b, worst)
        s.close()


def test_wide_step_matches_oracle_ragged_vocab():
    cfg = replace(syn.TINY_BF16, vocab=1100)
    w_cpu = syn.make_weights(cfg, seed=4, device="cpu")
    om = oracle_for(cfg, w_cpu)
    B, n = 5, 60
    prompts = syn.make_prompts(cfg.vocab, [3, 17, 40, 9, 130], seed=5)
    guesses = syn.make_guesses(cfg.vocab, B, n, seed=6)
    eng = engine_for(cfg, syn.weights_to(w_cpu, "cuda"), max_batch=B, max_seq=200, max_block=n)
    try:
        heads = eng.prefill(prompts)
        r = eng.jacobi_step(guesses, want_logits=True)
    finally:
        eng.close()
    for b, p in enumerate(prompts):
        s = om.session(len(p) + n + 1)
        orc.prefill(s, p)
        st = orc.jacobi_step(s, [int(heads[b])] + list(guesses[b][1:]), len(p), keep_logits=True)
        ok, worst = logits_ok(r["logits"][b], st.logits, "bf16")
        assert ok, (b, worst)
        for k in range(n):
            if st.gap[k] >= FLAG_GAP:
                assert r["next"][b][k] == st.pred[k]
            assert abs(r["gap"][b][k] - st.gap[k]) < FLAG_GAP
        s.close()


@pytest.mark.parametrize("hd,kv,lens", [
    (128, 2, [129, 128, 127, 1]), (128, 1, [385]), (64, 4, [256, 257]), (64, 2, [640, 130])])
def test_wide_attention_matches_oracle_at_tile_edges(hd, kv, lens):
    """Prompts around the 128-row tiles and 128-key chunks of the wide
    attention (last tile absent, one row, full), the wide tiles' outputs read
    back through a short step.  Weights of std 0.08 spread the scores over
    tens of units, so that running maxima move and accumulators are rescaled."""
    cfg = replace(syn.TINY_BF16, n_heads=256 // hd, n_kv_heads=kv, head_dim=hd)
    w_cpu = syn.make_weights(cfg, seed=11, device="cpu")
    for l in range(cfg.n_layers):
        for k in ("wq", "wk"):
            w_cpu[k][l] = w_cpu[k][l] * 4
    om = oracle_for(cfg, w_cpu)
    prompts = syn.make_prompts(cfg.vocab, lens, seed=12)
    n = 3
    guesses = syn.make_guesses(cfg.vocab, len(lens), n, seed=13)
    eng = engine_for(cfg, syn.weights_to(w_cpu, "cuda"), max_batch=len(lens), max_seq=max(lens) + 2 * n, max_block=n)
    try:
        heads = eng.prefill(prompts)
        r = eng.jacobi_step(guesses, want_logits=True)
    finally:
        eng.close()
    for b, p in enumerate(prompts):
        s = om.session(len(p) + n + 1)
        orc.prefill(s, p)
        st = orc.jacobi_step(s, [int(heads[b])] + list(guesses[b][1:]), len(p), keep_logits=True)
        ok, worst = logits_ok(r["logits"][b], st.logits, "bf16")
        assert ok, (b, worst)
        s.close()
