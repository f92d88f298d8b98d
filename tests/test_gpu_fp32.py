"""The fp32 engine's kernels at the shapes where they can go wrong: K slices
that are ragged or empty (ffn 8 and 40 over 8 slices), 8 / 9 / 17 token
columns, head_dim 128, grouped key/value heads, and contexts on both sides of
a 128-key chunk, so that a tile has one chunk (written directly) or several
(merged by the last one).  Logits against the oracle within the fp32 bound,
and the block step's rows bit for bit against one-row steps."""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2403_00835_gb300 import synthetic as syn
from tests.parity_util import engine_for, logits_ok, oracle_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,kv,ffn,vocab,n,lens", [
    (64, 4, 8, 130, 8, [1, 120, 121]),
    (64, 2, 40, 300, 9, [127, 128, 400]),
    (128, 1, 688, 2048, 17, [5, 111, 250]),
    (128, 2, 264, 257, 1, [127, 128, 129]),
])
def test_fp32_step_matches_oracle(hd, kv, ffn, vocab, n, lens):
    cfg = replace(syn.TINY, n_heads=256 // hd, n_kv_heads=kv, head_dim=hd, ffn=ffn, vocab=vocab)
    w_cpu = syn.make_weights(cfg, seed=3, device="cpu")
    w_gpu = syn.weights_to(w_cpu, "cuda")
    om = oracle_for(cfg, w_cpu)
    prompts = syn.make_prompts(cfg.vocab, lens, seed=4)
    guesses = syn.make_guesses(cfg.vocab, len(lens), n, seed=5)
    eng = engine_for(cfg, w_gpu, max_batch=len(lens), max_seq=max(lens) + 2 * n + 2, max_block=n)
    try:
        heads = eng.prefill(prompts)
        r = eng.jacobi_step(guesses, want_logits=True)
        for b, p in enumerate(prompts):
            s = om.session(len(p) + n + 1)
            head, _, _ = orc.prefill(s, p)
            assert heads[b] == head
            st = orc.jacobi_step(s, [head] + list(guesses[b][1:]), len(p), keep_logits=True)
            ok, worst = logits_ok(r["logits"][b], st.logits, "f32")
            assert ok, (b, worst)
            s.close()
        # a row's bits do not depend on the rows that share its launch
        eng.prefill(prompts)
        one = eng.jacobi_step([[g[0]] for g in guesses], want_logits=True)
        np.testing.assert_array_equal(one["logits"][:, 0], r["logits"][:, 0])
    finally:
        eng.close()
