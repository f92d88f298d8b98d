"""Performance cases of the Jacobi-decoding engine, through its public entry
points (``Engine`` of the Python binding and the C ABI's allocation-free GEMM).

Every case is one of four kinds:

- ``generate``: the whole call of a serving program, ``jacobi_decode`` of a
  batch of prompts (prefill, the device-resident loop, tokens back), then the
  logits of one more block with ``jacobi_step``.
- ``decode``: the loop alone on sequences that are already prefilled:
  ``decode_begin``, a few iterations of ``decode_run``, ``decode_read``, then
  the logits of one more block.
- ``prefill``: new prompts into the KV cache, then the logits of a short block
  that attends to all of it.
- ``gemm``: ``cllm_gemm_bf16_noalloc``, the library's weight GEMM on its own.

Models are the shapes of ``synthetic.py`` with seeded random weights.  Most
cases run a few layers of the 7B shape with a 2048-token vocabulary: a layer
costs what it costs at full depth, rounding does not travel through 32 layers,
and the logits that are compared stay small.  One case is the full model.
"""
from __future__ import annotations

import ctypes
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2403_00835_gb300 import cllm
from paper_2403_00835_gb300 import synthetic as syn

DEV = "cuda"
MODES = {"refill": cllm.CLLM_BLOCK_REFILL, "shrink": cllm.CLLM_BLOCK_SHRINK,
         "lookahead": cllm.CLLM_BLOCK_LOOKAHEAD}


def _engine_case(kind, model, layers, vocab, batch, lo, hi, n, steps, mode="refill", kv_heads=0, name=None):
    """steps: new tokens per sequence (generate) or loop iterations (decode)."""
    c = dict(kind=kind, model=model, layers=layers, vocab=vocab, batch=batch, lo=lo, hi=hi, n=n, steps=steps,
             mode=mode, kv_heads=kv_heads)
    if name:
        c["name"] = name
    return c


def listed():
    e = _engine_case
    return [
        # the smallest calls: a two-layer fp32 decoder, where launches and latency are everything
        e("generate", "tiny-f32", 2, 2048, 1, 32, 32, 8, 64, name="tiny_f32_generate"),
        # the same shapes in bf16, a small ragged batch
        e("generate", "tiny-bf16", 2, 2048, 3, 5, 60, 16, 48, name="tiny_bf16_generate"),
        # the whole 7B model: one user's request, the usual block of 16
        e("generate", "llama2-7b", 32, 32000, 1, 128, 128, 16, 16, name="llama7b_generate_n16"),
        # greedy decoding far into a long context: one row against 4096 cached keys
        e("decode", "llama2-7b", 4, 2048, 1, 4096, 4096, 1, 8, name="ar_long_context"),
        # a wide block of one sequence
        e("decode", "llama2-7b", 4, 2048, 1, 512, 512, 64, 6, name="wide_block_n64"),
        # a small batch of blocks: 128 rows
        e("decode", "llama2-7b", 4, 2048, 4, 1024, 1024, 32, 4, name="batch4_n32"),
        # the coder-style batch: ragged prompts, 256 rows
        e("decode", "coder-7b", 4, 2048, 8, 256, 1024, 32, 4, name="coder_batch8_n32"),
        # a full server: 16 sequences, 1024 rows
        e("decode", "llama2-7b", 4, 2048, 16, 256, 256, 64, 2, name="batch16_n64"),
        # prompts: one ordinary, a ragged batch, one long
        e("prefill", "llama2-7b", 2, 2048, 1, 500, 500, 4, 0, name="prefill_500"),
        e("prefill", "coder-7b", 2, 2048, 8, 256, 1024, 4, 0, name="prefill_ragged_batch8"),
        e("prefill", "llama2-7b", 2, 2048, 1, 4096, 4096, 4, 0, name="prefill_4096"),
        # one projection of 16 rows for a program that brings its own buffers
        dict(name="gemm_4096_t16", kind="gemm", m=4096, k=4096, t=16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """The same kinds over the range that the listed cases stand for: 1 to 1024
    block rows, contexts of 16 to 4096 tokens, prompts of up to 5120 tokens in
    all, both small decoders, grouped key/value heads among the 7B shapes."""
    u = rng.random()
    if u < 0.1:
        m, k = 128 * _log_int(rng, 1, 48), 8 * _log_int(rng, 8, 1376)
        t = _log_int(rng, 1, 256)
        while 128 * m * 40 + 4 * t * m > 4 << 20 and t > 1:  # well inside the call's 8 MiB of scratch
            t //= 2
        return dict(kind="gemm", m=m, k=k, t=t)
    if u < 0.3:
        b = rng.randint(1, 4)
        lo = _log_int(rng, 4, 60)
        return _engine_case("generate", rng.choice(("tiny-f32", "tiny-bf16")), 2, 2048, b, lo,
                            rng.randint(lo, 90), rng.randint(1, 16), rng.randint(16, 64),
                            mode=rng.choice(tuple(MODES)))
    model, kv = rng.choice(("llama2-7b", "coder-7b")), rng.choice((0, 0, 8))
    if u < 0.75:
        b = _log_int(rng, 1, 16)
        n = min(_log_int(rng, 1, 128), 1024 // b)
        hi = min(_log_int(rng, 16, 4096), 8192 // b)
        lo = hi if rng.random() < 0.5 else max(16, hi // rng.randint(2, 4))
        return _engine_case("decode", model, rng.randint(1, 4), 2048, b, min(lo, hi), hi, n, rng.randint(1, 3),
                            kv_heads=kv)
    b = _log_int(rng, 1, 16)
    hi = _log_int(rng, 16, min(4096, 5120 // b))
    lo = hi if b == 1 else max(16, hi // rng.randint(1, 4))
    return _engine_case("prefill", model, rng.randint(1, 2), 2048, b, min(lo, hi), hi, rng.randint(1, 8), 0,
                        kv_heads=kv)


# ---- inputs ------------------------------------------------------------------


def _config(case):
    cfg = syn.CONFIGS[case["model"]]
    cfg = replace(cfg, n_layers=case["layers"], vocab=case["vocab"])
    return replace(cfg, n_kv_heads=case["kv_heads"]) if case["kv_heads"] else cfg


def _lens(case, seed):
    if case["lo"] == case["hi"]:
        return [case["lo"]] * case["batch"]
    return syn.ragged_lens(case["batch"], case["lo"], case["hi"], seed=seed)


def _inputs(case, seed):
    cfg = _config(case)
    w = syn.make_weights(cfg, seed=seed, device=DEV)
    prompts = syn.make_prompts(cfg.vocab, _lens(case, seed + 1), seed=seed + 1)
    guess = np.asarray(syn.make_guesses(cfg.vocab, case["batch"], case["n"], seed=seed + 2), dtype=np.int32)
    return cfg, w, prompts, guess


def _gemm_inputs(case, seed):
    m, k, t = case["m"], case["k"], case["t"]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    w = (torch.randn(m, k, device=DEV, generator=gen) * 0.02).bfloat16()
    rows = (t + 15) // 16 * 16
    x = torch.randn(rows, k, device=DEV, generator=gen)
    hi = x.bfloat16()
    planes = torch.stack([hi, (x - hi.float()).bfloat16()]).contiguous()
    y0 = torch.randn(t, m, device=DEV, generator=gen)
    return w, planes, y0, rows


def prepare(case, seed):
    if case["kind"] == "gemm":
        w, planes, y0, rows = _gemm_inputs(case, seed)
        return dict(case=case, w=w, x=planes, y0=y0, y=torch.empty_like(y0), rows=rows, lib=cllm.load())
    cfg, w, prompts, guess = _inputs(case, seed)
    room = max(len(p) for p in prompts) + 2 * case["n"] + case["steps"] * (case["n"] if case["kind"] == "decode" else 1)
    eng = cllm.Engine(cfg, w, max_batch=case["batch"], max_seq=room + 8, max_block=case["n"])
    if case["kind"] == "decode":
        eng.prefill(prompts)
    return dict(case=case, eng=eng, prompts=prompts, guess=guess, seed=seed)


# ---- one pass ------------------------------------------------------------------


def run(state):
    case = state["case"]
    if case["kind"] == "gemm":
        y = state["y"]
        y.copy_(state["y0"])  # the call accumulates into Y
        rc = state["lib"].cllm_gemm_bf16_noalloc(
            state["w"].data_ptr(), state["x"].data_ptr(), y.data_ptr(), case["m"], case["k"], case["t"],
            state["rows"], ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != 0:
            raise RuntimeError(cllm.STATUS.get(rc, rc))
        return {"y": y}
    eng, n, out = state["eng"], case["n"], {}
    if case["kind"] == "generate":
        out["tokens"], out["iters"] = eng.jacobi_decode(state["prompts"], n, case["steps"], seed=state["seed"],
                                                        block_mode=MODES[case["mode"]])
    elif case["kind"] == "decode":
        eng.decode_begin(n, case["steps"] * n, seed=state["seed"], block_mode=MODES[case["mode"]])
        eng.decode_run(case["steps"])
        out["tokens"], out["iters"] = eng.decode_read()
    else:
        out["heads"] = eng.prefill(state["prompts"])
    step = eng.jacobi_step(state["guess"], want_gap=False, want_logits=True)
    out["next"], out["accepted"], out["logits"] = step["next"], step["accepted"], step["logits"]
    if case["kind"] == "generate":
        out.pop("iters")  # how soon the loop ends rests on the guesses that happen to hold, near ties among them
    return out


# ---- what a pass cannot do without ---------------------------------------------


def work(case):
    """Weights read once per forward, the cached keys and values of each row's
    sequence read once, new ones written, logits written; multiply-adds of the
    weights and of the causal attention.  (The activations' low-order plane is
    this engine's own choice and is not counted.)"""
    if case["kind"] == "gemm":
        m, k, t = case["m"], case["k"], case["t"]
        return {"bytes": 2 * m * k + 4 * t * k + 8 * t * m, "flops": 2.0 * m * k * t}
    cfg = _config(case)
    es, kes = (4, 4) if cfg.dtype == "f32" else (2, 2)
    d, dq, dkv = cfg.d_model, cfg.n_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim
    layer = d * dq + 2 * d * dkv + dq * d + 3 * d * cfg.ffn
    head = cfg.vocab * d
    b, n, mean = case["batch"], case["n"], (case["lo"] + case["hi"]) / 2

    def forward(rows, ctx, logit_rows):
        """rows new rows per sequence after ctx cached ones."""
        return (cfg.n_layers * (layer * es + 2 * dkv * kes * b * (ctx + rows)) + head * es + b * rows * d * es,
                2.0 * b * rows * cfg.n_layers * layer + 2.0 * b * logit_rows * head
                + 4.0 * cfg.n_layers * dq * b * rows * (ctx + rows / 2))

    total_b, total_f = forward(n, mean + (case["steps"] if case["kind"] != "prefill" else 0), n)
    total_b += 4 * b * n * cfg.vocab
    parts = []
    if case["kind"] != "decode":
        parts.append(forward(mean, 0, 1))
    # every iteration commits at least one token; with random weights, about one
    parts += [forward(n, mean + i, n) for i in range(case["steps"])]
    return {"bytes": total_b + sum(p[0] for p in parts), "flops": total_f + sum(p[1] for p in parts)}


def tolerance(case):
    """Four times the distance from 64 bits that the engines show: 6.6e-7 in
    fp32; in bf16 (activations as two bf16 planes; queries, keys, values and
    attention weights in fp16) 2.3e-4 for the small decoder, 1.2e-3 for a few
    layers of the 7B shape, 3.4e-3 for all 32.  Tokens differ where the two
    best logits are nearer than that."""
    if case["kind"] == "gemm":
        return {"rel": 2.6e-6}
    rel = {"tiny-f32": 3e-6, "tiny-bf16": 1e-3}.get(case["model"], 1.4e-2 if case["layers"] > 8 else 5e-3)
    return {"rel": rel, "differ": 0.01}


# ---- the same in 64 bits -------------------------------------------------------


def _mix(x):
    mask = (1 << 64) - 1
    x = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & mask
    x = ((x ^ (x >> 27)) * 0x94D049BB133111EB) & mask
    return x ^ (x >> 31)


def _guess(seed, b, step, slot, vocab):
    """Output (b<<40 | step<<16 | slot) + 1 of splitmix64, scaled to the vocabulary."""
    i = (b << 40 | step << 16 | slot) + 1
    return ((_mix((seed + i * 0x9E3779B97F4A7C15) & ((1 << 64) - 1)) >> 32) * vocab) >> 32


class _Decoder:
    """The pre-norm LLaMA decoder in fp64 with a key/value cache per sequence."""

    def __init__(self, cfg, w, batch):
        self.c, self.w = cfg, {k: ([t.double() for t in v] if isinstance(v, list) else v.double())
                               for k, v in w.items()}
        self.kv = [[None] * batch for _ in range(cfg.n_layers)]
        i = torch.arange(cfg.head_dim // 2, device=DEV, dtype=torch.float64)
        self.freq = float(cfg.rope_theta) ** (-2.0 * i / cfg.head_dim)

    def _norm(self, x, gain):
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + self.c.rms_eps) * gain

    def _rope(self, x, pos):
        ang = pos.double()[:, None] * self.freq
        cos, sin = ang.cos()[:, None, :], ang.sin()[:, None, :]
        a, b = x.chunk(2, -1)
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    def forward(self, blocks, starts, last_only=False):
        """Logits of each sequence's block (its last row only, if asked)."""
        c, w = self.c, self.w
        sizes = [len(t) for t in blocks]
        x = w["tok_emb"][torch.tensor(sum((list(map(int, t)) for t in blocks), []), device=DEV)]
        pos = torch.cat([torch.arange(s, s + k, device=DEV) for s, k in zip(starts, sizes)])
        for l in range(c.n_layers):
            h = self._norm(x, w["attn_norm"][l])
            q = self._rope((h @ w["wq"][l].T).view(-1, c.n_heads, c.head_dim), pos).split(sizes)
            k = self._rope((h @ w["wk"][l].T).view(-1, c.n_kv_heads, c.head_dim), pos).split(sizes)
            v = (h @ w["wv"][l].T).view(-1, c.n_kv_heads, c.head_dim).split(sizes)
            outs = []
            for b, (s, m) in enumerate(zip(starts, sizes)):
                old = self.kv[l][b]
                kk = k[b] if old is None else torch.cat([old[0][:s], k[b]])
                vv = v[b] if old is None else torch.cat([old[1][:s], v[b]])
                self.kv[l][b] = (kk, vv)
                g = c.n_heads // c.n_kv_heads
                kh, vh = kk.repeat_interleave(g, 1).transpose(0, 1), vv.repeat_interleave(g, 1).transpose(0, 1)
                sc = q[b].transpose(0, 1) @ kh.transpose(1, 2) / math.sqrt(c.head_dim)
                seen = torch.arange(s + m, device=DEV)[None, :] <= torch.arange(s, s + m, device=DEV)[:, None]
                p = sc.masked_fill_(~seen, -math.inf).softmax(-1)
                outs.append((p @ vh).transpose(0, 1).reshape(m, -1))
            x = x + torch.cat(outs) @ w["wo"][l].T
            h = self._norm(x, w["mlp_norm"][l])
            x = x + (torch.nn.functional.silu(h @ w["w_gate"][l].T) * (h @ w["w_up"][l].T)) @ w["w_down"][l].T
        if last_only:
            x = torch.stack([t[-1] for t in x.split(sizes)])
            sizes = [1] * len(sizes)
        return (self._norm(x, w["final_norm"]) @ w["lm_head"].T).split(sizes)


def exact(case, seed):
    """Logits (or Y) in 64 bits; tokens have no such value."""
    if case["kind"] == "gemm":
        w, planes, y0, _ = _gemm_inputs(case, seed)
        x = (planes[0].double() + planes[1].double())[:case["t"]]
        return {"y": y0.double() + x @ w.double().T}
    cfg, w, prompts, guess = _inputs(case, seed)
    dec = _Decoder(cfg, w, case["batch"])
    heads = [int(t[-1].argmax()) for t in dec.forward(prompts, [0] * len(prompts), last_only=True)]
    at = [len(p) for p in prompts]
    if case["kind"] == "generate":
        # any block policy's output is the greedy one: one token at a time gives the same state
        for _ in range(case["steps"]):
            heads_next = [int(t[-1].argmax()) for t in dec.forward([[h] for h in heads], at)]
            at, heads = [a + 1 for a in at], heads_next
    elif case["kind"] == "decode":
        n = case["n"]
        blocks = [[h] + [_guess(seed, b, 0, k, cfg.vocab) for k in range(1, n)] for b, h in enumerate(heads)]
        for it in range(1, case["steps"] + 1):
            for b, t in enumerate(dec.forward(blocks, at)):
                pred = t.argmax(-1).tolist()
                a = 1
                while a < n and blocks[b][a] == pred[a - 1]:
                    a += 1
                at[b], heads[b] = at[b] + a, pred[a - 1]
                blocks[b] = pred[a - 1:] + [_guess(seed, b, it, k, cfg.vocab) for k in range(n - a + 1, n)]
    last = [[h] + list(g[1:]) for h, g in zip(heads, guess.tolist())]
    logits = torch.stack(dec.forward(last, at))
    whole = {"generate": ("tokens",), "decode": ("tokens", "iters"), "prefill": ("heads",)}[case["kind"]]
    return {**{k: None for k in whole + ("next", "accepted")}, "logits": logits}
