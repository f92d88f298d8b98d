"""The bf16 weight GEMM (tcgen05 + TMA, split-K with fixed-order reduction) in
isolation: Y[t][m] = sum_k W[m][k] X[t][k] against an fp64 matmul of the same
bf16 values, over ragged M/K/T tiles, split and whole-tile work partitions; and,
up to 256 tokens, a token's column must be bit-identical whatever the number of
tokens in the launch (the property that makes a Jacobi step and an AR step
agree).  `engine` is the kernel that the engine launches (CTA pairs; the test
hook of include/cllm_testing.h), `noalloc` the allocation-free entry point's."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_00835_gb300 import cllm

pytestmark = pytest.mark.gpu


def _lib():
    lib = cllm.load()
    lib.cllm_test_gemm_bf16.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 4
    lib.cllm_test_gemm_bf16.restype = ctypes.c_int
    return lib


def split_hilo(x):
    """fp32 activations -> stacked bf16 planes [2][rows][K]: hi = bf16(x), lo = bf16(x - hi)."""
    hi = x.bfloat16()
    lo = (x - hi.float()).bfloat16()
    return torch.stack([hi, lo]).contiguous()


def run_gemm(W, X2, T, which="engine"):
    M, K = W.shape
    Y = torch.zeros(T, M, device="cuda", dtype=torch.float32)
    if which == "engine":
        rc = _lib().cllm_test_gemm_bf16(W.data_ptr(), X2.data_ptr(), Y.data_ptr(), M, K, T, X2.shape[1])
    else:
        rc = _lib().cllm_gemm_bf16_noalloc(W.data_ptr(), X2.data_ptr(), Y.data_ptr(), M, K, T, X2.shape[1],
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, cllm.STATUS.get(rc, rc)
    return Y


def x_rows(T):
    return max((T + 15) // 16 * 16, 256 if T > 256 else 0)


def check_fp64(W, X2, T, Y):
    Y = Y.cpu().double().numpy()
    Wd = W.cpu().double().numpy()
    Xd = (X2[0, :T].double() + X2[1, :T].double()).cpu().numpy()
    ref = Xd @ Wd.T
    bound = 1e-5 * (np.abs(Xd) @ np.abs(Wd).T) + 1e-7
    assert (np.abs(Y - ref) <= bound).all(), float((np.abs(Y - ref) / bound).max())


def inputs(M, K, rows, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = (torch.randn(M, K, device="cuda", generator=g) * 0.02).bfloat16()
    return W, split_hilo(torch.randn(rows, K, device="cuda", generator=g))


@pytest.mark.parametrize("M,K,T", [
    (128, 64, 1), (128, 64, 16), (768, 256, 8), (256, 688, 17), (512, 256, 100),
    (256, 512, 256), (384, 256, 300), (4096, 4096, 16), (4096, 11008, 64), (12288, 4096, 32),
    (256, 4096, 520)])
def test_gemm_matches_fp64(M, K, T):
    W, X2 = inputs(M, K, x_rows(T), M * 7 + K * 3 + T)
    check_fp64(W, X2, T, run_gemm(W, X2, T))


# 1, 2, 3, 5 and 11 weight tiles (a pair without its second tile, groups of 4
# that are not full) and the 7B projection; K = 2056, 688 and 4096 are cut over
# several CTAs' ranges, K = 72 is not
EDGE_T = (1, 16, 64, 65, 128, 129, 144, 256)


@pytest.mark.parametrize("M,K", [(128, 2056), (256, 688), (384, 72), (640, 4096), (1408, 688), (4096, 4096)])
def test_engine_gemm_at_tile_edges(M, K):
    """Every width of the pair kernel (stacked planes up to 128 tokens, two MMAs
    per chunk above) against fp64, and bit for bit against one another."""
    W, X2 = inputs(M, K, 256, M + K)
    ys = {T: run_gemm(W, X2, T) for T in EDGE_T}
    for T, Y in ys.items():
        check_fp64(W, X2, T, Y)
        assert torch.equal(Y, ys[256][:T]), T


@pytest.mark.parametrize("M,K,widths", [
    (128, 2056, EDGE_T), (256, 688, EDGE_T), (640, 1024, (1, 16, 64, 65)), (4096, 4096, (1, 16))])
def test_noalloc_gemm_at_tile_edges(M, K, widths):
    W, X2 = inputs(M, K, 256, M + K + 1)
    ys = {T: run_gemm(W, X2, T, "noalloc") for T in widths}
    for T, Y in ys.items():
        check_fp64(W, X2, T, Y)
        assert torch.equal(Y, ys[max(widths)][:T]), T


@pytest.mark.parametrize("M,K", [(4096, 4096), (768, 688)])
def test_gemm_column_independent_of_token_count(M, K):
    W, X2 = inputs(M, K, 256, 5)
    ys = {T: run_gemm(W, X2, T) for T in (1, 16, 48, 64, 256)}
    for T in (16, 48, 64, 256):
        assert torch.equal(ys[T][:1], ys[1])
    assert torch.equal(ys[64][:48], ys[48])
    assert torch.equal(ys[256][:64], ys[64])
