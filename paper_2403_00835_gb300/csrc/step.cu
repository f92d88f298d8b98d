// Per-iteration kernels around the block forward:
//   embed       - token rows of the block (or of a prefill) -> fp32 residual
//                 stream, first RMSNorm input and per-tile sums of squares,
//                 plus each row's position and sequence index
//   accept      - the fixed-point test of Alg. 3: longest prefix of the block
//                 reproduced by the predictions, commit (advance the committed
//                 length; the K/V already sit in the cache), new head, refill
//   decode_init - reset a decode to the prefill state, draw the first guesses
// Guesses come from a counter-based splitmix64 stream (Vigna): the
// ((b<<40 | iteration<<16 | slot) + 1)-th output for key `seed`.
#include "act.cuh"
#include "internal.cuh"
#include "ptx.cuh"
#include "step_items.cuh"

namespace cllm {

struct StepSync {
  __device__ void operator()() const { __syncthreads(); }
};

// One warp per (row, 128-column group): the same values and sums as embed_unit
// (a column per lane in each quarter of the group), without its block barrier
// and with 8 groups to a block.  A block per group was bound by launching
// blocks: 69 us for 2048 rows of 4096 columns (84 MB).
constexpr int kEmbedWarps = 8;

template <typename Act>
__global__ void __launch_bounds__(32 * kEmbedWarps) embed_kernel(const EmbedArgs a) {
  pdl_launch_dependents();
  pdl_wait();
  const int ngrp = a.d / 128, lane = threadIdx.x & 31;
  const int unit = blockIdx.x * kEmbedWarps + (threadIdx.x >> 5);
  if (unit >= a.T * ngrp) return;
  const int t = unit / ngrp, grp = unit - t * ngrp;
  int tok, pos, b;
  embed_row(a, t, tok, pos, b);
  if (tok < 0 || tok >= a.V) {
    if (lane == 0 && grp == 0) atomicOr(a.err, DERR_TOKEN);
    tok = 0;
  }
  const int m0 = grp * 128 + lane;
  const Act* src = static_cast<const Act*>(a.emb) + static_cast<size_t>(tok) * a.d + m0;
  const Act* gain = static_cast<const Act*>(a.gain) + m0;
  const size_t o = static_cast<size_t>(t) * a.d + m0;
  float e[4], g[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    e[q] = ld_act(src, 32 * q);
    g[q] = ld_act(gain, 32 * q);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    a.x[o + 32 * q] = e[q];
    st_gin(static_cast<Act*>(a.xg), o + 32 * q, a.plane, e[q] * g[q]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) e[q] = warp_sum(e[q] * e[q]);
  if (lane == 0) a.ssq[static_cast<size_t>(grp) * a.ldt + t] = ((e[0] + e[1]) + e[2]) + e[3];
  if (grp == 0) embed_meta(a, t, pos, b, lane, 32);
}

__global__ void __launch_bounds__(128) accept_kernel(const AcceptArgs a) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int s_act[4], s_com[4];
  accept_body(a, threadIdx.x, s_act, s_com, StepSync{});
}

__global__ void __launch_bounds__(128) decode_init_kernel(const AcceptArgs a) {
  const int tid = threadIdx.x;
  for (int b = tid; b < a.B; b += blockDim.x) {
    a.L[b] = a.plen[b];
    a.committed[b] = 0;
    a.iters[b] = 0;
    a.done[b] = 0;
    if (a.width != nullptr) a.width[b] = a.n;
    int* y = a.block + b * a.n;
    y[0] = a.head[b];
    for (int k = 1; k < a.n; ++k) y[k] = draw_guess(a, b, 0, k);
    if (a.acc_hist != nullptr) {
      a.win_end[b] = 0;
      a.win_cnt[b] = 0;
      for (int k = 0; k < a.n; ++k) a.st_pos[static_cast<size_t>(b) * a.n + k] = -1;
    }
  }
  if (a.acc_hist != nullptr) {
    for (int i = tid; i <= a.n; i += blockDim.x) {
      a.acc_hist[i] = 0;
      a.win_hist[i] = 0;
    }
    if (tid < 2) a.totals[tid] = 0;
  }
  for (size_t i = tid; i < static_cast<size_t>(a.B) * a.max_new; i += blockDim.x) a.out[i] = -1;
  if (tid == 0) {
    a.status[0] = a.B;
    a.status[1] = 0;
  }
}

__global__ void set_head_kernel(int* block, const int* head, int B, int n, int V, int* err) {
  const int b = threadIdx.x;
  if (b < B) {
    const int h = head[b];
    if (h < 0 || h >= V) atomicOr(err, DERR_TOKEN);
    block[b * n] = h;
  }
}

// Row `rows[b]` of the norm input (row_bytes per plane, 16-byte pieces; the lo
// plane, if any, plane bytes further) and of its statistics.  Every piece is
// one independent load, so a row costs one round trip (element by element it
// took 17 us).
__global__ void __launch_bounds__(256) gather_rows_kernel(const char* src, const float* ssq_src, char* dst,
                                                          float* ssq_dst, const int* rows, int row_bytes, int d,
                                                          int ldt_src, int ldt_dst, size_t plane_src,
                                                          size_t plane_dst) {
  const int b = blockIdx.x, row = rows[b];
  const int per = row_bytes / 16, n = plane_dst ? 2 * per : per;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 256) {
    const int pl = i >= per ? 1 : 0;
    const size_t o = static_cast<size_t>(i - pl * per) * 16;
    *reinterpret_cast<uint4*>(dst + pl * plane_dst + static_cast<size_t>(b) * row_bytes + o) =
        __ldcg(reinterpret_cast<const uint4*>(src + pl * plane_src + static_cast<size_t>(row) * row_bytes + o));
  }
  for (int i = threadIdx.x; i < d / 128; i += 256)
    ssq_dst[static_cast<size_t>(i) * ldt_dst + b] = __ldcg(ssq_src + static_cast<size_t>(i) * ldt_src + row);
}

// ---- launchers ----------------------------------------------------------------------

static void small_cfg(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, dim3 grid, dim3 block,
                      cudaStream_t s, bool pdl) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

cudaError_t launch_embed(const EmbedArgs& a, int act_bf16, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  small_cfg(cfg, attr, dim3((a.T * (a.d / 128) + kEmbedWarps - 1) / kEmbedWarps), dim3(32 * kEmbedWarps), s, pdl);
  if (act_bf16) return cudaLaunchKernelEx(&cfg, embed_kernel<__nv_bfloat16>, a);
  return cudaLaunchKernelEx(&cfg, embed_kernel<float>, a);
}

cudaError_t launch_accept(const AcceptArgs& a, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  small_cfg(cfg, attr, dim3(1), dim3(128), s, pdl);
  return cudaLaunchKernelEx(&cfg, accept_kernel, a);
}

cudaError_t launch_decode_init(const AcceptArgs& a, cudaStream_t s) {
  decode_init_kernel<<<1, 128, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_set_head(int* block, const int* head, int B, int n, int V, int* err,
                            cudaStream_t s) {
  set_head_kernel<<<1, 128, 0, s>>>(block, head, B, n, V, err);
  return cudaGetLastError();
}

cudaError_t launch_gather_rows(const void* xg_src, const float* ssq_src, void* xg_dst,
                               float* ssq_dst, const int* rows, int B, int d, int ldt_src,
                               int ldt_dst, size_t plane_src, size_t plane_dst, int act_bf16,
                               cudaStream_t s) {
  // (d is a multiple of 128, so rows and planes are whole 16-byte pieces)
  const size_t es = act_bf16 ? 2 : 4;
  gather_rows_kernel<<<B, 256, 0, s>>>(static_cast<const char*>(xg_src), ssq_src, static_cast<char*>(xg_dst), ssq_dst,
                                       rows, static_cast<int>(d * es), d, ldt_src, ldt_dst,
                                       act_bf16 ? plane_src * es : 0, act_bf16 ? plane_dst * es : 0);
  return cudaGetLastError();
}

}  // namespace cllm
