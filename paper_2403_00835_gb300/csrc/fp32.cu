// fp32 engine: the weight GEMMs and the block attention on CUDA cores.
//
// The fp32 decoders are small (a layer's weights sit in L2), so a launch is
// bound by latency: how long one SM takes to pull its share of the weights
// and how many dependent steps follow.  Both kernels therefore spread a tile
// over many threads and keep every load of a tile in flight at once.
#include <float.h>

#include "act.cuh"
#include "attn_item.cuh"
#include "epilogue.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace cllm {

// ---------------------------------------------------------------------------------
// GEMM: D[m][t] = sum_k W[m][k] X[t][k] with the fused epilogues.
//
// A cluster of kF32Split CTAs computes one 128-row x 16-token tile: CTA
// `rank` sums its slice of K (thread r owns row r, tokens in registers), the
// others push their sums into rank 0's shared memory, and rank 0 adds the
// slices in rank order and runs the epilogue.  A single CTA would pull the
// tile's 128 KB (K = 256) to 344 KB (K = 688) of weights through one SM's L2
// port, 2-6 us; eight pull them in 0.3-0.8 us.  Weight slabs travel by
// cp.async, 8 threads per 128-byte row piece (one CTA per tile with one thread
// per row reading its own row touched 32 lines per load and took 34-56 us per
// launch at 8 tokens; with this attention kernel, a decode of 64 tokens at
// n = 8 went from 22.2 to 4.9 ms), and the first slabs are requested before the previous kernel has
// finished.  The slices depend on K only, so a token's bits do not depend on
// the launch's token count.
// ---------------------------------------------------------------------------------

constexpr int kF32Split = 8;       // CTAs (K slices) per tile: the portable cluster limit
constexpr int kF32Slab = 32;       // K elements per slab
constexpr int kF32Ld = kF32Slab + 4;  // padded row: 16-byte reads of 8 rows fall in distinct banks

struct F32GemmSmem {
  float w[2][kBM][kF32Ld];
  float x[2][kEpiCols][kF32Slab];
  float part[kF32Split - 1][kEpiCols][kBM];  // rank 0: the other ranks' sums
  EpiSmem es;
};

__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// NC: token columns computed (8 when the launch has at most 8 tokens).
template <int KIND, int NC>
__global__ void __launch_bounds__(128) gemm_f32_kernel(const GemmArgs g, const EpiArgs e, int kslice) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  F32GemmSmem& sm = *reinterpret_cast<F32GemmSmem*>(smem_raw);
  const int rank = static_cast<int>(cluster_ctarank());
  const int mt = blockIdx.x / kF32Split, nt = blockIdx.y, r = threadIdx.x;
  const int t0 = nt * kEpiCols;
  const int k0 = rank * kslice, k1 = min(g.K, k0 + kslice);
  const int nslab = k1 > k0 ? (k1 - k0 + kF32Slab - 1) / kF32Slab : 0;
  pdl_launch_dependents();
  cluster_arrive();  // waited for before the first remote store: every CTA has started
  // weight row of tile row rr (null: past the matrix)
  auto row_ptr = [&](int rr) -> const float* {
    if (KIND == EPI_GATEUP) {
      const int f = mt * 64 + (rr & 63);
      if (f >= g.M) return nullptr;
      return static_cast<const float*>(rr < 64 ? g.A0 : g.A1) + static_cast<size_t>(f) * g.K;
    }
    const int m = mt * kBM + rr;
    if (m >= g.M) return nullptr;
    if (KIND == EPI_QKV) {
      if (m < g.rows_q) return static_cast<const float*>(g.A0) + static_cast<size_t>(m) * g.K;
      if (m < g.rows_qk) return static_cast<const float*>(g.A1) + static_cast<size_t>(m - g.rows_q) * g.K;
      return static_cast<const float*>(g.A2) + static_cast<size_t>(m - g.rows_qk) * g.K;
    }
    return static_cast<const float*>(g.A0) + static_cast<size_t>(m) * g.K;
  };
  constexpr int PPR = kF32Slab / 4;  // 16-byte pieces per row of a slab
  auto load_w = [&](int s) {
    const int kb = k0 + s * kF32Slab, pc = (r % PPR) * 4;
#pragma unroll
    for (int i = 0; i < kBM * PPR / 128; ++i) {
      const int rr = i * (128 / PPR) + r / PPR;
      const float* src = row_ptr(rr);
      float* dst = &sm.w[s & 1][rr][pc];
      if (src != nullptr && kb + pc < k1)
        cp_async16(dst, src + kb + pc);
      else
        *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto load_x = [&](int s) {
    const int kb = k0 + s * kF32Slab;
    const int j = r / PPR, pc = (r % PPR) * 4, t = t0 + j;
    if (j >= NC) return;
    float* dst = &sm.x[s & 1][j][pc];
    if (t < g.T && kb + pc < k1)
      cp_async16(dst, static_cast<const float*>(g.X) + static_cast<size_t>(t) * g.ldx + kb + pc);
    else
      *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
  };
  // weights do not depend on the previous kernel: the first two slabs now
  if (nslab > 0) load_w(0);
  if (nslab > 1) load_w(1);
  pdl_wait();
  if (nslab > 0) load_x(0);
  cp_async_commit();
  if (nslab > 1) load_x(1);
  cp_async_commit();
  if (r == 0) sm.es.prepared = 0;
  EpiPre pre;
  pre.ok = 0;
  if (KIND == EPI_RESID && rank == 0) epi_prefetch<KIND, float>(e, mt, t0, r, sm.es, pre);

  float v[kEpiCols];
#pragma unroll
  for (int j = 0; j < kEpiCols; ++j) v[j] = 0.f;
  for (int s = 0; s < nslab; ++s) {
    cp_async_wait_but1();
    __syncthreads();
    const float* wr = sm.w[s & 1][r];
#pragma unroll
    for (int kk = 0; kk < kF32Slab; kk += 4) {
      const float4 w = *reinterpret_cast<const float4*>(wr + kk);
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const float4 x = *reinterpret_cast<const float4*>(&sm.x[s & 1][j][kk]);
        v[j] = fmaf(w.x, x.x, v[j]);
        v[j] = fmaf(w.y, x.y, v[j]);
        v[j] = fmaf(w.z, x.z, v[j]);
        v[j] = fmaf(w.w, x.w, v[j]);
      }
    }
    __syncthreads();
    if (s + 2 < nslab) {
      load_w(s + 2);
      load_x(s + 2);
    }
    cp_async_commit();
  }
  cluster_wait();
  if (rank != 0) {
    const uint32_t dst = mapa_smem(&sm.part[rank - 1][0][r], 0);
#pragma unroll
    for (int j = 0; j < NC; ++j) st_cluster(dst + j * kBM * 4, v[j]);
    cluster_arrive();  // release: rank 0's wait sees the sums
    cluster_wait();
    return;
  }
  cluster_arrive();
  cluster_wait();
#pragma unroll
  for (int q = 0; q < kF32Split - 1; ++q)
#pragma unroll
    for (int j = 0; j < NC; ++j) v[j] += sm.part[q][j][r];
  epi_apply<KIND, float>(e, mt, t0, v, r, sm.es, &pre);
  if (KIND == EPI_ARGMAX) epi_argmax_finish(e, r, sm.es);
}

// ---------------------------------------------------------------------------------
// Attention: one CTA of 128 threads per (16-row query tile, head, chunk of
// 128 keys anchored at position 0).  K, V and Q of the chunk are staged in
// shared memory with one round trip; a thread owns a key for the scores and
// a dimension for P.V, and a warp reduces a row's softmax, so no step is a
// serial walk over the keys (a warp per row with a reduction per key took
// 46 us for 8 rows x 100 keys).  A row's sums are over its own keys in an
// order fixed by their positions.  A tile of one chunk writes its output
// directly; otherwise the last chunk of a (tile, head) to finish merges the
// partials in chunk order (self-resetting ticket), which saves a launch.
// ---------------------------------------------------------------------------------

template <int HD>
struct F32AttnSmem {
  float k[kAttnChunk][HD + 4];
  float v[kAttnChunk][HD];
  float q[kQTile][HD];
  float p[kQTile][kAttnChunk];  // scores, then probabilities
  float m[kQTile], l[kQTile];
  int last;
};

struct F32Sync {
  __device__ void operator()() const { __syncthreads(); }
};

constexpr int kF32MaxQTiles = 2048;

template <int HD>
__global__ void __launch_bounds__(128) attn_f32_kernel(const AttnArgs a, int* tickets) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  F32AttnSmem<HD>& sm = *reinterpret_cast<F32AttnSmem<HD>*>(smem_raw);
  int* pre = reinterpret_cast<int*>(smem_raw + (sizeof(F32AttnSmem<HD>) + 15) / 16 * 16);
  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int total = attn_item_prefix(a, pre, tid, F32Sync{}, 1);
  const int group = a.H / a.Hkv;
  const int ldq = a.H * HD;
  const float* Q = static_cast<const float*>(a.q);
  const float* KC = static_cast<const float*>(a.k_cache);
  const float* VC = static_cast<const float*>(a.v_cache);
  float* out = static_cast<float*>(a.out);
  constexpr int PPR = HD / 4;               // 16-byte pieces per row
  constexpr int DG = 128 / HD;              // row groups of the P.V step (2 at HD 64)
  constexpr int RPT = kQTile / DG;          // rows per thread there
  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    const int qi = attn_find_qtile(pre, a.n_qtiles, item);
    const int local = item - pre[qi];
    const int c = local / a.H, h = local - c * a.H;
    const int nch = (pre[qi + 1] - pre[qi]) / a.H;
    const int2 qt = a.qtiles[qi];
    const int b = qt.x, r0 = qt.y;
    const int nr = min(kQTile, a.seq_nrows[b] - r0);
    const int pos0 = a.seq_start[b] + r0;
    const int row_g0 = a.seq_row0[b] + r0;
    const int kb = c * kAttnChunk;
    if (pos0 + nr > a.max_seq && tid == 0) atomicOr(a.err, DERR_CAPACITY);
    const int nk = min(min(pos0 + nr, a.max_seq) - kb, kAttnChunk);  // keys of the chunk that some row sees
    const size_t kvbase = ((static_cast<size_t>(b) * a.Hkv + h / group) * a.max_seq + kb) * HD;
    // ---- stage: Q and K, then V ----
    for (int i = tid; i < kQTile * PPR; i += 128) {
      const int rr = i / PPR, pc = (i - rr * PPR) * 4;
      if (rr < nr)
        cp_async16(&sm.q[rr][pc], Q + static_cast<size_t>(row_g0 + rr) * ldq + h * HD + pc);
      else
        *reinterpret_cast<float4*>(&sm.q[rr][pc]) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int i = tid; i < nk * PPR; i += 128) {
      const int rr = i / PPR, pc = (i - rr * PPR) * 4;
      cp_async16(&sm.k[rr][pc], KC + kvbase + static_cast<size_t>(rr) * HD + pc);
    }
    cp_async_commit();
    for (int i = tid; i < nk * PPR; i += 128) {
      const int rr = i / PPR, pc = (i - rr * PPR) * 4;
      cp_async16(&sm.v[rr][pc], VC + kvbase + static_cast<size_t>(rr) * HD + pc);
    }
    cp_async_commit();
    cp_async_wait_but1();
    __syncthreads();
    // ---- scores: thread = key, 8 rows at a time ----
    const int key = kb + tid;
    for (int rb = 0; rb < nr; rb += 8) {
      float s[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) s[j] = 0.f;
      if (tid < nk) {
#pragma unroll 4
        for (int d = 0; d < HD; d += 4) {
          const float4 kv = *reinterpret_cast<const float4*>(&sm.k[tid][d]);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 qv = *reinterpret_cast<const float4*>(&sm.q[rb + j][d]);
            s[j] = fmaf(qv.x, kv.x, s[j]);
            s[j] = fmaf(qv.y, kv.y, s[j]);
            s[j] = fmaf(qv.z, kv.z, s[j]);
            s[j] = fmaf(qv.w, kv.w, s[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        sm.p[rb + j][tid] = (tid < nk && key <= pos0 + rb + j) ? s[j] * a.scale_log2 : -INFINITY;
    }
    __syncthreads();
    // ---- softmax of a row: one warp, 4 keys per lane ----
    for (int i = warp; i < nr; i += 4) {
      float x[4], mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = sm.p[i][lane + 32 * u];
        mx = fmaxf(mx, x[u]);
      }
      mx = warp_max(mx);
      float sum = 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = mx == -INFINITY ? 0.f : exp2f(x[u] - mx);  // (a row may see no key of the chunk)
        sm.p[i][lane + 32 * u] = x[u];
        sum += x[u];
      }
      sum = warp_sum(sum);
      if (lane == 0) {
        sm.m[i] = mx;
        sm.l[i] = sum;
      }
    }
    cp_async_wait_all();
    __syncthreads();
    // ---- P.V: thread = dimension (and row group) ----
    const int d = tid % HD, rg = (tid / HD) * RPT;
    float o[RPT];
#pragma unroll
    for (int j = 0; j < RPT; ++j) o[j] = 0.f;
    const bool work = rg < nr;
    int kk = 0;
    if (work) {
      for (; kk + 4 <= nk; kk += 4) {
        const float v0 = sm.v[kk][d], v1 = sm.v[kk + 1][d], v2 = sm.v[kk + 2][d], v3 = sm.v[kk + 3][d];
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          if (rg + j < nr) {
            const float4 p = *reinterpret_cast<const float4*>(&sm.p[rg + j][kk]);
            o[j] = fmaf(p.x, v0, o[j]);
            o[j] = fmaf(p.y, v1, o[j]);
            o[j] = fmaf(p.z, v2, o[j]);
            o[j] = fmaf(p.w, v3, o[j]);
          }
        }
      }
      for (; kk < nk; ++kk) {
        const float v0 = sm.v[kk][d];
#pragma unroll
        for (int j = 0; j < RPT; ++j)
          if (rg + j < nr) o[j] = fmaf(sm.p[rg + j][kk], v0, o[j]);
      }
    }
    if (nch == 1) {
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (rg + j < nr) out[static_cast<size_t>(row_g0 + rg + j) * ldq + h * HD + d] = o[j] / sm.l[rg + j];
      __syncthreads();  // the tile is reloaded by the next item
      continue;
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (rg + j < nr) {
        const size_t pidx = (static_cast<size_t>(row_g0 + rg + j) * a.H + h) * a.nch_max + c;
        a.part_o[pidx * HD + d] = o[j];
        if (d == 0) a.part_ml[pidx] = make_float2(sm.m[rg + j], sm.l[rg + j]);
      }
    __syncthreads();
    if (tid == 0) {
      int* tk = tickets + static_cast<size_t>(qi) * a.H + h;
      const int old = ticket_add(tk, 1);
      sm.last = old == nch - 1;
      if (sm.last) *tk = 0;
    }
    __syncthreads();
    if (!sm.last) continue;
    // ---- last chunk of the tile: merge a row's chunks 0..pos/128 in order ----
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if (rg + j >= nr) continue;
      const size_t base = (static_cast<size_t>(row_g0 + rg + j) * a.H + h) * a.nch_max;
      const int n = min((pos0 + rg + j) / kAttnChunk + 1, nch);
      float M = -INFINITY;
      for (int i = 0; i < n; ++i) M = fmaxf(M, __ldcg(&a.part_ml[base + i].x));
      float acc = 0.f, l = 0.f;
      for (int i = 0; i < n; ++i) {
        const float2 ml = __ldcg(&a.part_ml[base + i]);
        const float f = exp2f(ml.x - M);
        l = fmaf(f, ml.y, l);
        acc = fmaf(f, __ldcg(a.part_o + (base + i) * HD + d), acc);
      }
      out[static_cast<size_t>(row_g0 + rg + j) * ldq + h * HD + d] = acc / l;
    }
  }
}

// ---- launchers ----------------------------------------------------------------------

template <int HD>
constexpr size_t attn_f32_smem_bytes() {
  return (sizeof(F32AttnSmem<HD>) + 15) / 16 * 16 + sizeof(int) * (kF32MaxQTiles + 1);
}
static_assert(attn_f32_smem_bytes<128>() <= 227 * 1024, "fp32 attention shared memory");

template <int KIND>
static cudaError_t f32_set_kind() {
  cudaError_t err = cudaFuncSetAttribute(gemm_f32_kernel<KIND, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(F32GemmSmem)));
  if (err != cudaSuccess) return err;
  return cudaFuncSetAttribute(gemm_f32_kernel<KIND, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(sizeof(F32GemmSmem)));
}

cudaError_t f32_set_attributes() {
  cudaError_t err;
  if ((err = f32_set_kind<EPI_QKV>()) != cudaSuccess) return err;
  if ((err = f32_set_kind<EPI_GATEUP>()) != cudaSuccess) return err;
  if ((err = f32_set_kind<EPI_RESID>()) != cudaSuccess) return err;
  if ((err = f32_set_kind<EPI_ARGMAX>()) != cudaSuccess) return err;
  if ((err = cudaFuncSetAttribute(attn_f32_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(attn_f32_smem_bytes<64>()))) != cudaSuccess)
    return err;
  return cudaFuncSetAttribute(attn_f32_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(attn_f32_smem_bytes<128>()));
}

static void f32_cfg(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, dim3 grid, size_t smem, cudaStream_t s,
                    bool pdl, int cluster) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
}

template <int KIND>
static cudaError_t launch_f32_one(const GemmArgs& g, const EpiArgs& e, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  f32_cfg(cfg, attr, dim3(g.mtiles * kF32Split, g.ntiles), sizeof(F32GemmSmem), s, pdl, kF32Split);
  const int kslice = round_up(ceil_div(g.K, kF32Split), 4);
  if (g.T <= 8) return cudaLaunchKernelEx(&cfg, gemm_f32_kernel<KIND, 8>, g, e, kslice);
  return cudaLaunchKernelEx(&cfg, gemm_f32_kernel<KIND, 16>, g, e, kslice);
}

cudaError_t launch_gemm_f32(int kind, const GemmArgs& g, const EpiArgs& e, cudaStream_t s, bool pdl) {
  switch (kind) {
    case EPI_QKV: return launch_f32_one<EPI_QKV>(g, e, s, pdl);
    case EPI_GATEUP: return launch_f32_one<EPI_GATEUP>(g, e, s, pdl);
    case EPI_RESID: return launch_f32_one<EPI_RESID>(g, e, s, pdl);
    case EPI_ARGMAX: return launch_f32_one<EPI_ARGMAX>(g, e, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_attention_f32(const AttnArgs& a, int* tickets, int grid, cudaStream_t s, bool pdl) {
  if (a.n_qtiles > kF32MaxQTiles) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  if (a.hd == 64) {
    f32_cfg(cfg, attr, dim3(grid), attn_f32_smem_bytes<64>(), s, pdl, 1);
    return cudaLaunchKernelEx(&cfg, attn_f32_kernel<64>, a, tickets);
  }
  if (a.hd == 128) {
    f32_cfg(cfg, attr, dim3(grid), attn_f32_smem_bytes<128>(), s, pdl, 1);
    return cudaLaunchKernelEx(&cfg, attn_f32_kernel<128>, a, tickets);
  }
  return cudaErrorInvalidValue;
}

}  // namespace cllm
