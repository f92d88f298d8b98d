// Weight GEMMs of launches with more than 256 token rows (prefill, wide batches).
//
//   D[m][t] = sum_k W[m][k] X[t][k],  X in two bf16 planes (hi, lo)
//
// Here every weight tile meets many tokens, so the launch is bound by the
// tensor pipe -- if shared memory can be filled fast enough.  A CTA pair
// (tcgen05 cta_group::2) works on 512 weight rows x up to 128 tokens: each CTA
// holds two 128-row weight tiles and one plane of the activations (the pair's
// B operand is [hi rows | lo rows], one half in each CTA), so a 64-column
// chunk costs a CTA 48 KB of shared-memory fill for eight MMAs of M = 256,
// N = 256 (0.58 us at the dense rate).  The 128 x 256 tile of a single CTA
// with both planes cost 80 KB for the same MMA work and ran at the L2's
// bandwidth.
//
// The two weight tiles are two accumulators (hi and lo columns of each: 512
// tensor-memory columns) whose rows are chosen so that a lane holds what the
// epilogue combines: gate and up rows of the same feature, or the two halves
// of a rotate-half pair.  The epilogue's 8 warps first pull the whole
// accumulator into registers (128 sums per thread, ~0.4 us) and hand tensor
// memory back, so the next unit's MMAs run while they finish this one.
//
// Work split: unit u (token tiles of a row unit are neighbours, so that the
// clusters working at one time share weights through L2) goes to cluster
// u mod clusters for as many whole rounds as there are; the remaining units'
// (unit, K chunk) space is cut into equal contiguous ranges, one per cluster.
// A unit cut over several ranges is finished by whichever contributor is the
// last to arrive (a ticket); the others leave their sums in global partials.
// No cluster ever waits for another one, so the launch needs no co-residency
// (another engine's launches may hold part of the SMs), and the sums are added
// in range order, so the result does not depend on the order of arrival.
// (The first contributor waiting for the others saved the store of its own
// sums -- 500 rows 1.25 against 1.29 ms, 4096 rows 5.53 against 5.58 -- but two
// engines' launches, each with part of its clusters resident, could hold each
// other until the waits ran out.)
//
// Per launch at 2048 rows, 7B shape, against the single-CTA kernel: gate/up
// 757 -> 405 us (1.82 PFLOP/s counting both planes: near the power limit), QKV
// 555 -> 246, O and down together 511 -> 359.  Two pairs of a cluster sharing
// each weight tile by multicast loads would take gate/up to 384 us (4096-row
// prefill, 2 layers, 5.20 against 5.30 ms), but the ranks of a replica run load
// this library too, and a multicast load has no place in a multi-GPU program.
#include <float.h>
#include <limits.h>

#include <algorithm>

#include "act.cuh"
#include "epilogue.cuh"
#include "gemm_roles.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace cllm {

constexpr int kWStages = 4;
constexpr int kWATile = kBM * kBK * 2;           // one 128 x 64 weight tile
constexpr int kWBTile = kWideTokens * kBK * 2;   // one plane of 128 tokens
constexpr int kWStage = 2 * kWATile + kWBTile;   // 48 KB
// Warps 0-3: producer, MMA issuer, two idle; warps 4-11: epilogue.  The launch
// has 384 x 168 registers; the first warpgroup keeps 56 a thread and the
// epilogue's two take 224 (128 x 56 + 256 x 224 = 384 x 168), so a thread holds
// its 128 sums without spilling.
constexpr int kWThreads = 128 + 256;
constexpr int kWRegsLow = 56, kWRegsEpi = 224;
static_assert(128 * kWRegsLow + 256 * kWRegsEpi <= kWThreads * 168, "register split");

struct WideSmem {
  float rs[kWideTokens];
  int pos[kWideTokens];
  int bidx[kWideTokens];
  float red[2][2][4][4][kEpiCols];     // [group][accumulator][chunk][warp][column]
  float am[2][2][4][4][kEpiCols][3];
  uint64_t full[kWStages], empty[kWStages], tfull, tempty, drain;
  uint32_t tmem;
  int abort_flag;
  int issued;  // chunks this CTA's producer has loaded
  int ok[2];  // [0] the accumulator wait's result, [1] this cluster finishes the unit
};

constexpr size_t wide_smem_bytes() { return 1024 + kWStages * kWStage + sizeof(WideSmem); }
static_assert(kWideTokens == 8 * kEpiCols, "partial layout");
static_assert(wide_smem_bytes() <= 227 * 1024, "wide GEMM shared memory");

// (max, argmax, second max) of 16 columns over a warp's 32 rows; column c ends
// in lanes 2c and 2c + 1 (halving exchanges; the merge is exact).
__device__ __forceinline__ void warp_argmax16(float (&c1)[kEpiCols], int m, int lane, float& o1, int& oi, float& o2) {
  float c2[kEpiCols];
  int ci[kEpiCols];
#pragma unroll
  for (int j = 0; j < kEpiCols; ++j) {
    c2[j] = -INFINITY;
    ci[j] = m;
  }
#pragma unroll
  for (int o = 16, half = 8; o >= 2; o >>= 1, half >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float w1 = __shfl_xor_sync(0xffffffffu, hi ? c1[i] : c1[i + half], o);
      const int wj = __shfl_xor_sync(0xffffffffu, hi ? ci[i] : ci[i + half], o);
      const float w2 = __shfl_xor_sync(0xffffffffu, hi ? c2[i] : c2[i + half], o);
      float a1 = hi ? c1[i + half] : c1[i], a2 = hi ? c2[i + half] : c2[i];
      int ai = hi ? ci[i + half] : ci[i];
      am_merge(a1, ai, a2, w1, wj, w2);
      c1[i] = a1;
      ci[i] = ai;
      c2[i] = a2;
    }
  }
  o1 = c1[0];
  o2 = c2[0];
  oi = ci[0];
  am_merge(o1, oi, o2, __shfl_xor_sync(0xffffffffu, c1[0], 1), __shfl_xor_sync(0xffffffffu, ci[0], 1),
           __shfl_xor_sync(0xffffffffu, c2[0], 1));
}

// Epilogue of one finished unit: v0 / v1 = the two accumulators' sums of this
// thread's lane, chunk c = tokens t0 + (grp + 2c) * 16 .. + 15.
//   row0: first weight row of this CTA's accumulator 0 (accumulator 1 follows
//   at +128; GATEUP: feature index of both)
template <int KIND>
__device__ __forceinline__ void wide_apply(const EpiArgs& e, const GemmArgs& g, int row0, int t0, int lr, int grp,
                                           float (&v0)[4][kEpiCols], float (&v1)[4][kEpiCols], WideSmem& s) {
  const int lane = lr & 31, w4 = lr >> 5;
  if (KIND == EPI_GATEUP) {
    const int f = row0 + lr;
    if (f >= e.F) return;
    __nv_bfloat16* hp = static_cast<__nv_bfloat16*>(e.h_out) + f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int tl = (grp + 2 * c) * kEpiCols;
      if (tl >= g.bn) break;
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) {
        const int t = t0 + tl + j;
        const float rs = s.rs[tl + j];
        const float gt = v0[c][j] * rs, up = v1[c][j] * rs;
        if (tl + j < g.bn && t < e.T)
          st_gin(hp, static_cast<size_t>(t) * e.F, e.plane_h, __fdividef(gt, 1.f + __expf(-gt)) * up);
      }
    }
  } else if (KIND == EPI_QKV) {
    // accumulator 0: first halves of 256 / hd heads, accumulator 1: their second halves
    const int half = e.hd >> 1;
    const int hl = lr / half, i = lr - hl * half;
    const int hs = row0 / e.hd + hl;  // head slot: Q heads, K heads, V heads
    const int H = e.dq / e.hd, HK = e.n_kv_heads;
    if (hs >= H + 2 * HK) return;
    const int sec = hs < H ? 0 : (hs < H + HK ? 1 : 2);
    const size_t kvh = static_cast<size_t>(hs - (sec == 1 ? H : H + HK));
    __half* q = static_cast<__half*>(e.q_out) + hs * e.hd + i;
    __half* cache = static_cast<__half*>(sec == 1 ? e.k_cache : e.v_cache) + kvh * e.max_seq * e.hd + i;
    const size_t bstride = static_cast<size_t>(HK) * e.max_seq * e.hd;
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int tl = (grp + 2 * c) * kEpiCols;
      if (tl >= g.bn) break;
      if (sec < 2) {
        float2 cs[kEpiCols];
#pragma unroll
        for (int j = 0; j < kEpiCols; ++j)
          cs[j] = e.rope[static_cast<size_t>(min(max(s.pos[tl + j], 0), e.max_seq - 1)) * half + i];
#pragma unroll
        for (int j = 0; j < kEpiCols; ++j) {
          const float rs = s.rs[tl + j];
          const float a = v0[c][j] * rs, b = v1[c][j] * rs;
          v0[c][j] = a * cs[j].x - b * cs[j].y;
          v1[c][j] = b * cs[j].x + a * cs[j].y;
        }
      } else {
#pragma unroll
        for (int j = 0; j < kEpiCols; ++j) {
          v0[c][j] *= s.rs[tl + j];
          v1[c][j] *= s.rs[tl + j];
        }
      }
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) {
        const int t = t0 + tl + j;
        if (tl + j >= g.bn || t >= e.T) continue;
        __half* dst;
        if (sec == 0) {
          dst = q + static_cast<size_t>(t) * e.dq;
        } else {
          const int p = s.pos[tl + j];
          if (static_cast<unsigned>(p) >= static_cast<unsigned>(e.max_seq)) {
            bad = true;
            continue;
          }
          dst = cache + static_cast<size_t>(s.bidx[tl + j]) * bstride + static_cast<size_t>(p) * e.hd;
        }
        dst[0] = __float2half_rn(v0[c][j]);
        dst[half] = __float2half_rn(v1[c][j]);
      }
    }
    if (bad) atomicOr(e.err, DERR_CAPACITY);
  } else if (KIND == EPI_RESID || KIND == EPI_ACC) {
#pragma unroll
    for (int st = 0; st < 8; ++st) {
      const int a = st >> 2, c = st & 3;
      const int m = row0 + a * kBM + lr, tl = (grp + 2 * c) * kEpiCols;
      if (m >= g.M || tl >= g.bn) continue;  // whole tiles (M is a multiple of 128)
      float (&v)[4][kEpiCols] = a == 0 ? v0 : v1;
      const float gn = KIND == EPI_RESID ? ld_act(static_cast<const __nv_bfloat16*>(e.gnext), m) : 0.f;
      float* xp = e.x + static_cast<size_t>(t0 + tl) * e.d + m;
      __nv_bfloat16* gp = static_cast<__nv_bfloat16*>(e.xg) + static_cast<size_t>(t0 + tl) * e.d + m;
      float xi[kEpiCols], sq[kEpiCols];
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) {
        const bool live = tl + j < g.bn && t0 + tl + j < e.T;
        xi[j] = live ? __ldcg(xp + static_cast<size_t>(j) * e.d) : 0.f;
      }
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) {
        const bool live = tl + j < g.bn && t0 + tl + j < e.T;
        xi[j] += v[c][j];
        sq[j] = live ? xi[j] * xi[j] : 0.f;
        if (live) {
          const size_t o = static_cast<size_t>(j) * e.d;
          xp[o] = xi[j];
          if (KIND == EPI_RESID) st_gin(gp, o, e.plane_x, xi[j] * gn);
        }
      }
      if (KIND == EPI_ACC) continue;
      const float col = warp_colsum16(sq, lane);
      if ((lane & 1) == 0) s.red[grp][a][c][w4][lane >> 1] = col;
    }
    if (KIND == EPI_ACC) return;
    named_bar_sync(1 + grp, 128);
    {
      // thread -> (accumulator, chunk, column) of its group's tokens
      const int a = lr >> 6, c = (lr >> 4) & 3, j = lr & 15;
      const int tl = (grp + 2 * c) * kEpiCols + j, mt = row0 / kBM + a;
      if (tl < g.bn && t0 + tl < e.T && mt * kBM < g.M) {
        const float (&rd)[4][kEpiCols] = s.red[grp][a][c];
        e.ssq_out[static_cast<size_t>(mt) * e.ldt + t0 + tl] = ((rd[0][j] + rd[1][j]) + rd[2][j]) + rd[3][j];
      }
    }
  } else {  // EPI_ARGMAX
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int m = row0 + a * kBM + lr;
      const bool vrow = m < e.V;
      float (&v)[4][kEpiCols] = a == 0 ? v0 : v1;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int tl = (grp + 2 * c) * kEpiCols;
        if (tl >= g.bn) break;
#pragma unroll
        for (int j = 0; j < kEpiCols; ++j) {
          const int t = t0 + tl + j;
          const float lg = v[c][j] * s.rs[tl + j];
          if (e.logits != nullptr && vrow && tl + j < g.bn && t < e.T) e.logits[static_cast<size_t>(t) * e.V + m] = lg;
          v[c][j] = vrow ? lg : -INFINITY;
        }
        float o1, o2;
        int oi;
        warp_argmax16(v[c], m, lane, o1, oi, o2);
        if ((lane & 1) == 0) {
          float (&d)[3] = s.am[grp][a][c][w4][lane >> 1];
          d[0] = o1;
          d[1] = __int_as_float(oi);
          d[2] = o2;
        }
      }
    }
    named_bar_sync(1 + grp, 128);
    {
      const int a = lr >> 6, c = (lr >> 4) & 3, j = lr & 15;
      const int tl = (grp + 2 * c) * kEpiCols + j, mt = row0 / kBM + a;
      if (tl < g.bn && t0 + tl < e.T && mt < e.am_mtiles) {
        float b1 = s.am[grp][a][c][0][j][0], b2 = s.am[grp][a][c][0][j][2];
        int bi = __float_as_int(s.am[grp][a][c][0][j][1]);
        for (int w = 1; w < 4; ++w)
          am_merge(b1, bi, b2, s.am[grp][a][c][w][j][0], __float_as_int(s.am[grp][a][c][w][j][1]),
                   s.am[grp][a][c][w][j][2]);
        float* dst = e.am_part + (static_cast<size_t>(mt) * e.ldt + t0 + tl) * 3;
        dst[0] = b1;
        dst[1] = __int_as_float(bi);
        dst[2] = b2;
      }
    }
  }
}

__device__ __forceinline__ void part_add16_global(const float* part, int ch, int r, float (&v)[kEpiCols]) {
  const float4* p = reinterpret_cast<const float4*>(part) + static_cast<size_t>(ch) * 4 * kBM + r;
  float4 t[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) t[q] = __ldcg(p + q * kBM);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    v[4 * q] += t[q].x;
    v[4 * q + 1] += t[q].y;
    v[4 * q + 2] += t[q].z;
    v[4 * q + 3] += t[q].w;
  }
}

// A cluster's segments: its whole units, then its range of the remainder.
struct WideWork {
  int u, whole_end, clusters;  // next whole unit; end of the whole rounds
  int c, c1, cpc, kchunks;     // remainder chunks (unit whole_end + c / kchunks)
  __device__ WideWork(const GemmArgs& g, int cluster, int n_clusters) {
    const int units = g.mtiles * g.ntiles;
    kchunks = g.kchunks;
    cpc = g.cpc;
    clusters = n_clusters;
    whole_end = units / n_clusters * n_clusters;
    u = cluster;
    const int rest = (units - whole_end) * kchunks;
    c = min(rest, cluster * cpc);
    c1 = min(rest, c + cpc);
  }
  // chunks of all segments
  __device__ int chunks() const { return whole_end / clusters * kchunks + (c1 - c); }
  // first, last: contributing clusters of a remainder unit (first = last for a whole one)
  __device__ bool next(Segment& sg, int cluster, int& first, int& last) {
    if (u < whole_end) {
      sg = Segment{u, 0, kchunks};
      u += clusters;
      first = last = cluster;
      return true;
    }
    if (!next_segment(c, c1, kchunks, sg)) return false;
    first = (sg.unit * kchunks) / cpc;
    last = ((sg.unit + 1) * kchunks - 1) / cpc;
    sg.unit += whole_end;
    return true;
  }
};

template <int KIND>
__global__ void __launch_bounds__(kWThreads, 1)
    gemm_wide_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                     const __grid_constant__ CUtensorMap mA2, const __grid_constant__ CUtensorMap mB, const GemmArgs g,
                     const EpiArgs e) {
  extern __shared__ uint8_t smem_raw[];
  // (the same offset in every CTA of the cluster: dynamic shared memory starts alike)
  uint8_t* ring =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  WideSmem& s = *reinterpret_cast<WideSmem*>(ring + kWStages * kWStage);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t r = cluster_ctarank();  // CTA of the pair
  const bool leader = r == 0;
  const int cluster = blockIdx.x / 2;
  volatile int* abort = &s.abort_flag;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&mA0);
    tma_prefetch_desc(&mB);
    for (int i = 0; i < kWStages; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 1);
    }
    mbar_init(&s.tfull, 1);
    mbar_init(&s.tempty, 16);  // the 8 epilogue warps of both CTAs
    mbar_init(&s.drain, 1);
    s.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&s.tmem, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem = s.tmem;
  pdl_launch_dependents();

  WideWork work(g, cluster, gridDim.x / 2);
  const int n_chunks = work.chunks();
  const uint32_t cta_bytes = 2 * kWATile + static_cast<uint32_t>(g.bn) * kBK * 2;  // a chunk, one CTA
  Segment sg;
  int first, last;
  // first token and this CTA's first row of unit u (512 rows; GATEUP: 256 features)
  auto unit_tok = [&](int u) { return (u % g.ntiles) * g.bn; };
  auto unit_row = [&](int u) {
    const int ru = u / g.ntiles, half = static_cast<int>(r);
    return KIND == EPI_GATEUP ? ru * 256 + half * 128 : ru * 512 + half * 256;
  };

  if (warp < 4) {
    setmaxnreg_dec<kWRegsLow>();
    if (warp == 0 && lane == 0) {
      // Position of the next chunk to be loaded; a unit's coordinates are
      // worked out once (this one thread's divisions for every chunk took
      // longer than the chunk's MMAs: QKV at 2048 rows 323 instead of 257 us).
      struct Pos {
        WideWork w;
        Segment sg;
        int k, row0, tok;
        const CUtensorMap* m;  // QKV: the matrix that holds all of the CTA's rows (null: several do)
      };
      auto seek = [&](Pos& p) {
        int f, l;
        if (!p.w.next(p.sg, cluster, f, l)) return;
        p.k = p.sg.k0;
        p.row0 = unit_row(p.sg.unit);
        p.tok = unit_tok(p.sg.unit) + (r ? g.lo_rows : 0);
        if constexpr (KIND == EPI_QKV) {
          // (row0 becomes the row within that matrix)
          const int end = p.row0 + 2 * kBM;
          p.m = nullptr;
          if (end <= g.rows_q) {
            p.m = &mA0;
          } else if (p.row0 >= g.rows_qk) {
            p.m = &mA2;
            p.row0 -= g.rows_qk;
          } else if (p.row0 >= g.rows_q && end <= g.rows_qk) {
            p.m = &mA1;
            p.row0 -= g.rows_q;
          }
        }
      };
      auto advance = [&](Pos& p) {
        if (++p.k == p.sg.k1) seek(p);
      };
      const int half = e.hd >> 1;
      auto load_a = [&](const Pos& p, int st) {
        uint64_t* bar = &s.full[st];
        const int x = p.k * kBK;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          uint8_t* dst = ring + st * kWStage + a * kWATile;
          if constexpr (KIND == EPI_GATEUP) {
            const CUtensorMap* m = a == 0 ? &mA0 : &mA1;
            tma_load_2d_pair(dst, m, bar, x, p.row0);
            tma_load_2d_pair(dst + kWATile / 2, m, bar, x, p.row0 + 64);
          } else if constexpr (KIND == EPI_QKV) {
            // boxes of half a head: picking the matrix for every box took the
            // one thread longer than the chunk's MMAs (2048 rows 334 us)
            if (p.m != nullptr && half == 64) {
              tma_load_2d_pair(dst, p.m, bar, x, p.row0 + a * 64);
              tma_load_2d_pair(dst + 64 * kBK * 2, p.m, bar, x, p.row0 + 128 + a * 64);
              continue;
            }
            if (p.m != nullptr) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                tma_load_2d_pair(dst + j * 32 * kBK * 2, p.m, bar, x, p.row0 + j * 64 + a * 32);
              continue;
            }
            for (int i = 0, y = p.row0 + a * half; i < kBM; i += half, y += e.hd) {
              uint8_t* d = dst + i * kBK * 2;
              if (y < g.rows_q) tma_load_2d_pair(d, &mA0, bar, x, y);
              else if (y < g.rows_qk) tma_load_2d_pair(d, &mA1, bar, x, y - g.rows_q);
              else tma_load_2d_pair(d, &mA2, bar, x, y - g.rows_qk);  // (past V: the map's zero fill)
            }
          } else {
            tma_load_2d_pair(dst, &mA0, bar, x, p.row0 + a * kBM);
          }
        }
      };
      auto load_b = [&](const Pos& p, int st) {
        tma_load_2d_pair(ring + st * kWStage + 2 * kWATile, &mB, &s.full[st], p.k * kBK, p.tok);
      };
      // weights of the first stages do not depend on the previous kernel
      const int n = n_chunks, pre = min(n, kWStages);
      Pos pa{work, {}, 0, 0, 0, nullptr};
      seek(pa);
      Pos pb = pa;
      for (int j = 0; j < pre; ++j, advance(pa)) {
        if (leader) mbar_arrive_expect_tx(&s.full[j], 2 * cta_bytes);
        load_a(pa, j);
      }
      pdl_wait();
      for (int j = 0; j < pre; ++j, advance(pb)) load_b(pb, j);
      int j = pre;
      uint32_t ph = 0;  // parity of the use before this one
      for (int st = 0; j < n; ++j) {
        if (leader && g.hold == j + 1) break;  // test hook: as if the wait had run out
        if (!mbar_wait(&s.empty[st], ph, abort)) break;
        if (leader) mbar_arrive_expect_tx(&s.full[st], 2 * cta_bytes);
        load_a(pa, st);
        load_b(pa, st);
        advance(pa);
        if (++st == kWStages) {
          st = 0;
          ph ^= 1;
        }
      }
      // every load of the pair has landed (bounded) before the CTAs may leave
      s.issued = j;
      if (leader)
        for (int i = max(0, j - kWStages); i < j; ++i)
          mbar_wait(&s.full[i % kWStages], (i / kWStages) & 1, nullptr);
    }
    if (warp == 1 && lane == 0 && leader) {
      const uint32_t idesc = idesc_bf16_f32(256, 2 * g.bn);
      uint32_t accph = 0;
      int idx = 0;
      bool ok = true;
      while (ok && work.next(sg, cluster, first, last)) {
        if (!mbar_wait(&s.tempty, accph ^ 1, abort)) break;
        tc_fence_after();
        for (int k = sg.k0; k < sg.k1; ++k, ++idx) {
          const int st = idx % kWStages;
          if (!mbar_wait(&s.full[st], (idx / kWStages) & 1, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_addr = smem_u32(ring + st * kWStage), b_addr = a_addr + 2 * kWATile;
#pragma unroll
          for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              tc_mma_f16_pair(tmem + a * 256, sdesc_kmajor_sw128(a_addr + a * kWATile + kk * 32),
                              sdesc_kmajor_sw128(b_addr + kk * 32), idesc, (k > sg.k0 || kk > 0) ? 1u : 0u);
          tc_commit_pair(&s.empty[st], 3);
        }
        if (ok) tc_commit_pair(&s.tfull, 3);
        accph ^= 1;
      }
      // every issued MMA has completed (bounded)
      tc_commit_pair(&s.drain, 1);
      mbar_wait(&s.drain, 0, nullptr);
    }
  } else {
    setmaxnreg_inc<kWRegsEpi>();
    pdl_wait();
    const int et = threadIdx.x - 128;    // 0..255
    const int grp = et >> 7;             // token chunks grp, grp + 2, ...
    const int lr = (warp & 3) * 32 + lane;  // tensor-memory lane = row of a weight tile
    const uint32_t taddr = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint32_t tempty_leader = mapa_smem(&s.tempty, 0);
    auto joint = [&]() { named_bar_sync(3, 256); };
    uint32_t accph = 0;
    while (work.next(sg, cluster, first, last)) {
      const int t0 = unit_tok(sg.unit), row0 = unit_row(sg.unit);
      if (KIND != EPI_RESID && KIND != EPI_ACC) {
        // the unit's RMSNorm scales, positions and sequences, while its MMAs run
        const int tq = (et >> 3) * 4, part = et & 7;
        if ((et & ~31) / 2 < g.bn) {  // (a warp's 4 column quads; bn is a multiple of 16)
          const bool in = t0 + tq < e.T;
          float ss[4];
          epi_ssq_quad(e, in ? t0 + tq : 0, part, ss);
          if (part < 4)
            s.rs[tq + part] = t0 + tq + part < e.T
                                  ? rsqrtf((part == 0 ? ss[0] : part == 1 ? ss[1] : part == 2 ? ss[2] : ss[3]) * e.inv_d +
                                           e.eps)
                                  : 0.f;
        }
        if (KIND == EPI_QKV && et < g.bn) {
          s.pos[et] = t0 + et < e.T ? e.pos[t0 + et] : 0;
          s.bidx[et] = t0 + et < e.T ? e.bidx[t0 + et] : 0;
        }
      }
      if (et == 0) s.ok[0] = mbar_wait(&s.tfull, accph, abort) ? 1 : 0;
      joint();
      if (!s.ok[0]) break;
      accph ^= 1;
      tc_fence_after();
      float v0[4][kEpiCols], v1[4][kEpiCols];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int tl = (grp + 2 * q) * kEpiCols;
        if (tl < g.bn) {
          const uint32_t a = taddr + tl;
          tmem_ld16x4(a, a + g.bn, a + 256, a + 256 + g.bn, v0[q], v1[q]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(tempty_leader);  // the next unit's MMAs may start
      if (last > first) {
        // A cluster has at most two cut segments, one that begins its unit and
        // one that does not, with a partial slot each.
        int* ticket = &g.tickets[first * 2 + r];
        auto part_of = [&](int o) {
          return g.partial + (static_cast<size_t>(o * 2 + (o == first)) * 2 + r) * kWidePartFloats;
        };
        // The sums are added in range order.  The first two contributors may
        // add the others' to their registers (a + b = b + a); a later one starts
        // again from the partials, its own among them.
        const bool reload = cluster > first + 1;
        // (all the others' sums may be there already: no need to store)
        if (et == 0)
          s.ok[1] = !reload && static_cast<int>(ld_acquire_gpu(reinterpret_cast<unsigned*>(ticket))) == last - first;
        joint();
        if (!s.ok[1]) {
          float* part = part_of(cluster);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if ((grp + 2 * q) * kEpiCols < g.bn) {
              part_st16(part, grp + 2 * q, lr, v0[q]);
              part_st16(part, 8 + grp + 2 * q, lr, v1[q]);
            }
          }
          joint();  // every thread's stores precede the arrival
          if (et == 0) s.ok[1] = ticket_add(ticket, 1) == last - first;
          joint();
          if (!s.ok[1]) continue;
        }
        if (et == 0) *ticket = 0;
        if (reload) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int j = 0; j < kEpiCols; ++j) v0[q][j] = v1[q][j] = 0.f;
        }
        for (int o = first; o <= last; ++o) {
          if (o == cluster && !reload) continue;
          const float* part = part_of(o);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if ((grp + 2 * q) * kEpiCols < g.bn) {
              part_add16_global(part, grp + 2 * q, lr, v0[q]);
              part_add16_global(part, 8 + grp + 2 * q, lr, v1[q]);
            }
          }
        }
      }
      wide_apply<KIND>(e, g, row0, t0, lr, grp, v0, v1, s);
      joint();  // the tables are rewritten for the next unit
    }
  }
  // TMEM and barriers are shared by the pair: leave together
  __syncthreads();
  if (threadIdx.x == 0 && *abort) atomicOr(g.err, DERR_TIMEOUT);
  __syncwarp();
  tc_fence_before();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  if (threadIdx.x == 0 && leader && s.issued < n_chunks)
    pair_land_peer(s.full, kWStages, s.issued, mapa_smem(&s.issued, 1), cta_bytes);
  __syncwarp();
  if (warp == 1) tmem_dealloc_pair(tmem, 512);
  cluster_arrive();
  cluster_wait();
}

// Reduction of the LM head's per-tile maxima: 8 threads per token row.
__global__ void __launch_bounds__(128) argmax_reduce_kernel(const EpiArgs e) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * 16 + (threadIdx.x >> 3), part = threadIdx.x & 7;
  float v1 = -INFINITY, v2 = -INFINITY;
  int i1 = INT_MAX;
  if (t < e.T) {
#pragma unroll 8
    for (int mt = part; mt < e.am_mtiles; mt += 8) {
      const float* p = e.am_part + (static_cast<size_t>(mt) * e.ldt + t) * 3;
      am_merge(v1, i1, v2, p[0], __float_as_int(p[1]), p[2]);
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const float w1 = __shfl_xor_sync(0xffffffffu, v1, o);
    const int j1 = __shfl_xor_sync(0xffffffffu, i1, o);
    const float w2 = __shfl_xor_sync(0xffffffffu, v2, o);
    am_merge(v1, i1, v2, w1, j1, w2);
  }
  if (part == 0 && t < e.T) {
    e.pred[t] = i1;
    e.gap[t] = v1 - v2;
  }
}

// ---- launchers ----------------------------------------------------------------------

template <int KIND>
static cudaError_t wide_set_one() {
  return cudaFuncSetAttribute(gemm_wide_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(wide_smem_bytes()));
}

cudaError_t gemm_wide_set_attributes_acc() { return wide_set_one<EPI_ACC>(); }

cudaError_t gemm_wide_set_attributes() {
  cudaError_t err;
  if ((err = wide_set_one<EPI_QKV>()) != cudaSuccess) return err;
  if ((err = wide_set_one<EPI_GATEUP>()) != cudaSuccess) return err;
  if ((err = wide_set_one<EPI_RESID>()) != cudaSuccess) return err;
  return wide_set_one<EPI_ARGMAX>();
}

// Clusters that can be resident at once (0: none, or an error).
int gemm_wide_clusters() {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(2 * 64);
  cfg.blockDim = dim3(kWThreads);
  cfg.dynamicSmemBytes = wide_smem_bytes();
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, gemm_wide_kernel<EPI_ACC>, &cfg) == cudaSuccess ? n : 0;
}

WidePlan plan_wide(int kind, int M, int K, int T, int clusters, bool split) {
  WidePlan p{};
  p.row_units = ceil_div(M, kind == EPI_GATEUP ? 256 : 512);
  p.ntiles = ceil_div(T, kWideTokens);
  p.bn = round_up(ceil_div(T, p.ntiles), kEpiCols);
  p.kchunks = ceil_div(K, kBK);
  const int units = p.row_units * p.ntiles, rest = units % clusters;
  p.cpc = split ? std::max(1, ceil_div(rest * p.kchunks, clusters)) : p.kchunks;
  // (every cluster has a whole unit, or a part of the remainder)
  p.clusters = units >= clusters ? clusters : ceil_div(rest * p.kchunks, p.cpc);
  return p;
}

template <int KIND>
static cudaError_t launch_wide_one(const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int clusters,
                                   cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  cfg.gridDim = dim3(clusters * 2);
  cfg.blockDim = dim3(kWThreads);
  cfg.dynamicSmemBytes = wide_smem_bytes();
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, gemm_wide_kernel<KIND>, m.a0, m.a1, m.a2, m.b, g, e);
}

cudaError_t launch_gemm_wide(int kind, const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int clusters,
                             cudaStream_t s, bool pdl) {
  cudaError_t err;
  switch (kind) {
    case EPI_QKV: return launch_wide_one<EPI_QKV>(m, g, e, clusters, s, pdl);
    case EPI_GATEUP: return launch_wide_one<EPI_GATEUP>(m, g, e, clusters, s, pdl);
    case EPI_RESID: return launch_wide_one<EPI_RESID>(m, g, e, clusters, s, pdl);
    case EPI_ACC: return launch_wide_one<EPI_ACC>(m, g, e, clusters, s, pdl);
    case EPI_ARGMAX: break;
    default: return cudaErrorInvalidValue;
  }
  if ((err = launch_wide_one<EPI_ARGMAX>(m, g, e, clusters, s, pdl)) != cudaSuccess) return err;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((e.T + 15) / 16);
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, argmax_reduce_kernel, e);
}

}  // namespace cllm
