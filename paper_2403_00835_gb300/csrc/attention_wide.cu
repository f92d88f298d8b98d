// Block attention of launches with many rows per sequence (prefill, wide
// blocks): O = softmax(Q K^T / sqrt(hd)) V with a causal mask, on tcgen05.
//
// The 16-row tiles of attn_item.cuh re-read K and V from L2 for every 16 query
// rows and run on mma.sync; with 2048 rows and 4096 keys that took 0.7 ms of a
// layer.  Here a CTA owns 256 query rows of one head as two tiles of 128, so
// 64 KB of K and V (128 keys) serve 256 rows, and the two tiles hide each
// other's latency: while one tile's softmax runs on its 4 warps, the tensor
// cores work on the other.  Per tile and 128-key chunk: S = Q K^T into tensor
// memory (128 columns), a thread per row turns its 128 scores into fp16
// probabilities written back over S, and P V accumulates with P read from
// tensor memory (A operand) and V from shared memory (MN-major B operand).
// The output accumulator is rescaled when a row's running maximum has grown,
// which a warp votes on, so chunks after the first few rarely pay for it.  One thread issues every TMA load and MMA:
// the order of its waits also tells it when a K or V buffer is free.
//
// Compute: 2 x 128 x 128 x hd x 2 FLOP per tile and chunk, 0.26 us per MMA
// group at the dense rate; the softmax's 16384 exponentials of a tile take
// 0.5 us of the SM's special-function units, so the two are balanced.
// 4096-token prefill, mean of its two 2048-row launches: 444 us and 45 us of
// merging -> 109 us.
#include <float.h>

#include "act.cuh"
#include "attn_item.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace cllm {

// Warps 0-3 and 4-7: the tiles' softmax; warp 8 issues (9-11 idle).  Of the
// launch's 384 x 168 registers the last warpgroup keeps 56 a thread, the
// softmax warps take 224 (a row's 128 scores are held at once).
constexpr int kWAttnThreads = 256 + 128;
constexpr int kWAttnRegsLow = 56, kWAttnRegsRow = 224;
static_assert(128 * kWAttnRegsLow + 256 * kWAttnRegsRow <= kWAttnThreads * 168, "register split");
constexpr int kWQ = 128;                 // query rows per tile

template <int HD>
struct WideAttnSmem {
  alignas(1024) uint8_t q[2][kWQ * HD * 2];
  alignas(1024) uint8_t k[2][kAttnChunk * HD * 2];
  alignas(1024) uint8_t v[2][kAttnChunk * HD * 2];
  uint64_t qfull, kfull[2], vfull[2], sfull[2], pready[2], ofull[2], drain;
  uint32_t tmem;
  int abort_flag;
};

template <int HD>
constexpr size_t wide_attn_smem() { return sizeof(WideAttnSmem<HD>) + 1024; }
static_assert(wide_attn_smem<128>() <= 227 * 1024, "wide attention shared memory");

template <int HD>
__global__ void __launch_bounds__(kWAttnThreads, 1)
    attn_wide_kernel(const __grid_constant__ AttnMaps m, const AttnArgs a, int kv_row0) {
  extern __shared__ uint8_t smem_raw[];
  WideAttnSmem<HD>& s = *reinterpret_cast<WideAttnSmem<HD>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                             ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &s.abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&s.qfull, 1);
    mbar_init(&s.drain, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s.kfull[i], 1);
      mbar_init(&s.vfull[i], 1);
      mbar_init(&s.sfull[i], 1);
      mbar_init(&s.pready[i], 4);
      mbar_init(&s.ofull[i], 1);
    }
    s.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 8) {
    tmem_alloc(&s.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s.tmem;
  pdl_launch_dependents();
  pdl_wait();

  const int tile = blockIdx.x / a.H, h = blockIdx.x - tile * a.H;
  const int2 qt = a.qtiles[tile];
  const int b = qt.x, r0 = qt.y;
  const int nr = min(2 * kWQ, a.seq_nrows[b] - r0);
  const int pos0 = a.seq_start[b] + r0;
  const int row_g0 = a.seq_row0[b] + r0;
  if (pos0 + nr > a.max_seq && threadIdx.x == 0) atomicOr(a.err, DERR_CAPACITY);
  // rows and 128-key chunks of each tile (a tile's last row sees the most keys)
  auto tile_rows = [&](int t) { return min(max(nr - t * kWQ, 0), kWQ); };
  auto tile_chunks = [&](int t) {
    const int rows = tile_rows(t);
    return rows > 0 ? min((pos0 + t * kWQ + rows - 1) / kAttnChunk + 1, a.nch_max) : 0;
  };
  const int n0 = tile_chunks(0), n1 = tile_chunks(1), n = max(n0, n1);

  if (warp >= 8) {
    setmaxnreg_dec<kWAttnRegsLow>();
    if (warp == 8 && lane == 0 && n > 0) {
      const int kvrow = kv_row0 + (b * a.Hkv + h / (a.H / a.Hkv)) * a.max_seq;
      constexpr int NH = HD / 64;  // 64-column halves
      auto load_k = [&](int c) {
        uint64_t* bar = &s.kfull[c & 1];
        mbar_arrive_expect_tx(bar, NH * kAttnChunk * 128);
        for (int i = 0; i < NH; ++i)
          tma_load_2d_nohint(s.k[c & 1] + i * kAttnChunk * 128, &m.k, bar, i * 64, kvrow + c * kAttnChunk);
      };
      auto load_v = [&](int c) {
        uint64_t* bar = &s.vfull[c & 1];
        mbar_arrive_expect_tx(bar, NH * kAttnChunk * 128);
        for (int i = 0; i < NH; ++i)
          tma_load_2d_nohint(s.v[c & 1] + i * kAttnChunk * 128, &m.v, bar, i * 64, kvrow + c * kAttnChunk);
      };
      const int ntile = n1 > 0 ? 2 : 1;
      mbar_arrive_expect_tx(&s.qfull, ntile * NH * kWQ * 128);
      for (int t = 0; t < ntile; ++t)
        for (int i = 0; i < NH; ++i)
          tma_load_2d_nohint(s.q[t] + i * kWQ * 128, &m.qw, &s.qfull, h * HD + i * 64, row_g0 + t * kWQ);
      load_k(0);
      load_v(0);
      int loads_k = 1, loads_v = 1;
      if (n > 1) {
        load_k(1);
        load_v(1);
        loads_k = loads_v = 2;
      }
      constexpr uint32_t id_s = idesc_f16_f32(kWQ, kAttnChunk, false);
      constexpr uint32_t id_o = idesc_f16_f32(kWQ, HD, true);
      auto mma_s = [&](int t, int c) {
        const uint32_t qa = smem_u32(s.q[t]), ka = smem_u32(s.k[c & 1]);
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk) {
          const uint32_t off = (kk >> 2) * kWQ * 128 + (kk & 3) * 32;
          tc_mma_f16(tmem + t * 256, sdesc_kmajor_sw128(qa + off), sdesc_kmajor_sw128(ka + off), id_s, kk > 0);
        }
        tc_commit(&s.sfull[t]);
      };
      auto mma_o = [&](int t, int c) {
        const uint32_t va = smem_u32(s.v[c & 1]);
#pragma unroll
        for (int kk = 0; kk < kAttnChunk / 16; ++kk)
          tc_mma_f16_ts(tmem + t * 256 + 128, tmem + t * 256 + kk * 8,
                        sdesc_mnmajor_sw128(va + kk * 16 * 128, kAttnChunk * 128), id_o, c > 0 || kk > 0);
      };
      bool ok = mbar_wait(&s.qfull, 0, abort) && mbar_wait(&s.kfull[0], 0, abort);
      if (ok) {
        tc_fence_after();
        if (n0 > 0) mma_s(0, 0);
        if (n1 > 0) mma_s(1, 0);
      }
      for (int c = 0; ok && c < n; ++c) {
        const int nt[2] = {n0, n1};
        if (a.hold == c + 1) {  // test hook: as if this thread's wait had run out
          ok = false;
          break;
        }
        ok = mbar_wait(&s.vfull[c & 1], (c >> 1) & 1, abort);
        if (ok && c + 1 < n) ok = mbar_wait(&s.kfull[(c + 1) & 1], ((c + 1) >> 1) & 1, abort);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (!ok || c >= nt[t]) continue;
          ok = mbar_wait(&s.pready[t], c & 1, abort);
          if (!ok) break;
          tc_fence_after();
          mma_o(t, c);
          if (c + 1 < nt[t]) mma_s(t, c + 1);
          else tc_commit(&s.ofull[t]);
          // every S of chunk c is done (its P was ready), and so is every
          // P V of chunk c - 1 (issued before those S): their buffers are free
          if (t == 1 || c >= n1) {
            if (c + 2 < n) {
              load_k(c + 2);
              ++loads_k;
            }
            if (c >= 1 && c + 1 < n) {
              load_v(c + 1);
              ++loads_v;
            }
          }
        }
      }
      if (!ok) {
        // MMAs and loads in flight end (bounded) before the CTA leaves (otherwise
        // the tiles' last commits, which the softmax warps wait for, cover them)
        tc_commit(&s.drain);
        mbar_wait(&s.drain, 0, nullptr);
        mbar_wait(&s.qfull, 0, nullptr);
        for (int c = max(0, loads_k - 2); c < loads_k; ++c) mbar_wait(&s.kfull[c & 1], (c >> 1) & 1, nullptr);
        for (int c = max(0, loads_v - 2); c < loads_v; ++c) mbar_wait(&s.vfull[c & 1], (c >> 1) & 1, nullptr);
      }
    }
  } else {
    setmaxnreg_inc<kWAttnRegsRow>();
    const int t = warp >> 2;
    const int row = (warp & 3) * 32 + lane;
    const int nt = t == 0 ? n0 : n1;
    const int p_row = pos0 + t * kWQ + row;  // this row's position: it sees keys 0..p_row
    const int p_first = pos0 + t * kWQ;
    const uint32_t ts = tmem + t * 256 + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    // (one lane waits for its warp: lanes that gave up on their own would leave
    // the others at a warp-wide operation)
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) {
      int got = 0;
      if (lane == 0) got = mbar_wait(bar, parity, abort) ? 1 : 0;
      got = __shfl_sync(0xffffffffu, got, 0);
      __syncwarp();
      return got != 0;
    };
    float mx = -INFINITY, l = 0.f;
    bool ok = true;
    for (int c = 0; c < nt; ++c) {
      if (!warp_wait(&s.sfull[t], c & 1)) {
        ok = false;
        break;
      }
      tc_fence_after();
      float x0[64], x1[64];
      tmem_ld64(ts, x0);
      tmem_ld64(ts + 64, x1);
      const int kb = c * kAttnChunk;
      if (kb + kAttnChunk - 1 > p_first) {  // some row of the tile does not see every key
#pragma unroll
        for (int i = 0; i < 64; ++i) {
          if (kb + i > p_row) x0[i] = -INFINITY;
          if (kb + 64 + i > p_row) x1[i] = -INFINITY;
        }
      }
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < 64; i += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) m4[u] = fmaxf(m4[u], fmaxf(x0[i + u], x1[i + u]));
      const float cm = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * a.scale_log2;
      // (chunk 0 holds position 0, which every row sees)
      const bool grow = cm > mx;
      if (c == 0) {
        mx = cm;
      } else if (__any_sync(0xffffffffu, grow)) {
        const float nm = grow ? cm : mx;
        const float f = grow ? ex2_ftz(mx - nm) : 1.f;
        l *= f;
        mx = nm;
#pragma unroll 1
        for (int d = 0; d < HD; d += 64) {
          float o[64];
          tmem_ld64(ts + 128 + d, o);
          uint32_t r[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(o[i] * f);
          tmem_st32(ts + 128 + d, r);
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(o[32 + i] * f);
          tmem_st32(ts + 128 + d + 32, r);
        }
      }
      const float nm = mx == -INFINITY ? 0.f : -mx;
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t pk[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float p0 = ex2_ftz(fmaf(x0[2 * i], a.scale_log2, nm)), p1 = ex2_ftz(fmaf(x0[2 * i + 1], a.scale_log2, nm));
        sum[i & 3] += p0 + p1;
        pk[i] = pack_f16x2(p0, p1);
      }
      tmem_st32(ts, pk);
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float p0 = ex2_ftz(fmaf(x1[2 * i], a.scale_log2, nm)), p1 = ex2_ftz(fmaf(x1[2 * i + 1], a.scale_log2, nm));
        sum[i & 3] += p0 + p1;
        pk[i] = pack_f16x2(p0, p1);
      }
      tmem_st32(ts + 32, pk);
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.pready[t]);
    }
    if (ok && nt > 0) {
      ok = warp_wait(&s.ofull[t], 0);
      tc_fence_after();
      const bool live = ok && row < tile_rows(t);
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(a.out) +
                           (static_cast<size_t>(row_g0 + t * kWQ + row) * a.H + h) * HD;
#pragma unroll 1
      for (int d = 0; d < HD; d += 64) {
        float o[64];
        tmem_ld64(ts + 128 + d, o);
        if (live) {
#pragma unroll
          for (int i = 0; i < 64; i += 4)
            st_gin4(out, d + i, a.plane_out, make_float4(o[i] / l, o[i + 1] / l, o[i + 2] / l, o[i + 3] / l));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort) atomicOr(a.err, DERR_TIMEOUT);
  if (warp == 8) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---- launchers ----------------------------------------------------------------------

cudaError_t attention_wide_set_attributes() {
  const cudaError_t e = cudaFuncSetAttribute(attn_wide_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(wide_attn_smem<64>()));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(attn_wide_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(wide_attn_smem<128>()));
}

cudaError_t launch_attention_wide(const AttnArgs& a, const AttnMaps& m, int kv_row0, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(a.n_qtiles * a.H);
  cfg.blockDim = dim3(kWAttnThreads);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (a.hd == 64) {
    cfg.dynamicSmemBytes = wide_attn_smem<64>();
    return cudaLaunchKernelEx(&cfg, attn_wide_kernel<64>, m, a, kv_row0);
  }
  if (a.hd == 128) {
    cfg.dynamicSmemBytes = wide_attn_smem<128>();
    return cudaLaunchKernelEx(&cfg, attn_wide_kernel<128>, m, a, kv_row0);
  }
  return cudaErrorInvalidValue;
}

}  // namespace cllm
