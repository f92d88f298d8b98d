// Weight GEMMs of the engine's launches of up to 256 token rows, on CTA pairs.
//
// From about 64 rows on the activations are the traffic: a CTA that multiplies one
// 128 x 64 weight tile (16 KB) by all tokens fetches 32 KB (128 tokens) to
// 64 KB (256 tokens) of hi and lo activation planes with it, for every weight
// tile, and the launch runs at the L2's bandwidth.  The engine's work split
// keeps neighbouring CTAs on the same K range (groups of 4 tiles), so the two
// CTAs of a pair multiply their own weight tiles by the same activations in
// one tcgen05 cta_group::2 MMA (M = 256) and each holds only half of them:
// 32 instead of 48 KB per chunk at 128 tokens, 48 instead of 80 KB at 256.
//
// Work split, reductions and epilogues are those of the single-CTA kernels
// (gemm_roles.cuh): every output element is the same sums in the same order,
// so a token's bits do not depend on which kernel the launch's width selects.
#define CLLM_EPI_GROUPS 1
#include <algorithm>

#include "act.cuh"
#include "epilogue.cuh"
#include "gemm_roles.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace cllm {

// BNMAX 128: the pair's B operand is [hi rows | lo rows], one plane in each
// CTA, one MMA with N = 2 bn, two accumulators.  BNMAX 256: each CTA holds the
// same half of the tokens of both planes, two MMAs with N = bn, one accumulator.
template <int BNMAX>
struct PairCfg {
  static constexpr int STAGES = BNMAX == 128 ? 6 : 4;
  static constexpr int A_BYTES = kBM * kBK * 2;
  static constexpr int B_BYTES = (BNMAX == 128 ? 128 : 256) * kBK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr bool STACKED = BNMAX == 128;
  static constexpr int ACC_COLS = 2 * BNMAX;
  static constexpr int NACC = BNMAX == 128 ? 2 : 1;
  static constexpr int BN = BNMAX;
};

constexpr int kPairThreads = 64 + 256;
constexpr size_t kPairGroupBytes = (sizeof(EpiSmem) + 15) / 16 * 16;

template <int BNMAX>
constexpr size_t pair_smem_bytes() {
  return 1024 + static_cast<size_t>(PairCfg<BNMAX>::STAGES) * PairCfg<BNMAX>::STAGE_BYTES + 2 * kPairGroupBytes +
         tc_bar_bytes(PairCfg<BNMAX>::STAGES) + 2 * kPartRounds * 8 + 32;
}
static_assert(2 * kPartRounds * 4 * kPartChunkBytes <= PairCfg<128>::STAGES * PairCfg<128>::STAGE_BYTES &&
                  2 * kPartRounds * 4 * kPartChunkBytes <= PairCfg<256>::STAGES * PairCfg<256>::STAGE_BYTES,
              "partials' buffers fit the ring");
static_assert(pair_smem_bytes<128>() <= 227 * 1024 && pair_smem_bytes<256>() <= 227 * 1024, "pair GEMM shared memory");

template <int KIND, int BNMAX>
__global__ void __launch_bounds__(kPairThreads, 1)
    gemm_pair_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                     const __grid_constant__ CUtensorMap mA2, const __grid_constant__ CUtensorMap mB, const GemmArgs g,
                     const EpiArgs e) {
  using Cfg = PairCfg<BNMAX>;
  constexpr int S = Cfg::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* groups = ring + S * Cfg::STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(groups + 2 * kPairGroupBytes);
  TcPipe P{};
  P.full = bars;
  P.empty = bars + S;
  P.tfull = bars + 2 * S;
  P.tempty = P.tfull + 2;
  P.drain = P.tempty + 2;
  P.part_bar = P.drain + 1;
  P.ring_free = ring;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(P.part_bar + 2 * kPartRounds);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  P.abort = abort_flag;
  P.jflag = abort_flag + 1;
  int* issued = abort_flag + 2;  // chunks this CTA's producer has loaded
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t r = cluster_ctarank();
  const bool leader = r == 0;
  const int cta = blockIdx.x;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&mA0);
    tma_prefetch_desc(&mB);
    for (int i = 0; i < S; ++i) {
      mbar_init(&P.full[i], 1);
      mbar_init(&P.empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&P.tfull[i], 1);
      mbar_init(&P.tempty[i], 16);  // the 8 epilogue warps of both CTAs
    }
    mbar_init(P.drain, 1);
    for (int i = 0; i < 2 * kPartRounds; ++i) mbar_init(&P.part_bar[i], 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  P.tmem = *tmem_slot;
  pdl_launch_dependents();

  // both CTAs run over the even tile's range; a pair at the end of the rows may
  // have no odd tile (its loads are zero fill, its epilogue stores nothing)
  int c0, c1;
  cta_range(g, cta & ~1, c0, c1);
  const uint32_t b_rows = static_cast<uint32_t>(Cfg::STACKED ? g.bn : g.bn / 2);
  const uint32_t cta_bytes = Cfg::A_BYTES + (Cfg::STACKED ? 1u : 2u) * b_rows * kBK * 2;  // a chunk, one CTA

  if (warp == 0) {
    if (lane == 0) {
      int u = c0 / g.kchunks, ka = c0 - u * g.kchunks, kb = ka, mt = tile_of(g, u, cta);
      auto load_a = [&](int st) {
        uint8_t* dst = ring + st * Cfg::STAGE_BYTES;
        uint64_t* bar = &P.full[st];
        const int x = ka * kBK;
        if constexpr (KIND == EPI_GATEUP) {
          tma_load_2d_pair(dst, &mA0, bar, x, mt * 64);
          tma_load_2d_pair(dst + Cfg::A_BYTES / 2, &mA1, bar, x, mt * 64);
        } else if constexpr (KIND == EPI_QKV) {
          const int row = mt * kBM;
          if (row < g.rows_q) tma_load_2d_pair(dst, &mA0, bar, x, row);
          else if (row < g.rows_qk) tma_load_2d_pair(dst, &mA1, bar, x, row - g.rows_q);
          else tma_load_2d_pair(dst, &mA2, bar, x, row - g.rows_qk);
        } else {
          tma_load_2d_pair(dst, &mA0, bar, x, mt * kBM);
        }
        if (++ka == g.kchunks) {
          ka = 0;
          mt += 1 << g.gshift;
        }
      };
      auto load_b = [&](int st) {
        uint8_t* dst = ring + st * Cfg::STAGE_BYTES + Cfg::A_BYTES;
        uint64_t* bar = &P.full[st];
        const int x = kb * kBK;
        if constexpr (Cfg::STACKED) {
          tma_load_2d_pair(dst, &mB, bar, x, r ? g.lo_rows : 0);
        } else {
          const int y = static_cast<int>(r * b_rows);
          tma_load_2d_pair(dst, &mB, bar, x, y);
          tma_load_2d_pair(dst + Cfg::B_BYTES / 2, &mB, bar, x, g.lo_rows + y);
        }
        if (++kb == g.kchunks) kb = 0;
      };
      // weights of the first stages do not depend on the previous kernel
      const int n = c1 - c0, pre = min(n, S);
      for (int j = 0; j < pre; ++j) {
        if (leader) mbar_arrive_expect_tx(&P.full[j], 2 * cta_bytes);
        load_a(j);
      }
      pdl_wait();
      for (int j = 0; j < pre; ++j) load_b(j);
      int j = pre;
      uint32_t ph = 0;
      for (int st = 0; j < n; ++j) {
        if (leader && g.hold == j + 1) break;  // test hook: as if the wait had run out
        if (!mbar_wait(&P.empty[st], ph, P.abort)) break;
        if (leader) mbar_arrive_expect_tx(&P.full[st], 2 * cta_bytes);
        load_a(st);
        load_b(st);
        if (++st == S) {
          st = 0;
          ph ^= 1;
        }
      }
      // every load of the pair has landed (bounded) before the CTAs may leave
      *issued = j;
      if (leader)
        for (int i = max(0, j - S); i < j; ++i) mbar_wait(&P.full[i % S], (i / S) & 1, nullptr);
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      const uint32_t idesc = idesc_bf16_f32(256, Cfg::STACKED ? 2 * g.bn : g.bn);
      int acc = 0, st = 0, c = c0;
      uint32_t accph = 0, ph = 0;
      Segment sg;
      bool ok = true;
      while (ok && next_segment(c, c1, g.kchunks, sg)) {
        if (!mbar_wait(&P.tempty[acc], accph ^ 1, P.abort)) break;
        tc_fence_after();
        const uint32_t dt = P.tmem + static_cast<uint32_t>(acc * Cfg::ACC_COLS);
        for (int k = sg.k0; k < sg.k1; ++k) {
          if (!mbar_wait(&P.full[st], ph, P.abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_addr = smem_u32(ring + st * Cfg::STAGE_BYTES), b_addr = a_addr + Cfg::A_BYTES;
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            const uint64_t ad = sdesc_kmajor_sw128(a_addr + kk * 32);
            const uint32_t accum = (k > sg.k0 || kk > 0) ? 1u : 0u;
            tc_mma_f16_pair(dt, ad, sdesc_kmajor_sw128(b_addr + kk * 32), idesc, accum);
            if constexpr (!Cfg::STACKED)
              tc_mma_f16_pair(dt + Cfg::BN, ad, sdesc_kmajor_sw128(b_addr + Cfg::B_BYTES / 2 + kk * 32), idesc, accum);
          }
          tc_commit_pair(&P.empty[st], 3);
          if (++st == S) {
            st = 0;
            ph ^= 1;
          }
        }
        if (ok) tc_commit_pair(&P.tfull[acc], 3);
        if (++acc == Cfg::NACC) {
          acc = 0;
          accph ^= 1;
        }
      }
      // every issued MMA has completed (bounded)
      tc_commit_pair(P.drain, 1);
      mbar_wait(P.drain, 0, nullptr);
    }
  } else {
    pdl_wait();
    uint8_t* mine = groups + ((warp - 2) / 4) * kPairGroupBytes;
    EpiSmem& es = *reinterpret_cast<EpiSmem*>(mine);
    P.tempty_leader = mapa_smem(P.tempty, 0);
    int acc = 0;
    uint32_t accph = 0;
    tc_epilogue<KIND, Cfg, 2, true>(P, acc, accph, g, e, c0, c1, cta, es);
  }
  // TMEM and barriers are shared by the pair: leave together
  __syncthreads();
  if (threadIdx.x == 0 && *P.abort) atomicOr(g.err, DERR_TIMEOUT);
  __syncwarp();
  tc_fence_before();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  if (threadIdx.x == 0 && leader && *issued < c1 - c0)
    pair_land_peer(P.full, S, *issued, mapa_smem(issued, 1), cta_bytes);
  __syncwarp();
  if (warp == 1) tmem_dealloc_pair(P.tmem, 512);
  cluster_arrive();
  cluster_wait();
}

// ---- launchers ----------------------------------------------------------------------

template <int KIND>
static cudaError_t pair_set_kind() {
  const cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<KIND, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(pair_smem_bytes<128>()));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(gemm_pair_kernel<KIND, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(pair_smem_bytes<256>()));
}

cudaError_t gemm_pair_set_attributes() {
  cudaError_t err;
  if ((err = pair_set_kind<EPI_QKV>()) != cudaSuccess) return err;
  if ((err = pair_set_kind<EPI_GATEUP>()) != cudaSuccess) return err;
  if ((err = pair_set_kind<EPI_RESID>()) != cudaSuccess) return err;
  return pair_set_kind<EPI_ARGMAX>();
}

template <int BN>
static int pair_clusters() {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(2 * 64);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = pair_smem_bytes<BN>();
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, gemm_pair_kernel<EPI_QKV, BN>, &cfg) == cudaSuccess ? n : 0;
}

int gemm_pair_clusters() { return std::min(pair_clusters<128>(), pair_clusters<256>()); }

template <int KIND, int BN>
static cudaError_t launch_pair_one(const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int grid, cudaStream_t s,
                                   bool pdl) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = pair_smem_bytes<BN>();
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, gemm_pair_kernel<KIND, BN>, m.a0, m.a1, m.a2, m.b, g, e);
}

template <int KIND>
static cudaError_t launch_pair_kind(const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int grid, cudaStream_t s,
                                    bool pdl) {
  return g.bn <= 128 ? launch_pair_one<KIND, 128>(m, g, e, grid, s, pdl)
                     : launch_pair_one<KIND, 256>(m, g, e, grid, s, pdl);
}

cudaError_t launch_gemm_pair(int kind, const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int grid, cudaStream_t s,
                             bool pdl) {
  switch (kind) {
    case EPI_QKV: return launch_pair_kind<EPI_QKV>(m, g, e, grid, s, pdl);
    case EPI_GATEUP: return launch_pair_kind<EPI_GATEUP>(m, g, e, grid, s, pdl);
    case EPI_RESID: return launch_pair_kind<EPI_RESID>(m, g, e, grid, s, pdl);
    case EPI_ARGMAX: return launch_pair_kind<EPI_ARGMAX>(m, g, e, grid, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace cllm
