// The weight-streaming GEMM on its own (the allocation-free entry point up to 256
// tokens; the engine's launches run on CTA pairs, gemm_pair.cu and gemm_wide.cu,
// or inside the persistent kernel).  Y[t][m] += D[m][t]: the residual add alone.
//
//   D[m][t] = sum_k W[m][k] * X[t][k]      (W: [M][K] weights, X: [T][K] activations)
//
// At small token counts every weight byte is used T times, so the GEMM is
// bound by streaming W from HBM.  The kernel is "swap-AB": the weight tile is
// the MMA's A operand (M = 128 rows), the tokens are its N (16..256 columns),
// and the fp32 accumulator lives in tensor memory (TMEM).  A producer warp
// streams W and X tiles with TMA into a ring of shared-memory stages, one
// thread issues tcgen05.mma, and four epilogue warps read TMEM.  The grid is
// one CTA per SM; the (tile, k-chunk) space is cut into equal contiguous
// ranges, and a tile whose K range is split over several CTAs is reduced by
// its first contributor in a fixed order.  The partition depends only on the
// weight shape and SM count, never on T, so a token's result does not depend
// on how many rows share the launch.
#include <float.h>
#include <limits.h>

#define CLLM_EPI_GROUPS 1  // kernels of this unit may run two epilogue groups
#include "act.cuh"
#include "epilogue.cuh"
#include "gemm_roles.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace cllm {

// ---------------------------------------------------------------------------------
// tcgen05 kernel (bf16): one GEMM per launch
// ---------------------------------------------------------------------------------

// One CTA per SM with as many stages as fit: the weight stream is
// latency-bound by the bytes in flight per SM (~45 GB/s per SM at ~1.8 us
// loaded DRAM latency needs > 80 KB in flight).
template <int BNMAX>
using SoloCfg = TcCfg<BNMAX, BNMAX <= 32 ? 8 : (BNMAX <= 64 ? 6 : (BNMAX <= 128 ? 4 : 2))>;

constexpr int kSoloRedSlots = 2;  // split-K partial blocks staged per reduction round

// Epilogue groups: at 256 token columns one accumulator fills tensor memory,
// so the MMAs of a CTA's next unit wait for the whole epilogue of the last
// one (16 chunks); a second group of 4 warps halves that wait.
template <int BNMAX>
constexpr int solo_groups() { return BNMAX == 256 ? 2 : 1; }

constexpr size_t kSoloGroupBytes = (sizeof(EpiSmem) + 15) / 16 * 16 + kSoloRedSlots * kRedSlotBytes;

template <int BNMAX>
constexpr size_t solo_smem_bytes() {
  using Cfg = SoloCfg<BNMAX>;
  return 1024 + static_cast<size_t>(Cfg::STAGES) * Cfg::STAGE_BYTES + solo_groups<BNMAX>() * kSoloGroupBytes + 16 +
         tc_bar_bytes(Cfg::STAGES) + 16;
}
constexpr size_t kSmemLimit = 227 * 1024 - 256;  // minus static shared memory
static_assert(solo_smem_bytes<32>() <= kSmemLimit && solo_smem_bytes<64>() <= kSmemLimit &&
                  solo_smem_bytes<128>() <= kSmemLimit && solo_smem_bytes<256>() <= kSmemLimit,
              "per-GEMM kernel shared memory over the 227 KB limit");

template <int BNMAX>
__global__ void __launch_bounds__(64 + 128 * solo_groups<BNMAX>(), 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, const GemmArgs g,
                   const EpiArgs e) {
  using Cfg = SoloCfg<BNMAX>;
  constexpr int NG = solo_groups<BNMAX>();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // [ring][per group: EpiSmem, staging slots][barriers][shared flags, 16 bytes]
  uint8_t* groups = base + Cfg::STAGES * Cfg::STAGE_BYTES;
  uint8_t* bars = groups + NG * kSoloGroupBytes;
  int* jflag = reinterpret_cast<int*>(bars + tc_bar_bytes(Cfg::STAGES));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&mA);
    tma_prefetch_desc(&mB);
  }
  TcPipe P = tc_pipe_init<Cfg, NG>(base, bars);
  P.red_slots = kSoloRedSlots;
  P.jflag = jflag;
  // Every CTA of this grid is resident (one per SM): let the next kernel in
  // the stream start its independent prologue now.
  pdl_launch_dependents();
  int c0, c1;
  cta_range(g, blockIdx.x, c0, c1);
  if (warp == 0) {
    if (lane == 0) {
      tc_produce_drain<Cfg>(P, tc_produce<Cfg>(P, g, &mA, &mB, c0, c1, blockIdx.x));
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int idx = 0, acc = 0;
      uint32_t accph = 0;
      tc_mma<Cfg>(P, idx, acc, accph, g, c0, c1);
      tc_mma_drain(P);
    }
  } else {
    pdl_wait();
    const int gi = (warp - 2) / 4;  // epilogue group
    uint8_t* mine = groups + gi * kSoloGroupBytes;
    EpiSmem& es = *reinterpret_cast<EpiSmem*>(mine);
    TcPipe Pg = P;
    Pg.red = reinterpret_cast<float*>(mine + (sizeof(EpiSmem) + 15) / 16 * 16);
    int acc = 0;
    uint32_t accph = 0;
    tc_epilogue<EPI_ACC, Cfg, NG>(Pg, acc, accph, g, e, c0, c1, blockIdx.x, es);
  }
  tc_pipe_release<Cfg>(P);
  if (threadIdx.x == 0 && *P.abort) atomicOr(g.err, DERR_TIMEOUT);
}

// ---------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------

template <int BN>
static cudaError_t set_attr_one() {
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<BN>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(solo_smem_bytes<BN>()));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(gemm_tc_kernel<BN>,
                              cudaFuncAttributePreferredSharedMemoryCarveout,
                              static_cast<int>(cudaSharedmemCarveoutMaxShared));
}

cudaError_t gemm_tc_set_attributes(int bn_max) {
  switch (bn_max) {
    case 32: return set_attr_one<32>();
    case 64: return set_attr_one<64>();
    case 128: return set_attr_one<128>();
    default: return set_attr_one<256>();
  }
}

static void fill_launch(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, dim3 grid, dim3 block,
                        size_t smem, cudaStream_t s, bool pdl) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

template <int BN>
static cudaError_t launch_tc_one(const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int grid,
                                 cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  fill_launch(cfg, attr, dim3(grid), dim3(64 + 128 * solo_groups<BN>()), solo_smem_bytes<BN>(), s, pdl);
  return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<BN>, m.a0, m.b, g, e);
}

cudaError_t launch_gemm_tc(int bn_max, const GemmMaps& m, const GemmArgs& g, const EpiArgs& e, int grid,
                           cudaStream_t s, bool pdl) {
  switch (bn_max) {
    case 32: return launch_tc_one<32>(m, g, e, grid, s, pdl);
    case 64: return launch_tc_one<64>(m, g, e, grid, s, pdl);
    case 128: return launch_tc_one<128>(m, g, e, grid, s, pdl);
    case 256: return launch_tc_one<256>(m, g, e, grid, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace cllm
