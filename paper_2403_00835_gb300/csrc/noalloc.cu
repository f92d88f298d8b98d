// Allocation-free variant of the weight-streaming GEMM (cllm_gemm_bf16_noalloc).
//
// Some callers cannot call cudaMalloc: code running under a caching allocator
// that has reserved the device's memory for itself, or a latency-critical
// path where the implicit device synchronisation of cudaMalloc/cudaFree is
// not acceptable.  This entry point runs the same tcgen05/TMA GEMM kernel as
// the rest of the library, but every byte of scratch it needs (split-K
// partial tiles, arrival tickets and the device error word) lives in one
// file-scope device array of fixed size, so the call allocates nothing.  The caller still provides the inputs and output.
#include "../../include/cllm.h"
#include "internal.cuh"

using namespace cllm;

namespace {

constexpr size_t kNoAllocScratchBytes = size_t(8) << 20;  // 8 MiB, held by each device until exit

// One array per device that loads the library.  In host code this name is
// only a stand-in: its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of the scratch array in the current device's current
// context.  It is looked up on every call (a host-side table lookup, cheap):
// an address cached per device would be stale after cudaDeviceReset or in a
// second driver context on the same device, and the kernel would then write
// its partial sums into memory it does not own.  The first call in a context
// also loads the library's device code there.
int scratch_address(void** out) {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return CLLM_ECUDA;
  *out = p;
  return CLLM_OK;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

extern "C" int cllm_gemm_bf16_noalloc(const void* W, const void* X, float* Y, int M, int K, int T,
                                      int x_rows, void* cuda_stream) {
  if (!W || !X || !Y || M < 128 || M % 128 || K < 8 || K % 8 || T < 1) return CLLM_EINVAL;
  if (x_rows < round_up(T, 16) || (T > 256 && x_rows < 256)) return CLLM_EINVAL;
  if ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(X) |
       reinterpret_cast<uintptr_t>(Y)) & 15u)
    return CLLM_EINVAL;
  // the call synchronises its stream and reads the error word back, which a
  // stream capture cannot hold: refuse before touching the stream
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(static_cast<cudaStream_t>(cuda_stream), &cap) != cudaSuccess)
    return CLLM_ECUDA;
  if (cap != cudaStreamCaptureStatusNone) return CLLM_EUNSUPPORTED;
  // (three attributes: the whole property structure takes longer to fill than
  // the GEMM of 16 rows runs)
  int dev = 0, major = 0, minor = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return CLLM_ECUDA;
  if (major != 10 || minor != 3) return CLLM_EUNSUPPORTED;
  const int mtiles = M / kBM;
  const Part p = plan_gemm(mtiles, K, T, sms);
  // scratch inside the static array: partial tiles, tickets, the error word.
  // The limit also counts the side outputs that the engine's own epilogue
  // would write for this size (statistics, next inputs and their gains), so
  // which sizes are accepted does not depend on the epilogue.
  const size_t sz_part = align256(static_cast<size_t>(mtiles) * p.maxc * p.bn * kBM * 4);
  const size_t off_tick = sz_part;
  const size_t sz_tick = align256(static_cast<size_t>(mtiles) * 4);
  const size_t off_err = off_tick + sz_tick;
  const size_t sz_side = align256(static_cast<size_t>(mtiles) * round_up(T, 16) * 4) +
                         align256(static_cast<size_t>(2) * T * M * 2) + align256(static_cast<size_t>(M) * 2);
  if (off_err + 256 + sz_side > kNoAllocScratchBytes) return CLLM_ECAPACITY;

  void* base = nullptr;
  int rc = scratch_address(&base);
  if (rc != CLLM_OK) return rc;
  char* sb = static_cast<char*>(base);
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  // T > 256: whole units, which need no partials
  const bool wide = T > 256;
  WidePlan w{};
  if (wide) {
    if (gemm_wide_set_attributes_acc() != cudaSuccess) return CLLM_ECUDA;
    const int clusters = gemm_wide_clusters();
    if (clusters < 1) return CLLM_ECUDA;
    w = plan_wide(EPI_ACC, M, K, T, clusters, false);
  } else if (gemm_tc_set_attributes(p.bn_max) != cudaSuccess) {
    return CLLM_ECUDA;
  }
  GemmMaps maps{};
  if (!make_map(&maps.a0, W, K, M, kBM) || !make_map(&maps.b, X, K, 2 * x_rows, wide ? w.bn : p.bn))
    return CLLM_EINVAL;
  maps.a1 = maps.a2 = maps.a0;
  // the array keeps the previous call's contents: tickets and the error word
  // must start at zero (they are neighbours)
  if (cudaMemsetAsync(sb + off_tick, 0, sz_tick + 256, s) != cudaSuccess) return CLLM_ECUDA;

  GemmArgs g{};
  g.M = M;
  g.K = K;
  g.T = T;
  g.mtiles = p.mtiles;
  g.ntiles = p.ntiles;
  g.kchunks = p.kchunks;
  g.cpc = p.cpc;
  g.bn = p.bn;
  g.maxc = p.maxc;
  g.rows_q = M;
  g.rows_qk = M;
  g.lo_rows = x_rows;
  if (wide) w.apply(g);
  g.partial = reinterpret_cast<float*>(sb);
  g.tickets = reinterpret_cast<int*>(sb + off_tick);
  g.err = reinterpret_cast<int*>(sb + off_err);
  EpiArgs e{};
  e.T = T;
  e.x = Y;
  e.d = M;
  e.err = g.err;
  const cudaError_t le = wide ? launch_gemm_wide(EPI_ACC, maps, g, e, w.clusters, s, false)
                              : launch_gemm_tc(p.bn_max, maps, g, e, p.grid, s, false);
  if (le != cudaSuccess) return CLLM_ECUDA;
  int herr = 0;
  if (cudaMemcpyAsync(&herr, g.err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CLLM_ECUDA;
  if (herr) return (herr & DERR_TIMEOUT) ? CLLM_ETIMEOUT : CLLM_EDEVICE;
  return CLLM_OK;
}
