// The warp roles of the weight-streaming GEMM.  The stand-alone GEMM kernel uses
// all three; the persistent per-iteration kernel and the CTA-pair kernel have
// producers and MMA issuers of their own and share the epilogue, which carries
// its pipeline state across the persistent kernel's phases.
//
//   producer (one thread): TMA of weight tiles (A, evict-first) and the
//     activation tile's hi/lo planes (B, evict-last) into the stage ring.
//     Weight tiles do not depend on earlier work, so they are issued before
//     the previous kernel has finished; activation tiles only after.
//   MMA issuer (one thread): tcgen05.mma M=128 into a TMEM accumulator pair.
//   epilogue (warps 2..5, 128 threads): tcgen05.ld, split-K partials reduced in
//     a fixed order by the tile's first contributor, fused epilogue (epilogue.cuh).
#pragma once
#include "epilogue.cuh"

namespace cllm {

// Stage = one 128 x 64 weight tile + the hi and lo planes of a BNMAX x 64
// activation tile.
template <int BNMAX, int STAGES_>
struct TcCfg {
  static constexpr int STAGES = STAGES_;
  static constexpr int A_BYTES = kBM * kBK * 2;
  static constexpr int B_HALF = BNMAX * kBK * 2;
  static constexpr int B_BYTES = 2 * B_HALF;
  // The hi and lo products land in separate accumulator columns and are summed
  // in the epilogue, for every BNMAX, so a token's result is the same
  // whatever the launch's token count.  BNMAX <= 128: the lo rows follow the
  // bn hi rows in shared memory and one MMA with N = 2*bn covers both (lo at
  // column bn + t); BNMAX = 256: two MMAs, lo into columns 256 + t.
  static constexpr bool STACKED = BNMAX <= 128;
  static constexpr int ACC_COLS = 2 * BNMAX;
  static constexpr int NACC = ACC_COLS <= 256 ? 2 : 1;  // accumulators in TMEM (512 columns)
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = NACC * ACC_COLS;  // 128, 256, 512 or 512
  static constexpr int BN = BNMAX;
};

struct TcPipe {
  uint8_t* sA;  // STAGES x A_BYTES, 1024-aligned
  uint8_t* sB;  // STAGES x B_BYTES
  uint64_t* full;
  uint64_t* empty;
  uint64_t* tfull;   // [2]
  uint64_t* tempty;  // [2]
  uint64_t* drain;
  volatile int* abort;
  uint32_t tmem;
  // staging of split-K partials for the last arriver's reduction: red_slots
  // blocks of kEpiCols x kBM floats (set by the kernel after tc_pipe_init)
  float* red;
  int red_slots;
  int* jflag;  // two epilogue groups, shared memory: [0] the split-K wait's result, [1] the accumulator wait's
  // CTA pairs
  uint32_t tempty_leader;  // address of the even CTA's tempty
  uint8_t* ring_free;      // the stage ring, idle once the last segment's MMAs are done
  uint64_t* part_bar;      // [groups][kPartRounds]
};

constexpr size_t kRedSlotBytes = sizeof(float) * kEpiCols * kBM;

// Shared-memory bytes of the barrier block that follows the ring.
__host__ __device__ constexpr size_t tc_bar_bytes(int stages) { return 8 * (2 * stages + 5) + 16; }

// Carve the pipeline from shared memory and initialise it (all threads call).
// `bars` must be 8-byte aligned and hold tc_bar_bytes(STAGES) bytes.
// NG: epilogue groups of 4 warps (each warp releases the accumulator).
template <class Cfg, int NG = 1>
__device__ TcPipe tc_pipe_init(uint8_t* ring, uint8_t* bars) {
  constexpr int S = Cfg::STAGES;
  TcPipe P;
  P.sA = ring;
  P.sB = ring + S * Cfg::A_BYTES;
  uint64_t* b = reinterpret_cast<uint64_t*>(bars);
  P.full = b;
  P.empty = b + S;
  P.tfull = b + 2 * S;
  P.tempty = P.tfull + 2;
  P.drain = P.tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(P.drain + 1);
  P.abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&P.full[i], 1);
      mbar_init(&P.empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&P.tfull[i], 1);
      mbar_init(&P.tempty[i], 4 * NG);
    }
    mbar_init(P.drain, 1);
    *P.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  P.tmem = *tmem_slot;
  return P;
}

// Release TMEM (all threads call; every role has finished and drained).
template <class Cfg>
__device__ void tc_pipe_release(const TcPipe& P) {
  tc_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(P.tmem, Cfg::TMEM_COLS);
  }
}

// ---- the persistent kernel's dependency ------------------------------------------

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Persistent kernel: grid barrier counter >= target (every CTA finished the
// phases this one depends on).  Waits are bounded.
struct GridDep {
  const unsigned* counter;
  unsigned target;
  __device__ bool ready() const { return ld_acquire_gpu(counter) >= target; }
  __device__ bool wait(volatile int* abort) const {
    if (ready()) return true;
    const uint64_t t0 = globaltimer_ns();
    while (!ready()) {
      if (*abort) return false;
      if (globaltimer_ns() - t0 > kWaitBudgetNs) {
        *abort = 1;
        return false;
      }
      __nanosleep(32);
    }
    return true;
  }
  // global data written by other CTAs' generic stores is read next by TMA
  __device__ void after() const { asm volatile("fence.proxy.async.global;" ::: "memory"); }
};

// ---- work decomposition -----------------------------------------------------------

struct Segment {
  int unit, k0, k1;
};

// Work split of a launch.  The weight rows' 128-row tiles form groups of
// 1 << g.gshift tiles, and CTA `cta` works on tile `cta mod group size` of the
// groups: CTAs of one residue share a (group, k-chunk) space cut into equal
// contiguous ranges of g.cpc chunks, range cta >> gshift to this CTA.  (gshift
// 0: every tile is a group.  With 4 tiles a group, four neighbouring CTAs
// always work on the same K range, so a pair of them can share activations.)
__device__ __forceinline__ int tile_of(const GemmArgs& g, int group, int cta) {
  return (group << g.gshift) + (cta & ((1 << g.gshift) - 1));
}

// Iterate the (group, k-range) segments of the chunk range [c, c1).
__device__ __forceinline__ bool next_segment(int& c, int c1, int kchunks, Segment& sg) {
  if (c >= c1) return false;
  sg.unit = c / kchunks;
  sg.k0 = c - sg.unit * kchunks;
  const int end = min(c1, (sg.unit + 1) * kchunks);
  sg.k1 = end - sg.unit * kchunks;
  c = end;
  return true;
}

// Chunk range of CTA `cta` (up to the last group that has its tile).
__device__ __forceinline__ void cta_range(const GemmArgs& g, int cta, int& c0, int& c1) {
  const int size = 1 << g.gshift;
  const int total = ((g.mtiles - (cta & (size - 1)) + size - 1) >> g.gshift) * g.kchunks;
  c0 = min(total, (cta >> g.gshift) * g.cpc);
  c1 = min(total, c0 + g.cpc);
}

// ---- producer -------------------------------------------------------------------------

// Issue this CTA's chunks [c0, c1) of a launch of its own (stand-alone GEMM: one
// weight matrix).  Returns the number of chunks issued: fewer than asked for if
// a bounded wait gave up.
template <class Cfg>
__device__ int tc_produce(const TcPipe& P, const GemmArgs& g, const CUtensorMap* mA, const CUtensorMap* mB, int c0,
                          int c1, int cta) {
  constexpr int S = Cfg::STAGES;
  const int n = c1 - c0, pre = min(n, S);
  const uint64_t pol_w = l2_policy_evict_first();
  const uint64_t pol_x = l2_policy_evict_last();
  const uint32_t b_bytes = 2u * static_cast<uint32_t>(g.bn) * kBK * 2;
  auto load_a = [&](int j, int st) {
    const int c = c0 + j;
    const int u = c / g.kchunks, k = c - u * g.kchunks;
    mbar_arrive_expect_tx(&P.full[st], Cfg::A_BYTES + b_bytes);
    tma_load_2d(P.sA + st * Cfg::A_BYTES, mA, &P.full[st], k * kBK, tile_of(g, u, cta) * kBM, pol_w);
  };
  auto load_b = [&](int j, int st) {
    const int k = (c0 + j) % g.kchunks;
    uint8_t* dst = P.sB + st * Cfg::B_BYTES;
    tma_load_2d(dst, mB, &P.full[st], k * kBK, 0, pol_x);
    tma_load_2d(dst + (Cfg::STACKED ? g.bn * kBK * 2 : Cfg::B_HALF), mB, &P.full[st], k * kBK, g.lo_rows,
                pol_x);
  };
  // weights of the first stages do not depend on the previous kernel
  for (int j = 0; j < pre; ++j) load_a(j, j);
  pdl_wait();
  for (int j = 0; j < pre; ++j) load_b(j, j);
  for (int j = pre; j < n; ++j) {
    const int st = j % S;
    if (!mbar_wait(&P.empty[st], ((j / S) & 1) ^ 1, P.abort)) return j;
    load_a(j, st);
    load_b(j, st);
  }
  return max(n, 0);
}

// Before exit: every fully issued stage has landed (bounded).
template <class Cfg>
__device__ void tc_produce_drain(const TcPipe& P, int issued) {
  constexpr int S = Cfg::STAGES;
  for (int i = max(0, issued - S); i < issued; ++i) mbar_wait(&P.full[i % S], (i / S) & 1, nullptr);
}

// ---- MMA issuer ------------------------------------------------------------------------

template <class Cfg>
__device__ bool tc_mma(const TcPipe& P, int& idx, int& acc, uint32_t& accph, const GemmArgs& g, int c0, int c1) {
  constexpr int S = Cfg::STAGES;
  const uint32_t idesc = idesc_bf16_f32(kBM, Cfg::STACKED ? 2 * g.bn : g.bn);
  int c = c0;
  Segment sg;
  while (next_segment(c, c1, g.kchunks, sg)) {
    if (!mbar_wait(&P.tempty[acc], accph ^ 1, P.abort)) return false;
    tc_fence_after();
    const uint32_t dt = P.tmem + static_cast<uint32_t>(acc * Cfg::ACC_COLS);
    for (int k = sg.k0; k < sg.k1; ++k, ++idx) {
      const int st = idx % S;
      if (!mbar_wait(&P.full[st], (idx / S) & 1, P.abort)) return false;
      tc_fence_after();
      const uint32_t a_addr = smem_u32(P.sA + st * Cfg::A_BYTES);
      const uint32_t b_addr = smem_u32(P.sB + st * Cfg::B_BYTES);
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk) {
        const uint64_t ad = sdesc_kmajor_sw128(a_addr + kk * 32);
        tc_mma_f16(dt, ad, sdesc_kmajor_sw128(b_addr + kk * 32), idesc,
                   (k > sg.k0 || kk > 0) ? 1u : 0u);
        if (!Cfg::STACKED)
          tc_mma_f16(dt + Cfg::BN, ad, sdesc_kmajor_sw128(b_addr + Cfg::B_HALF + kk * 32), idesc,
                     (k > sg.k0 || kk > 0) ? 1u : 0u);
      }
      tc_commit(&P.empty[st]);
    }
    tc_commit(&P.tfull[acc]);
    if (++acc == Cfg::NACC) {
      acc = 0;
      accph ^= 1;
    }
  }
  return true;
}

// Before exit: every issued MMA has completed (bounded).
__device__ __forceinline__ void tc_mma_drain(const TcPipe& P) {
  tc_commit(P.drain);
  mbar_wait(P.drain, 0, nullptr);
}

// ---- epilogue (128 threads; r = TMEM lane = weight row of the tile) -------------------

__device__ __forceinline__ void red_release_gpu(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bounded wait until *p >= target (acquire).  On timeout sets *abort.
__device__ inline bool count_wait(const int* p, int target, volatile int* abort) {
  const uint64_t t0 = globaltimer_ns();
  while (static_cast<int>(ld_acquire_gpu(reinterpret_cast<const unsigned*>(p))) < target) {
    if (*abort) return false;
    if (globaltimer_ns() - t0 > kWaitBudgetNs) {
      *abort = 1;
      return false;
    }
    __nanosleep(32);
  }
  return true;
}


// hi + lo accumulator columns of 16 token columns (chunk ch) of this thread's row
template <class Cfg>
__device__ __forceinline__ void tmem_ld_sum_cfg(uint32_t taddr, int ch, int bn, float (&v)[kEpiCols]) {
  tmem_ld16(taddr + ch * kEpiCols, v);
  float vlo[kEpiCols];
  tmem_ld16(taddr + (Cfg::STACKED ? bn : Cfg::BN) + ch * kEpiCols, vlo);
#pragma unroll
  for (int j = 0; j < kEpiCols; ++j) v[j] += vlo[j];
}

// Split-K partials of the CTA-pair kernels: 16 columns of row r of chunk ch as
// four 16-byte pieces, a piece of the 128 rows contiguous.
__device__ __forceinline__ void part_st16(float* part, int ch, int r, const float (&v)[kEpiCols]) {
  float4* p = reinterpret_cast<float4*>(part) + static_cast<size_t>(ch) * 4 * kBM + r;
#pragma unroll
  for (int q = 0; q < 4; ++q) __stcg(p + q * kBM, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
}
// (from a copy of the chunk in shared memory)
__device__ __forceinline__ void part_add16(float (&v)[kEpiCols], const uint8_t* chunk, int r) {
  const float4* p = reinterpret_cast<const float4*>(chunk) + r;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 t = p[q * kBM];
    v[4 * q] += t.x;
    v[4 * q + 1] += t.y;
    v[4 * q + 2] += t.z;
    v[4 * q + 3] += t.w;
  }
}
constexpr int kPartChunkBytes = kEpiCols * kBM * 4;
constexpr int kPartRounds = 3;  // rounds of four chunks in flight per epilogue group

// Persistent kernel: publish a finished output tile (its stores are read next
// by other CTAs, some through TMA) on its completion flag.
__device__ __forceinline__ void epi_publish(const EpiArgs& e, int mt, int r) {
  if (e.tile_done == nullptr) return;
  asm volatile("fence.proxy.async.global;" ::: "memory");
  epi_sync();
  if (r == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(e.tile_done + mt) : "memory");
}

// NG = 2 (per-GEMM kernel, 256 token columns): two groups of 4 epilogue warps
// (warps 2-5 and 6-9, each with its own named barrier, EpiSmem and staging
// slots) take alternate 16-column chunks of each unit; a barrier over both
// groups orders their stores before the split-K release, the ticket reset
// and the argmax reduction.  Per column the arithmetic is unchanged.
// PAIR: the accumulators belong to a CTA pair, whose even CTA issues the MMAs;
// a CTA whose tile lies past the last one only hands its accumulator back.
template <int KIND, class Cfg, int NG = 1, bool PAIR = false>
__device__ bool tc_epilogue(const TcPipe& P, int& acc, uint32_t& accph, const GemmArgs& g,
                            const EpiArgs& e, int c0, int c1, int cta, EpiSmem& es) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = warp & 3;
  const int r = grp * 32 + lane;
  const int gi = NG > 1 ? (warp >= 6 ? 1 : 0) : 0;  // this thread's group
  auto joint = [&]() {
    if constexpr (NG > 1) named_bar_sync(3, 128 * NG);
    else epi_sync();
  };
  auto release = [&]() {  // this warp is done with the accumulator
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      if constexpr (PAIR) mbar_arrive_remote(P.tempty_leader + 8u * acc);
      else mbar_arrive(&P.tempty[acc]);
    }
  };
  if (c0 < c1) epi_prepare<KIND>(e, r, es, gi, NG);
  int c = c0;
  Segment sg;
  while (next_segment(c, c1, g.kchunks, sg)) {
    const int mt = tile_of(g, sg.unit, cta);
    EpiPre pre;
    const bool past = PAIR && mt >= g.mtiles;
    // (pairs, QKV: the tile's RoPE rows stay in L1, and its registers are needed)
    constexpr bool kPre = !(PAIR && KIND == EPI_QKV);
    const EpiPre* use_pre = kPre ? &pre : nullptr;
    if (kPre && !past) epi_prefetch<KIND, __nv_bfloat16>(e, mt, gi * kEpiCols, r, es, pre);
    bool seg_ok;
    if constexpr (NG > 1) {
      // one wait for both groups: a group that returned alone would leave the
      // other at the joint barrier, which has no time limit
      if (gi == 0 && r == 0) P.jflag[1] = mbar_wait(&P.tfull[acc], accph, P.abort) ? 1 : 0;
      joint();
      seg_ok = P.jflag[1] != 0;
      joint();  // read by all before the next unit's wait writes it again
    } else {
      if (r == 0) es.ok = mbar_wait(&P.tfull[acc], accph, P.abort) ? 1 : 0;
      epi_sync();
      seg_ok = es.ok != 0;
      epi_sync();
    }
    if (!seg_ok) return false;
    const bool dbg = e.dbg != nullptr && r == 0 && c >= c1;  // last segment
    if (dbg) e.dbg[cta] = globaltimer_ns();
    tc_fence_after();
    if (past) {
      release();
      if (++acc == Cfg::NACC) {
        acc = 0;
        accph ^= 1;
      }
      continue;
    }
    const int first = (sg.unit * g.kchunks) / g.cpc;
    const int last = ((sg.unit + 1) * g.kchunks - 1) / g.cpc;
    const int nc = last - first + 1;
    const int slot = (cta >> g.gshift) - first;
    const int nchunk = (e.T + kEpiCols - 1) / kEpiCols;
    const uint32_t taddr = P.tmem + (static_cast<uint32_t>(grp * 32) << 16) +
                           static_cast<uint32_t>(acc * Cfg::ACC_COLS);
    float* mypart = g.partial + (static_cast<size_t>(mt) * g.maxc + slot) * g.bn * kBM;
    // Split-K: the tile's contributors are ranges first..last (slots 0..nc-1).
    // Slot 0 -- for which this tile is the last segment of its range, so it
    // finishes with the phase -- owns the reduction: the others store their
    // partial sums and release a count; the owner waits for nc - 1, then adds
    // the partials to its own accumulator in slot order.
    const bool owner = nc > 1 && slot == 0;
    if (!owner) {
      for (int ch = gi; ch < nchunk; ch += NG) {
        float v[kEpiCols];
        tmem_ld_sum_cfg<Cfg>(taddr, ch, g.bn, v);
        if (nc == 1) {
          epi_apply<KIND, __nv_bfloat16>(e, mt, ch * kEpiCols, v, r, es, use_pre);
        } else {
          if constexpr (PAIR) {
            part_st16(mypart, ch, r, v);
          } else {
#pragma unroll
            for (int j = 0; j < kEpiCols; ++j) mypart[(ch * kEpiCols + j) * kBM + r] = v[j];
          }
        }
      }
      if (nc == 1) epi_publish(e, mt, r);
      release();
      if (nc > 1) {
        if constexpr (PAIR) asm volatile("fence.proxy.async.global;" ::: "memory");  // (read by bulk copies)
        joint();  // every thread's partial stores precede the release
        if (gi == 0 && r == 0) red_release_gpu(&g.tickets[mt], 1);
        if (dbg) e.dbg[e.dbg_stride + cta] = globaltimer_ns();
      } else if (KIND == EPI_ARGMAX) {
        if constexpr (NG > 1) joint();  // both groups' partial maxima are written
        if (gi == 0) epi_argmax_finish(e, r, es);
      }
    } else {
      bool got;
      if constexpr (NG > 1) {
        // one wait for both groups, so that they agree on its outcome
        if (gi == 0 && r == 0) *P.jflag = count_wait(&g.tickets[mt], nc - 1, P.abort) ? 1 : 0;
        joint();
        got = *P.jflag != 0;
      } else {
        if (r == 0) es.ok = count_wait(&g.tickets[mt], nc - 1, P.abort) ? 1 : 0;
        epi_sync();
        got = es.ok != 0;
        epi_sync();
      }
      if (!got) {
        release();
        return false;
      }
      if (dbg) e.dbg[e.dbg_stride + cta] = globaltimer_ns();
      if constexpr (PAIR) {
        // This is the CTA's last segment, so its ring is idle: the partials
        // of slots 1..nc-1 come through it by bulk copies (per-thread loads
        // reached 30 GB/s), a round of four chunks of one slot per buffer, three
        // rounds in flight per group; the totals go back to tensor memory
        // (the hi columns).
        const int mine = (nchunk - gi + NG - 1) / NG;  // this group's chunks
        const int per = nc - 1, rounds = (mine + 3) / 4 * per;
        uint8_t* buf = P.ring_free + gi * (kPartRounds * 4 * kPartChunkBytes);
        uint64_t* bar = P.part_bar + gi * kPartRounds;
        auto load_round = [&](int k) {
          const int cb = (k / per) * 4, s0 = 1 + k % per, n = min(4, mine - cb);
          const float* src = g.partial + (static_cast<size_t>(mt) * g.maxc + s0) * g.bn * kBM;
          uint64_t* b = bar + k % kPartRounds;
          mbar_arrive_expect_tx(b, n * kPartChunkBytes);
          for (int i = 0; i < n; ++i)
            bulk_load(buf + ((k % kPartRounds) * 4 + i) * kPartChunkBytes,
                      src + static_cast<size_t>(gi + (cb + i) * NG) * (kEpiCols * kBM), kPartChunkBytes, b);
        };
        asm volatile("fence.proxy.async.global;" ::: "memory");
        if (r == 0)
          for (int k = 0; k < min(rounds, kPartRounds); ++k) load_round(k);
        bool got_all = true;
        for (int k = 0, cb = 0; cb < mine; cb += 4) {
          float v[4][kEpiCols];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (cb + i < mine) tmem_ld_sum_cfg<Cfg>(taddr, gi + (cb + i) * NG, g.bn, v[i]);
          for (int s0 = 1; s0 < nc; ++s0, ++k) {
            // (bounded, and not cut short by another role's abort: the copy must land)
            got_all &= mbar_wait(bar + k % kPartRounds, (k / kPartRounds) & 1, nullptr);
            const uint8_t* b = buf + (k % kPartRounds) * 4 * kPartChunkBytes;
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (cb + i < mine) part_add16(v[i], b + i * kPartChunkBytes, r);
            epi_sync();  // the buffer has been read
            if (r == 0 && k + kPartRounds < rounds) load_round(k + kPartRounds);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (cb + i < mine) tmem_st16(taddr + (gi + (cb + i) * NG) * kEpiCols, v[i]);
        }
        tmem_st_wait();
        if (!got_all) *P.abort = 1;  // (the sums are incomplete: the launch reports a timeout)
        for (int ch = gi; ch < nchunk; ch += NG) {
          float v[kEpiCols];
          tmem_ld16(taddr + ch * kEpiCols, v);
          epi_apply<KIND, __nv_bfloat16>(e, mt, ch * kEpiCols, v, r, es, use_pre);
        }
      } else {
        for (int ch = gi; ch < nchunk; ch += NG) {
          float v[kEpiCols];
          tmem_ld_sum_cfg<Cfg>(taddr, ch, g.bn, v);
          // slots 1..nc-1: a group of up to red_slots partial blocks
          // (kEpiCols x kBM contiguous floats each) is copied to shared memory
          // by all 128 threads at once (cp.async at L2, no registers held),
          // then each thread adds its row
          for (int s0 = 1; s0 < nc; s0 += P.red_slots) {
            const int ns = min(P.red_slots, nc - s0);
            for (int q = 0; q < ns; ++q) {
              const float* src = g.partial + (static_cast<size_t>(mt) * g.maxc + s0 + q) * g.bn * kBM +
                                 static_cast<size_t>(ch) * kEpiCols * kBM;
              float* dst = P.red + q * (kEpiCols * kBM);
#pragma unroll
              for (int i = 0; i < kEpiCols * kBM / (4 * 128); ++i)
                cp_async16(dst + 4 * (i * 128 + r), src + 4 * (i * 128 + r));
            }
            cp_async_commit();
            // the chunk's own epilogue inputs travel in the same round trip
            if (ch > gi && s0 == 1)
              epi_prefetch<KIND, __nv_bfloat16>(e, mt, ch * kEpiCols, r, es, pre);
            cp_async_wait_all();
            epi_sync();
            for (int q = 0; q < ns; ++q) {
              const float* blk = P.red + q * (kEpiCols * kBM);
#pragma unroll
              for (int j = 0; j < kEpiCols; ++j) v[j] += blk[j * kBM + r];
            }
            epi_sync();
          }
          if (dbg && ch == 0) e.dbg[4 * e.dbg_stride + cta] = globaltimer_ns();
          epi_apply<KIND, __nv_bfloat16>(e, mt, ch * kEpiCols, v, r, es, use_pre);
        }
      }
      // (the count is reset before the tile is published: a later phase that
      // the flag opens may count on the same ticket)
      if constexpr (NG > 1) joint();  // both groups are past the wait and done
      if (gi == 0 && r == 0) g.tickets[mt] = 0;
      epi_publish(e, mt, r);
      release();
      if (KIND == EPI_ARGMAX && gi == 0) epi_argmax_finish(e, r, es);
    }
    if (dbg) e.dbg[2 * e.dbg_stride + cta] = globaltimer_ns();
    if (++acc == Cfg::NACC) {
      acc = 0;
      accph ^= 1;
    }
  }
  return true;
}

}  // namespace cllm
