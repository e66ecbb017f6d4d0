// Warp-specialized tcgen05 GEMM pipeline for the INT4 activation x INT4
// weight product, shared by the standalone GEMM and the fused kernel.
//
// acc[i][n] = sum_k qx[i][k] * qw[n][k] is an exact integer: |q| <= 7, so
// every product is an integer of magnitude <= 49 and, for K <= 16384, every
// partial sum stays below 2^24.  sm_103a has no integer tcgen05 MMA, so the
// codes ride on E4M3, which holds every integer in [-7, 7] exactly, through
// tcgen05.mma kind::f8f6f4 with fp32 accumulation in tensor memory; the
// integer accumulators come out exact as long as the fp32 sums are exact
// (checked bit for bit against the int64 oracle, +-7 codes at K = 16384).
// 8-bit codes (W4A8, W8A8) arrive as two E4M3 planes, 16 h and l with
// q = 16 h + l.  W4A8 multiplies both activation planes into one
// accumulator: every partial sum stays below 2^24 for K <= 16384 (at most
// (128 + 8) * 7 per code pair), so it is exact too.  W8A8 keeps two or three
// accumulators (SEP below) that are each exact and are added as integers.
// E2M3 operands (F6) take the same MMA with 6-bit formats.
//
// Persistent: one CTA per SM walks 128 (M) x BNT (N) tiles, or a pair of CTAs
// (CG 2, one cluster, tcgen05 cta_group::2) walks 256 x BNT tiles, in a static
// round-robin order, K step 128 codes.  Each operand arrives either as E4M3
// bytes, which TMA writes straight into the MMA operand buffer with the
// 128-byte swizzle, or as packed nibbles (APACK / BPACK), which TMA stages and
// unpack warps expand into that layout.  Each CTA of a pair loads its own 128
// rows of A and half of B's rows, all copies of a stage completing on the
// leader's barrier; the leader issues the MMAs, which read both CTAs' shared
// memory, and their completion signals the barriers of both.  Warp roles:
//   warp 4       TMA producer;
//   warps 6-13   unpack (only when an operand is packed; 448 threads);
//   warp 5       one lane (of the leader) issues tcgen05.mma (4 x K=32 per
//                stage) and commits stage and tile completion;
//   warps 0-3, 6-9 epilogue (warps 0-3 alone when an operand is packed or the
//                caller asks for four): warp w drains accumulator rows 32 * (w %
//                4) .. + 31 (the TMEM lanes its SM sub-partition may read), half
//                the columns each with eight: TMEM -> registers -> scale, bias,
//                round -> swizzled staging -> TMA tensor store.  Two TMEM
//                accumulators let the epilogue of tile i overlap the MMAs of
//                tile i + 1.
//   other warps  idle in this phase.
// What bounds it: the MMAs of a 128-code step take 542 clocks, the loop with its
// copies 587 (a pair, operands in L2).  Around it, at K = 1152 a tile takes
// about 5900 clocks instead of 5300 (the epilogue: without the stores of Y 8192 x
// 3456 x 1152 takes 20.1 us instead of 23.5, with half of B's copies still 23.5),
// the first MMA starts 1900 clocks after the launch wait and the last tile's
// epilogue adds 4000.  The stages matter most once operands come from further
// away: 4608 x 12288 x 3072 took 112.6 us with four 32 KB stages, 98.3 with
// five and 90.1 with six, which is why the staging buffers are 2 KB a warp.
// The epilogue warps keep their column data to themselves, no barrier joins them,
// and they load it and their row scales a tile ahead: at K = 1152 a tile's epilogue
// takes about as long as its MMAs, and those loads' latency stood at its head (8192
// x 3456 x 1152 with asymmetric activations 27.9 -> 23.6 us, symmetric in a layer,
// where rotate-quant has just written the scales, 32.1 -> 30.8 for both kernels).
// With `ready` counters (fused kernel), the producer waits until all rows of
// a tile's token block have been published before loading its A tiles.
// Every wait is bounded; on a timeout the roles drain their own copies and
// MMAs and return (status word: CLQ_ERR_TIMEOUT).
#pragma once

#include "gemm_common.cuh"
#include "clq_kernels.h"

namespace clq {
namespace gemm {

constexpr int NUM_UNPACK = 256;
constexpr int WARP_TMA = 4;
constexpr int WARP_MMA = 5;
constexpr int WARP_UNPACK0 = 6;
constexpr int MIN_THREADS = (WARP_UNPACK0 + NUM_UNPACK / 32) * 32;  // 448
constexpr int MAX_STAGES = 8;

// Tile BM x BNT a CTA (BNT 256, 192, 128 or 64; gemm_tile_n picks it).
// PA / PB: E4M3 planes per operand, 1 for 4-bit codes, 2 for 8-bit codes
// split as q = 16 h + l (plane 0 holds 16 h, plane 1 holds l; both E4M3
// values, so the MMAs of the two planes add up to q in one accumulator).
// EW: epilogue warps (0: 4 with unpack warps, else 8); SMAX: stage cap, for
// a CTA that keeps shared memory for other work.
// SEP (8-bit x 8-bit codes, PA = PB = 2): the plane products go to SEP = 2 or 3
// accumulators of BNT columns, so that each stays exact in fp32 (see pipeline()).
template <bool APACK, bool BPACK, int BNT = BN, int PA = 1, int PB = 1, int EW = 0,
          int SMAX = MAX_STAGES, int SEP = 0, int CG = 1>
struct Cfg {
  static constexpr bool UNPACK = APACK || BPACK;
  static constexpr int EPI_WARPS = EW != 0 ? EW : (UNPACK ? 4 : 8);
  static constexpr int THREADS = UNPACK ? MIN_THREADS : 32 * (EPI_WARPS + 2);
  static constexpr int EPI_NCOL = BNT * 4 / EPI_WARPS;  // columns per epilogue warp
  // a warp's column data: s_w / b, bias and (standalone kernel) zero-point sums
  static constexpr int COL_FLOATS = (EW != 0 ? 2 : 3) * EPI_NCOL;
  static constexpr int AU = PA * A_U;    // E4M3 A stage (all planes)
  static constexpr int BU = PB * (BNT / CG) * BK;  // E4M3 B stage (all planes)
  static constexpr int BP = BNT * BKP;   // packed B stage
  static constexpr int STAGE = AU + BU + (APACK ? A_P : 0) + (BPACK ? BP : 0);
  static constexpr int FIXED = EPI_WARPS * (EPI_BYTES + COL_FLOATS * 4);
  static constexpr int S0 = (222 * 1024 - FIXED) / STAGE;
  static constexpr int S = S0 > SMAX ? SMAX : S0;  // pipeline stages
  static constexpr size_t OFF_UA = 0;                           // E4M3 operands
  static constexpr size_t OFF_UB = OFF_UA + S * AU;
  static constexpr size_t OFF_PA = OFF_UB + S * BU;             // packed staging
  static constexpr size_t OFF_PB = OFF_PA + (APACK ? S * A_P : 0);
  static constexpr size_t OFF_EPI = OFF_PB + (BPACK ? S * BP : 0);
  static constexpr size_t OFF_COL = OFF_EPI + EPI_WARPS * EPI_BYTES;  // per warp
  static constexpr size_t BYTES = OFF_COL + EPI_WARPS * COL_FLOATS * sizeof(float);
  // bytes that complete on a stage's barrier (both CTAs' copies of a pair)
  static constexpr uint32_t TX = CG * ((APACK ? A_P : AU) + (BPACK ? BP : BU));
  // accumulator buffers (tiles in flight) of ACC columns; the power of two that
  // tcgen05.alloc takes
  static constexpr int ACC = (SEP > 0 ? SEP : 1) * BNT;
  static constexpr int NBUF = 2 * ACC <= 512 ? 2 : 1;
  static constexpr uint32_t TMEM = NBUF * ACC <= 128 ? 128u : NBUF * ACC <= 256 ? 256u : 512u;
  static_assert(S >= 2, "pipeline needs two stages");
  static_assert((PA == 1 || PA == 2) && (PB == 1 || PB == 2), "one or two planes");
  static_assert(!UNPACK || (PA == 1 && PB == 1), "8-bit planes come as E4M3 only");
  static_assert(EPI_WARPS == 4 || !UNPACK, "packed operands leave four epilogue warps");
  static_assert(EPI_NCOL % EPI_COLS == 0 && STAGE % 1024 == 0, "whole blocks, aligned staging");
  static_assert(SMAX <= MAX_STAGES, "barrier arrays hold MAX_STAGES stages");
  static_assert(CG == 1 || (CG == 2 && !UNPACK), "pairs: E4M3 / E2M3 operands only");
  static_assert((SEP != 0) == (PA == 2 && PB == 2) && (SEP == 0 || SEP == 2 || SEP == 3),
                "SEP: two or three accumulators, 8-bit x 8-bit codes");
  static_assert(ACC <= 512, "one buffer fits tensor memory");
};

struct __align__(8) Barriers {
  uint64_t tma_full[MAX_STAGES];  // operand bytes landed
  uint64_t unpacked[MAX_STAGES];  // packed operands expanded (unpack warps)
  uint64_t mma_done[MAX_STAGES];  // MMAs reading the stage completed
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t drained;
  uint32_t tmem_slot;
  int32_t abort;
};

struct Maps {
  const CUtensorMap* A;
  const CUtensorMap* B;
  const CUtensorMap* Y;   // null: direct stores
  const CUtensorMap* A2;  // second planes (PA / PB == 2), else unused
  const CUtensorMap* B2;
};

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Barrier init (thread 0) and TMEM allocation (warp WARP_MMA); the caller
// follows with tcgen05 fences around a CTA barrier.
template <bool APACK, bool BPACK, int BNT = BN, int PA = 1, int PB = 1, int EW = 0,
          int SMAX = MAX_STAGES, int SEP = 0, int CG = 1>
__device__ __forceinline__ void setup(Barriers* bars) {
  using C = Cfg<APACK, BPACK, BNT, PA, PB, EW, SMAX, SEP, CG>;
  constexpr int S = C::S;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&bars->tma_full[s], 1);
      mbar_init(&bars->unpacked[s], NUM_UNPACK);
      mbar_init(&bars->mma_done[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->acc_full[s], 1);
      mbar_init(&bars->acc_empty[s], CG * C::EPI_WARPS);
    }
    mbar_init(&bars->drained, 1);
    bars->abort = 0;
    fence_mbarrier_init();
  }
  if ((threadIdx.x >> 5) == WARP_MMA) {
    tmem_alloc<CG>(&bars->tmem_slot, C::TMEM);
    tmem_relinquish<CG>();
  }
}

// Wait (bounded) until all rows of token block m are published.
__device__ __forceinline__ bool wait_rows_ready(const uint32_t* ready, int m, uint32_t need,
                                                volatile int32_t* abort, int32_t* status) {
  const uint64_t t0 = global_timer_ns();
  while (ld_acquire_u32(ready + m) < need) {
    if (*abort != 0) return false;
    if (global_timer_ns() - t0 > kWaitLimitNs) {
      record_status(status, CLQ_ERR_TIMEOUT);
      *abort = 1;
      return false;
    }
    __nanosleep(128);
  }
  fence_proxy_async_global();
  return true;
}

// ASYM: asymmetric activation codes (zero-point epilogue, g.lo / g.wsum).
// EW / SMAX: as in Cfg (the same values as the setup() call).
// F6: both operands are E2M3 codes, 16 codes in 12 bytes in global memory;
// the tensor maps (type 16U6_ALIGN16B) pad every 12-byte group to 16 bytes on
// the way into shared memory, which is the layout tcgen05.mma kind::f8f6f4
// reads for 6-bit operands, so a stage holds the same 128 bytes per row and K
// step as with E4M3 while only 96 of them cross from L2 (the copies complete
// that many transaction bytes).
//
// SEP (W8A8): plane 0 holds 16 h and plane 1 l of each 8-bit code (q = 16 h
// + l), so q_x q_w = (16 h_x)(16 h_w) + [(16 h_x) l_w + l_x (16 h_w)] + l_x l_w.
// One fp32 accumulator would round once partial sums pass 2^24 (K > 896 at
// +-127).  The first term sums multiples of 256 below 2^28 (exact up to 2^32) for
// every K <= 16384 and gets its own accumulator.  The rest: |16 h| <= 128 and |l|
// <= 8 make a code pair's three products at most 2 * 1024 + 64 = 2112, so all of
// them together stay below 2^24, exact in any order, up to K = 7943; SEP = 2 puts
// them in one accumulator, and two tiles fit tensor memory, so the epilogue
// overlaps the next tile's MMAs.  SEP = 3, for larger K, keeps the cross terms
// (multiples of 16 below 2^25, exact up to 2^28) and l l (below 2^20) apart and
// one tile at a time.  The epilogue adds the accumulators as int32 (|q_x q_w| K
// <= 2^28).
template <typename OutT, bool APACK, bool BPACK, int BNT = BN, int PA = 1, int PB = 1, bool ASYM = false, int EW = 0, int SMAX = MAX_STAGES,
          bool F6 = false, int SEP = 0, int CG = 1>
__device__ __forceinline__ void pipeline(const Maps& maps, const GemmArgs& g, uint8_t* smem,
                                         Barriers* bars, uint32_t tmem, const uint32_t* ready) {
  using C = Cfg<APACK, BPACK, BNT, PA, PB, EW, SMAX, SEP, CG>;
  constexpr int S = C::S;
  static_assert(!ASYM || EW == 0, "zero-point column data: standalone kernel only");
  static_assert(!F6 || (!C::UNPACK && PA == 1 && PB == 1), "E2M3 operands come one plane each");
  constexpr uint32_t TX = F6 ? C::TX / 4 * 3 : C::TX;
  volatile int32_t* abort = &bars->abort;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int nk = (g.K + BK - 1) / BK;
  const int tiles_n = (g.N + BNT - 1) / BNT;
  constexpr int TM = CG * BM;  // rows of a tile
  const int tiles = ((g.M + TM - 1) / TM) * tiles_n;
  // A unit, one CTA or a pair, takes every units-th tile; `rank` is this CTA's
  // half of the pair's tile (rows) and of its B boxes.
  const int unit = static_cast<int>(blockIdx.x) / CG;
  const int units = static_cast<int>(gridDim.x) / CG;
  const int rank = CG == 2 ? static_cast<int>(cluster_ctarank()) : 0;

  if (warp == WARP_TMA) {
    if (elect_one()) {
      prefetch_tensor_map(maps.A);
      prefetch_tensor_map(maps.B);
      if (PA == 2) prefetch_tensor_map(maps.A2);
      if (PB == 2) prefetch_tensor_map(maps.B2);
      if (maps.Y != nullptr) prefetch_tensor_map(maps.Y);
      int it = 0;  // K steps issued so far (all tiles), stage it % S
      int s = 0;
      uint32_t phase = 1;  // of mma_done[s]: the first pass over the ring waits for nothing
      int ready_m = -1;
      bool ok = true;
      // a pair's copies complete on the leader's barriers
      const uint32_t full0 = CG == 2 ? cluster_addr(&bars->tma_full[0], 0) : 0;
      for (int t = unit; t < tiles && ok; t += units) {
        const int mb = t / tiles_n;
        const int m0 = mb * TM + rank * BM;
        const int n0 = (t - mb * tiles_n) * BNT + rank * (BNT / CG);
        if (ready != nullptr && mb != ready_m && m0 < g.M) {  // this CTA's 128 rows
          if (!wait_rows_ready(ready, mb * CG + rank, static_cast<uint32_t>(min(BM, g.M - m0)),
                               abort, g.status)) {
            ok = false;
            break;
          }
          ready_m = mb;
        }
        for (int kb = 0; kb < nk; ++kb, ++it) {
          if (!mbar_wait_bounded(&bars->mma_done[s], phase, abort, g.status, kWaitLimitNs)) {
            ok = false;
            break;
          }
          uint64_t* full = &bars->tma_full[s];
          if (CG == 1 || rank == 0) mbar_arrive_expect_tx(full, TX);
          auto load = [&](size_t off, const CUtensorMap* map, int x, int y) {
            if constexpr (CG == 2)
              tma_load_2d_pair(smem + off, map, x, y, full0 + 8u * s);
            else
              tma_load_2d(smem + off, map, x, y, full);
          };
          if (APACK)
            load(C::OFF_PA + s * A_P, maps.A, kb * BKP, m0);
          else
            load(C::OFF_UA + s * C::AU, maps.A, kb * BK, m0);
          if (PA == 2) load(C::OFF_UA + s * C::AU + A_U, maps.A2, kb * BK, m0);
          if (BPACK)
            load(C::OFF_PB + s * C::BP, maps.B, kb * BKP, n0);
          else
            load(C::OFF_UB + s * C::BU, maps.B, kb * BK, n0);
          if (PB == 2) load(C::OFF_UB + s * C::BU + BNT / CG * BK, maps.B2, kb * BK, n0);
          if (++s == S) {
            s = 0;
            phase ^= 1;
          }
        }
      }
      // On an abort, the copies already in flight must land before exit (those
      // of a pair's second CTA complete on the leader's barriers: it allows
      // them a millisecond).
      if (!ok && rank != 0) {
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 1000000ull) __nanosleep(1000);
      } else if (!ok) {
        for (int j = max(0, it - S); j < it; ++j)
          mbar_wait_bounded(&bars->tma_full[j % S], (j / S) & 1, nullptr, nullptr, 10000000ull);
      }
    }
    __syncwarp();
  } else if (warp == WARP_MMA) {
    if (rank == 0 && elect_one()) {
      constexpr uint32_t idesc = F6 ? idesc_f8f6f4_f32(TM, BNT, kFmtE2M3, kFmtE2M3)
                                    : idesc_e4m3_f32(TM, BNT);
      // Operand descriptors of stage 0; a stage, plane or K slice further adds
      // its bytes / 16 to the start-address field.
      const uint64_t adesc = sw128_desc(smem_addr(smem + C::OFF_UA));
      const uint64_t bdesc = sw128_desc(smem_addr(smem + C::OFF_UB));
      int s = 0, tc = 0;
      uint32_t phase = 0;  // of the stage's ready barrier
      bool ok = true;
      for (int t = unit; t < tiles && ok; t += units, ++tc) {
        const int buf = C::NBUF == 1 ? 0 : (tc & 1);
        const uint32_t use = C::NBUF == 1 ? tc : (tc >> 1);  // this buffer's earlier tiles
        if (!mbar_wait_bounded(&bars->acc_empty[buf], (use & 1) ^ 1, abort, g.status,
                               kWaitLimitNs)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + buf * C::ACC;
        for (int kb = 0; kb < nk; ++kb) {
          uint64_t* ready_bar = C::UNPACK ? &bars->unpacked[s] : &bars->tma_full[s];
          if (!mbar_wait_bounded(ready_bar, phase, abort, g.status, kWaitLimitNs)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t a0 = adesc + static_cast<uint32_t>(s * (C::AU / 16));
          const uint64_t b0 = bdesc + static_cast<uint32_t>(s * (C::BU / 16));
#pragma unroll
          for (int pa = 0; pa < PA; ++pa)
#pragma unroll
            for (int pb = 0; pb < PB; ++pb)
#pragma unroll
              for (int k = 0; k < BK / 32; ++k) {
                // SEP: accumulator 0 takes 16h x 16h; 3: 1 the cross terms, 2 l x l;
                // 2: 1 all of them.  A tile's first product into each replaces it.
                const int acc_i = SEP == 3 ? pa + pb : SEP == 2 ? (pa | pb) : 0;
                const bool first =
                    (kb | k) == 0 && (SEP == 0 ? (pa | pb) == 0
                                               : pa == 0 || (SEP == 3 && pb == 1));
                mma_e4m3<CG>(d + acc_i * BNT, a0 + (pa * A_U + k * 32) / 16,
                             b0 + (pb * (BNT / CG) * BK + k * 32) / 16, idesc, first ? 0u : 1u);
              }
          mma_commit<CG>(&bars->mma_done[s]);
          if (++s == S) {
            s = 0;
            phase ^= 1;
          }
        }
        if (ok) mma_commit<CG>(&bars->acc_full[buf]);
      }
      // Every MMA issued must complete before TMEM is released.
      mma_commit<CG>(&bars->drained);
      mbar_wait_bounded(&bars->drained, 0, nullptr, nullptr, 10000000ull);
    }
    __syncwarp();
  } else if (warp < 4 || (C::EPI_WARPS > 4 && warp >= 6 && warp < 2 + C::EPI_WARPS)) {
    // ---- epilogue ----
    const int quarter = warp & 3;
    const int part = warp < 4 ? 0 : 1 + ((warp - 6) >> 2);  // which NCOL columns of the tile
    const int ew = part * 4 + quarter;
    constexpr int NCOL = C::EPI_NCOL;
    const uint32_t empty0 = CG == 2 ? cluster_addr(&bars->acc_empty[0], 0) : 0;  // leader's
    uint8_t* staging = smem + C::OFF_EPI + ew * EPI_BYTES;
    float* col = reinterpret_cast<float*>(smem + C::OFF_COL) + ew * C::COL_FLOATS;
    // A tile's column data (s_w / b, bias, zero-point sums) and row scales, loaded
    // into registers a tile ahead.
    constexpr int NC = NCOL / 32;
    float sc[NC], bi[NC], wz[NC], nsx[4], nlo[4];
    auto load_scales = [&](int t) {
      const int mb = t / tiles_n;
      const int m0 = mb * TM + rank * BM;
      const int n0 = (t - mb * tiles_n) * BNT;
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const int cn = n0 + part * NCOL + 32 * j + lane;
        const bool in = t < tiles && cn < g.N;
        sc[j] = in ? __ldg(g.s_w + cn) : 0.f;
        bi[j] = in && g.bias != nullptr
                    ? Num<OutT>::to_f(__ldg(static_cast<const uint16_t*>(g.bias) + cn))
                    : 0.f;
        if (ASYM) wz[j] = in ? __ldg(g.wsum + cn) : 0.f;
      }
      // a thread's fragments hold rows 8 k + lane / 4 of the warp's 32
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int row = m0 + quarter * EPI_ROWS + 8 * k + (lane >> 2);
        const bool in = ready == nullptr && t < tiles && row < g.M;
        nsx[k] = in ? __ldg(g.s_x + row) : 0.f;
        if (ASYM) nlo[k] = in ? __ldg(g.lo + row) : 0.f;
      }
    };
    load_scales(unit);
    int tc = 0;
    for (int t = unit; t < tiles; t += units, ++tc) {
      const int mb = t / tiles_n;
      const int m0 = mb * TM + rank * BM;
      const int n0 = (t - mb * tiles_n) * BNT;
      const int buf = C::NBUF == 1 ? 0 : (tc & 1);
      const uint32_t use = C::NBUF == 1 ? tc : (tc >> 1);
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const float s = sc[j] * g.inv_b;
        col[32 * j + lane] = s;
        col[NCOL + 32 * j + lane] = bi[j];
        if (ASYM) col[2 * NCOL + 32 * j + lane] = wz[j] * s;
      }
      // Asymmetric codes: the value of code 0 is min + 2^(n-1) delta.
      float sx[4], zm[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        sx[k] = nsx[k];
        zm[k] = ASYM ? fmaf(g.zp_shift, sx[k], nlo[k]) : 0.f;
      }
      load_scales(t + units);
      __syncwarp();
      bool ok = mbar_wait_bounded(&bars->acc_full[buf], use & 1, abort, g.status,
                                  kWaitLimitNs);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      // In the fused kernel other CTAs of this grid write s_x: it is read from
      // L2 after the tile's MMAs have completed.
      if (ready != nullptr) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int row = m0 + quarter * EPI_ROWS + 8 * k + (lane >> 2);
          if (row < g.M) sx[k] = __ldcg(g.s_x + row);
        }
      }
      epilogue_part<OutT, NCOL, ASYM, SEP, BNT>(
          tmem + buf * C::ACC, quarter, part * NCOL, lane, m0, n0, g.M, g.N, sx, col, zm, staging,
          maps.Y, g.Y, g.acc_dbg, [&]() {
            tc_fence_before();
            __syncwarp();
            if (elect_one()) {
              if (CG == 2)
                mbar_arrive_cluster(empty0 + 8u * buf);
              else
                mbar_arrive(&bars->acc_empty[buf]);
            }
          });
      __syncwarp();  // every lane has read this tile's column data
    }
    if (elect_one()) bulk_wait_all();
    __syncwarp();
  } else if (C::UNPACK && warp >= WARP_UNPACK0 && warp < WARP_UNPACK0 + NUM_UNPACK / 32) {
    const int ut = threadIdx.x - WARP_UNPACK0 * 32;
    int it = 0;
    bool ok = true;
    for (int t = unit; t < tiles && ok; t += units) {
      for (int kb = 0; kb < nk; ++kb, ++it) {
        const int s = it % S;
        if (!mbar_wait_bounded(&bars->tma_full[s], (it / S) & 1, abort, g.status,
                               kWaitLimitNs)) {
          ok = false;
          break;
        }
        if (APACK)
          unpack_rows<BM, NUM_UNPACK>(smem + C::OFF_PA + s * A_P, smem + C::OFF_UA + s * C::AU,
                                      ut);
        if (BPACK)
          unpack_rows<BNT, NUM_UNPACK>(smem + C::OFF_PB + s * C::BP,
                                       smem + C::OFF_UB + s * C::BU, ut);
        fence_proxy_async_smem();
        mbar_arrive(&bars->unpacked[s]);
      }
    }
  }
}

// After a CTA (pair: cluster) barrier that follows pipeline(): release TMEM.
template <int CG = 1>
__device__ __forceinline__ void teardown(uint32_t tmem, uint32_t cols) {
  if ((threadIdx.x >> 5) == WARP_MMA) {
    tc_fence_after();
    tmem_dealloc<CG>(tmem, cols);
  }
}

}  // namespace gemm
}  // namespace clq
