// Pieces shared by the W4A4 GEMM and the fused rotate-quant + GEMM kernels:
// tile shape, nibble -> E4M3 unpacking into the tcgen05 operand layout, and
// the TMEM -> fp16/bf16 epilogue with TMA stores.
#pragma once

#include "clq_device.cuh"

namespace clq {
namespace gemm {

constexpr int BM = 128;           // rows of A (tokens) per tile
constexpr int BN = 256;           // rows of B (output channels) per tile (widest)
constexpr int BK = 128;           // codes per K step = one 128-byte swizzle row
constexpr int BKP = BK / 2;       // packed bytes per row per K step
constexpr int A_U = BM * BK;      // 16 KB unpacked A stage
constexpr int A_P = BM * BKP;     // 8 KB packed A stage
constexpr int EPI_COLS = 32;      // output columns per epilogue store
constexpr int EPI_ROWS = 32;      // rows per store: one warp's TMEM lanes
constexpr int EPI_BYTES = EPI_ROWS * EPI_COLS * 2;  // 2 KB staging buffer, one a warp

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

__device__ __forceinline__ uint32_t pack2(uint16_t lo, uint16_t hi) {
  return static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
}

// Eight 4-bit two's-complement codes (code j in nibble j) -> eight E4M3
// bytes.  Magnitude tables for the non-negative codes 0..7 and the negative
// codes -8..-1 are looked up with prmt on the low three bits of each nibble;
// the sign bit of each nibble, replicated to a byte mask by prmt's sign mode,
// selects between them.
__device__ __forceinline__ uint2 nibbles_to_e4m3(uint32_t w) {
  const uint32_t P0 = 0x44403800u, P1 = 0x4E4C4A48u;  // e4m3(0..7)
  const uint32_t N0 = 0xCACCCED0u, N1 = 0xB8C0C4C8u;  // e4m3(-8..-1)
  const uint32_t sel_lo = w & 0x7777u;
  const uint32_t sel_hi = (w >> 16) & 0x7777u;
  const uint32_t w4 = w << 4;
  const uint32_t m_lo = prmt(w4, w, 0xD9C8u);
  const uint32_t m_hi = prmt(w4, w, 0xFBEAu);
  const uint32_t p_lo = prmt(P0, P1, sel_lo), n_lo = prmt(N0, N1, sel_lo);
  const uint32_t p_hi = prmt(P0, P1, sel_hi), n_hi = prmt(N0, N1, sel_hi);
  return make_uint2((p_lo & ~m_lo) | (n_lo & m_lo), (p_hi & ~m_hi) | (n_hi & m_hi));
}

// Byte offset of 16-byte chunk c (0..7) of row r in a K-major E4M3 operand
// tile with the 128-byte swizzle: 8-row atoms of 1024 bytes.
__device__ __forceinline__ uint32_t sw128_offset(int r, int c) {
  return static_cast<uint32_t>((r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4));
}

// Unpack ROWS x 64 packed bytes (row-major staging) into the swizzled E4M3
// tile, NT threads cooperating (thread index t).
template <int ROWS, int NT>
__device__ __forceinline__ void unpack_rows(const uint8_t* __restrict__ src,
                                            uint8_t* __restrict__ dst, int t) {
#pragma unroll
  for (int i = 0; i < ROWS * 4 / NT; ++i) {
    const int q = t + NT * i;
    const int r = q >> 2;
    const int c = q & 3;
    const uint4 p = *reinterpret_cast<const uint4*>(src + r * BKP + c * 16);
    const uint2 e0 = nibbles_to_e4m3(p.x), e1 = nibbles_to_e4m3(p.y);
    const uint2 e2 = nibbles_to_e4m3(p.z), e3 = nibbles_to_e4m3(p.w);
    *reinterpret_cast<uint4*>(dst + sw128_offset(r, 2 * c)) = make_uint4(e0.x, e0.y, e1.x, e1.y);
    *reinterpret_cast<uint4*>(dst + sw128_offset(r, 2 * c + 1)) =
        make_uint4(e2.x, e2.y, e3.x, e3.y);
  }
}

// 16 TMEM lanes x 32 columns, one matrix fragment per 8 columns: thread t gets,
// of column group g, columns 8 g + 2 (t % 4) and + 1 of lane t / 4 in r[4 g],
// r[4 g + 1] and of lane t / 4 + 8 in r[4 g + 2], r[4 g + 3].
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// Four 8 x 8 matrices of 16-bit values to shared memory: lane l gives the
// address of row l % 8 of matrix l / 8, register m the pair at row l / 4,
// columns 2 (l % 4) and + 1 of matrix m.
__device__ __forceinline__ void stmatrix4(uint32_t addr, const uint32_t (&o)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr),
               "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3])
               : "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* smem_src,
                                             int32_t x, int32_t y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(smem_addr(smem_src)), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Wait for this thread's outstanding tcgen05.ld and make every register of
// r depend on that wait, so that no use of r is scheduled before it.
__device__ __forceinline__ void tmem_ld_wait_tie(uint32_t (&r)[16]) {
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));
}

// Byte offset of 16-byte chunk q (8 columns) of row r in a staging buffer: the
// tensor map's 64-byte swizzle, which also spreads the rows over the banks.
__device__ __forceinline__ int staged_chunk(int r, int q) {
  return r * 64 + ((q ^ ((r >> 1) & 3)) << 4);
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// A staged block (rows row0 .. row0 + 31, columns col0 .. col0 + 31) straight to
// Y when N % 8 != 0 rules the tensor store out: half a warp takes consecutive
// column pairs of one row, four-byte aligned whatever N's parity (in a row that
// starts at an odd element, pairs 1-2, 3-4, .., and the last lane takes columns
// 31 and 0).  Eight pairs are read before the first is stored: with loads and
// stores alternating, which may alias as far as the compiler knows, a block took
// about 4700 clocks.  What is left is instructions, so the swizzled rows' addresses
// are four registers and immediates, one load serves a pair (the next lane's comes
// by shuffle) and rows past M are skipped by halves: with addresses formed per load,
// two loads a pair and a divergent exit, a product of packed operands with 24 rows and
// 111 columns took 9.4 us, 1357 x 1184 -> 1003 8.5 and 8192 x 1152 -> 3455 51.1; now
// 6.9, 7.0 and 34.7 (stores by elements before that: 7.8 and 31.7).
__device__ __forceinline__ void store_block_direct(uint32_t staging, int lane, int row0, int M,
                                                   int col0, int N, uint16_t* Y) {
  const int ncol = min(EPI_COLS, N - col0);
  const int rows = min(EPI_ROWS, M - row0);      // warp-uniform
  const int p = lane & 15, h = lane >> 4;        // this lane's pair, of rows h, h + 2, ..
  const int next = (lane & 16) | ((p + 1) & 15);  // the lane of the next pair
  uint16_t* y = Y + static_cast<size_t>(row0 + h) * N + col0;
  const uint32_t odd0 = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(y) >> 1) & 1u;
  // row 2 i + h: its chunk c lies at (c ^ (i & 3)) << 4 (staged_chunk)
  uint32_t at[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) at[k] = staging + h * 64 + (((p >> 2) ^ k) << 4) + (p & 3) * 4;
  const int j = 2 * p + static_cast<int>(odd0);  // column of the low half
  // rows 2 i + h < M whose pair is stored whole, in its low half, or in its high half
  // (column 0 of a row that starts at an odd element)
  const int both = j + 1 < ncol ? rows - h : 0;
  const int low = j + 1 == ncol ? rows - h : 0;
  const int first = odd0 != 0 && p == 15 ? rows - h : 0;
#pragma unroll
  for (int i0 = 0; i0 < EPI_ROWS / 2; i0 += 8) {  // rows 2 i + h: the same parity for all i
    if (2 * i0 >= rows) break;
    uint32_t w[8];
#pragma unroll
    for (int i = i0; i < i0 + 8; ++i) {
      const uint32_t a = lds_u32(at[i & 3] + 128 * i);
      w[i - i0] = __funnelshift_r(a, __shfl_sync(0xffffffffu, a, next), 16u * odd0);
    }
#pragma unroll
    for (int i = i0; i < i0 + 8; ++i, y += 2 * static_cast<size_t>(N)) {
      if (2 * i < both) *reinterpret_cast<uint32_t*>(y + j) = w[i - i0];
      if (2 * i < low) y[j] = static_cast<uint16_t>(w[i - i0]);
      if (2 * i < first) y[0] = static_cast<uint16_t>(w[i - i0] >> 16);
    }
  }
}

// One warp's share of a tile's epilogue: TMEM lanes 32 * quarter .. + 31 (the
// warp's rows) and tile columns [col0, col0 + NCOL) in blocks of 32 columns:
// TMEM -> registers -> y = acc * s_x[row] * s_w[col] / b + bias[col], rounded to
// OutT -> the warp's swizzled staging buffer -> one bulk tensor store a block (or
// direct stores, mapY null).  `col` is the warp's column data (s_w / b, bias,
// zero-point sums; NCOL floats each); sx[k] belongs to row 8 k + lane / 4 of the
// 32.  ASYM (asymmetric activation codes, centered): sx is the row's step delta,
// zm the value of code 0, and y = acc * delta * s_w / b + zm * sum_k q_w * s_w /
// b + bias.  Once the last block is in registers, `release()` hands the
// accumulator back, so that the MMAs of the tile after next need not wait for
// the stores.
//
// What it costs is shared-memory time, which the MMAs' operands and the copies
// that bring them want too.  So the accumulators are read as matrix fragments:
// a thread's two columns of a group serve four rows, and 32 columns take 8
// eight-byte loads of column data a warp where one row a lane took 16
// sixteen-byte ones; the packed pairs leave by stmatrix.
//
// SEP > 0: the accumulator is the sum of SEP (2 or 3) TMEM accumulators BNT
// columns apart, each an exact integer in fp32 (the W8A8 plane products); they
// are added as int32 and the block goes on with that (exact) sum.
template <typename OutT, int NCOL, bool ASYM, int SEP, int BNT, typename Release>
__device__ __forceinline__ void epilogue_part(uint32_t tmem_acc, int quarter, int col0, int lane,
                                              int m0, int n0, int M, int N, const float (&sx)[4],
                                              const float* col, const float (&zm)[4],
                                              uint8_t* staging, const CUtensorMap* mapY, void* Y,
                                              int32_t* acc_dbg, Release release) {
  static_assert(NCOL % EPI_COLS == 0, "column share must be whole 32-column blocks");
  const uint32_t lane_base = tmem_acc + (static_cast<uint32_t>(quarter * 32) << 16);
  const int row0 = m0 + quarter * EPI_ROWS;
  // blocks that hold rows and columns of Y (warp-uniform)
  const int nblk =
      row0 < M ? max(0, min(NCOL / EPI_COLS, (N - n0 - col0 + EPI_COLS - 1) / EPI_COLS)) : 0;
  if (nblk == 0) {
    release();
    return;
  }
  const uint32_t stage_addr = smem_addr(staging);
#pragma unroll 1
  for (int i = 0; i < nblk; ++i) {
    const int c = col0 + i * EPI_COLS;  // tile column
    uint32_t r[2][16];                  // rows 0 .. 15 and 16 .. 31
    tmem_ld_frag(lane_base + c, r[0]);
    tmem_ld_frag(lane_base + (16u << 16) + c, r[1]);
    const float* cc = col + i * EPI_COLS + 2 * (lane & 3);
    float2 cs[4], cb[4], cz[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      cs[g] = *reinterpret_cast<const float2*>(cc + 8 * g);
      cb[g] = *reinterpret_cast<const float2*>(cc + NCOL + 8 * g);
      if (ASYM) cz[g] = *reinterpret_cast<const float2*>(cc + 2 * NCOL + 8 * g);
    }
    tmem_ld_wait_tie(r[0]);
    tmem_ld_wait_tie(r[1]);
    if constexpr (SEP > 0) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const uint32_t at = lane_base + (static_cast<uint32_t>(half * 16) << 16) + c;
        uint32_t r1[SEP - 1][16];
#pragma unroll
        for (int p = 1; p < SEP; ++p) tmem_ld_frag(at + p * BNT, r1[p - 1]);
#pragma unroll
        for (int p = 1; p < SEP; ++p) tmem_ld_wait_tie(r1[p - 1]);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          int sum = __float2int_rn(__uint_as_float(r[half][j]));
#pragma unroll
          for (int p = 1; p < SEP; ++p) sum += __float2int_rn(__uint_as_float(r1[p - 1][j]));
          r[half][j] = static_cast<uint32_t>(sum);
        }
      }
    }
    if (i == nblk - 1) release();
    if (acc_dbg != nullptr) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int row = row0 + 8 * k + (lane >> 2);
          const int cn = n0 + c + 8 * (j >> 1) + 2 * (lane & 3) + (j & 1);
          const uint32_t v = r[k >> 1][4 * (j >> 1) + 2 * (k & 1) + (j & 1)];
          if (row < M && cn < N)
            acc_dbg[static_cast<size_t>(row) * N + cn] =
                SEP > 0 ? static_cast<int32_t>(v) : __float2int_rn(__uint_as_float(v));
        }
    }
    // The store that last used the staging buffer has finished reading it.
    if (mapY != nullptr && elect_one()) bulk_wait_read<0>();
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // rows 8 k + lane / 4
      const float2 sx2 = make_float2(sx[k], sx[k]);
      uint32_t o[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const uint32_t v0 = r[k >> 1][4 * g + 2 * (k & 1)];
        const uint32_t v1 = r[k >> 1][4 * g + 2 * (k & 1) + 1];
        const float2 acc = SEP > 0 ? make_float2(static_cast<float>(static_cast<int32_t>(v0)),
                                                  static_cast<float>(static_cast<int32_t>(v1)))
                                    : make_float2(__uint_as_float(v0), __uint_as_float(v1));
        const float2 bias = ASYM ? __ffma2_rn(make_float2(zm[k], zm[k]), cz[g], cb[g]) : cb[g];
        const float2 y = __ffma2_rn(acc, __fmul2_rn(sx2, cs[g]), bias);
        o[g] = Num<OutT>::pack2(y.x, y.y);
      }
      stmatrix4(stage_addr + staged_chunk(8 * k + (lane & 7), lane >> 3), o);
    }
    if (mapY != nullptr) {
      fence_proxy_async_smem();
      __syncwarp();
      if (elect_one()) {
        tma_store_2d(mapY, staging, n0 + c, row0);
        bulk_commit();
      }
    } else {
      __syncwarp();
      store_block_direct(stage_addr, lane, row0, M, n0 + c, N, static_cast<uint16_t*>(Y));
      __syncwarp();
    }
  }
}

}  // namespace gemm
}  // namespace clq
