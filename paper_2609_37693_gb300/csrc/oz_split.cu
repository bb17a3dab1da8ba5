// oz_split.cu -- phases 1 (Scale) and 2 (Reduce) of Sec. "Structure".
//
// Scale (eq. convert): per vector (row of A, column of B) the exponent e with
// max|x| in [2^(e-1), 2^e), from the largest |x| bit pattern (for finite
// doubles the order of |x| is the order of its bits), and the shift
// s = beta - e (0 for a zero vector).
//
// Reduce: a' = trunc(x 2^s) taken straight from the IEEE fields: with the
// 53-bit significand f and exponent E, x 2^s = f 2^(E - 1075 + s), so a'
// is f shifted left or right (the right shift truncates toward zero). The
// residue modulo m (m <= 239) is formed in exact fp32 arithmetic (twice the
// integer issue rate): |a'| is cut once per entry into signed pieces, a first
// piece P0 of 22 bits and then pieces of 13 bits (P1..P3 when beta <= 61,
// P1..P4 when beta <= 64) or, for widened operands (beta up to 84, Sec. "Not
// True Emulation of DGEMM", a' in 128 bits), six of 12 bits. Per modulus
//   y = P0 + P1 c_1 + P2 c_2 + ...,   c_i = 2^(bits below piece i) mod m, |c_i| <= 119,
// an integer congruent to a' with |y| < 2^22 + 4 * 8191 * 119 < 2^23, so every
// partial sum is exact. One quotient q = rint(y * fl(1/m)) (an fma against
// the 1.5 * 2^23 rounding constant) is the integer nearest to y/m: the
// estimate is off by at most |y/m| 2^-24 < 1/(2m), and for odd m, y/m is at
// least 1/(2m) away from every half-integer. So r = y - q m is exactly the
// representative nearest zero. For the even modulus (236, always at index
// 2 of an INT8 plan) y/m can be a half-integer; the estimate then picks
// either neighbour, r is +-m/2, and +m/2 is mapped to -m/2: the result lies
// in [-floor(m/2), ceil(m/2) - 1] for every modulus. (The paper reduces a
// one-byte modulus in two 32-bit Barrett steps, Sec. "Around the GEMMs";
// this is the same reduction in the fp32 pipe: six fp32 operations per
// modulus and entry.)
//
// Planes are written K-major, Q planes of nvec_pad x k_pad entries, int8
// (two's complement, IMMA engine) or bf16 (TC engine; integers below 2^8 are
// exact in bf16).
#include <stdint.h>

#include <type_traits>

#include "oz_internal.h"
#include "oz_device.cuh"
#include "oz_launch.h"
#include "oz_pair.cuh"
#include "oz_sync.cuh"

namespace oz {
namespace {

// Signed pieces of a' as exact floats, NP of them: a 22-bit first piece,
// then 13-bit pieces (NP = 4: |a'| < 2^61; NP = 5: |a'| < 2^74) or 12-bit
// pieces (NP = 7, widened operands, |a'| < 2^84).
template <int NP>
struct Pieces {
  static constexpr int kW0 = 22;
  static constexpr int kBits = NP > 5 ? 12 : 13;
  float p[NP];
};

template <int NP>
__device__ __forceinline__ Pieces<NP> pieces_of(uint64_t bits, int32_t s) {
  Pieces<NP> P;
  constexpr int W0 = Pieces<NP>::kW0, PB = Pieces<NP>::kBits;
  constexpr uint32_t mask = (1u << PB) - 1u;
  if constexpr (NP > 5) {
    const TruncWide t = truncate_wide(bits, s);
    const float sg = t.neg ? -1.0f : 1.0f;
    const float off = t.neg ? 8388608.0f : -8388608.0f;
    P.p[0] = fmaf(__int_as_float(0x4B000000u | ((uint32_t)t.mag & ((1u << W0) - 1u))), sg, off);   // +-v, exact
#pragma unroll
    for (int i = 1; i < NP; ++i) {
      const uint32_t v = (uint32_t)(t.mag >> (W0 + PB * (i - 1))) & mask;
      P.p[i] = fmaf(__int_as_float(0x4B000000u | v), sg, off);
    }
  } else {
    const Trunc t = truncate(bits, s);
    const float sg = t.neg ? -1.0f : 1.0f;
    const float off = t.neg ? 8388608.0f : -8388608.0f;
    P.p[0] = fmaf(__int_as_float(0x4B000000u | ((uint32_t)t.mag & ((1u << W0) - 1u))), sg, off);
#pragma unroll
    for (int i = 1; i < NP; ++i) {
      const uint32_t v = (uint32_t)(t.mag >> (W0 + PB * (i - 1))) & mask;
      P.p[i] = fmaf(__int_as_float(0x4B000000u | v), sg, off);
    }
  }
  return P;
}

// The constants of one modulus, held in registers while a tile is reduced:
// c[i - 1] = 2^(bits below piece i) mod m, nearest zero.
template <int NP>
struct ModConst {
  float c[NP - 1];
  float invm, m;
};

template <int NP>
__device__ __forceinline__ ModConst<NP> mod_const(const OzTables& T, int q) {
  ModConst<NP> c;
#pragma unroll
  for (int i = 0; i < NP - 1; ++i) c.c[i] = NP > 5 ? T.c12f[i][q] : T.c13f[i][q];
  c.invm = T.invm[q];
  c.m = T.mf[q];
  return c;
}

// The tie of the even modulus (index 2): +m/2 becomes -m/2.
__device__ __forceinline__ float fix_tie(const OzTables& T, float r) {
  const float h = T.halfm[2];
  return r == h ? -h : r;
}

// Representatives of a' nearest zero modulo one modulus for EPT entries, as
// exact floats in [-m/2, m/2] (see the header; below m/2 in magnitude for an
// odd m): y = P0 + P1 c_1 + ..., q = rint(y / m) by one fma against the
// rounding constant, r = y - q m. Two entries go through each packed fp32
// operation (the f32x2 fma and add of sm_100 and later round each half as the
// scalar operation would), so the issued instructions are half those of the
// scalar chain and the results are the same bits.
template <int NP, int EPT>
__device__ __forceinline__ void residues_any(const ModConst<NP>& c, const Pieces<NP> (&P)[EPT], float (&r)[EPT]) {
  static_assert(EPT % 2 == 0, "entries in pairs");
  const float2 kC = make_float2(12582912.0f, 12582912.0f), kCn = make_float2(-12582912.0f, -12582912.0f);
  const float2 inv = make_float2(c.invm, c.invm), nm = make_float2(-c.m, -c.m);
  float2 ci[NP - 1];
#pragma unroll
  for (int i = 0; i < NP - 1; ++i) ci[i] = make_float2(c.c[i], c.c[i]);
#pragma unroll
  for (int e = 0; e < EPT; e += 2) {
    float2 y = make_float2(P[e].p[0], P[e + 1].p[0]);
#pragma unroll
    for (int i = 1; i < NP; ++i) y = __ffma2_rn(make_float2(P[e].p[i], P[e + 1].p[i]), ci[i - 1], y);
    const float2 qf = __fadd2_rn(__ffma2_rn(y, inv, kC), kCn);   // rint(y / m), exact
    const float2 rr = __ffma2_rn(qf, nm, y);
    r[e] = rr.x;
    r[e + 1] = rr.y;
  }
}

// Representatives in [-floor(m/2), ceil(m/2) - 1] of modulus q for EPT
// entries, q a compile-time index after unrolling: only q = 2 takes the tie
// fix.
template <int NP, int EPT>
__device__ __forceinline__ void residues_q(const OzTables& T, int q, const ModConst<NP>& c, const Pieces<NP> (&P)[EPT],
                                           float (&r)[EPT]) {
  residues_any<NP, EPT>(c, P, r);
  if (q == 2) {
#pragma unroll
    for (int e = 0; e < EPT; ++e) r[e] = fix_tie(T, r[e]);
  }
}

// bf16 bit pattern of the integers r (|r| < 2^8 needs at most 8 significand
// bits, so the upper half of the float is exact)
__device__ __forceinline__ uint32_t bf16_pair(float r_lo, float r_hi) {
  return __byte_perm(__float_as_uint(r_lo), __float_as_uint(r_hi), 0x7632u);
}

// two's-complement byte of r: r + 1.5 * 2^23 has r in its low byte
__device__ __forceinline__ uint32_t int8_bits(float r) { return __float_as_uint(r + 12582912.0f); }

__device__ __forceinline__ uint32_t int8_quad(float a, float b, float c, float d) {
  return __byte_perm(__byte_perm(int8_bits(a), int8_bits(b), 0x0040u), __byte_perm(int8_bits(c), int8_bits(d), 0x0040u),
                     0x5410u);
}

// The residues of EPT consecutive entries (pieces P) modulo every modulus,
// stored at planes[q plane + off]: one 16- or 8-byte store of bf16 (EPT = 8
// or 4), or 8 or 4 bytes of int8, per modulus. QT > 0: the modulus count is QT
// at compile time (no per-modulus test); QT = 0: T.Q at run time.
template <bool kBF16, int NP, int EPT, int QT>
__device__ __forceinline__ void store_residues(const OzTables& T, const Pieces<NP> (&P)[EPT], void* __restrict__ planes,
                                               int64_t plane, int64_t off) {
  static_assert(EPT == 4 || EPT == 8, "four or eight entries");
  const int Q = QT > 0 ? QT : T.Q;
#pragma unroll
  for (int q = 0; q < (QT > 0 ? QT : OZ_MAX_MODULI); ++q) {
    if (QT > 0 || q < Q) {
      const ModConst<NP> mc = mod_const<NP>(T, q);
      float r[EPT];
      residues_q<NP, EPT>(T, q, mc, P, r);
      const int64_t o = (int64_t)q * plane + off;
      if (kBF16) {
        uint16_t* dst = static_cast<uint16_t*>(planes) + o;
        if constexpr (EPT == 8)
          *reinterpret_cast<uint4*>(dst) = make_uint4(bf16_pair(r[0], r[1]), bf16_pair(r[2], r[3]),
                                                      bf16_pair(r[4], r[5]), bf16_pair(r[6], r[7]));
        else
          *reinterpret_cast<uint2*>(dst) = make_uint2(bf16_pair(r[0], r[1]), bf16_pair(r[2], r[3]));
      } else {
        int8_t* dst = static_cast<int8_t*>(planes) + o;
        if constexpr (EPT == 8)
          *reinterpret_cast<uint2*>(dst) = make_uint2(int8_quad(r[0], r[1], r[2], r[3]), int8_quad(r[4], r[5], r[6], r[7]));
        else
          *reinterpret_cast<uint32_t*>(dst) = int8_quad(r[0], r[1], r[2], r[3]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Contiguous vectors (rows of A, or of B^T): one CTA of 256 threads per
// vector. Pass 1 finds the max bits; pass 2 re-reads the row (from L2) and
// writes 8 consecutive entries per thread per plane.
// ---------------------------------------------------------------------------
template <bool kBF16, int NP, int QT>
__device__ __forceinline__ void split_row(const OzTables& T, int64_t v, int64_t nvec, int64_t len,
                                          const double* __restrict__ X, int64_t ld, int64_t nvec_pad, int64_t k_pad,
                                          int32_t* __restrict__ shifts, void* __restrict__ planes,
                                          int32_t* __restrict__ flag, bool given, bool mark = false) {
  __shared__ uint64_t red[8];
  __shared__ int32_t s_sh;
  const int tid = threadIdx.x;
  const bool live = v < nvec;
  const uint64_t* row = reinterpret_cast<const uint64_t*>(X) + (live ? v * ld : 0);

  int32_t s;
  if (given) {                      // block-uniform: the shift of the whole row is known
    s = live ? shifts[v] : 0;
  } else {
    uint64_t mx = 0;
    uint32_t bad = 0;
    if (live) row_absmax(row, len, tid, 256, mx, bad);
    mx = warp_max_u64(mx);
    bad = __any_sync(0xffffffffu, bad);
    if ((tid & 31) == 0) red[tid >> 5] = mx | (bad ? (1ull << 63) : 0);
    __syncthreads();
    if (tid == 0) {
      uint64_t m = 0, anybad = 0;
      for (int w = 0; w < 8; ++w) {
        anybad |= red[w] >> 63;
        uint64_t x = red[w] & kAbsMask;
        m = x > m ? x : m;
      }
      if (anybad && flag) atomicOr(flag, 1);
      int32_t s0 = live ? shift_from_maxbits(anybad ? 0 : m, T.bits) : 0;
      s_sh = s0;
      if (live) shifts[v] = s0 + (mark && anybad ? kBadMark : 0);
    }
    __syncthreads();
    s = s_sh;
  }

  const int64_t plane = nvec_pad * k_pad;
  const bool vec = live && ((reinterpret_cast<uintptr_t>(row) & 15) == 0);
  // eight entries per thread per pass
  for (int64_t h0 = (int64_t)tid * 8; h0 < k_pad; h0 += 256 * 8) {
    uint64_t b[8];
    if (vec && h0 + 8 <= len) {
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const ulonglong2 w = ld_dep(reinterpret_cast<const ulonglong2*>(row + h0 + e));
        b[e] = w.x;
        b[e + 1] = w.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) b[e] = (live && h0 + e < len) ? ld_dep(row + h0 + e) : 0ull;
    }
    Pieces<NP> P[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (((b[e] >> 52) & 0x7ff) == 0x7ff) b[e] = 0;  // non-finite: flagged above
      P[e] = pieces_of<NP>(b[e], s);
    }
    store_residues<kBF16, NP, 8, QT>(T, P, planes, plane, v * k_pad + h0);
  }
}

// The same for a short row (k_pad <= 1024 in one product's split, <= 4096
// in the grouped one): one warp per row, eight rows per block; the row's
// maximum is a warp reduction.
template <bool kBF16, int NP, int QT>
__device__ __forceinline__ void split_row_warp(const OzTables& T, int64_t v, int64_t nvec, int64_t len,
                                               const double* __restrict__ X, int64_t ld, int64_t nvec_pad,
                                               int64_t k_pad, int32_t* __restrict__ shifts,
                                               void* __restrict__ planes, int32_t* __restrict__ flag, bool given,
                                               bool pad, bool mark = false) {
  const int lane = threadIdx.x & 31;
  const bool live = v < nvec;
  if (!live && !pad) return;          // the whole warp shares v
  const uint64_t* row = reinterpret_cast<const uint64_t*>(X) + (live ? v * ld : 0);
  int32_t s;
  if (given) {
    s = live ? shifts[v] : 0;
  } else {
    uint64_t mx = 0;
    uint32_t bad = 0;
    if (live) row_absmax(row, len, lane, 32, mx, bad);
    mx = warp_max_u64(mx);
    bad = __any_sync(0xffffffffu, bad);
    s = live ? shift_from_maxbits(bad ? 0 : mx, T.bits) : 0;
    if (lane == 0) {
      if (bad && flag) atomicOr(flag, 1);
      if (live) shifts[v] = s + (mark && bad ? kBadMark : 0);
    }
  }
  const int64_t plane = nvec_pad * k_pad;
  const bool vec = live && ((reinterpret_cast<uintptr_t>(row) & 15) == 0);
  for (int64_t h0 = (int64_t)lane * 8; h0 < k_pad; h0 += 32 * 8) {
    uint64_t b[8];
    if (vec && h0 + 8 <= len) {
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const ulonglong2 w = ld_dep(reinterpret_cast<const ulonglong2*>(row + h0 + e));
        b[e] = w.x;
        b[e + 1] = w.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) b[e] = (live && h0 + e < len) ? ld_dep(row + h0 + e) : 0ull;
    }
    Pieces<NP> P[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (((b[e] >> 52) & 0x7ff) == 0x7ff) b[e] = 0;
      P[e] = pieces_of<NP>(b[e], s);
    }
    store_residues<kBF16, NP, 8, QT>(T, P, planes, plane, v * k_pad + h0);
  }
}

// (three blocks per SM: 113 us against 130 at 65536 x 256)
template <bool kBF16, int NP, int QT>
__global__ void __launch_bounds__(256, NP > 5 ? 2 : 3) split_rows_warp_kernel(const __grid_constant__ OzTables T, int64_t nvec,
                                                              int64_t len, const double* __restrict__ X, int64_t ld,
                                                              int64_t nvec_pad, int64_t k_pad,
                                                              int32_t* __restrict__ shifts,
                                                              void* __restrict__ planes, int32_t* __restrict__ flag,
                                                              bool given, bool pad) {
  const int64_t v = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  split_row_warp<kBF16, NP, QT>(T, v, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, given, pad);
}

// Grouped, short rows: block b holds rows 8 (b - rows_begin) .. + 7 of its
// problem; map[b] is the problem.
// (three blocks per SM where the registers allow it without spilling)
template <int NP, int QT>
__global__ void __launch_bounds__(256, (QT > 0 && NP == 4) ? 3 : 2) split_rows_warp_grouped_kernel(const __grid_constant__ OzTables T,
                                                                         const OzGroupProblem* __restrict__ probs,
                                                                         const int32_t* __restrict__ map) {
  const int64_t b = blockIdx.x;
  const OzGroupProblem& P = probs[__ldg(map + b)];
  const int64_t v = (b - P.rows_begin) * 8 + (threadIdx.x >> 5);
  split_row_warp<true, NP, QT>(T, v, P.m, P.k, P.A, P.lda, P.m_pad, P.k_pad, P.s, P.U, P.flag, false, false);
}

template <bool kBF16, int NP, int QT>
__global__ void __launch_bounds__(256, 3) split_rows_kernel(const __grid_constant__ OzTables T, int64_t nvec, int64_t len,
                                                         const double* __restrict__ X, int64_t ld,
                                                         int64_t nvec_pad, int64_t k_pad,
                                                         int32_t* __restrict__ shifts, void* __restrict__ planes,
                                                         int32_t* __restrict__ flag, bool given) {
  split_row<kBF16, NP, QT>(T, blockIdx.x, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, given);
}

// Grouped: block b is row b - rows_begin of its problem's A; map[b] is the problem.
template <int NP, int QT>
__global__ void __launch_bounds__(256, (QT > 0 && NP == 4) ? 3 : 2) split_rows_grouped_kernel(const __grid_constant__ OzTables T,
                                                                    const OzGroupProblem* __restrict__ probs,
                                                                    const int32_t* __restrict__ map) {
  const int64_t b = blockIdx.x;
  const OzGroupProblem& P = probs[__ldg(map + b)];
  split_row<true, NP, QT>(T, b - P.rows_begin, P.m, P.k, P.A, P.lda, P.m_pad, P.k_pad, P.s, P.U, P.flag, false);
}

// ---------------------------------------------------------------------------
// Strided vectors (columns of B, or of A^T).
// Pass 1: column maxima by atomicMax into colmax (zeroed by the launcher).
// Block (32 x 8): 32 consecutive columns, 8 warps over rows; each CTA covers
// 256 rows.
// ---------------------------------------------------------------------------
// mark: a non-finite entry sets bit 63 of its column's word instead of the flag.
__device__ __forceinline__ void colmax_block(int64_t bx, int64_t by, int tx, int ty, int64_t nvec, int64_t len,
                                             const double* __restrict__ X, int64_t ld,
                                             uint64_t* __restrict__ colmax, int32_t* __restrict__ flag,
                                             bool mark = false) {
  __shared__ uint64_t red[8][32];
  const int64_t j = bx * 32 + tx;
  const int64_t h0 = by * 256 + ty;
  uint64_t mx = 0;
  uint32_t bad = 0;
  if (j < nvec) {
    const uint64_t* col = reinterpret_cast<const uint64_t*>(X) + j;
    // 32 rows per thread, loads issued together (predicated, no early exit)
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int64_t h = h0 + 8 * i;
      const uint64_t b = h < len ? ld_dep(col + h * ld) & kAbsMask : 0ull;
      bad |= (uint32_t)((b >> 52) == 0x7ff);
      mx = b > mx ? b : mx;
    }
  }
  if (bad && flag) atomicOr(flag, 1);
  red[ty][tx] = bad ? (mark ? 1ull << 63 : 0ull) : mx;
  __syncthreads();
  if (ty == 0 && j < nvec) {
    uint64_t m = 0;
    for (int w = 0; w < 8; ++w) m = red[w][tx] > m ? red[w][tx] : m;
    if (m) atomicMax(reinterpret_cast<unsigned long long*>(colmax + j), (unsigned long long)m);
  }
}

__global__ void __launch_bounds__(256) colmax_kernel(int64_t nvec, int64_t len, const double* __restrict__ X,
                                                     int64_t ld, uint64_t* __restrict__ colmax,
                                                     int32_t* __restrict__ flag) {
  colmax_block(blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, nvec, len, X, ld, colmax, flag);
}

// Grouped: block b is block b - cm_begin of its problem's (ceil(n/32) x
// ceil(k/256)) grid, x fastest; map[b] is the problem.
__global__ void __launch_bounds__(256) colmax_grouped_kernel(const OzGroupProblem* __restrict__ probs,
                                                             const int32_t* __restrict__ map) {
  const int64_t b = blockIdx.x;
  const OzGroupProblem& P = probs[__ldg(map + b)];
  const int64_t l = b - P.cm_begin, nbx = (P.n + 31) / 32;
  colmax_block(l % nbx, l / nbx, threadIdx.x, threadIdx.y, P.n, P.k, P.B, P.ldb, P.colmax, P.flag);
}

__global__ void shifts_from_colmax_kernel(int64_t nvec, const uint64_t* __restrict__ colmax, int beta,
                                          int32_t* __restrict__ shifts) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nvec) shifts[j] = shift_from_maxbits(colmax[j], beta);
}

__global__ void shifts_grouped_kernel(const OzGroupProblem* __restrict__ probs, const int32_t* __restrict__ map,
                                      int beta) {
  const int64_t b = blockIdx.x;
  const OzGroupProblem& P = probs[__ldg(map + b)];
  const int64_t j = (b - P.sh_begin) * blockDim.x + threadIdx.x;
  if (j < P.n) P.t[j] = shift_from_maxbits(P.colmax[j], beta);
}

// Shifts of contiguous vectors without a split (a blocked call takes them over
// the whole row before splitting it slab by slab): one warp per row.
__global__ void __launch_bounds__(256) shifts_rows_kernel(int64_t nvec, int64_t len, const double* __restrict__ X,
                                                          int64_t ld, int beta, int32_t* __restrict__ shifts,
                                                          int32_t* __restrict__ flag) {
  const int64_t v = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (v >= nvec) return;                 // the whole warp shares v
  const uint64_t* row = reinterpret_cast<const uint64_t*>(X) + v * ld;
  uint64_t mx = 0;
  uint32_t bad = 0;
  row_absmax(row, len, lane, 32, mx, bad);
  mx = warp_max_u64(mx);
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    if (bad && flag) atomicOr(flag, 1);
    shifts[v] = shift_from_maxbits(bad ? 0 : mx, beta);
  }
}

// Pass 2: 64 (h) x 64 (vector) tiles; residues go through shared memory so
// that the planes, which are K-major per vector, are written along h.
// Thread t handles vector j = t % 64 and 16 consecutive h.
template <bool kBF16, int NP>
__device__ __forceinline__ void split_cols_block(const OzTables& T, int64_t bx, int64_t by, int64_t nvec,
                                                 int64_t len, const double* __restrict__ X, int64_t ld,
                                                 int64_t nvec_pad, int64_t k_pad,
                                                 const int32_t* __restrict__ shifts, void* __restrict__ planes) {
  constexpr int kPitchWords = kBF16 ? 33 : 17;   // 64 entries + 4 bytes of padding per row
  __shared__ uint32_t tile[2][64 * kPitchWords];
  const int tid = threadIdx.x;
  const int jl = tid & 63;
  const int hg = tid >> 6;                         // 0..3: h = hg*16 .. hg*16+15
  const int64_t j0 = bx * 64;
  const int64_t hbase = by * 64;
  const int64_t j = j0 + jl;
  const bool live = j < nvec;
  const int32_t s = live ? shifts[j] : 0;

  Pieces<NP> P[16];
  const uint64_t* Xb = reinterpret_cast<const uint64_t*>(X);
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    int64_t h = hbase + hg * 16 + e;
    uint64_t b = (live && h < len) ? __ldg(Xb + h * ld + j) : 0ull;
    if (((b >> 52) & 0x7ff) == 0x7ff) b = 0;
    P[e] = pieces_of<NP>(b, s);
  }
  const int Q = T.Q;
  const int64_t plane = nvec_pad * k_pad;
#pragma unroll 1
  for (int q = 0; q < Q; ++q) {
    uint32_t* tb = tile[q & 1];
    const ModConst<NP> mc = mod_const<NP>(T, q);
    float r[16];
    residues_any<NP, 16>(mc, P, r);
    if (q == 2) {                                    // block-uniform branch: the even modulus
#pragma unroll
      for (int e = 0; e < 16; ++e) r[e] = fix_tie(T, r[e]);
    }
    if (kBF16) {
#pragma unroll
      for (int w = 0; w < 8; ++w) tb[jl * kPitchWords + hg * 8 + w] = bf16_pair(r[2 * w], r[2 * w + 1]);
    } else {
#pragma unroll
      for (int w = 0; w < 4; ++w)
        tb[jl * kPitchWords + hg * 4 + w] = int8_quad(r[4 * w], r[4 * w + 1], r[4 * w + 2], r[4 * w + 3]);
    }
    __syncthreads();
    // write 64 rows of 64 entries: int8 -> 4 words of 16 B per row, bf16 -> 8
    constexpr int kChunks = kBF16 ? 8 : 4;          // 16-byte chunks per row
    for (int c = tid; c < 64 * kChunks; c += 256) {
      int row = c / kChunks, ch = c % kChunks;
      if (j0 + row >= nvec_pad) continue;
      uint4 o;
      o.x = tb[row * kPitchWords + ch * 4 + 0];
      o.y = tb[row * kPitchWords + ch * 4 + 1];
      o.z = tb[row * kPitchWords + ch * 4 + 2];
      o.w = tb[row * kPitchWords + ch * 4 + 3];
      const int64_t off = (int64_t)q * plane + (j0 + row) * k_pad + hbase;
      char* dst = static_cast<char*>(planes) + (off * (kBF16 ? 2 : 1)) + ch * 16;
      *reinterpret_cast<uint4*>(dst) = o;
    }
    // tile[q & 1] is rewritten two moduli later, after the next barrier
  }
}

template <bool kBF16, int NP>
__global__ void __launch_bounds__(256) split_cols_kernel(const __grid_constant__ OzTables T, int64_t nvec, int64_t len,
                                                         const double* __restrict__ X, int64_t ld,
                                                         int64_t nvec_pad, int64_t k_pad,
                                                         const int32_t* __restrict__ shifts,
                                                         void* __restrict__ planes) {
  split_cols_block<kBF16, NP>(T, blockIdx.x, blockIdx.y, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes);
}

// bf16 planes (TC engine): tiles of 32 vectors x 64 h. Lane l holds vector
// j0 + l, warp w the eight h = hbase + 8w .. + 7 (each load instruction reads
// 32 consecutive doubles of one row of X). The residues of every modulus are
// staged in shared memory, [q][32 vectors][64 h + 8 pad] bf16 (rows of 144
// bytes: the 16-byte stores and loads of a quarter-warp fall in distinct
// banks), and after one barrier each thread writes one 16-byte run per
// modulus, so the planes (K-major per vector) receive whole 128-byte rows.
constexpr int kColTileJ = 32, kColTileH = 64;
constexpr int kColPitchWords = 36;
constexpr int kColPlaneWords = kColTileJ * kColPitchWords;     // 1152 words = 4608 bytes per modulus

// Lane's eight entries of vector j at h0 .. h0 + 7 (zero past the operand).
__device__ __forceinline__ void load_col8(const uint64_t* Xb, int64_t ld, bool live, int64_t j, int64_t h0,
                                          int64_t len, uint64_t (&b)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) b[e] = (live && h0 + e < len) ? ld_dep(Xb + (h0 + e) * ld + j) : 0ull;
}

// One tile from the entries b of this thread (lane's vector, shift s), vectors
// below nstore.
template <int NP, int QT>
__device__ __forceinline__ void split_cols_entries(const OzTables& T, uint64_t (&b)[8], int32_t s, int64_t j0,
                                                   int64_t hbase, int64_t nstore, int64_t nvec_pad, int64_t k_pad,
                                                   uint16_t* __restrict__ planes, uint32_t* tile) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  Pieces<NP> P[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (((b[e] >> 52) & 0x7ff) == 0x7ff) b[e] = 0;   // non-finite: flagged by the column maxima
    P[e] = pieces_of<NP>(b[e], s);
  }
  const int Q = QT > 0 ? QT : T.Q;
  uint4* const mine = reinterpret_cast<uint4*>(tile + lane * kColPitchWords + 4 * w);
#pragma unroll
  for (int q = 0; q < (QT > 0 ? QT : OZ_MAX_MODULI); ++q) {
    if (QT > 0 || q < Q) {
      const ModConst<NP> mc = mod_const<NP>(T, q);
      float r[8];
      residues_q<NP, 8>(T, q, mc, P, r);
      mine[q * (kColPlaneWords / 4)] =
          make_uint4(bf16_pair(r[0], r[1]), bf16_pair(r[2], r[3]), bf16_pair(r[4], r[5]), bf16_pair(r[6], r[7]));
    }
  }
  __syncthreads();
  // thread t: vector row t / 8 of the tile, 16-byte chunk t % 8 of its 64 h
  const int row = threadIdx.x >> 3, ch = threadIdx.x & 7;
  if (j0 + row < nstore) {
    const int64_t plane = nvec_pad * k_pad;
    uint16_t* dst = planes + (j0 + row) * k_pad + hbase + 8 * ch;
    const uint4* src = reinterpret_cast<const uint4*>(tile + row * kColPitchWords + 4 * ch);
#pragma unroll 4
    for (int q = 0; q < Q; ++q)
      *reinterpret_cast<uint4*>(dst + q * plane) = src[q * (kColPlaneWords / 4)];
  }
}

template <int NP, int QT>
__device__ __forceinline__ void split_cols_tile(const OzTables& T, int64_t j0, int64_t hbase, int64_t nvec,
                                                int64_t len, const double* __restrict__ X, int64_t ld,
                                                int64_t nstore, int64_t nvec_pad, int64_t k_pad,
                                                const int32_t* __restrict__ shifts, uint16_t* __restrict__ planes,
                                                uint32_t* tile) {
  const int64_t j = j0 + (threadIdx.x & 31);
  const bool live = j < nvec;
  const int32_t s = live ? __ldg(shifts + j) : 0;
  uint64_t b[8];
  load_col8(reinterpret_cast<const uint64_t*>(X), ld, live, j, hbase + 8 * (threadIdx.x >> 5), len, b);
  split_cols_entries<NP, QT>(T, b, s, j0, hbase, nstore, nvec_pad, k_pad, planes, tile);
}

template <int NP, int QT>
__global__ void __launch_bounds__(256, NP > 5 ? 2 : 3) split_cols_bf16_kernel(const __grid_constant__ OzTables T, int64_t nvec,
                                                                int64_t len, const double* __restrict__ X, int64_t ld,
                                                                int64_t nstore, int64_t nvec_pad, int64_t k_pad,
                                                                const int32_t* __restrict__ shifts,
                                                                uint16_t* __restrict__ planes) {
  extern __shared__ uint4 col_tile[];
  split_cols_tile<NP, QT>(T, (int64_t)blockIdx.x * kColTileJ, (int64_t)blockIdx.y * kColTileH, nvec, len, X, ld,
                          nstore, nvec_pad, k_pad, shifts, planes, reinterpret_cast<uint32_t*>(col_tile));
}

// Grouped: block b is tile l = b - sc_begin of its problem's
// ceil(n / 32) x (k_pad / 64) grid, vectors fastest; map[b] is its problem.
template <int NP, int QT>
__global__ void __launch_bounds__(256, 3) split_cols_grouped_kernel(const __grid_constant__ OzTables T,
                                                                   const OzGroupProblem* __restrict__ probs,
                                                                   const int32_t* __restrict__ map) {
  extern __shared__ uint4 col_tile[];
  const int64_t b = blockIdx.x;
  const OzGroupProblem& P = probs[__ldg(map + b)];
  const int64_t l = b - P.sc_begin, nbx = (P.n + kColTileJ - 1) / kColTileJ;
  split_cols_tile<NP, QT>(T, (l % nbx) * kColTileJ, (l / nbx) * kColTileH, P.n, P.k, P.B, P.ldb, P.n, P.n_pad, P.k_pad,
                          P.t, static_cast<uint16_t*>(P.V), reinterpret_cast<uint32_t*>(col_tile));
}

// ---------------------------------------------------------------------------
// Both operands of a product together (oz_dgemm, bf16 planes).
//   Contiguous vectors: a block per row, or a warp per row when rows are
//     short, as the kernels above.
//   Strided vectors of at most kStripMaxK entries: a cluster of kStripCtas
//     blocks per strip of 32 vectors. Block r of the cluster holds the strip's
//     64-entry tiles r, r + kStripCtas, ...; it scans them for the maxima, the
//     blocks exchange these through distributed shared memory, and each then
//     splits its tiles (the last one from registers). No scratch, no second
//     launch: with the dependent launches, a 256^3 product in 28-30 us instead of
//     47 (19 since the call's host path was shortened too).
//   Longer strided vectors: a pass for the column maxima, then 32 x 64 tiles
//     with the shifts formed from them. (A block's tiles of a strip would run
//     one after another, with two barriers each: at 4096 the shared launch takes
//     189 us longer than the rows alone, the separate kernels for B 141 us.)
// The passes of a small product share one launch; those of a larger one with
// k_pad up to 1024 are launched one after another, since a shared launch costs
// the rows L1 (65536 x 256 rows beside a 256 x 256 B: 150 us against 121 us).
// Larger products of longer vectors, or of more than kStripEntries strided
// entries, keep the separate kernels above, and launches past kMergeEntries are
// in plain stream order (65536 x 256 x 256 with both operands transposed: 420 us
// with separate kernels, 577 in strips, 514 before either; with neither
// transposed 382 us in strips, 393 apart; 4096 x 4096 x 512 358 either way). In
// long products (split_both_suits) the launches are nothing, and ld.global.nc and plain
// launches are worth 0.8 % of an 8192^3 product.
// ---------------------------------------------------------------------------
struct SplitSide {
  const double* X;
  int64_t ld, nvec, nvec_pad;
  int32_t* shifts;
  uint16_t* planes;
  uint64_t* colmax;      // kSideTile: zeroed before the first launch
  int kind;              // kSideRow, kSideWarp, kSideStrip or kSideTile
  int blocks1, blocks2;  // rows and strips (a multiple of kStripCtas) or maxima; tiles
};
constexpr int kSideRow = 0, kSideWarp = 1, kSideStrip = 2, kSideTile = 3, kSideAny = -1;
constexpr int kStripCtas = 8;
constexpr int64_t kStripMaxK = 1024;
constexpr int64_t kStripEntries = (int64_t)2 << 20;   // of the strided operands of a larger product
constexpr int64_t kMergeEntries = (int64_t)4 << 20;   // of both operands: up to which their passes share a launch

template <int NP, int QT>
__device__ __forceinline__ void split_strip(const OzTables& T, const SplitSide& S, int64_t strip, int64_t len,
                                            int64_t k_pad, uint32_t* tile) {
  __shared__ uint64_t red[8][32];
  __shared__ uint64_t cmax[32];            // this block's column maxima, bit 63: a non-finite entry
  __shared__ int32_t sh[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t rank = cluster_rank();
  const int64_t j0 = strip * kColTileJ, j = j0 + lane;
  const bool live = j < S.nvec;
  const uint64_t* Xb = reinterpret_cast<const uint64_t*>(S.X);
  const int ntiles = (int)(k_pad / kColTileH);
  const int last = ntiles > (int)rank ? (int)rank + (ntiles - 1 - (int)rank) / kStripCtas * kStripCtas : -1;
  uint64_t b[8];
  uint64_t mx = 0, bad = 0;
  for (int i = (int)rank; i < ntiles; i += kStripCtas) {
    load_col8(Xb, S.ld, live, j, (int64_t)i * kColTileH + 8 * w, len, b);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint64_t a = b[e] & kAbsMask;
      bad |= (uint64_t)((a >> 52) == 0x7ff) << 63;
      mx = a > mx ? a : mx;
    }
  }
  red[w][lane] = mx | bad;
  __syncthreads();
  if (w == 0) {
    uint64_t m = 0, f = 0;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint64_t x = red[v][lane];
      f |= x & ~kAbsMask;
      m = (x & kAbsMask) > m ? (x & kAbsMask) : m;
    }
    cmax[lane] = m | f;
  }
  cluster_sync();
  if (w == 0) {
    uint64_t m = 0, f = 0;
#pragma unroll
    for (int r = 0; r < kStripCtas; ++r) {
      uint64_t x;
      asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(x) : "r"(mapa(smem_u32(&cmax[lane]), (uint32_t)r)) : "memory");
      f |= x & ~kAbsMask;
      m = (x & kAbsMask) > m ? (x & kAbsMask) : m;
    }
    const int32_t s = shift_from_maxbits(f ? 0 : m, T.bits);
    sh[lane] = s;
    if (rank == 0 && live) S.shifts[j] = s + (f ? kBadMark : 0);
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // done with the other blocks' maxima
  const int32_t s = sh[lane];
  for (int i = last; i >= 0; i -= kStripCtas) {
    if (i != last) load_col8(Xb, S.ld, live, j, (int64_t)i * kColTileH + 8 * w, len, b);
    split_cols_entries<NP, QT>(T, b, s, j0, (int64_t)i * kColTileH, S.nvec, S.nvec_pad, k_pad, S.planes, tile);
    if (i >= kStripCtas) __syncthreads();            // the tile is read before the next one is staged
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // no block leaves while its maxima may be read
}

__device__ __forceinline__ void colmax_side(const SplitSide& S, int64_t l, int64_t len) {
  const int64_t nbx = (S.nvec + 31) / 32;
  colmax_block(l % nbx, l / nbx, threadIdx.x & 31, threadIdx.x >> 5, S.nvec, len, S.X, S.ld, S.colmax, nullptr, true);
}

// Blocks of side b, then side a (status: cleared, when not null).
// KIND: the kind of every side, kSideWarp; kSideAny: each its own.
template <int NP, int QT, int KIND>
__global__ void __launch_bounds__(256, KIND == kSideAny && NP > 5 ? 2 : 3) split_both_kernel(
    const __grid_constant__ OzTables T, const __grid_constant__ SplitSide a, const __grid_constant__ SplitSide b,
    int64_t len, int64_t k_pad, int32_t* __restrict__ status) {
  extern __shared__ uint4 col_tile[];
  pdl_wait();
  pdl_trigger();
  if (status && blockIdx.x == 0 && threadIdx.x < 4) status[threadIdx.x] = 0;
  const bool second = (int)blockIdx.x < b.blocks1;
  const SplitSide& S = second ? b : a;
  const int64_t l = second ? blockIdx.x : (int)blockIdx.x - b.blocks1;
  const int kind = KIND == kSideAny ? S.kind : KIND;
  if (kind == kSideStrip)
    split_strip<NP, QT>(T, S, l / kStripCtas, len, k_pad, reinterpret_cast<uint32_t*>(col_tile));
  else if (kind == kSideTile)
    colmax_side(S, l, len);
  else if (kind == kSideWarp)
    split_row_warp<true, NP, QT>(T, l * 8 + (threadIdx.x >> 5), S.nvec, len, S.X, S.ld, S.nvec_pad, k_pad, S.shifts,
                                 S.planes, nullptr, false, false, true);
  else if (l < S.nvec)
    split_row<true, NP, QT>(T, l, S.nvec, len, S.X, S.ld, S.nvec_pad, k_pad, S.shifts, S.planes, nullptr, false, true);
}

// The tiles of the kSideTile sides, vectors fastest.
template <int NP, int QT>
__global__ void __launch_bounds__(256, NP > 5 ? 2 : 3) split_tiles_kernel(const __grid_constant__ OzTables T,
                                                             const __grid_constant__ SplitSide a,
                                                             const __grid_constant__ SplitSide b, int64_t len,
                                                             int64_t k_pad) {
  extern __shared__ uint4 col_tile[];
  const bool second = (int)blockIdx.x < b.blocks2;
  const SplitSide& S = second ? b : a;
  const int l = second ? blockIdx.x : (int)blockIdx.x - b.blocks2;
  const int nbx = (int)((S.nvec + kColTileJ - 1) / kColTileJ);
  const int64_t j0 = (int64_t)(l % nbx) * kColTileJ, hbase = (int64_t)(l / nbx) * kColTileH;
  const int64_t j = j0 + (threadIdx.x & 31);
  const bool live = j < S.nvec;
  pdl_wait();
  pdl_trigger();
  uint64_t v[8];
  load_col8(reinterpret_cast<const uint64_t*>(S.X), S.ld, live, j, hbase + 8 * (threadIdx.x >> 5), len, v);
  const uint64_t m = live ? ld_dep(S.colmax + j) : 0ull;
  const int32_t s = shift_from_maxbits(m >> 63 ? 0ull : m, T.bits);
  if (hbase == 0 && live && threadIdx.x < 32) S.shifts[j] = s + (m >> 63 ? kBadMark : 0);
  split_cols_entries<NP, QT>(T, v, s, j0, hbase, S.nvec, S.nvec_pad, k_pad, S.planes,
                             reinterpret_cast<uint32_t*>(col_tile));
}

// Transpose of a rows x cols block of doubles (row pitch ld) into cols x rows
// (row pitch rows), through 32 x 33 shared tiles: reads and writes both
// coalesced. Lets the column vectors of B be split as rows.
__global__ void __launch_bounds__(256) transpose_kernel(int64_t rows, int64_t cols, const double* __restrict__ X,
                                                        int64_t ld, double* __restrict__ Y) {
  __shared__ double tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;    // 32 x 8 threads
  const int64_t ctiles = (cols + 31) / 32;                   // block b: tile (b / ctiles, b % ctiles)
  const int64_t c0 = ((int64_t)blockIdx.x % ctiles) * 32, r0 = ((int64_t)blockIdx.x / ctiles) * 32;
#pragma unroll
  for (int i = 0; i < 32; i += 8) {
    const int64_t r = r0 + ty + i, c = c0 + tx;
    if (r < rows && c < cols) tile[ty + i][tx] = __ldg(X + r * ld + c);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 32; i += 8) {
    const int64_t c = c0 + ty + i, r = r0 + tx;
    if (r < rows && c < cols) Y[c * rows + r] = tile[tx][ty + i];
  }
}

// Rows v in [nvec, nvec_pad) of the strided layout are covered by the grid
// (grid.x spans nvec_pad), so no separate padding pass is needed.

}  // namespace

namespace {

// pieces per entry for a bit budget: 22 bits and three or four of 13 bits,
// or 22 bits and six of 12 (widened operands)
int pieces_for(int bits) { return bits <= 61 ? 4 : bits <= 64 ? 5 : 7; }

template <bool kBF16, int NP, int QT>
void split_rows_qt(const OzTables& t, int64_t nvec, int64_t len, const double* X, int64_t ld, int64_t nvec_pad,
                   int64_t k_pad, int32_t* shifts, void* planes, int32_t* flag, cudaStream_t st, bool given,
                   bool pad) {
  const int64_t rows = pad ? nvec_pad : nvec;
  if (k_pad <= 1024)                             // short rows: one warp per row
    split_rows_warp_kernel<kBF16, NP, QT><<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(
        t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, given, pad);
  else
    split_rows_kernel<kBF16, NP, QT><<<(unsigned)rows, 256, 0, st>>>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts,
                                                                          planes, flag, given);
}

// Q = 16 (the paper's INT8 configuration) with the modulus count fixed at
// compile time; other counts read it from the table
template <bool kBF16, int NP>
void split_rows_np(const OzTables& t, int64_t nvec, int64_t len, const double* X, int64_t ld, int64_t nvec_pad,
                   int64_t k_pad, int32_t* shifts, void* planes, int32_t* flag, cudaStream_t st, bool given,
                   bool pad) {
  if (t.Q == 16)
    split_rows_qt<kBF16, NP, 16>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad);
  else
    split_rows_qt<kBF16, NP, 0>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad);
}

template <int NP, int QT>
cudaError_t split_cols_bf16_qt(const OzTables& t, int64_t nvec, int64_t len, const double* X, int64_t ld,
                               int64_t nvec_pad, int64_t k_pad, const int32_t* shifts, void* planes, cudaStream_t st,
                               bool pad) {
  const int64_t nstore = pad ? nvec_pad : nvec;
  const int smem = (QT > 0 ? QT : t.Q) * kColPlaneWords * 4;
  cudaError_t e = cudaFuncSetAttribute(split_cols_bf16_kernel<NP, QT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (QT > 0 ? QT : OZ_MAX_MODULI) * kColPlaneWords * 4);
  if (e != cudaSuccess) return e;
  dim3 g((unsigned)((nstore + kColTileJ - 1) / kColTileJ), (unsigned)(k_pad / kColTileH));
  split_cols_bf16_kernel<NP, QT><<<g, 256, smem, st>>>(t, nvec, len, X, ld, nstore, nvec_pad, k_pad, shifts,
                                                       static_cast<uint16_t*>(planes));
  return cudaGetLastError();
}

template <bool kBF16, int NP>
cudaError_t split_cols_np(const OzTables& t, int64_t nvec, int64_t len, const double* X, int64_t ld, int64_t nvec_pad,
                          int64_t k_pad, const int32_t* shifts, void* planes, cudaStream_t st, bool pad) {
  if constexpr (kBF16) {
    if constexpr (NP <= 5)
      if (t.Q == 16) return split_cols_bf16_qt<NP, 16>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
    return split_cols_bf16_qt<NP, 0>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
  } else {
    dim3 g((unsigned)(nvec_pad / 64), (unsigned)(k_pad / 64));
    split_cols_kernel<kBF16, NP><<<g, 256, 0, st>>>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes);
    return cudaGetLastError();
  }
}

}  // namespace

namespace {

template <int NP, int QT>
cudaError_t split_both_qt(const OzTables& t, const SplitSide& a, const SplitSide& b, int64_t len, int64_t k_pad,
                          int32_t* status, cudaStream_t st) {
  const int tile = t.Q * kColPlaneWords * 4;
  for (auto kernel : {(const void*)split_both_kernel<NP, QT, kSideAny>, (const void*)split_tiles_kernel<NP, QT>}) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (QT > 0 ? QT : OZ_MAX_MODULI) * kColPlaneWords * 4);
    if (e != cudaSuccess) return e;
  }
  for (const SplitSide* s : {&a, &b})
    if (s->kind == kSideTile) {
      cudaError_t e = cudaMemsetAsync(s->colmax, 0, 8 * (size_t)s->nvec, st);
      if (e != cudaSuccess) return e;
    }
  cudaError_t e = cudaSuccess;
  const bool small = (a.nvec_pad + b.nvec_pad) * k_pad <= kMergeEntries;
  // one launch of the sides x, y (either may be empty)
  auto first = [&](SplitSide x, SplitSide y) {
    if (e != cudaSuccess || x.blocks1 + y.blocks1 == 0) return;
    const bool strips = (x.blocks1 && x.kind == kSideStrip) || (y.blocks1 && y.kind == kSideStrip);
    const bool warps = (!x.blocks1 || x.kind == kSideWarp) && (!y.blocks1 || y.kind == kSideWarp);
    e = launch_kernel(small, warps ? split_both_kernel<NP, QT, kSideWarp> : split_both_kernel<NP, QT, kSideAny>,
                      dim3((unsigned)(x.blocks1 + y.blocks1)), dim3(256), strips ? (size_t)tile : 0, st,
                      strips ? kStripCtas : 1, t, x, y, len, k_pad, status);
    status = nullptr;
  };
  if (small || (a.kind == kSideWarp && b.kind == kSideWarp)) {
    first(a, b);
  } else {
    const SplitSide none = {};
    first(none, b);
    first(a, none);
  }
  if (e != cudaSuccess || a.blocks2 + b.blocks2 == 0) return e;
  return launch_kernel(small, split_tiles_kernel<NP, QT>, dim3((unsigned)(a.blocks2 + b.blocks2)), dim3(256),
                       (size_t)tile, st, 1, t, a, b, len, k_pad);
}

SplitSide split_side(const SplitOperand& o, int64_t len, int64_t k_pad) {
  SplitSide s = {};
  s.X = o.X;
  s.ld = o.ld;
  s.nvec = o.nvec;
  s.nvec_pad = o.nvec_pad;
  s.shifts = o.shifts;
  s.planes = static_cast<uint16_t*>(o.planes);
  s.colmax = o.colmax;
  s.kind = o.contiguous ? (k_pad <= 1024 ? kSideWarp : kSideRow) : k_pad <= kStripMaxK ? kSideStrip : kSideTile;
  s.blocks2 = 0;
  switch (s.kind) {
    case kSideRow: s.blocks1 = (int)round_up(o.nvec, kStripCtas); break;
    case kSideWarp: s.blocks1 = (int)round_up((o.nvec + 7) / 8, kStripCtas); break;
    case kSideStrip: s.blocks1 = (int)((o.nvec + kColTileJ - 1) / kColTileJ) * kStripCtas; break;
    default:
      s.blocks1 = (int)((o.nvec + 31) / 32 * ((len + 255) / 256));
      s.blocks2 = (int)((o.nvec + kColTileJ - 1) / kColTileJ * (k_pad / kColTileH));
  }
  return s;
}

}  // namespace

bool split_both_suits(int64_t m_pad, int64_t n_pad, int64_t k_pad, bool a_strided, bool b_strided) {
  const int64_t strided = (a_strided ? m_pad : 0) + (b_strided ? n_pad : 0);
  return (m_pad + n_pad) * k_pad <= kMergeEntries || (k_pad <= kStripMaxK && strided * k_pad <= kStripEntries);
}

cudaError_t launch_split_both(const OzTables& t, const SplitOperand& A, const SplitOperand& B, int64_t len,
                              int64_t k_pad, int32_t* status, cudaStream_t st) {
  // block counts fit an int
  if ((A.nvec_pad + B.nvec_pad) / kColTileJ * (k_pad / kColTileH) > INT32_MAX || A.nvec_pad + B.nvec_pad > INT32_MAX / 2)
    return cudaErrorInvalidValue;
  const SplitSide a = split_side(A, len, k_pad), b = split_side(B, len, k_pad);
  switch (pieces_for(t.bits)) {
    case 4:
      return t.Q == 16 ? split_both_qt<4, 16>(t, a, b, len, k_pad, status, st)
                       : split_both_qt<4, 0>(t, a, b, len, k_pad, status, st);
    case 5: return split_both_qt<5, 0>(t, a, b, len, k_pad, status, st);
    default: return split_both_qt<7, 0>(t, a, b, len, k_pad, status, st);
  }
}

cudaError_t launch_split_rows(const OzTables& t, int64_t nvec, int64_t len, const double* X, int64_t ld,
                              int64_t nvec_pad, int64_t k_pad, int32_t* shifts, void* planes, int bf16,
                              int32_t* flag, cudaStream_t st, bool given, bool pad) {
  if (nvec_pad == 0 || (nvec == 0 && !pad)) return cudaSuccess;
  switch (pieces_for(t.bits) * 2 + (bf16 ? 1 : 0)) {
    case 9: split_rows_np<true, 4>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad); break;
    case 8: split_rows_np<false, 4>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad); break;
    case 11: split_rows_np<true, 5>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad); break;
    case 10: split_rows_np<false, 5>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad); break;
    case 15: split_rows_np<true, 7>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad); break;
    default: split_rows_np<false, 7>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, flag, st, given, pad); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_transpose(int64_t rows, int64_t cols, const double* X, int64_t ld, double* Y, cudaStream_t st) {
  if (rows == 0 || cols == 0) return cudaSuccess;
  const int64_t tiles = ((cols + 31) / 32) * ((rows + 31) / 32);
  if (tiles > INT32_MAX) return cudaErrorInvalidValue;
  transpose_kernel<<<(unsigned)tiles, 256, 0, st>>>(rows, cols, X, ld, Y);
  return cudaGetLastError();
}

cudaError_t launch_shifts_cols(int bits, int64_t nvec, int64_t len, const double* X, int64_t ld, int32_t* shifts,
                               int32_t* flag, uint64_t* colmax, cudaStream_t st) {
  if (nvec == 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(colmax, 0, sizeof(uint64_t) * (size_t)nvec, st);
  if (e != cudaSuccess) return e;
  if (len > 0) {
    dim3 g1((unsigned)((nvec + 31) / 32), (unsigned)((len + 255) / 256));
    colmax_kernel<<<g1, dim3(32, 8), 0, st>>>(nvec, len, X, ld, colmax, flag);
  }
  shifts_from_colmax_kernel<<<(unsigned)((nvec + 255) / 256), 256, 0, st>>>(nvec, colmax, bits, shifts);
  return cudaGetLastError();
}

cudaError_t launch_shifts_rows(int bits, int64_t nvec, int64_t len, const double* X, int64_t ld, int32_t* shifts,
                               int32_t* flag, cudaStream_t st) {
  if (nvec == 0) return cudaSuccess;
  shifts_rows_kernel<<<(unsigned)((nvec + 7) / 8), 256, 0, st>>>(nvec, len, X, ld, bits, shifts, flag);
  return cudaGetLastError();
}

cudaError_t launch_split_cols(const OzTables& t, int64_t nvec, int64_t len, const double* X, int64_t ld,
                              int64_t nvec_pad, int64_t k_pad, int32_t* shifts, void* planes, int bf16,
                              int32_t* flag, uint64_t* colmax, cudaStream_t st, bool given, bool pad) {
  if (nvec_pad == 0 || (nvec == 0 && !pad)) return cudaSuccess;
  if (!given) {
    cudaError_t e0 = launch_shifts_cols(t.bits, nvec, len, X, ld, shifts, flag, colmax, st);
    if (e0 != cudaSuccess) return e0;
  }
  switch (pieces_for(t.bits) * 2 + (bf16 ? 1 : 0)) {
    case 9: return split_cols_np<true, 4>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
    case 8: return split_cols_np<false, 4>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
    case 11: return split_cols_np<true, 5>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
    case 10: return split_cols_np<false, 5>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
    case 15: return split_cols_np<true, 7>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
    default: return split_cols_np<false, 7>(t, nvec, len, X, ld, nvec_pad, k_pad, shifts, planes, st, pad);
  }
}

// Long rows (one block per row, total_rows blocks, problems in map_rows) and
// short rows (eight per block, total_wrows blocks, map_wrows); each range has
// its own rows_begin numbering. The map entries index probs.
cudaError_t launch_split_rows_grouped(const OzTables& t, const OzGroupProblem* probs, const GroupMaps& maps,
                                      int64_t total_rows, int64_t total_wrows, cudaStream_t st) {
  if (total_rows > INT32_MAX || total_wrows > INT32_MAX || t.bits > 64) return cudaErrorInvalidValue;
  auto launch = [&](auto np, auto qt) {
    constexpr int NP = decltype(np)::value, QT = decltype(qt)::value;
    if (total_rows > 0)
      split_rows_grouped_kernel<NP, QT><<<(unsigned)total_rows, 256, 0, st>>>(t, probs, maps.rows);
    if (total_wrows > 0)
      split_rows_warp_grouped_kernel<NP, QT><<<(unsigned)total_wrows, 256, 0, st>>>(t, probs, maps.wrows);
  };
  using I4 = std::integral_constant<int, 4>;
  using I5 = std::integral_constant<int, 5>;
  if (t.bits <= 61) {   // 22 bits and three 13-bit pieces
    if (t.Q == 16) launch(I4{}, std::integral_constant<int, 16>{});
    else if (t.Q == 15) launch(I4{}, std::integral_constant<int, 15>{});
    else launch(I4{}, std::integral_constant<int, 0>{});
  } else {
    launch(I5{}, std::integral_constant<int, 0>{});
  }
  return cudaGetLastError();
}

// column maxima, shifts and split of the B operands (colmax zeroed by the caller)
cudaError_t launch_split_cols_grouped(const OzTables& t, const OzGroupProblem* probs, const GroupMaps& maps,
                                      int64_t total_cm, int64_t total_sh, int64_t total_sc, cudaStream_t st) {
  if (total_cm > INT32_MAX || total_sh > INT32_MAX || total_sc > INT32_MAX || t.bits > 64) return cudaErrorInvalidValue;
  if (total_cm > 0) colmax_grouped_kernel<<<(unsigned)total_cm, dim3(32, 8), 0, st>>>(probs, maps.cm);
  if (total_sh > 0) shifts_grouped_kernel<<<(unsigned)total_sh, 256, 0, st>>>(probs, maps.sh, t.bits);
  if (total_sc == 0) return cudaGetLastError();
  auto launch = [&](auto np, auto qt) {
    constexpr int NP = decltype(np)::value, QT = decltype(qt)::value;
    const int smem = (QT > 0 ? QT : t.Q) * kColPlaneWords * 4;
    cudaError_t e = cudaFuncSetAttribute(split_cols_grouped_kernel<NP, QT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (QT > 0 ? QT : OZ_MAX_MODULI) * kColPlaneWords * 4);
    if (e != cudaSuccess) return e;
    split_cols_grouped_kernel<NP, QT><<<(unsigned)total_sc, 256, smem, st>>>(t, probs, maps.sc);
    return cudaGetLastError();
  };
  using I4 = std::integral_constant<int, 4>;
  using I5 = std::integral_constant<int, 5>;
  if (t.bits <= 61) {
    if (t.Q == 16) return launch(I4{}, std::integral_constant<int, 16>{});
    if (t.Q == 15) return launch(I4{}, std::integral_constant<int, 15>{});
    return launch(I4{}, std::integral_constant<int, 0>{});
  }
  return launch(I5{}, std::integral_constant<int, 0>{});
}

}  // namespace oz
