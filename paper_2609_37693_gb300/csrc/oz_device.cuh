// oz_device.cuh -- device helpers shared by the kernels: the IEEE-field view
// of eq. convert (split kernels, INT8 and float-format planes) and the
// modular byte sum of the blocked call's epilogues.
#pragma once

#include <stdint.h>

namespace oz {

constexpr uint64_t kAbsMask = 0x7fffffffffffffffull;

// Shift s from the largest |x| bit pattern.
static __device__ __forceinline__ int32_t shift_from_maxbits(uint64_t mb, int beta) {
  if (mb == 0) return 0;
  int eb = (int)(mb >> 52);
  int e = eb ? eb - 1022 : (64 - __clzll((long long)mb)) - 1074;  // frexp exponent
  return beta - e;
}

// Programmatic dependent launch: a kernel launched dependent (launch_kernel in
// oz_launch.h, which names these kernels) may start while the kernel before it on
// the stream is still running. Each of them therefore waits here, before its first
// access to global memory, until that kernel has finished and its writes are
// visible, and then lets its own successor be scheduled. Both are no-ops after a
// plain launch, the only one that kernels without the wait may have.
static __device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
static __device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A load of what an earlier kernel of the stream may have written: an ordinary
// one, which stays below pdl_wait. (ld.global.nc wants its data unwritten for
// the kernel's whole life, part of which a dependent launch spends beside its
// predecessor; so no __ldg, and no const __restrict__ kernel parameter.)
template <typename T>
static __device__ __forceinline__ T ld_dep(const T* p) {
  return *p;
}

// The mark of a vector that holds a non-finite entry: oz_dgemm's split adds it
// to the vector's shift (shifts lie within about +-1200), and the GEMM
// kernel takes it off again and sets bit 0 of the status word. The split can
// so clear the status word itself instead of a memset ahead of it.
constexpr int32_t kBadMark = 1 << 24;

// Thread `tid` of `threads`: unmark the shifts of both operands.
static __device__ __forceinline__ void unmark_shifts(int32_t* __restrict__ s, int m, int32_t* __restrict__ t, int n,
                                                     int32_t* status, int tid, int threads) {
  for (int i = tid; i < m + n; i += threads) {
    int32_t* p = i < m ? s + i : t + (i - m);
    const int32_t v = *p;
    if (v > kBadMark / 2) {
      *p = v - kBadMark;
      atomicOr(status, 1);
    }
  }
}

// Decoded truncated integer of one entry: |a'| and its sign.
struct Trunc {
  uint64_t mag;
  uint32_t neg;
};

static __device__ __forceinline__ Trunc truncate(uint64_t bits, int32_t s) {
  Trunc t;
  t.neg = (uint32_t)(bits >> 63);
  int eb = (int)((bits >> 52) & 0x7ff);
  uint64_t f = bits & ((1ull << 52) - 1);
  uint64_t mant = eb ? (f | (1ull << 52)) : f;
  int sh = (eb ? eb - 1075 : -1074) + s;   // a' = mant * 2^sh, |a'| < 2^beta <= 2^64
  if (sh >= 0) t.mag = mant << sh;         // sh <= 11 when beta <= 64 (wider: truncate_wide)
  else t.mag = (-sh) >= 64 ? 0ull : (mant >> (-sh));
  return t;
}

// The same for a widened budget (beta up to 84): |a'| < 2^84 needs 128 bits.
struct TruncWide {
  unsigned __int128 mag;
  uint32_t neg;
};

static __device__ __forceinline__ TruncWide truncate_wide(uint64_t bits, int32_t s) {
  TruncWide t;
  t.neg = (uint32_t)(bits >> 63);
  int eb = (int)((bits >> 52) & 0x7ff);
  uint64_t f = bits & ((1ull << 52) - 1);
  uint64_t mant = eb ? (f | (1ull << 52)) : f;
  int sh = (eb ? eb - 1075 : -1074) + s;   // a' = mant * 2^sh, |a'| < 2^beta <= 2^84
  if (sh >= 0) t.mag = (unsigned __int128)mant << sh;   // sh <= 31
  else t.mag = (-sh) >= 64 ? 0 : (unsigned __int128)(mant >> (-sh));
  return t;
}

// 64-bit max across a warp.
static __device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    uint64_t w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// The largest |x| bit pattern over row[h], h = t, t + step, ... (t < step),
// and whether any of those entries is not finite: 16-byte loads (two
// entries) when the row is 16-byte aligned, four of them in flight per
// iteration, so that a short row's maximum is not a chain of load latencies.
static __device__ __forceinline__ void row_absmax(const uint64_t* row, int64_t len, int t, int step,
                                           uint64_t& mx, uint32_t& bad) {
  auto fold = [&](uint64_t b) {
    b &= kAbsMask;
    bad |= (uint32_t)((b >> 52) == 0x7ff);
    mx = b > mx ? b : mx;
  };
  if ((reinterpret_cast<uintptr_t>(row) & 15) == 0) {
    const ulonglong2* r2 = reinterpret_cast<const ulonglong2*>(row);
    const int64_t np = len >> 1;
    int64_t p = t;
    for (; p + 3 * (int64_t)step < np; p += 4 * (int64_t)step) {
      ulonglong2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = ld_dep(r2 + p + u * step);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        fold(v[u].x);
        fold(v[u].y);
      }
    }
    for (; p < np; p += step) {
      const ulonglong2 v = ld_dep(r2 + p);
      fold(v.x);
      fold(v.y);
    }
    if ((len & 1) && t == 0) fold(ld_dep(row + len - 1));
  } else {
    for (int64_t h = t; h < len; h += step) fold(ld_dep(row + h));
  }
}

// (a + b) mod m in each byte, for bytes a, b in [0, m) and m < 256 given as
// mm = m * 0x01010101: a - (m - b), plus m in the bytes where that borrows.
// The GEMM epilogues of a blocked call add a slab's digits into the earlier
// slabs' this way.
static __device__ __forceinline__ uint32_t addmod_bytes(uint32_t a, uint32_t b, uint32_t mm) {
  const uint32_t c = __vsub4(mm, b);
  const uint32_t lt = __vcmpltu4(a, c);
  return __vadd4(__vsub4(a, c), lt & mm);
}

}  // namespace oz
