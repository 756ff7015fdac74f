// ig_fixed.cuh -- sums of doubles in integer arithmetic: every addend becomes a 64-bit fixed-point number
// whose scale is the largest addend's exponent, the integers are added exactly, and the total is rounded
// once. Any order of the additions gives the same bits.
//
// An FP64 instruction occupies its SM sub-partition for 64 cycles, so a tree over a warp and the warps
// after it took some 9 of those, one after another, to add a value over 152 tiles; the integer sum of a
// warp is one maximum, four additions by redux and some forty integer instructions, whatever the
// number of addends per lane. In the resident solve (ig_resident.cu): 5,917 rows, k = 1, 8.3 -> 6.3 us an
// iteration, 66,049 rows, k = 1, 8.3 -> 7.4 us.
//
// Error: an addend is cut below 2^-62 of the largest one, so 160 addends lose less than 2^-54 of it: less
// than one FP64 addition rounds.
#pragma once

#include <cuda_runtime.h>

namespace ig {
namespace {

__device__ __forceinline__ unsigned exponent_bits(double v) { return (unsigned)__double2hiint(v) & 0x7ff00000u; }

// v in units of 2^-62 of the power of two of exponent bits `top` (at least those of v, and `fixed_range`:
// a zero or a denormal, taken as of exponent 0, is then cut to 0).
__device__ __forceinline__ long long fixed_point(double v, unsigned top) {
  const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
  const unsigned long long m =
      ((unsigned long long)(__funnelshift_l(l, h, 11) | 0x80000000u) << 32) | (unsigned long long)(l << 11);
  unsigned long long f;
  asm("shr.u64 %0, %1, %2;" : "=l"(f) : "l"(m), "r"(((top - (h & 0x7ff00000u)) >> 20) + 1u));  // 0 from 64 on
  const long long s = (long long)((int)h >> 31);
  return ((long long)f ^ s) - s;
}
__device__ __forceinline__ bool fixed_range(unsigned top) { return top >= (64u << 20) && top < 0x7ff00000u; }

// The double nearest to t * 2^32 + l in units of 2^(field - 1023 - 95); ok is cleared when that is none of
// normal size.
__device__ __forceinline__ double nearest_double(long long t, unsigned l, int field, bool& ok) {
  const unsigned s = (unsigned)(int)(t >> 63);
  unsigned h = (unsigned)(int)(t >> 32) ^ s, m = (unsigned)t ^ s;
  l ^= s;
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (h == 0u) {
      h = m;
      m = l;
      l = 0u;
      field -= 32;
    }
  if (h == 0u) return 0.0;
  const int c = __clz((int)h);
  field -= c;
  ok = ok && field >= 1 && field <= 2045;
  const unsigned mh = __funnelshift_l(m, h, c), ml = __funnelshift_l(l, m, c);
  const unsigned long long r = ((((unsigned long long)mh << 32) | ml) >> 11) + (unsigned long long)((ml >> 10) & 1u);
  const unsigned long long b = ((unsigned long long)(unsigned)(field - 1) << 52) + r;
  return __longlong_as_double((long long)(b | ((unsigned long long)(s & 0x80000000u) << 32)));
}

__device__ __forceinline__ double warp_sum_fp64(double a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// A lane's addends; a warp's have to be 65,535 at most (the uppermost limb).
struct FixedSum {
  long long h = 0;           // upper words
  unsigned long long l = 0;  // lower words
  __device__ __forceinline__ void add(double v, unsigned top) {
    const long long f = fixed_point(v, top);
    h += f >> 32;
    l += (unsigned)f;
  }
  // the sum over the warp as four 16-bit limbs with room for carries (the uppermost is signed)
  __device__ __forceinline__ void warp_limbs(unsigned (&s)[4]) const {
    const long long t = h + (long long)(l >> 32);
    s[0] = __reduce_add_sync(0xffffffffu, (unsigned)l & 0xffffu);
    s[1] = __reduce_add_sync(0xffffffffu, (unsigned)l >> 16);
    s[2] = __reduce_add_sync(0xffffffffu, (unsigned)t & 0xffffu);
    s[3] = (unsigned)__reduce_add_sync(0xffffffffu, (int)(t >> 16));
  }
  __device__ static __forceinline__ double from_limbs(const unsigned (&s)[4], unsigned top, bool& ok) {
    const unsigned long long a = s[0] + ((unsigned long long)s[1] << 16);
    const long long t = (long long)(a >> 32) + (long long)s[2] + (long long)(int)s[3] * 65536;
    return nearest_double(t, (unsigned)a, (int)(top >> 20) + 33, ok);
  }
};

// The sum of v[0..J) over the lanes of a warp, on every lane. Addends out of the fixed-point range (tiny
// ones only, or an infinity or a NaN) are added in FP64.
template <int J>
__device__ __forceinline__ double warp_sum_fixed(const double (&v)[J]) {
  unsigned top = 0u, any = 0u;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    top = max(top, exponent_bits(v[j]));
    any |= ((unsigned)__double2hiint(v[j]) << 1) | (unsigned)__double2loint(v[j]);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  bool ok = fixed_range(top);
  double a = 0.0;
  if (ok) {
    FixedSum f;
#pragma unroll
    for (int j = 0; j < J; ++j) f.add(v[j], top);
    unsigned s[4];
    f.warp_limbs(s);
    a = FixedSum::from_limbs(s, top, ok);
  }
  if (!ok) {
    if (!__any_sync(0xffffffffu, any != 0u)) return 0.0;
    a = 0.0;
#pragma unroll
    for (int j = 0; j < J; ++j) a += v[j];
    a = warp_sum_fp64(a);
  }
  return a;
}

}  // namespace
}  // namespace ig
