// Float64 inner products on the integer pipe (block fixed point).
//
// GB300 issues 2 float64 FMAs per clock and SM but 64 32 x 32 + 64-bit integer
// multiply-adds (measured: 1.99 against 63.6 lanes/clk/SM), so the inner
// products V_c . x and V_c . w of a hybrid step -- two thirds of its float64
// work -- run as exact integer sums.  A block of values is scaled by the power
// of two of its largest magnitude and each value cut into two limbs,
//     v = (vh 2^32 + vl) 2^(E - 58),   |vh| <= 2^27,  -2^31 <= vl < 2^31
// (E the exponent of the block's largest magnitude: 59 bits below it; a float64
// product of it rounds at 2^-54 of it).  A product takes three multiply-adds,
//     vh xh 2^64 + (vh xl + vl xh) 2^32
// (vl xl, of either sign and below 2^-56 of the largest product, is left out),
// summed exactly over a lane's points of a piece and over the warp's lanes
// (below 2^62) and then added in float64 once per piece.  So an inner product
// sees one float64 rounding per 32 lanes x points of a piece instead of two per
// value: its error is below that of float64 FMA chains.  The blocks: of a basis
// column, the CTA's share of it (its largest magnitude is kept from the pass
// that wrote it); of x and w, the piece.  Infinities and NaNs give finite
// garbage here; w . w, kept in float64, carries them to the step's checks.
#pragma once

#include "lsa_internal.cuh"

namespace lsa {

// |v| as an integer key: the high word without its sign (its exponent is the key >> 20).
__device__ __forceinline__ unsigned fx_key(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// The block's shift base: (base - key(v)) >> 20 is 5 plus the exponents between v and the block's largest.
__device__ __forceinline__ unsigned fx_base(unsigned maxkey) { return (maxkey | 0xfffffu) + (5u << 20); }

// The two limbs of v in a block of shift base `base` (floor of the scaled value).  Zeros and subnormal values
// keep an implicit leading one, which the shift removes unless the whole block is below 2^-960.
__device__ __forceinline__ void fx_split(double v, unsigned base, int& h, int& l) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;      // mantissa with its leading one at bit 63
  const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 11);
  unsigned long long s;
  asm("shr.u64 %0, %1, %2;" : "=l"(s) : "l"(m), "r"((base - fx_key(v)) >> 20));   // shifts beyond 63 give 0
  const unsigned sg = (unsigned)((int)hi >> 31);
  l = (int)((unsigned)s ^ sg);                                        // balanced: its top bit is carried into h
  h = (int)((unsigned)(s >> 32) ^ sg) + (int)((unsigned)l >> 31);
}

// As fx_split for the x and w of a piece, whose zeros give exactly 0.
__device__ __forceinline__ void fx_split0(double v, unsigned base, int& h, int& l) {
  fx_split(v, base, h, l);
  if (fx_key(v) < 0x100000u) h = l = 0;
}

// 2^(E - 26) for a block of largest key k: half the scale of a product's sum, so that neither half leaves the range
// of float64 before the product does.  0 for a block of zeros and subnormal values.
__device__ __forceinline__ double fx_scale(unsigned k) {
  const int e = (int)(k >> 20) - 26;                                  // biased exponent
  if (k < 0x100000u) return 0.0;
  return e > 0 ? __hiloint2double(e << 20, 0) : __longlong_as_double(1LL << (51 + e));
}

// sum 2^(Ev + Ex - 52): a sum of products (in units of 2^64 limb units) of blocks with the largest keys kv and
// kx.  It underflows where the float64 products would: the squares of a start vector of 1e-150 count.
__device__ __forceinline__ double fx_value(long long sum, unsigned kv, unsigned kx) {
  return (double)sum * fx_scale(min(kv, kx)) * fx_scale(max(kv, kx));
}

// Warp sums of NV 64-bit integers at once (warp_sum_many's scheme): lane l gets the sum of value
// l >> (5 - log2 NV).
template <int NV>
__device__ __forceinline__ long long warp_sum_many_s64(long long (&v)[NV]) {
  const unsigned lane = threadIdx.x & 31u;
  int s = 16;
#pragma unroll
  for (int h = NV / 2; h >= 1; h >>= 1, s >>= 1) {
    const bool up = (lane & (unsigned)s) != 0u;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const long long send = up ? v[i] : v[i + h];
      const long long keep = up ? v[i + h] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  long long r = v[0];
#pragma unroll
  for (; s >= 1; s >>= 1) r += __shfl_xor_sync(0xffffffffu, r, s);
  return r;
}

}  // namespace lsa
