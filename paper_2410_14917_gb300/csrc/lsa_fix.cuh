// Float64 inner products on the integer pipe (block fixed point).
//
// GB300 issues 2 float64 FMAs per clock and SM but 64 32 x 32 + 64-bit integer
// multiply-adds (measured: 1.99 against 63.6 lanes/clk/SM), so the inner
// products V_c . x and V_c . w of a hybrid step -- two thirds of its float64
// work -- run as exact integer sums.  A block of values (up to 256, the piece of
// a vector that one warp sums; of the single-cluster kernel the CTA's tile) is
// scaled by a power of two S that its Euclidean norm stays below (to 6 %), and
// each value rounded to 58 bits below S and cut into two limbs,
//     v = (vh 2^28 + vl) S 2^-58,   |vh| <= 2^30,  -2^27 <= vl < 2^27.
// A product takes three multiply-adds,
//     vh xh 2^56 + (vh xl + vl xh) 2^28
// (and for x . x and x . w of the vector's own block a fourth, vl xl: those of
// x . x all have one sign), summed exactly over the lane's points and over the
// warp's lanes, then added in float64 once per block.  By Cauchy and Schwarz no
// partial sum of the products exceeds 1.13 2^116, so the sums of vh xh stay
// below 2^61 whatever the values.
//
// Error of a block's sum, in units of Sv Sx (at most 8 |v| |x|; 3 for uniform
// values): rounding of the values 2^-60 each, vl xl left out 2^-59.6, a lane's
// sum rounded to 2^-60 once 2^-59.3 over the warp.  That is 2^-58.5 Sv Sx, below
// half a float64 rounding unit of |v| |x|, for a peak over a background as for
// values of one size, and summed over the blocks of a vector the same of its
// norms.  Float64 FMA chains round every partial sum.  Blocks by their largest
// value instead of their norm, one per share of a vector and without any vl xl,
// lost 2^-42 of |x|^2 for a peak over a background of 1e-4 on 192^3.
// On uniform data the orthogonality of the basis is that of float64 products
// (Gray-Scott 512^2, m = 32, 24 start vectors: 1.3e-14 and 1.5e-14 in the mean).
// The blocks' scales, the rounding and the fourth product cost 1 to 5 % of a
// call (ADR 256^3 53.8 to 55.2 ms, 64 x 64 in the cluster kernel 345 to 358 us).
// Infinities and NaNs give finite garbage here; w . w, kept in float64, carries
// them to the step's checks.
#pragma once

#include "lsa_internal.cuh"

namespace lsa {

// |v| as an integer key: the high word without its sign (its biased exponent is the key >> 20).
__device__ __forceinline__ unsigned fx_key(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// A block's shift base is (biased exponent of S + 4) << 20 | 0xfffff; (base - key(v)) >> 20 then is the number of
// mantissa bits of v that lie below 59 bits under S.  0 stands for a block of zeros and subnormal values.
// k: the block's largest key; q: the sum of fx_square over its values.
__device__ __forceinline__ unsigned fx_base(unsigned k, unsigned q) {
  const int b = 32 - __clz((int)(q - 1));                             // ceil(log2 q), q >= 2^21
  return k < 0x100000u ? 0u : (((k >> 20) + 5u + (unsigned)((b - 21) >> 1)) << 20) | 0xfffffu;
}
// 2^22 (v / 2^(E(k) + 1))^2 to the power of two next to it (E the exponent): at most twice and at least 0.89 times as
// much; values eleven exponents below the largest count as zero.
__device__ __forceinline__ unsigned fx_square(double v, unsigned k) {
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(1u << 22), "r"(((k | 0xfffffu) - fx_key(v)) >> 19));   // beyond 31: 0
  return r;
}
// The shift bases of the blocks of the warp's lanes' values x and w.
template <int V>
__device__ __forceinline__ void fx_blocks(const double (&x)[V], const double (&w)[V], unsigned& bx, unsigned& bw) {
  unsigned kx = 0, kw = 0, qx = 0, qw = 0;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    kx = max(kx, fx_key(x[i]));
    kw = max(kw, fx_key(w[i]));
  }
  kx = __reduce_max_sync(0xffffffffu, kx);
  kw = __reduce_max_sync(0xffffffffu, kw);
#pragma unroll
  for (int i = 0; i < V; ++i) {
    qx += fx_square(x[i], kx);
    qw += fx_square(w[i], kw);
  }
  qx = __reduce_add_sync(0xffffffffu, qx);
  qw = __reduce_add_sync(0xffffffffu, qw);
  bx = fx_base(kx, qx);
  bw = fx_base(kw, qw);
}
template <int V>
__device__ __forceinline__ unsigned fx_block(const double (&v)[V]) {
  unsigned k = 0, q = 0;
#pragma unroll
  for (int i = 0; i < V; ++i) k = max(k, fx_key(v[i]));
  k = __reduce_max_sync(0xffffffffu, k);
#pragma unroll
  for (int i = 0; i < V; ++i) q += fx_square(v[i], k);
  return fx_base(k, __reduce_add_sync(0xffffffffu, q));
}

// The two limbs of v, rounded to nearest, in a block of shift base `base`.  Zeros and subnormal values keep an
// implicit leading one, which the shift removes unless the whole block is below 2^-960, where products underflow.
__device__ __forceinline__ void fx_split(double v, unsigned base, int& h, int& l) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;      // mantissa with its leading one at bit 63
  const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 11);
  unsigned long long t;                                               // 59 bits below S
  asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"((base - fx_key(v)) >> 20));   // shifts beyond 63 give 0
  const int sg = ((int)hi >> 31) | 1;
  h = (int)((t + (1ULL + (1ULL << 28))) >> 29) * sg;                  // balanced: vl's top bit is carried into it
  l = ((int)((unsigned)t * 8u + 8u) >> 4) * sg;
}

// Sums of the products of a lane's limbs of a column (h, l) with those of x and w, in units of 2^56 limb units.
// self: the column is x, and the products of the low limbs count too.
template <int VL>
__device__ __forceinline__ void fx_dot(const int (&h)[VL], const int (&l)[VL], const int (&xh)[VL], const int (&xl)[VL],
                                       const int (&wh)[VL], const int (&wl)[VL], bool self, long long& tx, long long& tw) {
  static_assert(VL <= 8, "a block has 256 values at most");
  long long xx = 0, xc = 1LL << 27, ww = 0, wc = 1LL << 27;
#pragma unroll
  for (int k = 0; k < VL; ++k) {
    xx += (long long)h[k] * xh[k];
    xc += (long long)h[k] * xl[k];
    xc += (long long)l[k] * xh[k];
    ww += (long long)h[k] * wh[k];
    wc += (long long)h[k] * wl[k];
    wc += (long long)l[k] * wh[k];
  }
  if (self) {
    long long xs = 0, ws = 0;
#pragma unroll
    for (int k = 0; k < VL; ++k) {
      xs += (long long)l[k] * xl[k];
      ws += (long long)l[k] * wl[k];
    }
    xc += xs >> 28;
    wc += ws >> 28;
  }
  tx = xx + (xc >> 28);
  tw = ww + (wc >> 28);
}

// S 2^-30 of a block of shift base b: half the scale of a product's sum, so that neither half leaves the range of
// float64 before the product does.
__device__ __forceinline__ double fx_scale(unsigned b) {
  const int e = (int)(b >> 20) - 34;                                  // biased exponent
  if (b == 0) return 0.0;
  return e > 0 ? __hiloint2double(e << 20, 0) : __longlong_as_double(1LL << (51 + e));
}

// A sum of products (fx_dot's units) of blocks with the shift bases bv and bx.  It underflows where the float64
// products would: the squares of a start vector of 1e-150 count.  (One multiplication as a rule: pass B's stencil
// keeps the float64 unit busy.)
__device__ __forceinline__ double fx_value(long long sum, unsigned bv, unsigned bx) {
  const int w = (int)(bv >> 20) + (int)(bx >> 20) - (2 * 34 + 1023);   // biased exponent of the sum's unit
  if (w < 1 || w > 2046) return (double)sum * fx_scale(min(bv, bx)) * fx_scale(max(bv, bx));
  return (double)sum * __hiloint2double(w << 20, 0);
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
