// Two-phase hybrid step of the float32 form with the streaming kernel's sums
// (lsa_stream.cuh): the same basis and products to the last bit, in flat passes
// of plain 16-byte loads.
//
// The streaming kernel reads the basis once a step, but its tasks are a chain
// (stage, projection, barrier, stencil and inner products of the plane before)
// on one CTA per SM, and it projects every tile's halo again.  Where a basis is
// short or small, reading it twice with nothing between the loads is faster
// (the figures are at strip_grid in lsa_api.cu):
//
//   pass A    x_j = a w_{j-1} - sum_c c_c x_c, four points a thread, the columns
//             in the streaming kernel's four chains (c mod 4), stored; barrier;
//   pass B1   w_j = A x_j, four points a thread, stored; barrier;
//   pass B2   inner products.  A warp takes two rows of the planes of one rank
//             (the tiles of one CTA of the streaming kernel) in order, a lane
//             a quad of four points and columns c, c + 4 nq, ..., so that every
//             Kahan sum has its terms in the streaming kernel's order.  (CTAs
//             that shared a rank's columns instead of its rows were a fifth of
//             the pass apart.)
//
// Pass A goes through the points backwards, so that the passes after it, which
// go forwards, start on what it left in L2.  Pass A runs at 5.6 TB/s (256^3),
// pass B2 at 3.8: its order leaves a lane the loads of a few planes at a time,
// whose sums wait for them.  Products and sums are packed float32 pairs, which
// took pass B2 from 440 to 390 us; a second batch of planes in flight spills.
#pragma once

#include "lsa_ordered.cuh"
#include "lsa_stream.cuh"

namespace lsa {

template <class Op>
struct StripPass : OrderedPass<Op> {
  using Base = OrderedPass<Op>;
  using Stream = StreamEngine<Op>;
  using E = typename Base::E;
  using Base::e;
  using Base::e0;
  using Base::e1;
  using Base::G0;
  static constexpr int KU = 8;                 // column slots of a thread in one walk over the planes
  struct Buf {
    typename Base::Buf base;
    double wred[NW][2][SQ_NG * KU];          // a warp's inner products
  };
  __host__ __device__ static constexpr size_t smem_bytes() { return Base::offset() + sizeof(Buf); }

  double (*wred)[2][SQ_NG * KU];
  int nq;                // warps that share a block's columns: a power of two, 8 / nq ranks a unit
  int units;             // units of pass B2

  __device__ StripPass(E& en, Buf& bu, int ranks) : Base(en, bu.base), wred(bu.wred) {
    G0 = min(ranks, e.gsize);
    nq = 1;
    while (nq < NW && (2 * nq * G0 + NW - 1) / NW * NW <= e.gsize) nq *= 2;
    units = (nq * G0 + NW - 1) / NW * NW;
    e.nrows = units;
  }

  __device__ __forceinline__ static float4 ld4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ static void axpy(float4& x, float c, const float4& v) {
    x.x = fmaf(c, v.x, x.x); x.y = fmaf(c, v.y, x.y); x.z = fmaf(c, v.z, x.z); x.w = fmaf(c, v.w, x.w);
  }

  // x = a src - sum_c coef_c V_c in four chains of columns c = g, g + 4, ..., added in pairs
  // (StreamEngine::proj_quad_n, quad_sum).
  __device__ void project4(int nc, float a, const float* src, float* xout) {
    const long long N = e.P.op.N, n4 = N / 4;
    const float* V = reinterpret_cast<const float*>(e.P.V);
    const long long chunks = (n4 + NT - 1) / NT;
    for (long long ch = chunks - 1 - e.grank; ch >= 0; ch -= e.gsize) {
      const long long q = ch * NT + e.tid;
      if (q >= n4) continue;
      const float* Vq = V + 4 * q;
      float4 x[SQ_NG];
      const float4 s = ld4(src + 4 * q);
      x[0] = make_float4(a * s.x, a * s.y, a * s.z, a * s.w);
      x[1] = x[2] = x[3] = make_float4(0.f, 0.f, 0.f, 0.f);
      int c = 0;
      auto block = [&](auto cn, auto chain) {        // CN columns, their loads before their FMAs
        constexpr int CN = decltype(cn)::value, G = decltype(chain)::value;
        float4 v[CN];
#pragma unroll
        for (int i = 0; i < CN; ++i) v[i] = ld4(Vq + (long long)(c + i) * N);
#pragma unroll
        for (int i = 0; i < CN; ++i) axpy(x[(G + i) & 3], -e.S.coefc[c + i], v[i]);
        c += CN;
      };
      using std::integral_constant;
#pragma unroll 1
      while (c + 8 <= nc) block(integral_constant<int, 8>(), integral_constant<int, 0>());
      const int rest = nc - c;
      if (rest & 4) block(integral_constant<int, 4>(), integral_constant<int, 0>());
      if (rest & 2) block(integral_constant<int, 2>(), integral_constant<int, 0>());
      if (rest & 1) {
        if (rest & 2) block(integral_constant<int, 1>(), integral_constant<int, 2>());
        else block(integral_constant<int, 1>(), integral_constant<int, 0>());
      }
      float4 o;
      o.x = (x[0].x + x[1].x) + (x[2].x + x[3].x);
      o.y = (x[0].y + x[1].y) + (x[2].y + x[3].y);
      o.z = (x[0].z + x[1].z) + (x[2].z + x[3].z);
      o.w = (x[0].w + x[1].w) + (x[2].w + x[3].w);
      *reinterpret_cast<float4*>(xout + 4 * q) = o;
    }
  }

  // w = A x (OrderedPass::stencil's values), four consecutive points of a row a thread.
  __device__ void stencil4(const float* x, float* w) {
    const DevOp& d = e.P.op;
    const int n4 = (int)(d.N / 4), nxy = d.nx * d.ny;
    for (int g = e.grank * NT + e.tid; g < n4; g += e.gsize * NT) {
      const int q = 4 * g, r = q / d.nx, ix = q - r * d.nx;
      int iy = r, iz = 0;
      float4 zm = make_float4(0.f, 0.f, 0.f, 0.f), zp = zm, f = zm;
      if constexpr (Op::DIM == 3) {
        iz = r / d.ny;
        iy = r - iz * d.ny;
        zm = ldx(x + (iz == 0 ? q + (d.nz - 1) * nxy : q - nxy));
        zp = ldx(x + (iz == d.nz - 1 ? q - (d.nz - 1) * nxy : q + nxy));
      }
      const float4 c = ldx(x + q), s = ldx(x + (iy == 0 ? q + (d.ny - 1) * d.nx : q - d.nx)),
                   n = ldx(x + (iy == d.ny - 1 ? q - (d.ny - 1) * d.nx : q + d.nx));
      const float west = x[ix == 0 ? q + d.nx - 1 : q - 1], east = x[ix + 4 == d.nx ? q + 4 - d.nx : q + 4];
      if constexpr (Op::NF == 1) f = __ldg(reinterpret_cast<const float4*>(d.g0 + q));
      float4 o;
      o.x = point(zm.x, s.x, west, c.x, c.y, n.x, zp.x, f.x);
      o.y = point(zm.y, s.y, c.x, c.y, c.z, n.y, zp.y, f.y);
      o.z = point(zm.z, s.z, c.y, c.z, c.w, n.z, zp.z, f.z);
      o.w = point(zm.w, s.w, c.z, c.w, east, n.w, zp.w, f.w);
      *reinterpret_cast<float4*>(w + q) = o;
    }
  }
  __device__ __forceinline__ static float4 ldx(const float* p) { return *reinterpret_cast<const float4*>(p); }
  __device__ __forceinline__ float point(float below, float south, float west, float c, float east, float north,
                                         float above, float f) const {
    const float c5[5] = {south, west, c, east, north};
    float zm[3] = {0.f, 0.f, below}, zp[3] = {0.f, 0.f, above}, out[1];
    Op::template apply_f<float, 2, 5>(this->b.cf, zm, c5, zp, 2, f, 0.f, out);
    return out[0];
  }

  // Unit u: block u % 8 (two rows, eight quads) of the planes of ranks (8 / nq) (u / 8) + 0, 1, ..., one after the
  // other in x as a rule, so that a unit reads longer runs of memory than one tile's rows.  Its inner products of x
  // and w with the column slots k0 .. k0 + nk - 1 (nk <= K), and with `self` x.x, x.w, w.w (w null: x.x alone, no
  // columns).  Warp: rank (8 / nq) (u / 8) + warp / nq, columns c0 + 4 nq k with c0 = lane group + 4 (warp % nq).
  template <int K>
  struct Sums {                              // Kahan sums of the columns' products with x and w, in pairs
    unsigned long long s[K], c[K];
    float self[3], selfc[3];
  };
  template <int K>
  struct Place {                             // where a lane is in its rank's planes
    int r, ti, z, ZS, nxy, at, base;
    const float *x, *w, *V;
    long long step;
    bool on[K];
  };
  template <int K, int NP>
  struct Planes {
    float4 x[NP], w[NP], v[NP][K];
  };
  template <int K, int NP>
  __device__ __forceinline__ void load(Place<K>& l, Planes<K, NP>& b) const {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      if (l.z == l.ZS) { l.z = 0; l.base = this->tile(l.r, ++l.ti).base + l.at; }
      const int i = l.base + l.nxy * l.z;
      ++l.z;
      b.x[p] = ld4(l.x + i);
      b.w[p] = ld4(l.w + i);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        b.v[p][k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (l.on[k]) b.v[p][k] = ld4(l.V + k * l.step + i);
      }
    }
  }
  template <int K, int NP>
  __device__ __forceinline__ static void add(Sums<K>& f, const Planes<K, NP>& b, bool self, int g) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const float4 xq = b.x[p], wq = b.w[p];
      const unsigned long long xlo = Stream::pack2(xq.x, xq.y), xhi = Stream::pack2(xq.z, xq.w);
      const unsigned long long wlo = Stream::pack2(wq.x, wq.y), whi = Stream::pack2(wq.z, wq.w);
#pragma unroll
      for (int k = 0; k < K; ++k) {            // (v0 x0 + v2 x2) + (v1 x1 + v3 x3)
        const unsigned long long lo = Stream::pack2(b.v[p][k].x, b.v[p][k].y);
        const unsigned long long hi = Stream::pack2(b.v[p][k].z, b.v[p][k].w);
        const float2 tx = Stream::unpack2(Stream::ffma2(hi, xhi, Stream::fmul2(lo, xlo)));
        const float2 tw = Stream::unpack2(Stream::ffma2(hi, whi, Stream::fmul2(lo, wlo)));
        kahan2(f.s[k], f.c[k], Stream::pack2(tx.x + tx.y, tw.x + tw.y));
      }
      if (self) {                              // point g of the quad
        const float xg = g == 0 ? xq.x : g == 1 ? xq.y : g == 2 ? xq.z : xq.w;
        const float wg = g == 0 ? wq.x : g == 1 ? wq.y : g == 2 ? wq.z : wq.w;
        E::kahan(f.self[0], f.selfc[0], xg * xg);
        E::kahan(f.self[1], f.selfc[1], xg * wg);
        E::kahan(f.self[2], f.selfc[2], wg * wg);
      }
    }
  }
  __device__ __forceinline__ static unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
  }
  // Kahan sums of a pair of values at once (s the sums, nc the negated compensations): Engine::kahan's roundings.
  __device__ __forceinline__ static void kahan2(unsigned long long& s, unsigned long long& nc, unsigned long long v) {
    const unsigned long long minus = 0xbf800000bf800000ULL;
    const unsigned long long y = add2(v, nc), t = add2(s, y);
    nc = Stream::ffma2(Stream::ffma2(s, minus, t), minus, y);        // y - (t - s)
    s = t;
  }
  template <int K>
  __device__ __forceinline__ void walk(int unit, int k0, int nk, int nd, bool self, const float* x, const float* w,
                                       double* part) {
    const DevOp& d = e.P.op;
    const long long N = d.N;
    const int sub = e.warp % nq, q = (unit % NW) * 8 + (e.lane & 7), g = e.lane >> 3;
    const int r = (NW / nq) * (unit / NW) + e.warp / nq, np = r < G0 ? this->planes(r) : 0;
    const int ZS = this->zs(), nxy = d.nx * d.ny, at = (q & 3) * 4 + d.nx * (q >> 2);
    const int cstep = SQ_NG * nq, c0 = g + SQ_NG * sub + cstep * k0;
    const long long vstep = N * cstep;
    const float* V = reinterpret_cast<const float*>(e.P.V) + c0 * N;
    const bool selves = self;
    self = self && sub == 0;
    Sums<K> f;
    Place<K> pl;
    pl.r = r; pl.ti = -1; pl.z = pl.ZS = ZS; pl.nxy = nxy; pl.at = at;
    pl.x = x; pl.w = w ? w : x; pl.V = V; pl.step = vstep;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      f.s[k] = f.c[k] = 0ull;
      pl.on[k] = k < nk && c0 + cstep * k < nd;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) f.self[i] = f.selfc[i] = 0.f;
    constexpr int NP = K <= 2 ? 4 : K <= 3 ? 3 : K <= 6 ? 2 : 1;     // planes in flight
    int left = np;
#pragma unroll 1
    for (; left >= NP; left -= NP) {
      Planes<K, NP> a;
      load(pl, a);
      add(f, a, self, g);
    }
    if constexpr (NP > 1) {
#pragma unroll 1
      for (; left > 0; --left) {
        Planes<K, 1> a;
        load(pl, a);
        add(f, a, self, g);
      }
    }
    __syncthreads();                           // (an earlier range's reads of wred)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float2 sum = Stream::unpack2(f.s[k]), neg = Stream::unpack2(f.c[k]);
      float s = sum.x, se = neg.x, t = sum.y, te = neg.y;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const float os = __shfl_xor_sync(0xffffffffu, s, o), ose = __shfl_xor_sync(0xffffffffu, se, o);
        const float ot = __shfl_xor_sync(0xffffffffu, t, o), ote = __shfl_xor_sync(0xffffffffu, te, o);
        float es, et;
        s = two_sum(s, os, es);
        se = (se + ose) + es;
        t = two_sum(t, ot, et);
        te = (te + ote) + et;
      }
      if ((e.lane & 7) == 0) {
        wred[e.warp][0][SQ_NG * k + g] = (double)s + (double)se;
        wred[e.warp][1][SQ_NG * k + g] = (double)t + (double)te;
      }
    }
    if (self) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double s = Base::comp_sum(f.self[i], -f.selfc[i]);
        if (e.lane == 0) e.S.bred[e.warp][i] = s;
      }
    }
    __syncthreads();
    for (int t = e.tid; t < 2 * cstep * nk; t += NT) {
      const int kind = t & 1, s = t >> 1, k = s / cstep, cs = s - k * cstep, c = cstep * k0 + s;
      if (c >= nd) continue;
      double acc = 0.0;
      for (int i = cs / SQ_NG; i < NW; i += nq) acc += wred[i][kind][SQ_NG * k + cs % SQ_NG];
      part[kind * nd + c] = acc;
    }
    if (selves && e.tid < 3) {
      double acc = 0.0;
      for (int i = 0; i < NW; i += nq) acc += e.S.bred[i][e.tid];
      part[2 * nd + e.tid] = acc;
    }
  }
  __device__ int sums(int nd, const float* x, const float* w) {
    if (e.grank >= units) return 2 * nd + 3;
    const int kn = (nd + SQ_NG * nq - 1) / (SQ_NG * nq);
    double* part = e.part_row();
    int k0 = 0;
    do {
      const int nk = min(KU, kn - k0);
      switch (nk) {
        case 8: case 7: walk<8>(e.grank, k0, nk, nd, k0 == 0, x, w, part); break;
        case 6: walk<6>(e.grank, k0, nk, nd, k0 == 0, x, w, part); break;
        case 5: walk<5>(e.grank, k0, nk, nd, k0 == 0, x, w, part); break;
        case 4: walk<4>(e.grank, k0, nk, nd, k0 == 0, x, w, part); break;
        case 3: walk<3>(e.grank, k0, nk, nd, k0 == 0, x, w, part); break;
        case 2: walk<2>(e.grank, k0, nk, nd, k0 == 0, x, w, part); break;
        default: walk<1>(e.grank, k0, nk, nd, k0 == 0, x, w, part);
      }
      k0 += KU;
    } while (k0 < kn);
    return 2 * nd + 3;
  }

  // Alg. 4 (StreamEngine::run_hybrid, pass for pass; column 0 holds the start vector).
  __device__ void run() {
    const ArnoldiParams& P = e.P;
    float* V = reinterpret_cast<float*>(P.V);
    float* Wb[2] = {reinterpret_cast<float*>(P.W0), reinterpret_cast<float*>(P.W1)};
    const long long N = P.op.N;
    const int m = P.m;
    if (e.tid == 0) { e.S.a = 1.f; e.S.done = 0; e.S.fallback_pending = 0; e.S.syncs_c = 0; }
    __syncthreads();
    for (int j = 1; j <= m; ++j) {
      float* x = V + (long long)(j - 1) * N;
      if (j > 1) {
        project4(j - 1, e.S.a, Wb[(j - 1) & 1], x);
        if (!e.sync_only()) return;
      }
      stencil4(x, Wb[j & 1]);
      if (!this->barrier()) return;
      if (!e.reduce_all(sums(j - 1, x, Wb[j & 1]), [&] { e.hybrid_step(j); })) return;
      if (e.S.done) return;
      if (e.S.fallback_pending) {     // explicit norm of the projected vector (in the buffer of w_{j-1}, now free)
        if (!norm_pass(j, Wb[j & 1], Wb[(j - 1) & 1], [&] { e.hybrid_fallback_finish(j); })) return;
        if (e.S.done) return;
      }
    }
    norm_pass(m, Wb[m & 1], V + (long long)m * N, [&] { e.hybrid_final_finish(); });
  }
  template <class Fn>
  __device__ bool norm_pass(int nc, const float* src, float* xout, Fn fn) {
    project4(nc, e.S.a, src, xout);
    if (!this->barrier()) return false;
    if (e.grank < units) walk<1>(e.grank, 0, 0, 0, true, xout, nullptr, e.part_row());
    return e.reduce_all(3, fn);
  }
};

template <class Op>
__global__ void __launch_bounds__(NT, 2) k_arnoldi_strip(ArnoldiParams P, int ranks) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using F = StripPass<Op>;
  using E = typename F::E;
  E e(P, *reinterpret_cast<typename E::Smem*>(smem_raw), reinterpret_cast<double*>(smem_raw + E::small_offset()));
  e.redundant_steps();
  F f(e, *reinterpret_cast<typename F::Buf*>(smem_raw + F::offset()), ranks);
  f.run();
}

// `ranks`: the CTAs that the streaming kernel would have.
template <class Op>
cudaError_t launch_arnoldi_strip_t(const ArnoldiParams& P, int G, int ranks, cudaStream_t s) {
  ArnoldiParams Pc = P;
  void* args[2] = {&Pc, &ranks};
  auto k = k_arnoldi_strip<Op>;
  const size_t sm = StripPass<Op>::smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel((void*)k, dim3(G), dim3(NT), args, sm, s);
}

// Resident CTAs per SM.
template <class Op>
int strip_blocks_per_sm_t() {
  int nb = 0;
  auto k = k_arnoldi_strip<Op>;
  const size_t sm = StripPass<Op>::smem_bytes();
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, NT, sm) != cudaSuccess) return 0;
  return nb;
}

}  // namespace lsa
