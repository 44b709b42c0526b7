// Two-phase hybrid step of the float32 form over the tiles' planes, with every
// sum in the order of the tile passes (Engine::run_hybrid, step form 1): the
// same basis, H and products to the last bit, on all SMs.
//
// The tile passes give each CTA whole tile columns, so a grid of few tile
// columns (75 x 50 x 41: 20) leaves most SMs idle and walks its planes one after
// another, three barriers and two round trips to L2 each (160 us a step there).
// Their sums are Kahan sums per lane and column of runs of eight products, one
// run a plane (a 2D tile is one plane).  Here the runs of a chunk of planes are
// formed in parallel (warps take planes) and only the Kahan additions go plane
// by plane (warps take columns, from shared memory):
//
//   pass A    x_j on equal flat shares, stored; grid barrier;
//   pass B1   w_j = A x_j on the same shares, stored; grid barrier;
//   pass B2   units of one tile-pass CTA ("rank": the tiles r, r + G0, ...) and
//             up to sixteen columns, or of one rank's self terms.
//
// Every pass is bound by the loads in flight: pass A issues 32 of a thread
// before their FMAs (with one point a thread and the last columns one by one it
// took 1.25 times as long), pass B2 four columns of a plane.  Sixteen columns a
// unit, so that x and w are read again once every sixteen columns.  A step of
// 75 x 50 x 41 (m = 20) takes 22 us, of which the passes are 8, the barriers 8
// and the reduction and step function the rest.
#pragma once

#include <type_traits>

#include "lsa_engine.cuh"

namespace lsa {

template <class Op>
struct OrderedPass {
  using E = Engine<Op, float, float, false, false>;
  static_assert(Op::NS == 1, "the single-species operators");
  static constexpr int K = NT / 32;          // points of a lane and plane
  static constexpr int CG = 16, PCH = 16;    // columns of a unit at most, planes of their chunk

  struct Buf {
    float2 run[CG * PCH * 32];               // [column][plane][lane]: runs of a chunk
    Coef<float> cf;
  };
  __host__ __device__ static constexpr size_t offset() { return (E::smem_bytes() + 127) & ~(size_t)127; }
  __host__ __device__ static constexpr size_t smem_bytes() { return offset() + sizeof(Buf); }

  E& e;
  Buf& b;
  long long e0, e1;      // this CTA's share of the points (passes A and B1)
  int G0;                // ranks: the CTAs of the tile passes
  unsigned rtx;          // 2^32 / tiles_x, rounded down

  __device__ OrderedPass(E& en, Buf& bu) : e(en), b(bu) {
    const long long N = e.P.op.N;
    long long per = (N + e.gsize - 1) / e.gsize;
    per = (per + 31) & ~31LL;
    e0 = min(N, (long long)e.grank * per);
    e1 = min(N, e0 + per);
    G0 = min(e.gsize, e.P.tl.ntiles);
    rtx = e.P.tl.tiles_x > 1 ? (unsigned)((1ULL << 32) / e.P.tl.tiles_x) : 0xffffffffu;
    e.nrows = G0;
    if (e.tid == 0) b.cf = e.cf;
    __syncthreads();
  }

  // x = a src - sum_c coef_c V_c on the share, stored (Engine::project_flat's operations for every value:
  // eight columns at a time, two alternating accumulators).  U points of a thread: 8 U loads in flight.
  template <int U>
  __device__ __forceinline__ void project_points(long long q0, int nc, float a, bool unit, const double* src64,
                                                 const float* src, float* xout) {
    constexpr int CB = 8;
    const long long N = e.P.op.N;
    const float* V = reinterpret_cast<const float*>(e.P.V) + q0;
    float x[U], xb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      x[u] = src64 ? (float)__ldg(src64 + q0 + u * NT) : __ldcg(src + q0 + u * NT);
      if (!unit) x[u] = a * x[u];
      xb[u] = 0.f;
    }
    int c = 0;
    auto block = [&](auto cn) {              // CN columns, their loads before their FMAs
      constexpr int CN = decltype(cn)::value;
      float v[CN][U];
#pragma unroll
      for (int i = 0; i < CN; ++i)
#pragma unroll
        for (int u = 0; u < U; ++u) v[i][u] = __ldcg(V + (long long)(c + i) * N + u * NT);
#pragma unroll
      for (int i = 0; i < CN; ++i) {
        const float cc = e.S.coefc[c + i];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (CN == CB && (i & 1)) xb[u] = fma(-cc, v[i][u], xb[u]);
          else x[u] = fma(-cc, v[i][u], x[u]);
        }
      }
      c += CN;
    };
#pragma unroll 1
    while (c + CB <= nc) block(std::integral_constant<int, CB>());
    const int rest = nc - c;
    if (rest & 4) block(std::integral_constant<int, 4>());
    if (rest & 2) block(std::integral_constant<int, 2>());
    if (rest & 1) block(std::integral_constant<int, 1>());
#pragma unroll
    for (int u = 0; u < U; ++u) xout[q0 + u * NT] = x[u] + xb[u];
  }
  __device__ void project(int nc, float a, bool unit, const double* src64, const float* src, float* xout) {
    long long q = e0 + e.tid;
    for (; q + 3 * NT < e1; q += 4 * NT) project_points<4>(q, nc, a, unit, src64, src, xout);
    for (; q < e1; q += NT) project_points<1>(q, nc, a, unit, src64, src, xout);
  }

  // w = A x at the points g, g + NT, ... (U of them, below e1): all their loads, then the values.
  template <int U>
  __device__ __forceinline__ void stencil_points(long long g, const float* x, float* w) {
    const DevOp& d = e.P.op;
    const int nxy = d.nx * d.ny;
    float c5[U][5], z[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = (int)g + u * NT, r = q / d.nx, ix = q - r * d.nx;
      int iy = r;
      if constexpr (Op::DIM == 3) {
        const int iz = r / d.ny;
        iy = r - iz * d.ny;
        z[u][0] = x[iz == 0 ? q + (d.nz - 1) * nxy : q - nxy];
        z[u][1] = x[iz == d.nz - 1 ? q - (d.nz - 1) * nxy : q + nxy];
      }
      c5[u][0] = x[iy == 0 ? q + (d.ny - 1) * d.nx : q - d.nx];
      c5[u][1] = x[ix == 0 ? q + (d.nx - 1) : q - 1];
      c5[u][2] = x[q];
      c5[u][3] = x[ix == d.nx - 1 ? q - (d.nx - 1) : q + 1];
      c5[u][4] = x[iy == d.ny - 1 ? q - (d.ny - 1) * d.nx : q + d.nx];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float zm[3] = {0.f, 0.f, 0.f}, zp[3] = {0.f, 0.f, 0.f}, out[1];
      if constexpr (Op::DIM == 3) {
        zm[2] = z[u][0];
        zp[2] = z[u][1];
      }
      Op::template apply<float, 2, 5>(d, b.cf, zm, c5[u], zp, 2, g + u * NT, out);
      w[g + u * NT] = out[0];
    }
  }
  __device__ void stencil(const float* x, float* w) {
    long long g = e0 + e.tid;
    for (; g + 3 * NT < e1; g += 4 * NT) stencil_points<4>(g, x, w);
    for (; g < e1; g += NT) stencil_points<1>(g, x, w);
  }

  __device__ __forceinline__ int planes(int r) const {
    const Tiling& tl = e.P.tl;
    return ((tl.ntiles - 1 - r) / G0 + 1) * zs();   // (ZS divides nz: make_tiling)
  }
  __device__ __forceinline__ int zs() const { return Op::DIM == 2 ? 1 : e.P.tl.ZS; }
  // The ti-th tile of a rank.
  struct Tile {
    int w, h, base, mul;      // (i * mul >> 16 = i / w for i < 256, w <= 16)
  };
  // (the quotient by tiles_x through its reciprocal, rounded down: one too small at most)
  __device__ __forceinline__ Tile tile(int r, int ti) const {
    const DevOp& d = e.P.op;
    const Tiling& tl = e.P.tl;
    const int t = r + ti * G0;
    int rr = __umulhi(t, rtx);
    rr += t - rr * tl.tiles_x >= tl.tiles_x;
    const int bx = t - rr * tl.tiles_x, bz = Op::DIM == 2 ? 0 : rr / tl.tiles_y, by = rr - bz * tl.tiles_y;
    Tile o;
    o.w = min(TX, d.nx - bx * TX);
    o.h = min(TY, d.ny - by * TY);
    o.mul = o.w == TX ? 65536 / TX : (65536 + o.w - 1) / o.w;
    o.base = bx * TX + d.nx * (by * TY + d.ny * bz * tl.ZS);
    return o;
  }
  // Place i of a tile's planes relative to its base; -1 beyond a ragged tile.
  __device__ __forceinline__ int place(const Tile& o, int i) const {
    const int ly = (i * o.mul) >> 16, lx = i - ly * o.w;
    return ly < o.h ? lx + e.P.op.nx * ly : -1;
  }

  // Sum over the warp's lanes of compensated pairs, as write_partials' transposed sums pair the lanes.
  __device__ __forceinline__ static double comp_sum(float s, float ec) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
      const float os = __shfl_xor_sync(0xffffffffu, s, d), oe = __shfl_xor_sync(0xffffffffu, ec, d);
      float err;
      s = two_sum(s, os, err);
      ec = (ec + oe) + err;
    }
    return (double)s + (double)ec;
  }

  // Inner products of columns c0 .. c0 + min(NC, nd - c0) - 1 with x and w over rank r's planes: a warp takes a
  // plane, with up to four columns' loads in flight; then a warp adds up a column's runs.
  template <int NC>
  __device__ void dots(int r, int c0, int nd, const float* x, const float* w, double* part) {
    constexpr int PC = CG * PCH / NC < 32 ? CG * PCH / NC : 32, LC = NC < 4 ? NC : 4;
    const int nc = min(NC, nd - c0), np = planes(r), ZS = zs(), nxy = e.P.op.nx * e.P.op.ny;
    const long long N = e.P.op.N;
    const float* V = reinterpret_cast<const float*>(e.P.V) + (long long)c0 * N;
    float4 a[(NC + NW - 1) / NW];                    // this warp's columns: Kahan pairs of x and w
#pragma unroll
    for (int i = 0; i < (NC + NW - 1) / NW; ++i) a[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p0 = 0; p0 < np; p0 += PC) {
      const int n = min(PC, np - p0);
      int cur = -1, base = 0, off[K];
#pragma unroll 1
      for (int p = e.warp; p < n; p += NW) {
        const int ti = (p0 + p) / ZS;
        if (ti != cur) {
          cur = ti;
          const Tile o = tile(r, ti);
          base = o.base;
#pragma unroll
          for (int k = 0; k < K; ++k) off[k] = place(o, e.lane + 32 * k);
        }
        const int q = base + nxy * (p0 + p - ti * ZS);
        float xv[K], wv[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
          xv[k] = off[k] < 0 ? 0.f : __ldcg(x + q + off[k]);
          wv[k] = off[k] < 0 ? 0.f : __ldcg(w + q + off[k]);
        }
#pragma unroll 1
        for (int cb = 0; cb < nc; cb += LC) {
          float v[LC][K];
#pragma unroll
          for (int c = 0; c < LC; ++c) {
            const float* vc = V + (long long)(cb + c) * N + q;
#pragma unroll
            for (int k = 0; k < K; ++k) v[c][k] = cb + c < nc ? __ldcg(vc + max(off[k], 0)) : 0.f;
          }
#pragma unroll
          for (int c = 0; c < LC; ++c) {
            float px = 0.f, pw = 0.f;
#pragma unroll
            for (int k = 0; k < K; ++k) {
              px = fmaf(v[c][k], xv[k], px);
              pw = fmaf(v[c][k], wv[k], pw);
            }
            if (cb + c < nc) b.run[((cb + c) * PC + p) * 32 + e.lane] = make_float2(px, pw);
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < (NC + NW - 1) / NW; ++i) {
        const int c = e.warp + NW * i;
        if (c < nc) {
          const float2* run = b.run + c * PC * 32 + e.lane;
#pragma unroll 4
          for (int p = 0; p < n; ++p) {
            const float2 v = run[32 * p];
            E::kahan(a[i].x, a[i].y, v.x);
            E::kahan(a[i].z, a[i].w, v.y);
          }
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < (NC + NW - 1) / NW; ++i) {
      const int c = e.warp + NW * i;
      if (c < nc) {
        const double sx = comp_sum(a[i].x, -a[i].y), sw = comp_sum(a[i].z, -a[i].w);
        if (e.lane == 0) {
          part[c0 + c] = sx;
          part[nd + c0 + c] = sw;
        }
      }
    }
  }

  // Self terms x.x, x.w, w.w of rank r (w null: x.x only), a thread per place of the planes.
  __device__ void self(int r, int nd, const float* x, const float* w, double* part) {
    const int np = planes(r), ZS = zs(), nxy = e.P.op.nx * e.P.op.ny;
    int cur = -1, base = 0, off = -1;
    float f[3] = {0.f, 0.f, 0.f}, c[3] = {0.f, 0.f, 0.f};
    constexpr int U = 8;
    for (int p0 = 0; p0 < np; p0 += U) {
      float xv[U], wv[U];
      bool in[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int p = p0 + u, ti = p / ZS;
        if (p < np && ti != cur) {
          cur = ti;
          const Tile o = tile(r, ti);
          base = o.base;
          off = place(o, e.tid);
        }
        const int q = base + nxy * (p - ti * ZS) + off;
        in[u] = p < np && off >= 0;
        xv[u] = in[u] ? __ldcg(x + q) : 0.f;
        wv[u] = in[u] && w ? __ldcg(w + q) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (in[u]) {
          E::kahan(f[0], c[0], xv[u] * xv[u]);
          if (w) {
            E::kahan(f[1], c[1], xv[u] * wv[u]);
            E::kahan(f[2], c[2], wv[u] * wv[u]);
          }
        }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double s = comp_sum(f[i], -c[i]);
      if (e.lane == 0) e.S.bred[e.warp][i] = s;
    }
    __syncthreads();
    if (e.tid < 3) {
      double acc = 0;
      for (int i = 0; i < NW; ++i) acc += e.S.bred[i][e.tid];
      part[2 * nd + e.tid] = acc;
    }
    __syncthreads();
  }

  // Pass B2: every CTA takes units in turn; returns the number of reduction slots.
  __device__ int sums(int nd, const float* x, const float* w) {
    // columns per unit: as few as give every CTA at most one unit
    int cg = 1;
    while (cg < CG && G0 * ((nd + cg - 1) / cg) > e.gsize - G0) cg *= 2;
    const int per = 1 + (nd + cg - 1) / cg, units = G0 * per;
    for (int u = e.grank; u < units; u += e.gsize) {
      const int r = u % G0, k = u / G0;
      double* part = e.part_row(r);
      if (k == 0) self(r, nd, x, w, part);
      else if (cg == 1) dots<1>(r, k - 1, nd, x, w, part);
      else if (cg == 2) dots<2>(r, 2 * (k - 1), nd, x, w, part);
      else if (cg == 4) dots<4>(r, 4 * (k - 1), nd, x, w, part);
      else if (cg == 8) dots<8>(r, 8 * (k - 1), nd, x, w, part);
      else dots<16>(r, 16 * (k - 1), nd, x, w, part);
    }
    return 2 * nd + 3;
  }

  __device__ bool barrier() {
    e.bt1 += (unsigned)e.gsize;
    return e.arrive_wait(&e.P.ctl->arrive, e.bt1, true);
  }

  // Alg. 4 (Engine::run_hybrid, pass for pass).
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
      project(j - 1, j == 1 ? 1.f : e.S.a, j == 1 || (double)e.S.a == 1.0, j == 1 ? P.vin : nullptr, Wb[(j - 1) & 1], x);
      if (!e.sync_only()) return;
      stencil(x, Wb[j & 1]);
      if (!barrier()) return;
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
    project(nc, e.S.a, (double)e.S.a == 1.0, nullptr, src, xout);
    if (!barrier()) return false;
    for (int r = e.grank; r < G0; r += e.gsize) self(r, 0, xout, nullptr, e.part_row(r));
    return e.reduce_all(3, fn);
  }
};

template <class Op>
__global__ void __launch_bounds__(NT, 2) k_arnoldi_ordered(ArnoldiParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using F = OrderedPass<Op>;
  using E = typename F::E;
  E e(P, *reinterpret_cast<typename E::Smem*>(smem_raw), reinterpret_cast<double*>(smem_raw + E::small_offset()));
  if (!e.place()) return;
  e.redundant_steps();
  F f(e, *reinterpret_cast<typename F::Buf*>(smem_raw + F::offset()));
  f.run();
}

template <class Op>
cudaError_t launch_arnoldi_ordered_t(const ArnoldiParams& P, int G, cudaStream_t s) {
  ArnoldiParams Pc = P;
  void* args[1] = {&Pc};
  auto k = k_arnoldi_ordered<Op>;
  const size_t sm = OrderedPass<Op>::smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel((void*)k, dim3(G), dim3(NT), args, sm, s);
}

// Resident CTAs per SM.
template <class Op>
int ordered_blocks_per_sm_t() {
  int nb = 0;
  auto k = k_arnoldi_ordered<Op>;
  const size_t sm = OrderedPass<Op>::smem_bytes();
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, NT, sm) != cudaSuccess) return 0;
  return nb;
}

}  // namespace lsa
