// Flat two-phase hybrid step (Alg. 4): both passes of a step run over equal
// contiguous shares of the grid points, one share per CTA and every species of
// a point together.
//
//   pass A   x_j = a w_{j-1} - sum_i c_i x_i on the share (no halo), stored;
//            a grid barrier without a reduction;
//   pass B   w_j = A x_j with the neighbours of x read through L2, and the
//            inner products of the basis columns with x_j and w_j; then the
//            reduction and the O(j^2) step of the engine.
//
// There is no halo to project again, no tile chain and no tile-count
// imbalance; the price is the second barrier and a second reading of the
// basis.  Pass A is bound by the float64 unit (one FMA per column value) or,
// with the float32 basis, by memory.  In pass B of the float64 form a warp takes
// a piece of 32 VP points on its own: it forms w at them, keeps x and w in
// registers and streams the columns, eight at a time with one transposed warp
// sum for their sixteen inner products, so that no CTA barrier keeps one warp's
// stencil (float64 unit) from another's inner products (integer unit, memory:
// lsa_fix.cuh).  The columns come through a ring of asynchronous copies, in
// which a warp keeps 6 KB in flight (in registers, 2 to 4 KB: ADR 256^3 70 against
// 73 ms a phi product; with the limbs kept instead of converted 55 ms; the float64
// products it replaces took 94).  It walks its share backwards, so that it
// starts on the x that pass A left in L2 (and, where the columns are converted in
// place, on theirs).
#pragma once

#include <type_traits>

#include "lsa_engine.cuh"
#include "lsa_fix.cuh"

namespace lsa {

constexpr int FLAT_CG = 8;                // columns of a pass-B group (one transposed warp sum)
constexpr int FLAT_RING = 6144;           // bytes of a warp's ring of columns in flight

__device__ __forceinline__ unsigned flat_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
template <int BYTES>
__device__ __forceinline__ void flat_copy(unsigned dst, const void* src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void flat_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void flat_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <class Op, class Tc, bool AUG = false>
struct FlatPass {
  using E = Engine<Op, Tc, Tc, AUG, sizeof(Tc) == 4>;   // (float32: the tile passes for its norm passes)
  static constexpr int NS = Op::NS;
  static constexpr bool F64 = sizeof(Tc) == 8;
  static constexpr int VW = F64 ? 2 : 4;                 // values of a 16-byte load
  static constexpr int NGRP = MMAX / FLAT_CG;
  static_assert(FLAT_CG == 8, "the transposed warp sums below take 16 values");

  // Shared memory after the engine's.  float64: the warps' inner products and the
  // rings of columns in flight; float32: every lane's Kahan pairs and the chunk's x and
  // w.  And the stencil's coefficients, converted once: in registers the
  // compiler converts them again at every use, on the float64 pipe.
  struct Buf64 {
    alignas(16) unsigned char ring[NW][FLAT_RING];
    double sum[NW][NGRP * 16];
    Coef<double> cf;
  };
  struct Buf32 {
    float4 acc[KMAX][NT];
    float xw[4 * NS * NT];
    Coef<float> cf;
  };
  using Buf = typename std::conditional<F64, Buf64, Buf32>::type;
  __host__ __device__ static constexpr size_t offset() { return (E::smem_bytes() + 127) & ~(size_t)127; }
  __host__ __device__ static constexpr size_t smem_bytes() { return offset() + sizeof(Buf); }

  E& e;
  Buf& b;
  long long e0, e1;      // this CTA's share of the grid points
  bool vec;              // every column starts on a 16-byte boundary

  __device__ FlatPass(E& en, Buf& bu) : e(en), b(bu) {
    const long long np = e.P.op.npts;
    long long per = (np + e.gsize - 1) / e.gsize;
    per = (per + 31) & ~31LL;                  // shares start on a 32-point boundary
    e0 = min(np, (long long)e.grank * per);
    e1 = min(np, e0 + per);
    vec = np % VW == 0 && ((size_t)e.P.V & 15) == 0;
    if (e.tid == 0) b.cf = e.cf;
    __syncthreads();
  }

  // -------------------------------------------------------------------------
  // Pass A on `NU` units of one thread: unit u is VW consecutive values at
  // g[u] (32 lanes: 32 VW values).  Columns in ascending order with one
  // accumulator per value (float32: two, alternating), CB columns' loads in
  // flight before their FMAs.
  template <int W, int NU>
  __device__ __forceinline__ void project_units(const PassT<Tc>& ps, const long long (&g)[NU], const bool (&on)[NU]) {
    constexpr int CB = 8;
    const long long N = e.P.op.N;
    const Tc a = (Tc)ps.a;
    const bool unit = ps.a == 1.0;
    Tc x[NU][W], xb[NU][W];
#pragma unroll
    for (int u = 0; u < NU; ++u) {
#pragma unroll
      for (int i = 0; i < W; ++i) xb[u][i] = (Tc)0;
      if (ps.src64) {
#pragma unroll
        for (int i = 0; i < W; ++i) x[u][i] = (Tc)__ldg(ps.src64 + g[u] + i);
      } else {
        load<W>(ps.srcB + g[u], x[u]);
      }
#pragma unroll
      for (int i = 0; i < W; ++i)
        if (!unit) x[u][i] = a * x[u][i];
    }
    const Tc* Vb = reinterpret_cast<const Tc*>(e.P.V);
    int c = ps.c0;
    // CN columns, their loads before their FMAs (float32: the odd ones of a whole block in the second accumulator)
    auto block = [&](auto cn, int c) {
      constexpr int CN = decltype(cn)::value;
      Tc v[CN][NU][W];
#pragma unroll
      for (int k = 0; k < CN; ++k)
#pragma unroll
        for (int u = 0; u < NU; ++u) load<W>(Vb + (long long)(c + k) * N + g[u], v[k][u]);
#pragma unroll
      for (int k = 0; k < CN; ++k) {
        const Tc cc = e.S.coefc[c + k];
#pragma unroll
        for (int u = 0; u < NU; ++u)
#pragma unroll
          for (int i = 0; i < W; ++i) {
            if (!F64 && CN == CB && (k & 1)) xb[u][i] = fma(-cc, v[k][u][i], xb[u][i]);
            else x[u][i] = fma(-cc, v[k][u][i], x[u][i]);
          }
      }
    };
#pragma unroll 1
    for (; c + CB <= ps.c1; c += CB) block(std::integral_constant<int, CB>(), c);
    // the last columns: blocks of four, two and one (Gray-Scott 512^2 5.66 to 5.62 ms, ADR 256^3 54.97 to 53.82); the
    // augmented kernel, with less registers to spare, takes them one by one (6.84 ms in blocks, 6.64 so)
    if constexpr (AUG) {
#pragma unroll 1
      for (; c < ps.c1; ++c) block(std::integral_constant<int, 1>(), c);
    } else {
      const int rest = ps.c1 - c;
      if (rest & 4) block(std::integral_constant<int, 4>(), c);
      if (rest & 2) block(std::integral_constant<int, 2>(), c + (rest & 4));
      if (rest & 1) block(std::integral_constant<int, 1>(), c + (rest & 6));
    }
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      if (!on[u]) continue;
#pragma unroll
      for (int i = 0; i < W; ++i) {
        if (!F64) x[u][i] += xb[u][i];
        if (ps.self & SELF_XX) e.self_add(0, x[u][i], x[u][i]);
      }
      if (ps.xout) store<W>(ps.xout + g[u], x[u]);
    }
  }

  template <int W>
  __device__ __forceinline__ static void load(const Tc* p, Tc (&v)[W]) {
    if constexpr (W == 1) v[0] = __ldcg(p);
    else if constexpr (F64) {
      const double2 q = __ldcg(reinterpret_cast<const double2*>(p));
      v[0] = q.x; v[1] = q.y;
    } else {
      const float4 q = __ldcg(reinterpret_cast<const float4*>(p));
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
  }
  template <int W>
  __device__ __forceinline__ static void store(Tc* p, const Tc (&v)[W]) {
    if constexpr (W == 1) *p = v[0];
    else if constexpr (F64) *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    else *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }

  // Pass A over the share: warps take units of 32 W values of one species in
  // turn, two at a time, so that the tail of a short share leaves whole warps
  // without work instead of lanes.
  template <int W>
  __device__ __forceinline__ void project_w(const PassT<Tc>& ps) {
    constexpr int UW = 32 * W;
    const int cnt = (int)(e1 - e0);
    const int per = (cnt + UW - 1) / UW, units = NS * per;
    const long long np = e.P.op.npts;
    auto at = [&](int u, bool& on) {
      const int sp = NS == 1 ? 0 : u / per;
      const int q = (u - sp * per) * UW + e.lane * W;
      on = q < cnt;
      return sp * np + e0 + (on ? q : 0);
    };
    int u = e.warp;
#pragma unroll 1
    for (; u + NW < units; u += 2 * NW) {
      bool on[2];
      const long long g[2] = {at(u, on[0]), at(u + NW, on[1])};
      project_units<W, 2>(ps, g, on);
    }
    if (u < units) {
      bool on[1];
      const long long g[1] = {at(u, on[0])};
      project_units<W, 1>(ps, g, on);
    }
  }
  __device__ void project(const PassT<Tc>& ps) {
    if (vec) project_w<VW>(ps);
    else project_w<1>(ps);
  }

  // -------------------------------------------------------------------------
  // The stencil's x at point q: per species [south, west, centre, east, north], below and above at index 2 of
  // z.  Other CTAs' values of pass A: ordinary loads, which the grid barrier's acquire orders (it drops the
  // L1 lines of earlier steps), so that neighbouring points share L1 lines.
  struct Nbr {
    Tc c5[5 * NS], z[Op::DIM == 3 ? 2 : 1];
  };
  __device__ __forceinline__ void gather(const Tc* x, int q, Nbr& n) {
    const DevOp& d = e.P.op;
    const int r = q / d.nx, ix = q - r * d.nx;
    const int iz = r / d.ny, iy = r - iz * d.ny;
    const int qw = ix == 0 ? q + (d.nx - 1) : q - 1;
    const int qe = ix == d.nx - 1 ? q - (d.nx - 1) : q + 1;
    const int qs = iy == 0 ? q + (d.ny - 1) * d.nx : q - d.nx;
    const int qn = iy == d.ny - 1 ? q - (d.ny - 1) * d.nx : q + d.nx;
#pragma unroll
    for (int sp = 0; sp < NS; ++sp) {
      const Tc* xs = x + (long long)sp * d.npts;
      n.c5[5 * sp + 0] = xs[qs];
      n.c5[5 * sp + 1] = xs[qw];
      n.c5[5 * sp + 2] = xs[q];
      n.c5[5 * sp + 3] = xs[qe];
      n.c5[5 * sp + 4] = xs[qn];
    }
    if constexpr (Op::DIM == 3) {
      const int nxy = d.nx * d.ny;
      n.z[0] = x[iz == 0 ? q + (d.nz - 1) * nxy : q - nxy];
      n.z[1] = x[iz == d.nz - 1 ? q - (d.nz - 1) * nxy : q + nxy];
    }
  }
  // w = A x at point q (every species), returned; `own`: also stored and added to the self terms.
  __device__ __forceinline__ void stencil(const PassT<Tc>& ps, int q, const Nbr& n, bool own, Tc (&wv)[NS]) {
    const DevOp& d = e.P.op;
    Tc zm[3], zp[3], out[NS];
    zm[0] = zm[1] = zm[2] = zp[0] = zp[1] = zp[2] = (Tc)0;
    if constexpr (Op::DIM == 3) { zm[2] = n.z[0]; zp[2] = n.z[1]; }
    Op::template apply<Tc, 2, 5>(d, b.cf, zm, n.c5, zp, 2, (long long)q, out);
    if constexpr (AUG) {         // + B x_bot (augmented operator)
      const int p = e.P.naug;
#pragma unroll
      for (int sp = 0; sp < NS; ++sp)
        for (int k = 0; k < p; ++k)
          out[sp] = fma((Tc)e.S.xi[k], (Tc)__ldg(e.P.baug + (long long)(p - k) * d.N + sp * d.npts + q), out[sp]);
    }
#pragma unroll
    for (int sp = 0; sp < NS; ++sp) {
      wv[sp] = out[sp];
      if (!own) continue;
      ps.wout[(long long)sp * d.npts + q] = out[sp];
      if constexpr (!F64) {        // (float64: x . x and x . w as the inner products of column j)
        e.self_add(0, n.c5[5 * sp + 2], n.c5[5 * sp + 2]);
        e.self_add(1, n.c5[5 * sp + 2], out[sp]);
      }
      e.self_add(2, out[sp], out[sp]);
    }
  }

  // x . x and x . w of a piece, as the inner products of column nv (x itself).
  template <int VL>
  __device__ __forceinline__ void self_products(const int (&xh)[VL], const int (&xl)[VL], const int (&wh)[VL],
                                                const int (&wl)[VL], unsigned kx, unsigned kw, int nv) {
    long long t[2];
    fx_dot(xh, xl, xh, xl, wh, wl, true, t[0], t[1]);
    const long long s = warp_sum_many_s64<2>(t);         // lane l: value l >> 4
    if ((e.lane & 15) == 0) b.sum[e.warp][2 * nv + (e.lane >> 4)] += fx_value(s, kx, e.lane ? kw : kx);
  }

  // One piece of pass B with the limbs of the basis kept in P.F: lane l takes the VP points
  // p0 + 2 l + 64 k + {0, 1} of the share.  Pass B of step j writes the limbs of x_j and the shift base of each of
  // its pieces, and every later step reads them: eight bytes a value like the float64 column, 16-byte copies at any
  // N (the columns of F are padded), and no conversion, which takes three times the multiply-adds' time.
  template <int VP>
  __device__ __forceinline__ void piece_fixed(const PassT<Tc>& ps, int p0, int nc, int cs, int CS) {
    constexpr int VL = VP * NS;                      // values per lane
    const long long npf = (e.P.op.npts + 1) & ~1LL, NF = npf * NS;
    const int nv = nc - 1, cnt = (int)(e1 - e0);
    // the ring of columns in flight: every lane copies its own values to places that only it reads
    constexpr int CB = VL * 32 * 8, D = FLAT_RING / CB < 8 ? FLAT_RING / CB : 8;
    static_assert(D >= 2, "two columns in flight");
    const unsigned ring = flat_smem(b.ring[e.warp]) + e.lane * 16u;
    unsigned wr = ring, rd = ring;
    int2* const mine = e.P.F + e0 + p0 + 2 * e.lane;  // this lane's first value of column 0
    const int2* src = mine + (long long)cs * FLAT_CG * NF;
    int ic = cs * FLAT_CG;                           // next column to issue
    auto issue = [&]() {
      if (ic < nv) {
#pragma unroll
        for (int sp = 0; sp < NS; ++sp)
#pragma unroll
          for (int k = 0; k < VP / 2; ++k) flat_copy<16>(wr + (sp * (VP / 2) + k) * 512, src + sp * npf + 64 * k);
      }
      flat_commit();
      wr = wr == ring + (D - 1) * CB ? ring : wr + CB;
      src += NF;
      if ((++ic & (FLAT_CG - 1)) == 0) {
        ic += (CS - 1) * FLAT_CG;
        src += (CS - 1) * FLAT_CG * NF;
      }
    };
#pragma unroll
    for (int i = 0; i < D; ++i) issue();
    int xh[VL], xl[VL], wh[VL], wl[VL];
    unsigned* const keys = limb_keys(e.P.F, e.P.op, e.P.m) + (e0 + p0) / 32 * limb_key_stride(e.P.m);
    unsigned kx, kw;
    {
      double x[VL], w[VL];
      constexpr int GB = VP < 4 ? VP : 4;            // points whose loads are in flight together
#pragma unroll
      for (int k0 = 0; k0 < VP; k0 += GB) {
        Nbr n[GB];
        int q[GB];
        bool in[GB];
#pragma unroll
        for (int i = 0; i < GB; ++i) {
          const int pl = p0 + 2 * e.lane + 64 * ((k0 + i) / 2) + (i & 1);
          in[i] = pl < cnt;
          q[i] = in[i] ? (int)e0 + pl : 0;           // (beyond the share: any point, x and w count as zero)
          gather(ps.srcB, q[i], n[i]);
        }
#pragma unroll
        for (int i = 0; i < GB; ++i) {
          double wv[NS];
#pragma unroll
          for (int sp = 0; sp < NS; ++sp) wv[sp] = 0.0;
          if (in[i]) stencil(ps, q[i], n[i], cs == 0, wv);
#pragma unroll
          for (int sp = 0; sp < NS; ++sp) {
            const int v = sp * VP + k0 + i;
            w[v] = wv[sp];
            x[v] = in[i] ? n[i].c5[5 * sp + 2] : 0.0;
          }
        }
      }
      fx_blocks(x, w, kx, kw);
#pragma unroll
      for (int v = 0; v < VL; ++v) {
        fx_split(x[v], kx, xh[v], xl[v]);
        fx_split(w[v], kw, wh[v], wl[v]);
      }
      if (cs == 0) {
        // (two points a store: a share ends at an even point, or at the last one and its padding)
        if (e.lane == 0) keys[nv] = kx;
#pragma unroll
        for (int k = 0; k < VP; k += 2)
          if (p0 + 2 * e.lane + 32 * k < cnt)
#pragma unroll
            for (int sp = 0; sp < NS; ++sp) {
              const int v = sp * VP + k;
              *reinterpret_cast<int4*>(mine + nv * NF + sp * npf + 32 * k) = make_int4(xl[v], xh[v], xl[v + 1], xh[v + 1]);
            }
      }
    }
    if (cs == 0) self_products<VL>(xh, xl, wh, wl, kx, kw, nv);
#pragma unroll 1
    for (int g = cs; g * FLAT_CG < nv; g += CS) {
      const int c0 = g * FLAT_CG, kc = c0 + (e.lane >> 2);
      const unsigned kv = kc < nv ? __ldcg(keys + kc) : kx;    // of the column whose sum this lane gets
      long long t[16];
#pragma unroll
      for (int i = 0; i < FLAT_CG; ++i) {
        const int c = c0 + i;
        t[2 * i] = t[2 * i + 1] = 0;
        if (c < nv) {
          int h[VL], l[VL];
          flat_wait<D - 1>();
#pragma unroll
          for (int sp = 0; sp < NS; ++sp)
#pragma unroll
            for (int k = 0; k < VP / 2; ++k) {
              const int v = sp * VP + 2 * k;
              asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                           : "=r"(l[v]), "=r"(h[v]), "=r"(l[v + 1]), "=r"(h[v + 1])
                           : "r"(rd + (sp * (VP / 2) + k) * 512)
                           : "memory");
            }
          fx_dot(h, l, xh, xl, wh, wl, false, t[2 * i], t[2 * i + 1]);
        }
        rd = rd == ring + (D - 1) * CB ? ring : rd + CB;
        issue();
      }
      const long long s = warp_sum_many_s64<16>(t);      // lanes 2k, 2k + 1: value k
      if ((e.lane & 1) == 0)
        b.sum[e.warp][g * 16 + (e.lane >> 1)] += fx_value(s, kv, (e.lane & 2) ? kw : kx);
    }
    flat_wait<0>();        // (columns beyond the last group: nothing in flight into the next piece's slots)
  }
  // Warps that take the columns of one of np pieces in turn: as many as leave no warp without a piece (columns
  // permitting).
  __device__ __forceinline__ static int sharing(int np, int nc) {
    int CS = 1;
    while (2 * CS * np <= NW && 2 * CS * FLAT_CG <= nc + FLAT_CG) CS *= 2;
    return CS;
  }

  // The same without the kept limbs: VP points p0 + l + 32 k per lane, the float64 columns converted here.
  template <int VP>
  __device__ __forceinline__ void piece_float64(const PassT<Tc>& ps, int p0, int nc, int cs, int CS) {
    constexpr int VL = VP * NS;
    const long long N = e.P.op.N, npts = e.P.op.npts;
    const int nv = nc - 1, cnt = (int)(e1 - e0);
    const double* Vb = reinterpret_cast<const double*>(e.P.V);
    constexpr int CB = VL * 32 * 8, D = FLAT_RING / CB < 8 ? FLAT_RING / CB : 8;
    const unsigned ring = flat_smem(b.ring[e.warp]) + e.lane * 8u;
    unsigned wr = ring, rd = ring;
    int q[VP];
    bool in[VP];
#pragma unroll
    for (int k = 0; k < VP; ++k) {
      const int pl = p0 + e.lane + 32 * k;
      in[k] = pl < cnt;
      q[k] = in[k] ? (int)e0 + pl : 0;               // (beyond the share: any point, x and w count as zero)
    }
    int ic = cs * FLAT_CG;
    auto issue = [&]() {
      if (ic < nv) {
#pragma unroll
        for (int sp = 0; sp < NS; ++sp) {
          const double* p = Vb + (long long)ic * N + (long long)sp * npts;
#pragma unroll
          for (int k = 0; k < VP; ++k) flat_copy<8>(wr + (sp * VP + k) * 256, p + q[k]);
        }
      }
      flat_commit();
      wr = wr == ring + (D - 1) * CB ? ring : wr + CB;
      if ((++ic & (FLAT_CG - 1)) == 0) ic += (CS - 1) * FLAT_CG;
    };
#pragma unroll
    for (int i = 0; i < D; ++i) issue();
    int xh[VL], xl[VL], wh[VL], wl[VL];
    unsigned kx, kw;
    {
      Nbr n[VP];
      double x[VL], w[VL];
#pragma unroll
      for (int k = 0; k < VP; ++k) gather(ps.srcB, q[k], n[k]);
#pragma unroll
      for (int k = 0; k < VP; ++k) {
        double wv[NS];
#pragma unroll
        for (int sp = 0; sp < NS; ++sp) wv[sp] = 0.0;
        if (in[k]) stencil(ps, q[k], n[k], cs == 0, wv);
#pragma unroll
        for (int sp = 0; sp < NS; ++sp) {
          const int v = sp * VP + k;
          w[v] = wv[sp];
          x[v] = in[k] ? n[k].c5[5 * sp + 2] : 0.0;
        }
      }
      fx_blocks(x, w, kx, kw);
#pragma unroll
      for (int v = 0; v < VL; ++v) {
        fx_split(x[v], kx, xh[v], xl[v]);
        fx_split(w[v], kw, wh[v], wl[v]);
      }
    }
    if (cs == 0) self_products<VL>(xh, xl, wh, wl, kx, kw, nv);
#pragma unroll 1
    for (int g = cs; g * FLAT_CG < nv; g += CS) {
      const int c0 = g * FLAT_CG;
      long long t[16];
      unsigned kv = kx;                                  // of the column whose sum this lane gets
#pragma unroll
      for (int i = 0; i < FLAT_CG; ++i) {
        const int c = c0 + i;
        t[2 * i] = t[2 * i + 1] = 0;
        if (c < nv) {
          double v[VL];
          int h[VL], l[VL];
          flat_wait<D - 1>();
#pragma unroll
          for (int k = 0; k < VL; ++k) asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v[k]) : "r"(rd + k * 256) : "memory");
#pragma unroll
          for (int k = 0; k < VP; ++k)
            if (!in[k])                                  // (a copy of another point: not in the block)
#pragma unroll
              for (int sp = 0; sp < NS; ++sp) v[sp * VP + k] = 0.0;
          const unsigned kc = fx_block(v);
          if (e.lane >> 2 == i) kv = kc;
#pragma unroll
          for (int k = 0; k < VL; ++k) fx_split(v[k], kc, h[k], l[k]);
          fx_dot(h, l, xh, xl, wh, wl, false, t[2 * i], t[2 * i + 1]);
        }
        rd = rd == ring + (D - 1) * CB ? ring : rd + CB;
        issue();
      }
      const long long s = warp_sum_many_s64<16>(t);
      if ((e.lane & 1) == 0)
        b.sum[e.warp][g * 16 + (e.lane >> 1)] += fx_value(s, kv, (e.lane & 2) ? kw : kx);
    }
    flat_wait<0>();
  }
  template <int VP, bool FIXED>
  __device__ __forceinline__ void pieces(const PassT<Tc>& ps, int nc) {
    const int np = ((int)(e1 - e0) + 32 * VP - 1) / (32 * VP), CS = sharing(np, nc);
#pragma unroll 1
    for (int u = e.warp; u < np * CS; u += NW) {
      const int p0 = (np - 1 - u / CS) * 32 * VP;
      if constexpr (FIXED) piece_fixed<VP>(ps, p0, nc, u % CS, CS);
      else piece_float64<VP>(ps, p0, nc, u % CS, CS);
    }
  }

  // float64: pass B over the share, the inner products with columns 0..nc-1 (the last one is x itself); writes
  // the CTA's partial sums and returns the number of reduction slots.
  __device__ int pass_fixed(const PassT<Tc>& ps) {
    const int nc = ps.d1;
    for (int i = e.lane; i < (nc + FLAT_CG - 1) / FLAT_CG * 16; i += 32) b.sum[e.warp][i] = 0.0;
    __syncwarp();
    // eight values per lane where at least half the warps have a piece of them, else two points; without
    // room for the limbs of the basis four values, whose conversion takes the registers
    constexpr int VP = 8 / NS;
    if (e.P.F == nullptr) pieces<VP / 2, false>(ps, nc);
    else if (e1 - e0 > 32 * VP * (NW / 2 - 1)) pieces<VP, true>(ps, nc);
    else pieces<2, true>(ps, nc);
    return partials_fixed(nc);
  }

  // float32: pass B over the share in chunks of FCH points, warps taking columns.  Lane l takes the points
  // l + 32 k of a chunk: eight products in one float32 run, the runs in a Kahan sum per lane and column, in
  // the order of the points -- the float32 basis repeats only if these sums do to the last bit, since one that
  // rounds the other way moves a value of the basis by 6e-8.  The next column's values are loaded while one is
  // consumed.
  static constexpr int FCH = 2 * NT, FQ = FCH / NT;
  __device__ int pass_float(const PassT<Tc>& ps) {
    const int nd = ps.d1;
    const long long np = e.P.op.npts, step = e.P.op.N * NW;
#pragma unroll
    for (int kk = 0; kk < KMAX; ++kk) b.acc[kk][e.tid] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (long long base = e0; base < e1; base += FCH) {
      const int nv = (int)min((long long)FCH, e1 - base);
      Nbr n[FQ];
#pragma unroll
      for (int u = 0; u < FQ; ++u) gather(ps.srcB, (int)base + min(e.tid + u * NT, nv - 1), n[u]);
      __syncthreads();                     // the last chunk's reads
#pragma unroll
      for (int u = 0; u < FQ; ++u) {
        const int pl = e.tid + u * NT;
        const bool in = pl < nv;
        Tc wv[NS];
#pragma unroll
        for (int sp = 0; sp < NS; ++sp) wv[sp] = (Tc)0;
        if (in) stencil(ps, (int)base + pl, n[u], true, wv);
#pragma unroll
        for (int sp = 0; sp < NS; ++sp) {
          b.xw[sp * FCH + pl] = in ? (float)n[u].c5[5 * sp + 2] : 0.f;
          b.xw[(NS + sp) * FCH + pl] = (float)wv[sp];
        }
      }
      __syncthreads();
      if (e.warp >= nd) continue;
#pragma unroll 1
      for (int sp = 0; sp < NS; ++sp) {
        const float* x = b.xw + sp * FCH + e.lane;
        auto load = [&](const float* p, float (&v)[FCH / 32]) {
#pragma unroll
          for (int k = 0; k < FCH / 32; ++k) v[k] = e.lane + 32 * k < nv ? __ldcg(p + 32 * k) : 0.f;
        };
        auto dot = [&](const float (&v)[FCH / 32], int kk) {
          float4 a = b.acc[kk][e.tid];
#pragma unroll
          for (int g = 0; g < FCH / 256; ++g) {
            float px = 0.f, pw = 0.f;
#pragma unroll
            for (int k = 8 * g; k < 8 * g + 8; ++k) {
              px = fmaf(v[k], x[32 * k], px);
              pw = fmaf(v[k], x[NS * FCH + 32 * k], pw);
            }
            E::kahan(a.x, a.y, px);
            E::kahan(a.z, a.w, pw);
          }
          b.acc[kk][e.tid] = a;
        };
        const float* col = reinterpret_cast<const float*>(e.Vc(e.warp)) + (long long)sp * np + base + e.lane;
        float v0[FCH / 32], v1[FCH / 32];
        load(col, v0);
        int c = e.warp, kk = 0;
#pragma unroll 1
        for (;;) {
          const bool m1 = c + NW < nd;
          if (m1) load(col + step, v1);
          dot(v0, kk);
          if (!m1) break;
          const bool m2 = c + 2 * NW < nd;
          if (m2) load(col + 2 * step, v0);
          dot(v1, kk + 1);
          if (!m2) break;
          c += 2 * NW;
          col += 2 * step;
          kk += 2;
        }
      }
    }
    float vs[2 * KMAX], ve[2 * KMAX];        // Kahan keeps sum = s - c: e = -c
#pragma unroll
    for (int kk = 0; kk < KMAX; ++kk) {
      const float4 a = b.acc[kk][e.tid];
      vs[2 * kk] = a.x; ve[2 * kk] = -a.y;
      vs[2 * kk + 1] = a.z; ve[2 * kk + 1] = -a.w;
    }
    warp_sum_many_comp<2 * KMAX>(vs, ve);    // lanes 2k, 2k + 1: value k (column k / 2 of the warp, x or w)
    const int k = e.lane >> 1, c = e.warp + NW * (k >> 1);
    if ((e.lane & 1) == 0 && c < nd) e.part_row()[(k & 1) ? nd + c : c] = (double)vs[0] + (double)ve[0];
    return e.write_self(ps, nd);
  }
  __device__ int pass(const PassT<Tc>& ps) {
    e.zero_acc();
    if constexpr (F64) return pass_fixed(ps);
    else return pass_float(ps);
  }

  // float64: per-CTA partial sums to global memory in the engine's layout: x_i . x and x_i . w of the earlier
  // columns, then x . x, x . w (column nc - 1) and w . w.
  __device__ int partials_fixed(int nc) {
    double* part = e.part_row();
    const int np = nc - 1;
    const double ww = warp_sum(e.sww);
    if (e.lane == 0) e.S.bred[e.warp][2] = ww;
    __syncthreads();
    for (int s = e.tid; s < 2 * nc; s += NT) {
      const int c = s >> 1, isw = s & 1;
      double t = 0.0;
#pragma unroll
      for (int i = 0; i < NW; ++i) t += b.sum[i][s];
      if constexpr (AUG) {
        if (e.grank == 0) t += e.aug_dot(c, isw ? e.S.xw : e.S.xi);
      }
      part[c == np ? 2 * np + isw : isw * np + c] = t;
    }
    if (e.tid == NT - 1) {
      double t = 0.0;
      for (int i = 0; i < NW; ++i) t += e.S.bred[i][2];
      if constexpr (AUG) {
        if (e.grank == 0) t += e.aug_self(2);
      }
      part[2 * np + 2] = t;
    }
    return 2 * np + 3;
  }

  // Alg. 4 with the flat passes (Engine::run_hybrid, pass for pass).
  __device__ void run() {
    const ArnoldiParams& P = e.P;
    Tc* V = reinterpret_cast<Tc*>(P.V);
    Tc* Wb[2] = {reinterpret_cast<Tc*>(P.W0), reinterpret_cast<Tc*>(P.W1)};
    const long long N = P.op.N;
    const int m = P.m;
    if (e.tid == 0) { e.S.a = (Tc)1; e.S.done = 0; e.S.fallback_pending = 0; e.S.syncs_c = 0; }
    __syncthreads();
    PassT<Tc> ps;
    ps.dmode = DOT_X | DOT_W;
    for (int j = 1; j <= m; ++j) {
      ps.c0 = 0; ps.c1 = j - 1;
      ps.a = (j == 1) ? 1.0 : (double)e.S.a;
      ps.src64 = (j == 1) ? P.vin : nullptr;
      ps.srcB = (j == 1) ? nullptr : Wb[(j - 1) & 1];
      ps.xout = V + (long long)(j - 1) * N;
      ps.wout = Wb[j & 1];
      ps.d0 = ps.d1 = 0;
      ps.self = 0;
      if constexpr (AUG) e.aug_begin(ps);
      project(ps);
      if (!e.sync_only()) return;
      ps.c0 = ps.c1 = 0;
      ps.a = 1.0;
      ps.src64 = nullptr;
      ps.srcB = ps.xout;
      ps.xout = nullptr;
      ps.d1 = F64 ? j : j - 1;         // float64: the last column is x_j itself
      ps.self = F64 ? SELF_WW : SELF_XX | SELF_XW | SELF_WW;
      const int ns = pass(ps);
      if (!e.reduce_all(ns, [&] { e.hybrid_step(j); })) return;
      if (e.S.done) return;
      if (e.S.fallback_pending) {     // explicit norm of the projected vector (extra reduction of Alg. 4)
        if (!norm_pass(j, Wb[j & 1], nullptr, [&] { e.hybrid_fallback_finish(j); })) return;
        if (e.S.done) return;
      }
    }
    // v_{m+1} and its norm (one more reduction)
    norm_pass(m, Wb[m & 1], V + (long long)m * N, [&] { e.hybrid_final_finish(); });
  }

  // x = a src - sum_{c < nc} coef_c V_c and x . x, reduced; x stored when xout is given.
  template <class Fn>
  __device__ bool norm_pass(int nc, const Tc* src, Tc* xout, Fn fn) {
    PassT<Tc> ps;
    ps.c0 = 0; ps.c1 = nc; ps.a = (double)e.S.a;
    ps.src64 = nullptr; ps.srcB = src; ps.xout = xout; ps.wout = nullptr;
    ps.d0 = ps.d1 = 0; ps.dmode = 0; ps.self = SELF_XX;
    if constexpr (!F64) return e.reduce_all(e.run_pass(ps), fn);
    e.zero_acc();
    if constexpr (AUG) e.aug_begin(ps);
    project(ps);
    return e.reduce_all(e.write_self(ps, 0), fn);
  }
};

template <class Op, class Tc, bool AUG>
__global__ void __launch_bounds__(NT, 2) k_arnoldi_flat(ArnoldiParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using F = FlatPass<Op, Tc, AUG>;
  using E = typename F::E;
  typename E::Smem& S = *reinterpret_cast<typename E::Smem*>(smem_raw);
  E e(P, S, reinterpret_cast<double*>(smem_raw + E::small_offset()));
  if (!e.place()) return;
  e.redundant_steps();
  F f(e, *reinterpret_cast<typename F::Buf*>(smem_raw + F::offset()));
  f.run();
}

template <class Op, class Tc, bool AUG>
cudaError_t launch_arnoldi_flat_t(const ArnoldiParams& P, int G, cudaStream_t s) {
  ArnoldiParams Pc = P;
  void* args[1] = {&Pc};
  auto k = k_arnoldi_flat<Op, Tc, AUG>;
  const size_t sm = FlatPass<Op, Tc, AUG>::smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel((void*)k, dim3(G), dim3(NT), args, sm, s);
}

// Resident CTAs per SM.
template <class Op, class Tc, bool AUG>
int flat_blocks_per_sm_t() {
  int nb = 0;
  auto k = k_arnoldi_flat<Op, Tc, AUG>;
  const size_t sm = FlatPass<Op, Tc, AUG>::smem_bytes();
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, NT, sm) != cudaSuccess) return 0;
  return nb;
}

}  // namespace lsa
