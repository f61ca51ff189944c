// The Wilson-clover stencil on even-odd ordered half lattices.
//
// One thread computes one output site of parity p for one right-hand side:
//
//   H psi(x) = sum_mu [ U_mu(x) (1 - g_mu) psi(x+mu) + U_mu(x-mu)^dag (1 + g_mu) psi(x-mu) ]
//
// (projectors swapped for the adjoint, since g5 (1 -/+ g_mu) g5 = (1 +/- g_mu)),
// with the two-component spin projection so that only half spinors are
// transported by the links, and the time-boundary factor on hops that cross
// x0 = T-1 <-> 0.  The mode picks what is done with H psi:
//
//   HOP_DW : out = A in2 - 1/2 H in                  (one parity of D psi)
//   HOP_P1 : out = A^{-1} (-1/2 H in)                (D_oo^{-1} D_oe psi_e)
//   HOP_P2 : out = A in2 + 1/2 H in                  (D_ee psi_e - D_eo t_o)
//
// and the epilogue fuses the vector work of the solvers into the store
// (norm of the output, the CG update of x and r, or the binary64 residual
// eta - out of a reset step) with a deterministic binary64 grid reduction.
#pragma once
#include "df_pack.cuh"
#include "reduce.cuh"

namespace oq {

// Accumulate one transported hop with weight w (times the time-boundary
// factor when the hop crosses it).
template <int MU, int S, typename R>
__device__ __forceinline__ void hop_accum(Spinor<R>& acc, HalfSpinor<R>& t, R w, bool cr, float bc_t) {
  accum_reconstruct<MU, S>(acc, t, cr ? w * (R)bc_t : w);
}

// fnext / fprev (sub-domain launches, this rhs and output parity): the time
// faces that replace the hops leaving the sub-domain (HopArgs::halo_next)
template <int P, int FMT, int MU, bool DAG, bool NC = false>
__device__ __forceinline__ void hop_dir(const HopArgs& a, const char* in, int p, long i, const int x[4],
                                        Spinor<typename PrecTraits<P>::R>& acc,
                                        typename PrecTraits<P>::R w, const char* fnext = nullptr,
                                        const char* fprev = nullptr) {
  typedef typename PrecTraits<P>::R R;
  constexpr int SF = DAG ? +1 : -1;  // projector sign of the forward hop
  bool cr;
  // forward: U_mu(x) (1 -/+ g) psi(x + mu)
  {
    long j = eo_neighbour(a.g, x, MU, +1, &cr);
    HalfSpinor<R> h, t;
    float sg = a.g.bc_t;
    if (MU == 0 && cr && fnext) {
      // x0 = T-1: the projected neighbour comes from the next sub-domain
      const long Fs = a.g.Vh / a.g.L[0];
      load_half<R>(fnext, Fs, i - (long)x[0] * Fs, h);
      sg = a.halo_sign_next;
    } else {
      Spinor<R> nb;
      load_spinor<P, NC>(in, a.g.Vh, j, nb);
      project<MU, SF>(nb, h);
    }
    Su3<R> u;
    load_link<R, FMT>(a.links, a.g.Vh, p, MU, i, u);
    su3_mul(u, h, t);
    hop_accum<MU, SF>(acc, t, w, cr, sg);
  }
  // backward: U_mu(x - mu)^dag (1 +/- g) psi(x - mu)
  {
    long j = eo_neighbour(a.g, x, MU, -1, &cr);
    HalfSpinor<R> t;
    float sg = a.g.bc_t;
    if (MU == 0 && cr && fprev) {
      // x0 = 0: link and projection were applied by the previous sub-domain
      load_half<R>(fprev, a.g.Vh / a.g.L[0], i, t);
      sg = a.halo_sign_prev;
    } else {
      Spinor<R> nb;
      load_spinor<P, NC>(in, a.g.Vh, j, nb);
      HalfSpinor<R> h;
      project<MU, -SF>(nb, h);
      Su3<R> u;
      load_link<R, FMT>(a.links, a.g.Vh, 1 - p, MU, j, u);
      su3_dag_mul(u, h, t);
    }
    hop_accum<MU, -SF>(acc, t, w, cr, sg);
  }
}

// The double-float site, one right-hand side per thread, two lanes per
// instruction (df_pack.cuh).  In the hops the lanes are the two spins of the
// half spinor (the link is shared, the upper and lower spin pairs of the sum
// are two lanes each); in the clover term they are the two chiral blocks.  No
// lane belongs to another right-hand side, so the kernel keeps the registers
// of a scalar one (the two-rhs form of hop_df2.cuh needs 255).
//
// The hopping sum is one runtime loop over the 8 hops: unrolled, the
// double-float stencil is far beyond the instruction cache.  The spin
// projection for hop (mu, projector sign S) is h0 = p0 + i^c0 p[q0],
// h1 = p1 + i^c1 p[q1], the reconstruction acc2 += i^d0 t[r0],
// acc3 += i^d1 t[r1] (the maps of project / accum_reconstruct as tables;
// S = +1 adds 2 to every power): c0 and c1 (d0 and d1) are both even or both
// odd, so a power of i is one exchange of the real and imaginary pairs and
// per-lane signs.  A backward hop reads the link transposed and moves the
// conjugation into signed copies of h.
// 12 rhs on 48x24^3, both Dhat passes: 4.0 ms against 4.7 ms for the scalar
// form (16.5k instructions per site, 55 % of the binary32 pipe), each in its best
// launch; 1 rhs: 420 against 475 us.
namespace dfs {
using namespace df2;

// (sign of the real part, of the imaginary part) that i^c brings, see i_pow
__device__ __forceinline__ float ic_re(int c) { return (c & 3) == 1 || (c & 3) == 2 ? -1.f : 1.f; }
__device__ __forceinline__ float ic_im(int c) { return (c & 3) >= 2 ? -1.f : 1.f; }
// z i^c per lane: odd = the powers are odd, (sr, si) their signs
__device__ __forceinline__ C2 i_pow(const C2& z, bool odd, F2 sr, F2 si) {
  return C2{dsign(odd ? z.im : z.re, sr), dsign(odd ? z.re : z.im, si)};
}
// complex chunks of two components as a pair
__device__ __forceinline__ C2 pair(const float4& a, const float4& b) {
  return C2{D2{make_float2(a.x, b.x), make_float2(a.y, b.y)}, D2{make_float2(a.z, b.z), make_float2(a.w, b.w)}};
}

// up[c], lo[c]: colour c of the spin pairs (0, 1) and (2, 3); the hops are
// added without renormalising
template <bool DAG>
__device__ __forceinline__ void hop_loop(const HopArgs& a, const float4* in, int p, long i, const int x[4],
                                         C2 (&up)[3], C2 (&lo)[3]) {
  constexpr int SF = DAG ? +1 : -1;  // projector sign of the forward hop
  const long Vh = a.g.Vh;
#pragma unroll 1
  for (int k = 0; k < 8; ++k) {
    const int mu = k >> 1;
    const bool fwd = (k & 1) == 0;
    const int sh = ((fwd ? SF : -SF) > 0) ? 2 : 0;
    bool cr;
    const long j = eo_neighbour_rt(a.g, x, mu, fwd ? +1 : -1, &cr);
    // the link's elements (row r, column c), transposed for a backward hop
    const float4* ub =
        reinterpret_cast<const float4*>(a.links) + ((long)((fwd ? p : 1 - p) * 4 + mu) * 9) * Vh + (fwd ? i : j);
    const long sr = fwd ? 3 * Vh : Vh, sc = fwd ? Vh : 3 * Vh;
    float4 u[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) u[r][c] = ldg_nc(ub + r * sr + c * sc);
    const bool swq = (mu == 1 || mu == 2);  // q0 = 3, q1 = 2 (r0 = 1, r1 = 0)
    const int c0 = ((mu == 1 || mu == 3) ? 1 : 0) + sh;
    const int c1 = (mu == 0 ? 0 : mu == 1 ? 1 : mu == 2 ? 2 : 3) + sh;
    const F2 csr = make_float2(ic_re(c0), ic_re(c1)), csi = make_float2(ic_im(c0), ic_im(c1));
    const float4* nb = in + j;
    const float4* nq0 = nb + (swq ? 9 : 6) * Vh;
    const float4* nq1 = nb + (swq ? 6 : 9) * Vh;
    C2 h[3], g[3];  // the half spinor; its copy for the imaginary parts of the link
    const F2 cj = bc(fwd ? 1.f : -1.f);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const C2 n = pair(ldg_nc(nb + c * Vh), ldg_nc(nb + (3 + c) * Vh));
      const C2 m = i_pow(pair(ldg_nc(nq0 + c * Vh), ldg_nc(nq1 + c * Vh)), c0 & 1, csr, csi);
      h[c] = C2{add_lazy(n.re, m.re), add_lazy(n.im, m.im)};
      // u h = (ur + i s ui) h: re += ui (-s h.im), im += ui (s h.re), s = +-1
      g[c] = C2{dsign(h[c].re, cj), dneg(dsign(h[c].im, cj))};
    }
    const bool flip = cr && a.g.bc_t < 0.f;
    const int d0 = (mu == 0 ? 0 : mu == 1 ? 3 : mu == 2 ? 2 : 3) + sh;
    const int d1 = (mu == 0 ? 0 : mu == 1 ? 3 : mu == 2 ? 0 : 1) + sh;
    const F2 dsr = make_float2(ic_re(d0), ic_re(d1)), dsi = make_float2(ic_im(d0), ic_im(d1));
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      Acc re, im;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const dfloat ur(u[r][b].x, u[r][b].y), ui(u[r][b].z, u[r][b].w);
        if (b == 0) {
          acc_first(re, ur, h[b].re);
          acc_first(im, ur, h[b].im);
        } else {
          acc_add(re, ur, h[b].re);
          acc_add(im, ur, h[b].im);
        }
        acc_add(re, ui, g[b].im);
        acc_add(im, ui, g[b].re);
      }
      C2 t{acc_get(re), acc_get(im)};
      if (flip) t = cneg(t);
      up[r] = C2{add_lazy(up[r].re, t.re), add_lazy(up[r].im, t.im)};
      if (swq) {  // exchange the lanes
        t.re = D2{make_float2(t.re.hi.y, t.re.hi.x), make_float2(t.re.lo.y, t.re.lo.x)};
        t.im = D2{make_float2(t.im.hi.y, t.im.hi.x), make_float2(t.im.lo.y, t.im.lo.x)};
      }
      const C2 l = i_pow(t, d0 & 1, dsr, dsi);
      lo[r] = C2{add_lazy(lo[r].re, l.re), add_lazy(lo[r].im, l.im)};
    }
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    up[r] = C2{dnorm(up[r].re), dnorm(up[r].im)};
    lo[r] = C2{dnorm(lo[r].re), dnorm(lo[r].im)};
  }
}

// y = K x for both chiral blocks of a site (lane b: block b, component r =
// 3 (local spin) + colour); every component's products are summed in the order
// of its row (diagonal first), one entry of the blocks in registers at a time
__device__ __forceinline__ void clover(const void* base, long Vh, int p, long i, const C2 (&x)[6], C2 (&y)[6]) {
  const float4* q = reinterpret_cast<const float4*>(base) + (long)p * 36 * Vh + i;
  Acc re[6], im[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 w0 = ldg_nc(q + k * Vh), w1 = ldg_nc(q + (18 + k) * Vh);
    const D2 da{make_float2(w0.x, w1.x), make_float2(w0.y, w1.y)}, db{make_float2(w0.z, w1.z), make_float2(w0.w, w1.w)};
    acc_first(re[2 * k], da, x[2 * k].re);
    acc_first(im[2 * k], da, x[2 * k].im);
    acc_first(re[2 * k + 1], db, x[2 * k + 1].re);
    acc_first(im[2 * k + 1], db, x[2 * k + 1].im);
  }
  int n = 0;
#pragma unroll
  for (int r = 0; r < 6; ++r)
#pragma unroll
    for (int c = r + 1; c < 6; ++c) {
      const C2 o = pair(ldg_nc(q + (3 + n) * Vh), ldg_nc(q + (21 + n) * Vh));
      ++n;
      // y[r] += o x[c]
      acc_add(re[r], o.re, x[c].re);
      acc_add(re[r], o.im, dneg(x[c].im));
      acc_add(im[r], o.re, x[c].im);
      acc_add(im[r], o.im, x[c].re);
      // y[c] += conj(o) x[r]
      acc_add(re[c], o.re, x[r].re);
      acc_add(re[c], o.im, x[r].im);
      acc_add(im[c], o.re, x[r].im);
      acc_add(im[c], o.im, dneg(x[r].re));
    }
#pragma unroll
  for (int r = 0; r < 6; ++r) y[r] = C2{acc_get(re[r]), acc_get(im[r])};
}

// lanes (spin 0, spin 1) / (2, 3) of colour c <-> lanes (block 0, block 1) of
// component r = 3 s + c
__device__ __forceinline__ D2 lanes(D2 a, int la, D2 b, int lb) {
  return D2{make_float2(la ? a.hi.y : a.hi.x, lb ? b.hi.y : b.hi.x),
            make_float2(la ? a.lo.y : a.lo.x, lb ? b.lo.y : b.lo.x)};
}
__device__ __forceinline__ C2 lanes(const C2& a, int la, const C2& b, int lb) {
  return C2{lanes(a.re, la, b.re, lb), lanes(a.im, la, b.im, lb)};
}
__device__ __forceinline__ cx<dfloat> lane(const C2& z, int l) {
  return cx<dfloat>{dfloat(l ? z.re.hi.y : z.re.hi.x, l ? z.re.lo.y : z.re.lo.x),
                    dfloat(l ? z.im.hi.y : z.im.hi.x, l ? z.im.lo.y : z.im.lo.x)};
}

// One output site i (parity p) of right-hand side rhs; the site's
// contribution to the residual epilogue's norm (0 otherwise).  A in2 / w is
// formed first (w = +-1/2, so the scaling is exact), the unweighted hops add
// onto it and one final scaling gives A in2 + w H in.
template <int MODE, bool DAG, int EPI>
__device__ __forceinline__ double site(const HopArgs& a, long i, int rhs, int p) {
  int x[4];
  eo_coords(a.g, p, i, x);
  const long Vh = a.g.Vh;
  const long par_in = (MODE == HOP_DW) ? (long)(1 - p) * a.half_bytes : 0;
  const long par_out = (MODE == HOP_DW) ? (long)p * a.half_bytes : 0;
  const float4* in = reinterpret_cast<const float4*>((const char*)a.in + rhs * a.in_stride + par_in);
  constexpr float w = (MODE == HOP_P2) ? 0.5f : -0.5f;
  C2 up[3], lo[3], v[6], y[6];
  if constexpr (MODE != HOP_P1) {
    const float4* l = reinterpret_cast<const float4*>((const char*)a.in2 + rhs * a.in2_stride + par_out) + i;
#pragma unroll
    for (int r = 0; r < 6; ++r) v[r] = pair(ldg_nc(l + r * Vh), ldg_nc(l + (6 + r) * Vh));
    clover(a.clov, Vh, p, i, v, y);
#pragma unroll
    for (int r = 0; r < 6; ++r) y[r] = C2{dscale(y[r].re, 1.f / w), dscale(y[r].im, 1.f / w)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      up[c] = lanes(y[c], 0, y[3 + c], 0);
      lo[c] = lanes(y[c], 1, y[3 + c], 1);
    }
  } else {
    const D2 z{bc(0.f), bc(0.f)};
#pragma unroll
    for (int c = 0; c < 3; ++c) up[c] = lo[c] = C2{z, z};
  }
  hop_loop<DAG>(a, in, p, i, x, up, lo);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    up[c] = C2{dscale(up[c].re, w), dscale(up[c].im, w)};
    lo[c] = C2{dscale(lo[c].re, w), dscale(lo[c].im, w)};
  }
  Spinor<dfloat> res;
  if constexpr (MODE == HOP_P1) {
#pragma unroll
    for (int r = 0; r < 6; ++r) v[r] = lanes(up[r % 3], r / 3, lo[r % 3], r / 3);
    clover(a.cinv, Vh, p, i, v, y);
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      res.c[r / 3][r % 3] = lane(y[r], 0);
      res.c[2 + r / 3][r % 3] = lane(y[r], 1);
    }
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      res.c[0][c] = lane(up[c], 0);
      res.c[1][c] = lane(up[c], 1);
      res.c[2][c] = lane(lo[c], 0);
      res.c[3][c] = lane(lo[c], 1);
    }
  }
  double red = 0.0;
  if constexpr (EPI == EPI_RESID64) {
    Spinor<dfloat> e;
    load_spinor<P_DF64>((const char*)a.ep_eta + rhs * a.ep_eta_stride, Vh, i, e);
    // the site's 24 squares summed in double-float, one conversion
    dfloat acc2(0.f);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        res.c[s][c] = e.c[s][c] - res.c[s][c];
        acc2 = fma(res.c[s][c].re, res.c[s][c].re, fma(res.c[s][c].im, res.c[s][c].im, acc2));
      }
    red = (double)acc2;
  }
  store_spinor<P_DF64>((char*)a.out + rhs * a.out_stride + par_out, Vh, i, res);
  return red;
}

}  // namespace dfs

// value type of a site's reduction contribution: binary32 for the
// binary32-arithmetic types (their per-site norms are binary32 sums), else
// binary64 (see warp_total)
template <int P>
using RedT = typename std::conditional<P == P_F64 || P == P_DF64, double, float>::type;

// One output site i (parity p) of right-hand side rhs: the stencil, the
// clover term and the epilogue.  Returns the site's contribution to the
// epilogue's reduction (0 if none).
template <int P, int FMT, int MODE, bool DAG, int EPI>
__device__ __forceinline__ RedT<P> hop_site(const HopArgs& a, long i, int rhs, int p) {
  if constexpr (P == P_DF64) {
    return dfs::site<MODE, DAG, EPI>(a, i, rhs, p);
  } else {
    typedef typename PrecTraits<P>::R R;
    RedT<P> red = 0;
    int x[4];
    eo_coords(a.g, p, i, x);
    const long par_in = (MODE == HOP_DW) ? (long)(1 - p) * a.half_bytes : 0;
    const long par_out = (MODE == HOP_DW) ? (long)p * a.half_bytes : 0;
    const char* in = (const char*)a.in + rhs * a.in_stride + par_in;
    Spinor<R> acc;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc.c[s][c] = cx<R>{0, 0};
    const R w = (MODE == HOP_P2) ? (R)0.5 : (R)-0.5;
    const char* fn = nullptr;
    const char* fp = nullptr;
    if (a.halo_next) {  // sub-domain launch: faces of this rhs and output parity
      const long po = (MODE == HOP_DW) ? (long)p * a.halo_pstride : 0;
      fn = (const char*)a.halo_next + rhs * a.halo_stride + po;
      fp = (const char*)a.halo_prev + rhs * a.halo_stride + po;
    }
    // F32 Dw on 12-real links reads its neighbours by the non-coherent path, which
    // lets the compiler keep more of them in flight (32x24^3, 1 rhs: 65 against 76 us,
    // 3 rhs 153 against 184); on 18-real links it takes longer that way (83 against 73
    // us), elsewhere the path makes no difference.
    constexpr bool NC = P == P_F32 && FMT == LINK_12 && MODE == HOP_DW;
    hop_dir<P, FMT, 0, DAG, NC>(a, in, p, i, x, acc, w, fn, fp);
    hop_dir<P, FMT, 1, DAG, NC>(a, in, p, i, x, acc, w);
    hop_dir<P, FMT, 2, DAG, NC>(a, in, p, i, x, acc, w);
    hop_dir<P, FMT, 3, DAG, NC>(a, in, p, i, x, acc, w);

    Spinor<R> res;
    if constexpr (MODE == HOP_P1) {
      clover_apply<R>(a.cinv, a.g.Vh, p, i, acc, res);
    } else if constexpr (std::is_same<R, double>::value) {
      // binary64: A in2 added onto the sum of the hops by its own FMAs (24
      // additions fewer on the binary64 pipe than a sum of the two).  Hops added
      // onto A in2, the larger of the two, would round at its size every time:
      // error of Dw with a diagonal A against quadruple precision 1.4e-16, in
      // this order 8.3e-17, summed apart 9.5e-17 (8x6x4x10).
      Spinor<R> loc;
      load_spinor<P>((const char*)a.in2 + rhs * a.in2_stride + par_out, a.g.Vh, i, loc);
      res = acc;
      clover_apply<R, true>(a.clov, a.g.Vh, p, i, loc, res);
    } else {
      const char* in2 = (const char*)a.in2 + rhs * a.in2_stride + par_out;
      Spinor<R> loc, al;
      load_spinor<P>(in2, a.g.Vh, i, loc);
      clover_apply<R>(a.clov, a.g.Vh, p, i, loc, al);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) res.c[s][c] = al.c[s][c] + acc.c[s][c];
    }

    if constexpr (EPI == EPI_NONE || EPI == EPI_NORM) {
      store_spinor<P>((char*)a.out + rhs * a.out_stride + par_out, a.g.Vh, i, res);
      if constexpr (EPI == EPI_NORM) red = (RedT<P>)site_norm2(res);
    } else if constexpr (EPI == EPI_CG) {
      // q = res; x += alpha p; r -= alpha q  (x in F64 for F64 solves, else F32)
      constexpr int XP = (P == P_F64) ? P_F64 : P_F32;
      typedef typename PrecTraits<XP>::R RX;
      const CgState& st = a.cg[rhs];
      const R al = (R)st.alpha;
      Spinor<R> pv, rv;
      Spinor<RX> xv;
      load_spinor<P>((const char*)a.ep_p + rhs * a.ep_p_stride, a.g.Vh, i, pv);
      load_spinor<P>((const char*)a.ep_r + rhs * a.ep_r_stride, a.g.Vh, i, rv);
      load_spinor<XP>((const char*)a.ep_x + rhs * a.ep_x_stride, a.g.Vh, i, xv);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          xv.c[s][c].re = fma((RX)al, (RX)pv.c[s][c].re, xv.c[s][c].re);
          xv.c[s][c].im = fma((RX)al, (RX)pv.c[s][c].im, xv.c[s][c].im);
          rv.c[s][c].re = fma(-al, res.c[s][c].re, rv.c[s][c].re);
          rv.c[s][c].im = fma(-al, res.c[s][c].im, rv.c[s][c].im);
        }
      // the norm of what is stored (rounded to the storage type)
      round_trip<P>(rv);
      store_spinor<XP>((char*)a.ep_x + rhs * a.ep_x_stride, a.g.Vh, i, xv);
      store_spinor<P>((char*)a.ep_r + rhs * a.ep_r_stride, a.g.Vh, i, rv);
      red = (RedT<P>)site_norm2(rv);
    } else if constexpr (EPI == EPI_RESID64) {
      Spinor<R> e;
      load_spinor<P>((const char*)a.ep_eta + rhs * a.ep_eta_stride, a.g.Vh, i, e);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) res.c[s][c] = e.c[s][c] - res.c[s][c];
      store_spinor<P>((char*)a.out + rhs * a.out_stride, a.g.Vh, i, res);
      double acc2 = 0.0;
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double re = (double)res.c[s][c].re, im = (double)res.c[s][c].im;
          acc2 += re * re + im * im;
        }
      red = acc2;
    }
    return red;
  }
}

template <int P, int FMT, int MODE, bool DAG, int EPI>
__device__ __forceinline__ void hop_kernel_body(const HopArgs& a, double* red_smem) {
  // CTA = blockDim.x sites x blockDim.y right-hand sides (one rhs per row:
  // the rows read the same links and clover blocks, served by L1).  The
  // grid index runs fastest over the rhs tiles of one site block, then (for
  // HOP_DW) over the two parities, then over site blocks, so that CTAs that
  // read the same links are resident at the same time and share them in L2.
  const unsigned ntile = (a.nrhs + blockDim.y - 1) / blockDim.y;
  const unsigned tile = blockIdx.x % ntile;
  const unsigned rest = blockIdx.x / ntile;
  const long blk = (MODE == HOP_DW) ? (long)(rest >> 1) : (long)rest;
  const long i = blk * blockDim.x + threadIdx.x;
  const int rhs = tile * blockDim.y + threadIdx.y;
  const int p = (MODE == HOP_DW) ? (int)(rest & 1) : a.p;
  record_live(a);
  const bool off = a.cg && rhs < a.nrhs && a.cg[rhs].mode != a.gate;  // gated off by the solver state
  const bool live = (i < a.g.Vh) && (rhs < a.nrhs) && !off;
  RedT<P> red = 0;
  if (live) red = hop_site<P, FMT, MODE, DAG, EPI>(a, i, rhs, p);
  if constexpr (EPI != EPI_NONE) {
    grid_reduce(red, a.red, rhs, a.nrhs, red_smem, (unsigned)blk, gridDim.x / ntile, off);
  }
}

template <int P, int FMT, int MODE, bool DAG, int EPI>
__global__ void __launch_bounds__(256) hop_kernel(const HopArgs a) {
  extern __shared__ double red_smem[];
  hop_kernel_body<P, FMT, MODE, DAG, EPI>(a, red_smem);
}

// double-float only: at most 128 threads and 128 registers per thread, so
// that 16 warps fit on an SM (the tuner weighs it against hop_kernel), or
// 168 registers for 12 warps (fewer spills)
template <int P, int FMT, int MODE, bool DAG, int EPI>
__global__ void __launch_bounds__(128, 4) hop_kernel_capped(const HopArgs a) {
  extern __shared__ double red_smem[];
  hop_kernel_body<P, FMT, MODE, DAG, EPI>(a, red_smem);
}
template <int P, int FMT, int MODE, bool DAG, int EPI>
__global__ void __launch_bounds__(128, 3) hop_kernel_capped3(const HopArgs a) {
  extern __shared__ double red_smem[];
  hop_kernel_body<P, FMT, MODE, DAG, EPI>(a, red_smem);
}

// Batched form over several systems (lattices / operators of any size, one
// right-hand side each): CTA t takes tile t = (system, site block); every
// system has its own arguments, solver state and reduction scratch in device
// memory.  For HOP_DW the block index carries the parity in its lowest bit.
// Double-float: 64 sites per CTA at 168 registers (12 warps per SM).  (A grid
// of 8 CTAs per SM walking the list left its last round to few SMs: the F16
// batch of 8^4 and 32x16^3 systems 20.6 against 19.8 ms.)
template <int P, int FMT, int MODE, bool DAG, int EPI>
__global__ void __launch_bounds__(P == P_DF64 ? 64 : 256, P == P_DF64 ? 6 : 1)
    hop_batch_kernel(const HopArgs* __restrict__ sys, const int2* __restrict__ tiles) {
  extern __shared__ double red_smem[];
  const int2 tl = tiles[blockIdx.x];
  const HopArgs& a = sys[tl.x];
  if (a.cg && a.cg[0].mode != a.gate) return;  // the system is gated off by its solver state, in all of its CTAs
  const long blk = (MODE == HOP_DW) ? (long)(tl.y >> 1) : (long)tl.y;
  const int p = (MODE == HOP_DW) ? (tl.y & 1) : a.p;
  const long i = blk * blockDim.x + threadIdx.x;
  RedT<P> red = 0;
  if (i < a.g.Vh) red = hop_site<P, FMT, MODE, DAG, EPI>(a, i, 0, p);
  if constexpr (EPI != EPI_NONE) {
    const unsigned nblk = (unsigned)((a.g.Vh + blockDim.x - 1) / blockDim.x);
    grid_reduce(red, a.red, 0, 1, red_smem, (unsigned)blk, nblk);
  }
}

template <int P, int FMT, int MODE, bool DAG, int EPI>
static cudaError_t launch_one(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  dim3 block(L.bx, L.by, 1);
  const unsigned nb = (unsigned)((a.g.Vh + L.bx - 1) / L.bx);
  const unsigned ntile = (unsigned)((a.nrhs + L.by - 1) / L.by);
  dim3 grid((MODE == HOP_DW ? 2u * nb : nb) * ntile, 1u, 1u);
  size_t smem = (EPI == EPI_NONE) ? 0 : sizeof(double) * (L.bx / 32) * L.by;
  if (L.sys) {  // the binary32-arithmetic types run batches in hop_pair_batch_kernel
    if constexpr (P == P_F64 || P == P_DF64) {
      dim3 bblock(L.bx, 1, 1);
      if (P == P_DF64 && L.bx > 64) return cudaErrorInvalidValue;
      hop_batch_kernel<P, FMT, MODE, DAG, EPI>
          <<<L.ntiles, bblock, (EPI == EPI_NONE) ? 0 : sizeof(double) * (L.bx / 32), s>>>(L.sys, L.tiles);
      return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
  }
  if constexpr (P == P_DF64) {
    if (L.regcap) {
      if (L.bx * L.by > 128) return cudaErrorInvalidValue;
      if (L.regcap == 2)
        hop_kernel_capped3<P, FMT, MODE, DAG, EPI><<<grid, block, smem, s>>>(a);
      else
        hop_kernel_capped<P, FMT, MODE, DAG, EPI><<<grid, block, smem, s>>>(a);
      return cudaGetLastError();
    }
  }
  hop_kernel<P, FMT, MODE, DAG, EPI><<<grid, block, smem, s>>>(a);
  return cudaGetLastError();
}

template <int P, int FMT, bool DAG>
static cudaError_t dispatch_mode_epi(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  switch (L.mode) {
    case HOP_DW:
      if (L.epi == EPI_NONE) return launch_one<P, FMT, HOP_DW, DAG, EPI_NONE>(L, a, s);
      break;
    case HOP_P1:
      if (L.epi == EPI_NONE) return launch_one<P, FMT, HOP_P1, DAG, EPI_NONE>(L, a, s);
      break;
    case HOP_P2:
      if (L.epi == EPI_NONE) return launch_one<P, FMT, HOP_P2, DAG, EPI_NONE>(L, a, s);
      if constexpr (P != P_DF64) {
        if (L.epi == EPI_NORM) return launch_one<P, FMT, HOP_P2, DAG, EPI_NORM>(L, a, s);
        if (L.epi == EPI_CG) return launch_one<P, FMT, HOP_P2, DAG, EPI_CG>(L, a, s);
      }
      if constexpr (P == P_F64 || P == P_DF64)
        if (L.epi == EPI_RESID64) return launch_one<P, FMT, HOP_P2, DAG, EPI_RESID64>(L, a, s);
      break;
  }
  return cudaErrorInvalidValue;
}

template <int P, int FMT>
static cudaError_t dispatch_dag(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  return L.dagger ? dispatch_mode_epi<P, FMT, true>(L, a, s) : dispatch_mode_epi<P, FMT, false>(L, a, s);
}

}  // namespace oq
