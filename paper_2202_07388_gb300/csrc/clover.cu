// Clover term: A(x) = (4 + m0) + c_sw (i/4) sum_{mu,nu} sigma_{mu nu} F_{mu nu}(x)
// (QCD+QED with separate coefficients: c_sw F -> c_sw F^{SU(3)} + c_sw^QED
// F^{U(1)} 1_colour; Schroedinger-functional lattices: 4 + m0 + c_F - 1 at
// x0 = 1 and T-1)
// with the clover-leaf field strength F = (Q - Q^dag)/8, Q the sum of the four
// plaquettes at x in the (mu, nu) plane.  In the chiral basis
// sigma_{0k} = diag(s_k, -s_k) and sigma_{jk} = -eps_{jkl} diag(s_l, s_l), so A
// splits into two Hermitian 6x6 blocks (index 3*spin + colour):
//
//   block(+) = c0 + sum_k s_k (x) (i c_sw / 2)(F_0k - Fd_k)
//   block(-) = c0 - sum_k s_k (x) (i c_sw / 2)(F_0k + Fd_k)
//
// with Fd_1 = F_23, Fd_2 = -F_13, Fd_3 = F_12 and c0 = 4 + m0.  Everything
// is built and inverted in binary64, then stored in binary64 and binary32.
//
// The build is bound by the binary64 pipe (2 lanes per SM and clock on
// GB300), so it is arranged to do each product once: a thread per plaquette
// (not per leaf) forms U_mu(x) U_nu(x+mu) and U_nu(x) U_mu(x+nu) and from them
// the anti-Hermitian parts of the plaquette seen from its four corners
// (clover_plaq_kernel), a thread per site sums the four plaquettes around it
// (clover_gather_kernel), and the blocks are inverted in registers by
// symmetric elimination on their upper triangles (clover_block_kernel).
// That is ~5.9k binary64 operations per site, against ~12.5k and 9.9 KB of
// local memory per thread when one thread formed the 24 leaves of its site
// and ran Gauss-Jordan on the 6x12 systems: 32^4 takes 11 ms instead of 38.8
// (9.8 ms of binary64 operations at 0.63 T per second).
// The intermediate fields live in the output arrays: the corner matrices of
// two planes in the 72 reals per site of the inverse, the six field strengths
// in those of A, so the build needs no memory of its own.
#include "oq_internal.h"
#include "oq_kernels.h"

namespace oq {

typedef cx<double> cd;
struct M3 {
  cd m[3][3];
};

__device__ __forceinline__ M3 mul(const M3& a, const M3& b) {
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cd s = a.m[i][0] * b.m[0][j];
      cfma(s, a.m[i][1], b.m[1][j]);
      cfma(s, a.m[i][2], b.m[2][j]);
      c.m[i][j] = s;
    }
  return c;
}
// a^dag * b
__device__ __forceinline__ M3 dmul(const M3& a, const M3& b) {
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cd s = cmulc(a.m[0][i], b.m[0][j]);
      cfmac(s, a.m[1][i], b.m[1][j]);
      cfmac(s, a.m[2][i], b.m[2][j]);
      c.m[i][j] = s;
    }
  return c;
}

// y += d mu (d = -1, 0, +1) on the periodic lattice, with the x1 shift of a
// C* boundary when the step wraps
__device__ __forceinline__ void displace(const Geom& g, int y[4], int mu, int d) {
  if (!d) return;
  int v = y[mu] + d;
  const bool wrap = v < 0 || v >= g.L[mu];
  y[mu] = (v + g.L[mu]) % g.L[mu];
  if (wrap) y[1] = cs_x1(g, mu, y[1]);
}

// the link U_mu(y), y = x + d1 mu1 + d2 mu2; with au1 times exp(i q A_mu(y))
__device__ __forceinline__ M3 link_at(const Geom& g, const double2* u64, const int x[4], int mu, int d1, int mu1,
                                      int d2, int mu2, const double* au1 = nullptr, double q = 0.0) {
  int y[4] = {x[0], x[1], x[2], x[3]};
  displace(g, y, mu1, d1);
  displace(g, y, mu2, d2);
  const int p = (y[0] + y[1] + y[2] + y[3]) & 1;
  const long j = eo_index(g, y);
  Su3<double> u;
  load_link<double, LINK_18>(u64, g.Vh, p, mu, j, u);
  cd ph = cd{1.0, 0.0};
  if (au1) {
    double sn, cs;
    sincos(q * au1[(long)(p * 4 + mu) * g.Vh + j], &sn, &cs);
    ph = cd{cs, sn};
  }
  M3 r;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) r.m[a][b] = au1 ? u.m[a][b] * ph : u.m[a][b];
  return r;
}

// U(1) angle A_mu(y) at y = x + d1 mu1 + d2 mu2 (packed [parity][mu][site])
__device__ __forceinline__ double angle_at(const Geom& g, const double* au1, const int x[4], int mu, int d1,
                                           int mu1, int d2, int mu2) {
  int y[4] = {x[0], x[1], x[2], x[3]};
  displace(g, y, mu1, d1);
  displace(g, y, mu2, d2);
  const int p = (y[0] + y[1] + y[2] + y[3]) & 1;
  return au1[(long)(p * 4 + mu) * g.Vh + eo_index(g, y)];
}

// invert a general 6x6 complex matrix in place (Gauss-Jordan, partial pivoting)
__device__ __noinline__ bool invert6(cd a[6][6], cd inv[6][6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) inv[i][j] = cd{i == j ? 1.0 : 0.0, 0.0};
  for (int c = 0; c < 6; ++c) {
    int piv = c;
    double best = a[c][c].re * a[c][c].re + a[c][c].im * a[c][c].im;
    for (int r = c + 1; r < 6; ++r) {
      double v = a[r][c].re * a[r][c].re + a[r][c].im * a[r][c].im;
      if (v > best) { best = v; piv = r; }
    }
    if (!(best > 0.0)) return false;
    if (piv != c) {
      for (int j = 0; j < 6; ++j) {
        cd t = a[c][j]; a[c][j] = a[piv][j]; a[piv][j] = t;
        t = inv[c][j]; inv[c][j] = inv[piv][j]; inv[piv][j] = t;
      }
    }
    cd d = a[c][c];
    double n2 = d.re * d.re + d.im * d.im;
    cd dinv = cd{d.re / n2, -d.im / n2};
    for (int j = 0; j < 6; ++j) {
      a[c][j] = a[c][j] * dinv;
      inv[c][j] = inv[c][j] * dinv;
    }
    for (int r = 0; r < 6; ++r) {
      if (r == c) continue;
      cd f = a[r][c];
      for (int j = 0; j < 6; ++j) {
        a[r][j] = a[r][j] - f * a[c][j];
        inv[r][j] = inv[r][j] - f * inv[c][j];
      }
    }
  }
  return true;
}

// An anti-Hermitian 3x3 matrix as 9 reals: the imaginary diagonal parts, then
// re, im of the entries (0,1), (0,2), (1,2).
struct Ah3 {
  double v[9];
};

// The anti-Hermitian part M - M^dag of M = a b^dag (AD = false: rows of both)
// or M = a^dag b (AD = true: columns of both)
template <bool AD>
__device__ __forceinline__ Ah3 ah_product(const M3& a, const M3& b) {
  Ah3 k;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double im = 0.0;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      const cd x = AD ? conj(a.m[l][i]) : a.m[i][l], y = AD ? b.m[l][i] : conj(b.m[i][l]);
      im = fma(x.re, y.im, fma(x.im, y.re, im));
    }
    k.v[i] = 2.0 * im;
  }
  int n = 3;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i + 1; j < 3; ++j) {
      // M_ij - conj(M_ji)
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        const cd x = AD ? conj(a.m[l][i]) : a.m[i][l], y = AD ? b.m[l][j] : conj(b.m[j][l]);
        re = fma(x.re, y.re, fma(-x.im, y.im, re));
        im = fma(x.re, y.im, fma(x.im, y.re, im));
        const cd z = AD ? conj(a.m[l][j]) : a.m[j][l], w = AD ? b.m[l][i] : conj(b.m[i][l]);
        re = fma(-z.re, w.re, fma(z.im, w.im, re));
        im = fma(z.re, w.im, fma(z.im, w.re, im));
      }
      k.v[n++] = re;
      k.v[n++] = im;
    }
  return k;
}

// the planes in the order F_01, F_02, F_03, F_12, F_13, F_23
__device__ __forceinline__ void plane_dirs(int plane, int* mu, int* nu) {
  *mu = plane < 3 ? 0 : plane < 5 ? 1 : 2;
  *nu = plane < 3 ? plane + 1 : plane < 5 ? plane - 1 : 3;
}

// The plaquette of planes plane0 + blockIdx.z at every site, seen from its
// corners: K = L - L^dag of the leaf L of F_{mu nu} that runs around it,
//   corner x        : U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
//   corner x+mu     : U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag U_mu(x)
//   corner x+mu+nu  : U_mu(x+nu)^dag U_nu(x)^dag U_mu(x) U_nu(x+mu)
//   corner x+nu     : U_nu(x)^dag U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag
// stored at corner[parity][36 z + 9 corner + r][site].  au1: the links times
// exp(i q A).  sin1: also sin(q theta) of the plaquette's U(1) angle (the
// separate QED clover) into real z of pair chunk 27 + plane0 / 2 of the
// per-site 36 pairs (the field strengths use the first 27).
__global__ void __launch_bounds__(128) clover_plaq_kernel(Geom g, const double2* __restrict__ u64,
                                                          const double* __restrict__ au1, double q, int plane0,
                                                          int phase, double* __restrict__ corner, double* sin1) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = blockIdx.y, z = blockIdx.z;
  if (i >= g.Vh) return;
  int x[4], mu, nu;
  eo_coords(g, p, i, x);
  plane_dirs(plane0 + z, &mu, &nu);
  const double* ph = phase ? au1 : nullptr;
  double* out = corner + ((long)p * 72 + 36 * z) * g.Vh + i;
  auto store = [&](int c, const Ah3& k) {
#pragma unroll
    for (int r = 0; r < 9; ++r) out[(9 * c + r) * g.Vh] = k.v[r];
  };
  const M3 umx = link_at(g, u64, x, mu, 0, 0, 0, 0, ph, q);
  const M3 un_xpm = link_at(g, u64, x, nu, +1, mu, 0, 0, ph, q);
  const M3 unx = link_at(g, u64, x, nu, 0, 0, 0, 0, ph, q);
  const M3 um_xpn = link_at(g, u64, x, mu, +1, nu, 0, 0, ph, q);
  const M3 lo = mul(umx, un_xpm), hi = mul(unx, um_xpn);
  store(0, ah_product<false>(lo, hi));
  store(2, ah_product<true>(hi, lo));
  // corner x+mu: U_nu(x+mu) (hi^dag U_mu(x)), the second factor's dagger U_mu(x)^dag hi
  store(1, ah_product<false>(un_xpm, dmul(umx, hi)));
  // corner x+nu: (U_nu(x)^dag lo) U_mu(x+nu)^dag
  store(3, ah_product<false>(dmul(unx, lo), um_xpn));
  if (sin1) {
    const double th = angle_at(g, au1, x, mu, 0, 0, 0, 0) + angle_at(g, au1, x, nu, +1, mu, 0, 0) -
                      angle_at(g, au1, x, mu, +1, nu, 0, 0) - angle_at(g, au1, x, nu, 0, 0, 0, 0);
    sin1[(((long)p * 36 + 27 + plane0 / 2) * g.Vh + i) * 2 + z] = sin(q * th);
  }
}

// c_sw F of planes plane0 and plane0 + 1 at every site: the sum of the four
// plaquettes around it, 18 reals in pair chunks 9 plane0 / 2 .. + 8 of f
// (the layout of A: [parity][36][site] pairs).  sin1: + i c_sw^QED / 4 times
// the sum of the plaquettes' sin(q theta) on the diagonal (the U(1) clover
// leaves of exp(i q A), (Q - Q^*) / 8).
__global__ void __launch_bounds__(128) clover_gather_kernel(Geom g, const double* __restrict__ corner,
                                                            double csw, double csw_qed, int plane0,
                                                            const double* sin1, double2* f) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = blockIdx.y;
  if (i >= g.Vh) return;
  int x[4];
  eo_coords(g, p, i, x);
  double v[18];
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    int mu, nu;
    plane_dirs(plane0 + z, &mu, &nu);
    double e = 0.0;
#pragma unroll
    for (int r = 0; r < 9; ++r) v[9 * z + r] = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      // the plaquette whose corner c is x starts at x, x-mu, x-mu-nu, x-nu
      int y[4] = {x[0], x[1], x[2], x[3]};
      if (c == 1 || c == 2) displace(g, y, mu, -1);
      if (c == 2 || c == 3) displace(g, y, nu, -1);
      const int py = (y[0] + y[1] + y[2] + y[3]) & 1;
      const long j = eo_index(g, y);
      const double* k = corner + ((long)py * 72 + 36 * z + 9 * c) * g.Vh + j;
#pragma unroll
      for (int r = 0; r < 9; ++r) v[9 * z + r] += k[r * g.Vh];
      if (sin1) e += sin1[(((long)py * 36 + 27 + plane0 / 2) * g.Vh + j) * 2 + z];
    }
#pragma unroll
    for (int r = 0; r < 9; ++r) v[9 * z + r] *= 0.125 * csw;
    if (sin1) {
#pragma unroll
      for (int r = 0; r < 3; ++r) v[9 * z + r] += 0.25 * csw_qed * e;
    }
  }
  double2* o = f + ((long)p * 36 + 9 * (plane0 / 2)) * g.Vh + i;
#pragma unroll
  for (int k = 0; k < 9; ++k) o[k * g.Vh] = make_double2(v[2 * k], v[2 * k + 1]);
}

// index of the upper entry (r, c), r < c, among the 15 in row-major order
__host__ __device__ constexpr int up6(int r, int c) { return r * 5 - r * (r - 1) / 2 + (c - r - 1); }

// A Hermitian 6x6 block: real diagonal and the 15 upper entries.
struct H6 {
  double d[6];
  cd o[15];
};

__device__ __forceinline__ cd h6_get(const H6& m, int r, int c) {  // r != c
  return r < c ? m.o[up6(r, c)] : conj(m.o[up6(c, r)]);
}
// exponent-and-leading-bits word of |v|
__device__ __forceinline__ int mag_hi(double v) { return __double2hiint(v) & 0x7fffffff; }

// Invert in place by symmetric elimination without pivoting (one "sweep" per
// index; the matrix stays Hermitian, ~70 binary64 operations each).  False,
// with m undefined, if a pivot is zero, not finite, or below about half of the
// largest entry of its column, when growth would cost accuracy.
__device__ __forceinline__ bool h6_invert(H6& m) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double d = m.d[k];
    cd v[6], w[6];
    int top = 0;
#pragma unroll
    for (int r = 0; r < 6; ++r)
      if (r != k) {
        v[r] = h6_get(m, r, k);
        top = max(top, max(mag_hi(v[r].re), mag_hi(v[r].im)));
      }
    const int hd = mag_hi(d);
    ok = ok && hd >= 0x00100000 && hd < 0x7ff00000 && top <= hd + (1 << 20);
    const double inv = 1.0 / d;
#pragma unroll
    for (int r = 0; r < 6; ++r)
      if (r != k) w[r] = inv * v[r];
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      if (r == k) continue;
      m.d[r] = fma(-w[r].re, v[r].re, fma(-w[r].im, v[r].im, m.d[r]));
#pragma unroll
      for (int c = r + 1; c < 6; ++c) {
        if (c == k) continue;
        // a_rc -= w_r conj(v_c)
        cd& o = m.o[up6(r, c)];
        o.re = fma(-w[r].re, v[c].re, fma(-w[r].im, v[c].im, o.re));
        o.im = fma(-w[r].im, v[c].re, fma(w[r].re, v[c].im, o.im));
      }
    }
#pragma unroll
    for (int r = 0; r < 6; ++r)
      if (r != k) m.o[r < k ? up6(r, k) : up6(k, r)] = r < k ? w[r] : conj(w[r]);
    m.d[k] = -inv;
  }
#pragma unroll
  for (int r = 0; r < 6; ++r) m.d[r] = -m.d[r];
#pragma unroll
  for (int r = 0; r < 15; ++r) m.o[r] = -m.o[r];
  return ok;
}

// the general inversion (Gauss-Jordan with partial pivoting) of a Hermitian
// block, Hermitian part of the result; false if singular
__device__ __noinline__ bool h6_invert_pivoted(const double* in, double* out) {
  cd a[6][6], inv[6][6];
  for (int r = 0; r < 6; ++r)
    for (int c = 0; c < 6; ++c) {
      const int k = 6 + 2 * (r < c ? up6(r, c) : up6(c, r));
      a[r][c] = r == c ? cd{in[r], 0.0} : cd{in[k], r < c ? in[k + 1] : -in[k + 1]};
    }
  const bool ok = invert6(a, inv);
  for (int r = 0; r < 6; ++r) {
    out[r] = inv[r][r].re;
    for (int c = r + 1; c < 6; ++c) {
      out[6 + 2 * up6(r, c)] = 0.5 * (inv[r][c].re + inv[c][r].re);
      out[7 + 2 * up6(r, c)] = 0.5 * (inv[r][c].im - inv[c][r].im);
    }
  }
  return ok;
}

// one Hermitian block into the packed arrays
__device__ __forceinline__ void store_block(const Geom& g, int p, long i, int b, const H6& m, double2* a64,
                                            float4* a32) {
  double r[36];
#pragma unroll
  for (int k = 0; k < 6; ++k) r[k] = m.d[k];
#pragma unroll
  for (int k = 0; k < 15; ++k) {
    r[6 + 2 * k] = m.o[k].re;
    r[7 + 2 * k] = m.o[k].im;
  }
  double2* q64 = a64 + (long)p * 36 * g.Vh;
#pragma unroll
  for (int c = 0; c < 18; ++c) q64[(18 * b + c) * g.Vh + i] = make_double2(r[2 * c], r[2 * c + 1]);
  float4* q32 = a32 + (long)p * 18 * g.Vh;
#pragma unroll
  for (int c = 0; c < 9; ++c)
    q32[(9 * b + c) * g.Vh + i] =
        make_float4(narrow(r[4 * c]), narrow(r[4 * c + 1]), narrow(r[4 * c + 2]), narrow(r[4 * c + 3]));
}

// A and A^{-1} from the six field strengths c_sw F that a64 holds in its first
// 27 pair chunks (a thread reads and overwrites its own site only)
__global__ void __launch_bounds__(128) clover_block_kernel(Geom g, double c0, double cF, double2* a64, float4* a32,
                                                           double2* i64, float4* i32, int* status) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = blockIdx.y;
  if (i >= g.Vh) return;
  int x[4];
  eo_coords(g, p, i, x);
  double f[54];
  const double2* src = a64 + (long)p * 36 * g.Vh + i;
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    const double2 w = src[k * g.Vh];
    f[2 * k] = w.x;
    f[2 * k + 1] = w.y;
  }
  // Schroedinger-functional boundary improvement: + (c_F - 1) at x0 = 1, T-1
  if (g.bc_t == 0.f && (x[0] == 1 || x[0] == g.L[0] - 1)) c0 += cF - 1.0;
#pragma unroll 1
  for (int b = 0; b < 2; ++b) {
    // G_k = F_0k - Fd_k (b = 0) or -(F_0k + Fd_k) (b = 1): 9 reals each;
    // X_k = (i / 2) G_k is Hermitian: diagonal -G/2, upper entries i G / 2
    const double sa = b == 0 ? 1.0 : -1.0;
    double gk[3][9];
#pragma unroll
    for (int r = 0; r < 9; ++r) {
      gk[0][r] = fma(sa, f[r], -f[45 + r]);       // F_01, F_23
      gk[1][r] = fma(sa, f[9 + r], f[36 + r]);    // F_02, F_13
      gk[2][r] = fma(sa, f[18 + r], -f[27 + r]);  // F_03, F_12
    }
    H6 m;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double t = -0.5 * gk[2][a];
      m.d[a] = c0 + t;
      m.d[a + 3] = c0 - t;
      // the diagonal of Y = X1 - i X2
      m.o[up6(a, a + 3)] = cd{-0.5 * gk[0][a], 0.5 * gk[1][a]};
    }
    int n = 3;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int c = a + 1; c < 3; ++c) {
        const cd x1 = cd{-0.5 * gk[0][n + 1], 0.5 * gk[0][n]}, x2 = cd{-0.5 * gk[1][n + 1], 0.5 * gk[1][n]},
                 x3 = cd{-0.5 * gk[2][n + 1], 0.5 * gk[2][n]};
        m.o[up6(a, c)] = x3;
        m.o[up6(a + 3, c + 3)] = -x3;
        m.o[up6(a, c + 3)] = x1 - times_i(x2);
        m.o[up6(c, a + 3)] = conj(x1) - times_i(conj(x2));  // X is Hermitian
        n += 2;
      }
    store_block(g, p, i, b, m, a64, a32);
    H6 w = m;
    if (!h6_invert(w)) {
      double pk[36], iv[36];
#pragma unroll
      for (int r = 0; r < 6; ++r) pk[r] = m.d[r];
#pragma unroll
      for (int r = 0; r < 15; ++r) {
        pk[6 + 2 * r] = m.o[r].re;
        pk[7 + 2 * r] = m.o[r].im;
      }
      if (!h6_invert_pivoted(pk, iv)) atomicExch(status, 1);
#pragma unroll
      for (int r = 0; r < 6; ++r) w.d[r] = iv[r];
#pragma unroll
      for (int r = 0; r < 15; ++r) w.o[r] = cd{iv[6 + 2 * r], iv[7 + 2 * r]};
    }
    store_block(g, p, i, b, w, i64, i32);
  }
}

// qed: 0 = F of the links alone; 1 = F of the links times exp(i q A) (the
// U(3) clover); 2 = csw F(links) + csw_qed F(exp(i q A)) 1_colour
cudaError_t build_clover(const Geom& g, const double* links, const double* au1, double q, int qed_split,
                         double kappa, double csw, double csw_qed, double cF, double* a64, float* a32,
                         double* i64, float* i32, int* status_dev, cudaStream_t s) {
  const double c0 = 1.0 / (2.0 * kappa);
  const int qed = au1 ? (qed_split ? 2 : 1) : 0;
  const double2* u = reinterpret_cast<const double2*>(links);
  double* sin1 = qed == 2 ? a64 : nullptr;
  dim3 block(128), grid((unsigned)((g.Vh + 127) / 128), 2), grid2(grid.x, 2, 2);
  for (int plane0 = 0; plane0 < 6; plane0 += 2) {
    clover_plaq_kernel<<<grid2, block, 0, s>>>(g, u, au1, q, plane0, qed == 1, i64, sin1);
    clover_gather_kernel<<<grid, block, 0, s>>>(g, i64, csw, csw_qed, plane0, sin1,
                                                reinterpret_cast<double2*>(a64));
  }
  clover_block_kernel<<<grid, block, 0, s>>>(g, c0, cF, reinterpret_cast<double2*>(a64),
                                             reinterpret_cast<float4*>(a32), reinterpret_cast<double2*>(i64),
                                             reinterpret_cast<float4*>(i32), status_dev);
  return cudaGetLastError();
}

}  // namespace oq
