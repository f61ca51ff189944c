// Schwarz alternating procedure (Sec. 3, Figs. 2-3) as one kernel per colour.
//
// The lattice is cut into blocks of bs[0] x ... x bs[3] sites; block colour =
// parity of the sum of its block coordinates (an even number of blocks per
// direction, so blocks of one colour never touch).  One CTA handles one block
// of the requested colour, one thread per block site:
//
//   1. r_i = (rho - D phi)_i with the full stencil (neighbours in the
//      other-colour blocks carry the latest boundary values; phi of this
//      colour is only written by this CTA, at the end);
//   2. MR steps on the block operator D_i (Dirichlet: hops leaving the block
//      dropped, clover kept), with r_i in shared memory ([component][site]
//      for conflict-free neighbour reads), p = D_i r in registers:
//      omega = <p, r> / <p, p>, x += omega r, r -= omega p;
//      the adaptive variant (Sec. 3.2) leaves the loop when, after at least
//      4 steps, ||r|| > alpha ||r_prev||, when ||r|| grew, or when ||r|| fell
//      below tol = res ||eta|| / n_blocks; every decision is block-uniform;
//   3. phi_i += x.
// sap_block_eo_kernel replaces 2 by MR steps on the block's even-odd Schur
// complement (see below).  Arithmetic and storage are binary32, the norms of the
// adaptive exit tests binary64.
// sap_block_kernel (the default) keeps a site's links in registers and the
// block's clover in shared memory; sap_kernel reads them from global memory.
#include "oq_internal.h"
#include "oq_kernels.h"
#include "hop_impl.cuh"

namespace oq {

struct SapArgs {
  Geom g;
  int bs[4];
  int nb[4];
  int colour;
  int first;           // first cycle: phi is zero on this colour (colour 0: everywhere)
  const void* links;   // binary32 packed links
  const void* clov;    // binary32 packed clover
  const void* clov_inv;  // binary32 packed inverse clover (even-odd block solver)
  SapBlocked blk;        // copies of a site's own links and clover in block order (null: none)
  const char* rho;     // packed binary32 full field
  char* phi;           // packed binary32 full field, updated in place
  long half_bytes;
  int nmr;
  int adaptive;
  float alpha;
  double tol;          // adaptive exit 3 (absolute block norm)
  unsigned* mr_steps;  // accumulated MR steps over all blocks (may be null)
};

__device__ __forceinline__ void load_smem(const float* sm, int nsite, int t, Spinor<float>& s) {
#pragma unroll
  for (int k = 0; k < 12; ++k) s.c[k / 3][k % 3] = cx<float>{sm[(2 * k) * nsite + t], sm[(2 * k + 1) * nsite + t]};
}
__device__ __forceinline__ void store_smem(float* sm, int nsite, int t, const Spinor<float>& s) {
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    sm[(2 * k) * nsite + t] = s.c[k / 3][k % 3].re;
    sm[(2 * k + 1) * nsite + t] = s.c[k / 3][k % 3].im;
  }
}

// The block sums of an MR step, result in every thread.  The three sums
// that give the MR coefficient omega = <D p, r> / <D p, D p> are binary32
// (a preconditioner coefficient: a tree of warp shuffles, then the warp
// partials in a fixed order; ~5e-7 relative for 256 sites); binary64
// arithmetic runs at 1/64 of the binary32 rate on GB300, and these sums with
// a binary64 division per thread had kept its FP64 pipe 36 % busy.  The
// adaptive exit tests keep one binary64 sum (block_sum1).
__device__ __forceinline__ void block_sum3(float& a, float& b, float& c, double* red_d) {
  float* red = reinterpret_cast<float*>(red_d);
  a = warp_sum_f(a);
  b = warp_sum_f(b);
  c = warp_sum_f(c);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    red[3 * w] = a;
    red[3 * w + 1] = b;
    red[3 * w + 2] = c;
  }
  __syncthreads();
  a = b = c = 0.f;
  for (int k = 0; k < nw; ++k) {
    a += red[3 * k];
    b += red[3 * k + 1];
    c += red[3 * k + 2];
  }
}
__device__ __forceinline__ double block_sum1(double a, double* red) {
  a = warp_sum(a);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = a;
  __syncthreads();
  a = 0.0;
  for (int k = 0; k < nw; ++k) a += red[k];
  return a;
}

// in-block hop along +mu / -mu from smem (Dirichlet: outside neighbours dropped)
template <int FMT, int MU>
__device__ __forceinline__ void block_hop(const SapArgs& a, const float* sm, int nsite, int t, const int l[4],
                                          const int x[4], int p, long i, Spinor<float>& acc) {
  int stride = 1;
  for (int nu = 3; nu > MU; --nu) stride *= a.bs[nu];
  if (l[MU] + 1 < a.bs[MU]) {
    Spinor<float> nb;
    load_smem(sm, nsite, t + stride, nb);
    HalfSpinor<float> h, r;
    project<MU, -1>(nb, h);
    Su3<float> u;
    load_link<float, FMT>(a.links, a.g.Vh, p, MU, i, u);
    su3_mul(u, h, r);
    accum_reconstruct<MU, -1>(acc, r, -0.5f);
  }
  if (l[MU] > 0) {
    Spinor<float> nb;
    load_smem(sm, nsite, t - stride, nb);
    HalfSpinor<float> h, r;
    project<MU, +1>(nb, h);
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[MU] -= 1;
    Su3<float> u;
    load_link<float, FMT>(a.links, a.g.Vh, 1 - p, MU, eo_index(a.g, y), u);
    su3_dag_mul(u, h, r);
    accum_reconstruct<MU, +1>(acc, r, -0.5f);
  }
}

// MINB = 2 caps registers so that two 256-thread CTAs fit on an SM (a few
// spills to L1), MINB = 1 lets the compiler use ~200 registers (one CTA)
template <int FMT, int MINB>
__global__ void __launch_bounds__(256, MINB) sap_kernel(const SapArgs a) {
  extern __shared__ float sm[];
  const int nsite = a.bs[0] * a.bs[1] * a.bs[2] * a.bs[3];
  double* red = reinterpret_cast<double*>(sm + 24 * nsite);
  const int t = threadIdx.x;
  const bool act = t < nsite;
  // which block: the blockIdx.x-th block of colour a.colour
  const int half3 = a.nb[3] / 2;
  int row = blockIdx.x / half3;
  const int m = blockIdx.x % half3;
  const int bc2 = row % a.nb[2];
  row /= a.nb[2];
  const int bc1 = row % a.nb[1];
  const int bc0 = row / a.nb[1];
  const int bc3 = 2 * m + ((a.colour + bc0 + bc1 + bc2) & 1);
  int l[4], x[4];
  {
    int tt = act ? t : 0;
    l[3] = tt % a.bs[3];
    tt /= a.bs[3];
    l[2] = tt % a.bs[2];
    tt /= a.bs[2];
    l[1] = tt % a.bs[1];
    l[0] = tt / a.bs[1];
  }
  x[0] = bc0 * a.bs[0] + l[0];
  x[1] = bc1 * a.bs[1] + l[1];
  x[2] = bc2 * a.bs[2] + l[2];
  x[3] = bc3 * a.bs[3] + l[3];
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const long i = eo_index(a.g, x);

  // 1. block residual r = rho - D phi (full stencil)
  Spinor<float> r;
  if (act) {
    HopArgs ha;
    ha.g = a.g;
    ha.links = a.links;
    const char* nbf = a.phi + (long)(1 - p) * a.half_bytes;
    Spinor<float> acc;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc.c[s][c] = cx<float>{0.f, 0.f};
    hop_dir<P_F32, FMT, 0, false>(ha, nbf, p, i, x, acc, -0.5f);
    hop_dir<P_F32, FMT, 1, false>(ha, nbf, p, i, x, acc, -0.5f);
    hop_dir<P_F32, FMT, 2, false>(ha, nbf, p, i, x, acc, -0.5f);
    hop_dir<P_F32, FMT, 3, false>(ha, nbf, p, i, x, acc, -0.5f);
    Spinor<float> ph, aph, rh;
    load_spinor<P_F32>(a.phi + (long)p * a.half_bytes, a.g.Vh, i, ph);
    clover_apply<float>(a.clov, a.g.Vh, p, i, ph, aph);
    load_spinor<P_F32>(a.rho + (long)p * a.half_bytes, a.g.Vh, i, rh);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) r.c[s][c] = rh.c[s][c] - (aph.c[s][c] + acc.c[s][c]);
    store_smem(sm, nsite, t, r);
  }
  double n0 = 0.0;
  if (a.adaptive) {
    if (act) n0 = site_norm2(r);
    n0 = block_sum1(n0, red);  // also the barrier after the block residual is stored
  } else {
    __syncthreads();
  }
  double rn_prev = sqrt(n0);

  // 2. MR on D_i
  Spinor<float> xs;
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) xs.c[s][c] = cx<float>{0.f, 0.f};
  int steps = 0;
  for (int k = 1; k <= a.nmr; ++k) {
    Spinor<float> pv;
    float pr_re = 0.f, pr_im = 0.f, pp = 0.f;
    if (act) {
      Spinor<float> own;
      load_smem(sm, nsite, t, own);
      clover_apply<float>(a.clov, a.g.Vh, p, i, own, pv);
      block_hop<FMT, 0>(a, sm, nsite, t, l, x, p, i, pv);
      block_hop<FMT, 1>(a, sm, nsite, t, l, x, p, i, pv);
      block_hop<FMT, 2>(a, sm, nsite, t, l, x, p, i, pv);
      block_hop<FMT, 3>(a, sm, nsite, t, l, x, p, i, pv);
      float ar = 0.f, ai = 0.f, a2 = 0.f;
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          cx<float> q = pv.c[s][c], v = own.c[s][c];
          ar += q.re * v.re + q.im * v.im;
          ai += q.re * v.im - q.im * v.re;
          a2 += q.re * q.re + q.im * q.im;
        }
      pr_re = ar;
      pr_im = ai;
      pp = a2;
    }
    block_sum3(pr_re, pr_im, pp, red);  // contains __syncthreads: all neighbour reads done
    float om_re = 0.f, om_im = 0.f;
    if (pp > 0.f) {
      om_re = pr_re / pp;
      om_im = pr_im / pp;
    }
    const cx<float> om{om_re, om_im};
    double n1 = 0.0;
    if (act) {
      Spinor<float> own;
      load_smem(sm, nsite, t, own);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          cfma(xs.c[s][c], om, own.c[s][c]);
          own.c[s][c] = own.c[s][c] - om * pv.c[s][c];
        }
      store_smem(sm, nsite, t, own);
      n1 = site_norm2(own);
    }
    steps = k;
    if (a.adaptive) {
      n1 = block_sum1(n1, red);
      const double rn_new = sqrt(n1);
      if ((k >= 4 && rn_new > (double)a.alpha * rn_prev) || rn_new > rn_prev || rn_new < a.tol) break;
      rn_prev = rn_new;
    } else {
      __syncthreads();  // the updated residual is read by the neighbours next step
    }
  }
  // 3. phi_i += x
  if (act) {
    char* pp = a.phi + (long)p * a.half_bytes;
    Spinor<float> ph;
    load_spinor<P_F32>(pp, a.g.Vh, i, ph);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) ph.c[s][c] = ph.c[s][c] + xs.c[s][c];
    store_spinor<P_F32>(pp, a.g.Vh, i, ph);
  }
  if (a.mr_steps && t == 0) atomicAdd(a.mr_steps, (unsigned)steps);
}

// ---------------------------------------------------------------------------
// The default block solve.  A site's thread keeps its four forward links (18
// reals each) and its residual in registers; the block's clover is staged in
// shared memory once.  The backward hop of x along mu is U_mu(x-mu)^dag times
// the projected residual of x-mu, both of which the thread of x-mu holds: every
// thread transports its own residual along its four links and leaves the half
// spinors in shared memory for its forward neighbours ("sends"), next to the
// residual itself, from which the forward hops read.  An MR step then moves
// 288 words per site through shared memory (24 + 48 written, 4 x 24 residuals,
// 48 received, 72 clover), all in 16-byte accesses, against 456 in 4-byte and
// 8-byte ones when every hop read the neighbour's residual and a link, and needs
// two barriers instead of three.  Hops that leave the block are dropped by a
// zero weight rather than a branch, so that the loads of several hops overlap.
//
// The block residual rho - D phi takes the in-block part of D phi through the
// same shared-memory operator and reads only the neighbours outside the block
// from global memory.  In the first cycle phi is zero on the blocks of
// this colour (and, with colour 0, everywhere), so those terms are left out.
// BLK: own links and clover from the block-ordered copies (sap_blocked_kernel).
// Bound by latency at one block of 8 warps per SM (255 registers, 147 KB): an MR
// step runs two thirds of the issue slots (20 us of a launch, 48x24^3 in 4^4
// blocks), loading a block and the hops from outside it overlap with nothing.
// 5 MR steps there: 204 us a launch; 338 us with links and residual in shared
// memory and the operands in packed order.  Two threads per site (512 at 128
// registers) took 287 against 228 us, both directions' outside operands
// requested together 243, and an L2 prefetch of the next block 210 against 204.
// Shared memory: 72 + 24 + 48 floats per block site.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(float4* smem, const float4* gmem) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// where a site's own links and clover lie: packed order (parity p, field stride V,
// index i) or, with block-ordered copies, the same expression with the block's
// number, its volume and the thread's position
struct OwnAt {
  long p, V, i;
};
template <bool BLK>
__device__ __forceinline__ OwnAt own_at(const SapArgs& a, int nsite, int block, int t, int p, long i) {
  if (BLK) return OwnAt{block, nsite, t};
  return OwnAt{p, a.g.Vh, i};
}
// coordinates of the n-th block of the colour, and its number among all blocks
__device__ __forceinline__ int colour_block(const SapArgs& a, int n, int (&bc)[4]) {
  const int half3 = a.nb[3] / 2;
  int row = n / half3;
  bc[2] = row % a.nb[2];
  row /= a.nb[2];
  bc[1] = row % a.nb[1];
  bc[0] = row / a.nb[1];
  bc[3] = 2 * (n % half3) + ((a.colour + bc[0] + bc[1] + bc[2]) & 1);
  return ((bc[0] * a.nb[1] + bc[1]) * a.nb[2] + bc[2]) * a.nb[3] + bc[3];
}
struct SapShared {
  float4* a;  // [18][nsite] clover (two blocks: 6 diagonal + 15 complex each)
  float4* r;  // [6][nsite] residual, two complex components per chunk
  float4* s;  // [mu][3][nsite] half spinors sent to the site above along mu
  int nsite;
};

__device__ __forceinline__ void sm4_load(const float4* b, int nsite, int t, Spinor<float>& v) {
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const float4 w = b[c * nsite + t];
    v.c[(2 * c) / 3][(2 * c) % 3] = cx<float>{w.x, w.y};
    v.c[(2 * c + 1) / 3][(2 * c + 1) % 3] = cx<float>{w.z, w.w};
  }
}
__device__ __forceinline__ void sm4_store(float4* b, int nsite, int t, const Spinor<float>& v) {
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const cx<float> x = v.c[(2 * c) / 3][(2 * c) % 3], y = v.c[(2 * c + 1) / 3][(2 * c + 1) % 3];
    b[c * nsite + t] = make_float4(x.re, x.im, y.re, y.im);
  }
}

// out = A in, one clover block at a time from shared memory
__device__ __forceinline__ void sm4_clover(const float4* a, int nsite, int t, const Spinor<float>& in,
                                           Spinor<float>& out) {
  const cx<float>* v = &in.c[0][0];
  cx<float>* o = &out.c[0][0];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    float r[36];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float4 w = a[(9 * b + k) * nsite + t];
      r[4 * k] = w.x;
      r[4 * k + 1] = w.y;
      r[4 * k + 2] = w.z;
      r[4 * k + 3] = w.w;
    }
    const cx<float>* x = v + 6 * b;
    cx<float>* y = o + 6 * b;
#pragma unroll
    for (int r0 = 0; r0 < 6; ++r0) y[r0] = r[r0] * x[r0];
    int k = 0;
#pragma unroll
    for (int r0 = 0; r0 < 6; ++r0)
#pragma unroll
      for (int c0 = r0 + 1; c0 < 6; ++c0) {
        const cx<float> off{r[6 + 2 * k], r[7 + 2 * k]};
        cfma(y[r0], off, x[c0]);
        cfmac(y[c0], off, x[r0]);
        ++k;
      }
  }
}

// the sends of a site: U_mu(x)^dag (1 + g_mu) v for its forward neighbours
template <int MU>
__device__ __forceinline__ void sm4_send(const SapShared& m, int t, const Su3<float>& u, const Spinor<float>& v) {
  HalfSpinor<float> h, y;
  project<MU, +1>(v, h);
  su3_dag_mul(u, h, y);
  const cx<float>* c = &y.c[0][0];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    m.s[(MU * 3 + k) * m.nsite + t] = make_float4(c[2 * k].re, c[2 * k].im, c[2 * k + 1].re, c[2 * k + 1].im);
}
__device__ __forceinline__ void sm4_publish(const SapShared& m, int t, const Su3<float> (&u)[4],
                                            const Spinor<float>& v) {
  sm4_store(m.r, m.nsite, t, v);
  sm4_send<0>(m, t, u[0], v);
  sm4_send<1>(m, t, u[1], v);
  sm4_send<2>(m, t, u[2], v);
  sm4_send<3>(m, t, u[3], v);
}

// acc += the in-block hops along mu of the published field, from the positions
// tu (above) and td (below); up / down: the site has such a neighbour in the
// block (where not, the position is its own and the weight zero)
template <int MU>
__device__ __forceinline__ void sm4_hop(const SapShared& m, int tu, int td, bool up, bool down, const Su3<float>& u,
                                        Spinor<float>& acc) {
  Spinor<float> nb;
  sm4_load(m.r, m.nsite, tu, nb);
  HalfSpinor<float> h, y, z;
  cx<float>* c = &z.c[0][0];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 w = m.s[(MU * 3 + k) * m.nsite + td];
    c[2 * k] = cx<float>{w.x, w.y};
    c[2 * k + 1] = cx<float>{w.z, w.w};
  }
  project<MU, -1>(nb, h);
  su3_mul(u, h, y);
  accum_reconstruct<MU, -1>(acc, y, up ? -0.5f : 0.f);
  accum_reconstruct<MU, +1>(acc, z, down ? -0.5f : 0.f);
}

// p = D_i v for the published field v (own value passed in registers)
__device__ __forceinline__ void sm4_apply(const SapShared& m, int t, const int (&stride)[4], unsigned up,
                                          unsigned down, const Su3<float> (&u)[4], const Spinor<float>& v,
                                          Spinor<float>& p) {
  sm4_clover(m.a, m.nsite, t, v, p);
  sm4_hop<0>(m, up & 1 ? t + stride[0] : t, down & 1 ? t - stride[0] : t, up & 1, down & 1, u[0], p);
  sm4_hop<1>(m, up & 2 ? t + stride[1] : t, down & 2 ? t - stride[1] : t, up & 2, down & 2, u[1], p);
  sm4_hop<2>(m, up & 4 ? t + stride[2] : t, down & 4 ? t - stride[2] : t, up & 4, down & 4, u[2], p);
  sm4_hop<3>(m, up & 8 ? t + stride[3] : t, down & 8 ? t - stride[3] : t, up & 8, down & 8, u[3], p);
}

// the hops along mu that come from outside the block, from global memory
template <int FMT, int MU>
__device__ __forceinline__ void outer_hop(const SapArgs& a, const char* nbf, int p, const int x[4], bool up,
                                          bool down, const Su3<float>& u, Spinor<float>& acc) {
  bool cr;
  if (!up) {
    const long j = eo_neighbour(a.g, x, MU, +1, &cr);
    Spinor<float> nb;
    load_spinor<P_F32>(nbf, a.g.Vh, j, nb);
    HalfSpinor<float> h, y;
    project<MU, -1>(nb, h);
    su3_mul(u, h, y);
    hop_accum<MU, -1>(acc, y, -0.5f, cr, a.g.bc_t);
  }
  if (!down) {
    const long j = eo_neighbour(a.g, x, MU, -1, &cr);
    Spinor<float> nb;
    load_spinor<P_F32>(nbf, a.g.Vh, j, nb);
    Su3<float> v;
    load_link<float, FMT>(a.links, a.g.Vh, 1 - p, MU, j, v);
    HalfSpinor<float> h, y;
    project<MU, +1>(nb, h);
    su3_dag_mul(v, h, y);
    hop_accum<MU, +1>(acc, y, -0.5f, cr, a.g.bc_t);
  }
}

template <int FMT, bool BLK>
__global__ void __launch_bounds__(256, 1) sap_block_kernel(const SapArgs a) {
  extern __shared__ float4 sm4[];
  const int nsite = a.bs[0] * a.bs[1] * a.bs[2] * a.bs[3];
  SapShared m;
  m.nsite = nsite;
  m.a = sm4;
  m.r = sm4 + 18 * nsite;
  m.s = sm4 + 24 * nsite;
  float* red = reinterpret_cast<float*>(sm4 + 36 * nsite);  // 3 partials per warp (binary64: block_sum1)
  const int t = threadIdx.x;
  const bool act = t < nsite;
  int bc[4];
  const int block = colour_block(a, blockIdx.x, bc);
  const int stride[4] = {a.bs[1] * a.bs[2] * a.bs[3], a.bs[2] * a.bs[3], a.bs[3], 1};
  int l[4], x[4];
  {
    int tt = act ? t : 0;
    l[3] = tt % a.bs[3];
    tt /= a.bs[3];
    l[2] = tt % a.bs[2];
    tt /= a.bs[2];
    l[1] = tt % a.bs[1];
    l[0] = tt / a.bs[1];
  }
  x[0] = bc[0] * a.bs[0] + l[0];
  x[1] = bc[1] * a.bs[1] + l[1];
  x[2] = bc[2] * a.bs[2] + l[2];
  x[3] = bc[3] * a.bs[3] + l[3];
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const long i = eo_index(a.g, x);
  const OwnAt own = own_at<BLK>(a, nsite, block, t, p, i);
  unsigned up = 0, down = 0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    if (l[mu] + 1 < a.bs[mu]) up |= 1u << mu;
    if (l[mu] > 0) down |= 1u << mu;
  }
  const int w = t >> 5, nw = (blockDim.x + 31) >> 5;

  Spinor<float> r, xs;
  Su3<float> u[4];
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) r.c[s][c] = xs.c[s][c] = cx<float>{0.f, 0.f};
  char* phi = a.phi + (long)p * a.half_bytes;
  if (act) {
    const float4* q = reinterpret_cast<const float4*>(BLK ? a.blk.clov : a.clov) + own.p * 18 * own.V + own.i;
#pragma unroll
    for (int k = 0; k < 18; ++k) cp_async16(m.a + k * nsite + t, q + k * own.V);
    cp_async_commit();
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
      load_link<float, FMT>(BLK ? a.blk.links : a.links, own.V, (int)own.p, mu, own.i, u[mu]);
    // 1. block residual rho - D phi: the hops from outside the block
    if (!(a.first && a.colour == 0)) {
      const char* nbf = a.phi + (long)(1 - p) * a.half_bytes;
      outer_hop<FMT, 3>(a, nbf, p, x, up & 8, down & 8, u[3], r);
      outer_hop<FMT, 2>(a, nbf, p, x, up & 4, down & 4, u[2], r);
      outer_hop<FMT, 1>(a, nbf, p, x, up & 2, down & 2, u[1], r);
      outer_hop<FMT, 0>(a, nbf, p, x, up & 1, down & 1, u[0], r);
    }
    Spinor<float> rh;
    load_spinor<P_F32>(a.rho + (long)p * a.half_bytes, a.g.Vh, i, rh);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) r.c[s][c] = rh.c[s][c] - r.c[s][c];
    if (!a.first) {
      load_spinor<P_F32>(phi, a.g.Vh, i, xs);  // the block's phi
      sm4_publish(m, t, u, xs);
    }
    cp_async_wait();
  }
  __syncthreads();  // the staged clover (each site reads its own) and the published phi
  if (!a.first) {
    // the part of D phi inside the block
    if (act) {
      Spinor<float> pv;
      sm4_apply(m, t, stride, up, down, u, xs, pv);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          r.c[s][c] = r.c[s][c] - pv.c[s][c];
          xs.c[s][c] = cx<float>{0.f, 0.f};
        }
    }
    __syncthreads();  // every read of the published phi is done
  }
  double rn_prev = 0.0;
  if (a.adaptive) rn_prev = sqrt(block_sum1(act ? site_norm2(r) : 0.0, reinterpret_cast<double*>(red)));

  // 2. MR on D_i
  int steps = 0;
  for (int k = 1; k <= a.nmr; ++k) {
    if (act) sm4_publish(m, t, u, r);
    __syncthreads();
    Spinor<float> pv;
    float d0 = 0.f, d1 = 0.f, d2 = 0.f;  // <p, r>, <p, p>
    if (act) {
      sm4_apply(m, t, stride, up, down, u, r, pv);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const cx<float> q = pv.c[s][c], v = r.c[s][c];
          d0 += q.re * v.re + q.im * v.im;
          d1 += q.re * v.im - q.im * v.re;
          d2 += q.re * q.re + q.im * q.im;
        }
    }
    d0 = warp_sum_f(d0);
    d1 = warp_sum_f(d1);
    d2 = warp_sum_f(d2);
    if ((t & 31) == 0) {
      red[3 * w] = d0;
      red[3 * w + 1] = d1;
      red[3 * w + 2] = d2;
    }
    __syncthreads();  // the partial sums; every read of the published residual is done
    d0 = d1 = d2 = 0.f;
    for (int j = 0; j < nw; ++j) {
      d0 += red[3 * j];
      d1 += red[3 * j + 1];
      d2 += red[3 * j + 2];
    }
    cx<float> om{0.f, 0.f};
    if (d2 > 0.f) om = cx<float>{d0 / d2, d1 / d2};
    if (act) {
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          cfma(xs.c[s][c], om, r.c[s][c]);
          r.c[s][c] = r.c[s][c] - om * pv.c[s][c];
        }
    }
    steps = k;
    if (a.adaptive) {
      const double rn_new = sqrt(block_sum1(act ? site_norm2(r) : 0.0, reinterpret_cast<double*>(red)));
      if ((k >= 4 && rn_new > (double)a.alpha * rn_prev) || rn_new > rn_prev || rn_new < a.tol) break;
      rn_prev = rn_new;
    }
  }
  // 3. phi_i += x
  if (act) {
    if (!a.first) {
      Spinor<float> ph;
      load_spinor<P_F32>(phi, a.g.Vh, i, ph);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) xs.c[s][c] = ph.c[s][c] + xs.c[s][c];
    }
    store_spinor<P_F32>(phi, a.g.Vh, i, xs);
  }
  if (a.mr_steps && t == 0) atomicAdd(a.mr_steps, (unsigned)steps);
}

__device__ __forceinline__ void zero_spinor(Spinor<float>& v) {
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) v.c[s][c] = cx<float>{0.f, 0.f};
}

// Two binary32 lanes of one packed instruction, for the even-odd kernel.  A spinor
// is held as six complex pairs, lanes spin s and s + 2; links as pairs of directions
// (0, 1) and (2, 3); a site's two clover blocks as one block of pairs.  A packed FMA
// takes the pipe twice as long as a scalar one, so what it saves is issue: the
// even-odd kernel, one warp per scheduler in each half pass, gained (93 to 77 us a
// colour on 24x16^3); sap_block_kernel, two warps and 23 % fewer instructions, takes
// 252 us instead of 239, waiting for the longer latency, and stays scalar.
namespace eop {
typedef float2 F2;
struct C2 {
  F2 re, im;
};
struct Sp6 {
  C2 c[6];  // [3 s + colour]
};
struct Link2 {
  C2 m[3][3];
};
__device__ __forceinline__ F2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ F2 ffma2(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ F2 fmul2(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ F2 fsub2(F2 a, F2 b) { return __ffma2_rn(b, bc2(-1.f), a); }
__device__ __forceinline__ C2 pair_of(cx<float> a, cx<float> b) { return C2{{a.re, b.re}, {a.im, b.im}}; }
__device__ __forceinline__ Sp6 pack6(const Spinor<float>& v) {
  Sp6 o;
#pragma unroll
  for (int k = 0; k < 6; ++k) o.c[k] = pair_of(v.c[k / 3][k % 3], v.c[2 + k / 3][k % 3]);
  return o;
}
__device__ __forceinline__ Spinor<float> spinor_of(const Sp6& v) {
  Spinor<float> o;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    o.c[k / 3][k % 3] = cx<float>{v.c[k].re.x, v.c[k].im.x};
    o.c[2 + k / 3][k % 3] = cx<float>{v.c[k].re.y, v.c[k].im.y};
  }
  return o;
}
template <int L>
__device__ __forceinline__ Su3<float> link_of(const Link2& u) {
  Su3<float> o;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      o.m[a][b] = L ? cx<float>{u.m[a][b].re.y, u.m[a][b].im.y} : cx<float>{u.m[a][b].re.x, u.m[a][b].im.x};
  return o;
}
template <int FMT, bool BLK>
__device__ __forceinline__ void load_link2(const SapArgs& a, const OwnAt& own, int q, Link2& u) {
  const void* b = BLK ? a.blk.links : a.links;
  Su3<float> v, w;
  load_link<float, FMT>(b, own.V, (int)own.p, 2 * q, own.i, v);
  load_link<float, FMT>(b, own.V, (int)own.p, 2 * q + 1, own.i, w);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int d = 0; d < 3; ++d) u.m[c][d] = pair_of(v.m[c][d], w.m[c][d]);
}
__device__ __forceinline__ void sm4_load(const float4* b, int nsite, int t, Sp6& v) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 w = b[k * nsite + t];
    v.c[k] = C2{{w.x, w.y}, {w.z, w.w}};
  }
}
__device__ __forceinline__ void sm4_store(float4* b, int nsite, int t, const Sp6& v) {
#pragma unroll
  for (int k = 0; k < 6; ++k) b[k * nsite + t] = make_float4(v.c[k].re.x, v.c[k].re.y, v.c[k].im.x, v.c[k].im.y);
}

// The staged clover blocks of a site, made pairs in place: slot(q) holds the reals
// 2q and 2q + 1 of both blocks (6 diagonal, then 15 complex).
__device__ __forceinline__ int clover_slot(int q) { return (q & 1) ? 9 + q / 2 : q / 2; }
__device__ __forceinline__ void sm4_clover_pairs(float4* a, int nsite, int t) {
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const float4 v = a[k * nsite + t], w = a[(9 + k) * nsite + t];
    a[k * nsite + t] = make_float4(v.x, w.x, v.y, w.y);
    a[(9 + k) * nsite + t] = make_float4(v.z, w.z, v.w, w.w);
  }
}
// out = A in
__device__ __forceinline__ void sm4_clover(const float4* a, int nsite, int t, const Sp6& in, Sp6& out) {
  const F2 m1 = bc2(-1.f);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float4 w = a[clover_slot(q) * nsite + t];
    out.c[2 * q] = C2{fmul2({w.x, w.y}, in.c[2 * q].re), fmul2({w.x, w.y}, in.c[2 * q].im)};
    out.c[2 * q + 1] = C2{fmul2({w.z, w.w}, in.c[2 * q + 1].re), fmul2({w.z, w.w}, in.c[2 * q + 1].im)};
  }
  F2 nre[5], nim[5];  // -Re in[0 .. 4], -Im in[1 .. 5]: a packed FMA has no negated operand
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    nre[k] = fmul2(m1, in.c[k].re);
    nim[k] = fmul2(m1, in.c[k + 1].im);
  }
  int q = 3;
#pragma unroll
  for (int r = 0; r < 6; ++r)
#pragma unroll
    for (int c = r + 1; c < 6; ++c) {
      const float4 w = a[clover_slot(q) * nsite + t];
      const F2 ore{w.x, w.y}, oim{w.z, w.w};
      C2 &y = out.c[r], &z = out.c[c];
      const C2 &x = in.c[c], &v = in.c[r];
      y.re = ffma2(oim, nim[c - 1], ffma2(ore, x.re, y.re));
      y.im = ffma2(oim, x.re, ffma2(ore, x.im, y.im));
      z.re = ffma2(oim, v.im, ffma2(ore, v.re, z.re));
      z.im = ffma2(oim, nre[r], ffma2(ore, v.im, z.im));
      ++q;
    }
}

// y = U h or U^dag h for both directions of a pair.  APART: the caller stores the two
// directions apart, so the last operation of each real is done per lane (a lane of
// a pair costs a move where four reals of one direction have to be neighbours).
template <bool DAG, bool APART>
__device__ __forceinline__ void link2_mul(const Link2& u, const HalfSpinor<float>& h0, const HalfSpinor<float>& h1,
                                          HalfSpinor<float>& y0, HalfSpinor<float>& y1) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      // U: re = p - n, im = s;  U^dag: re = s, im = p - n
      F2 sum, pos, neg;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const C2 w = DAG ? u.m[b][a] : u.m[a][b], h = pair_of(h0.c[s][b], h1.c[s][b]);
        const F2 f = DAG ? h.re : h.im, g = DAG ? h.im : h.re;
        if (b == 0) {
          sum = ffma2(w.im, g, fmul2(w.re, f));
          pos = fmul2(w.re, g);
          neg = fmul2(w.im, f);
        } else {
          pos = ffma2(w.re, g, pos);
          neg = ffma2(w.im, f, neg);
          sum = ffma2(w.re, f, sum);
          if (b < 2 || !APART) sum = ffma2(w.im, g, sum);
          else sum = F2{fmaf(w.im.x, g.x, sum.x), fmaf(w.im.y, g.y, sum.y)};
        }
      }
      const F2 dif = APART ? F2{pos.x - neg.x, pos.y - neg.y} : fsub2(pos, neg);
      y0.c[s][a] = DAG ? cx<float>{sum.x, dif.x} : cx<float>{dif.x, sum.x};
      y1.c[s][a] = DAG ? cx<float>{sum.y, dif.y} : cx<float>{dif.y, sum.y};
    }
}

// the sends of a site: U_mu(x)^dag (1 + g_mu) v for its forward neighbours
template <int Q>
__device__ __forceinline__ void sm4_send(const SapShared& m, int t, const Link2& u, const Spinor<float>& v) {
  HalfSpinor<float> h[2], y[2];
  project<2 * Q, +1>(v, h[0]);
  project<2 * Q + 1, +1>(v, h[1]);
  link2_mul<true, true>(u, h[0], h[1], y[0], y[1]);
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const cx<float>* c = &y[d].c[0][0];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      m.s[((2 * Q + d) * 3 + k) * m.nsite + t] =
          make_float4(c[2 * k].re, c[2 * k].im, c[2 * k + 1].re, c[2 * k + 1].im);
  }
}
__device__ __forceinline__ void sm4_publish(const SapShared& m, int t, const Link2 (&u)[2], const Sp6& v) {
  sm4_store(m.r, m.nsite, t, v);
  const Spinor<float> w = spinor_of(v);
  sm4_send<0>(m, t, u[0], w);
  sm4_send<1>(m, t, u[1], w);
}

// acc += the in-block hops along 2Q and 2Q + 1 of the published field, from the
// positions tu (above) and td (below); up / down: the site has such a neighbour in
// the block (where not, the position is its own and the weight zero)
template <int Q>
__device__ __forceinline__ void sm4_hops(const SapShared& m, const int (&tu)[4], const int (&td)[4], unsigned up,
                                         unsigned down, const Link2& u, Spinor<float>& acc) {
  HalfSpinor<float> h[2], y[2], z[2];
  Sp6 n;
  sm4_load(m.r, m.nsite, tu[2 * Q], n);
  project<2 * Q, -1>(spinor_of(n), h[0]);
  sm4_load(m.r, m.nsite, tu[2 * Q + 1], n);
  project<2 * Q + 1, -1>(spinor_of(n), h[1]);
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    cx<float>* c = &z[d].c[0][0];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 w = m.s[((2 * Q + d) * 3 + k) * m.nsite + td[2 * Q + d]];
      c[2 * k] = cx<float>{w.x, w.y};
      c[2 * k + 1] = cx<float>{w.z, w.w};
    }
  }
  link2_mul<false, false>(u, h[0], h[1], y[0], y[1]);
  accum_reconstruct<2 * Q, -1>(acc, y[0], up >> (2 * Q) & 1 ? -0.5f : 0.f);
  accum_reconstruct<2 * Q, +1>(acc, z[0], down >> (2 * Q) & 1 ? -0.5f : 0.f);
  accum_reconstruct<2 * Q + 1, -1>(acc, y[1], up >> (2 * Q + 1) & 1 ? -0.5f : 0.f);
  accum_reconstruct<2 * Q + 1, +1>(acc, z[1], down >> (2 * Q + 1) & 1 ? -0.5f : 0.f);
}

__device__ __forceinline__ double norm2_of(const Sp6& v) { return site_norm2(spinor_of(v)); }
// a -= b
__device__ __forceinline__ void sp6_sub(Sp6& a, const Sp6& b) {
#pragma unroll
  for (int k = 0; k < 6; ++k) a.c[k] = C2{fsub2(a.c[k].re, b.c[k].re), fsub2(a.c[k].im, b.c[k].im)};
}
__device__ __forceinline__ void sp6_zero(Sp6& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) a.c[k] = C2{{0.f, 0.f}, {0.f, 0.f}};
}
// a site's part of <p, r> = d0 + i d1 and <p, p> = d2
__device__ __forceinline__ void mr_dots(const Sp6& p, const Sp6& r, float& d0, float& d1, float& d2) {
  F2 s{0.f, 0.f}, v = s, w = s, n = s;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    s = ffma2(p.c[k].im, r.c[k].im, ffma2(p.c[k].re, r.c[k].re, s));
    v = ffma2(p.c[k].re, r.c[k].im, v);
    w = ffma2(p.c[k].im, r.c[k].re, w);
    n = ffma2(p.c[k].im, p.c[k].im, ffma2(p.c[k].re, p.c[k].re, n));
  }
  d0 = s.x + s.y;
  d1 = (v.x - w.x) + (v.y - w.y);
  d2 = n.x + n.y;
}
// x += om r, r -= om p
__device__ __forceinline__ void mr_update(cx<float> om, const Sp6& p, Sp6& x, Sp6& r) {
  const F2 wr = bc2(om.re), wi = bc2(om.im), nr = bc2(-om.re), ni = bc2(-om.im);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    x.c[k].re = ffma2(ni, r.c[k].im, ffma2(wr, r.c[k].re, x.c[k].re));
    x.c[k].im = ffma2(wi, r.c[k].re, ffma2(wr, r.c[k].im, x.c[k].im));
    r.c[k].re = ffma2(wi, p.c[k].im, ffma2(nr, p.c[k].re, r.c[k].re));
    r.c[k].im = ffma2(ni, p.c[k].re, ffma2(nr, p.c[k].im, r.c[k].im));
  }
}

}  // namespace eop

// ---------------------------------------------------------------------------
// Even-odd reduced block solver (openQCD's choice for SAP, Sec. 3): per block
//   rhat_e = r_e - D_eo A_oo^{-1} r_o,
//   MR steps on Dhat_i = A_ee - D_eo A_oo^{-1} D_oe (even block sites),
//   delta_o = A_oo^{-1} (r_o - D_oe delta_e),
// D_eo, D_oe the in-block hops.  Links in registers and sends as in
// sap_block_kernel; the staged clover is A at even and A^{-1} at odd sites.  An
// MR step is two half passes: the odd threads form A^{-1} D_oe of the published
// even residual and publish it, the even threads form D_eo of that.  Latency
// and issue of one warp per scheduler bound it: a half pass keeps 4 of an SM's
// 8 warps busy, and one block fills an SM (255 registers).  (A colour of 24x16^3
// in 4^4 blocks, 4 MR steps: 77 us; with links and clover in shared memory and
// both hops of a link multiplied by their reader it took 128 us.)
// ---------------------------------------------------------------------------
// The block's sites are held parity-sorted: position k < nsite/2 is the
// block-local-even site with in-block lexicographic index n = 2k + c, c
// fixing the parity (bs[3] even, so the sites of one parity alternate along
// x3), positions from nsite/2 on the local-odd sites.  A half pass then runs
// whole warps instead of every other lane.
__device__ __forceinline__ int eo_pos(int n, int par, int half) { return par * half + (n >> 1); }
// coordinates in the block and in-block index of the k-th site of a parity
__device__ __forceinline__ int eo_site(const SapArgs& a, int k, int par, int (&l)[4]) {
  int rr = (2 * k) / a.bs[3];  // the row (l0, l1, l2) of in-block index 2k + c
  l[2] = rr % a.bs[2];
  rr /= a.bs[2];
  l[1] = rr % a.bs[1];
  l[0] = rr / a.bs[1];
  const int c = (par + l[0] + l[1] + l[2]) & 1;
  l[3] = (2 * k) % a.bs[3] + c;
  return 2 * k + c;
}

template <int FMT, bool BLK>
__global__ void __launch_bounds__(256, 1) sap_block_eo_kernel(const SapArgs a) {
  extern __shared__ float4 sm4[];
  const int nsite = a.bs[0] * a.bs[1] * a.bs[2] * a.bs[3];
  SapShared m;
  m.nsite = nsite;
  m.a = sm4;
  m.r = sm4 + 18 * nsite;
  m.s = sm4 + 24 * nsite;
  float* red = reinterpret_cast<float*>(sm4 + 36 * nsite);  // 3 partials per warp (binary64: block_sum1)
  const int t = threadIdx.x;
  const bool act = t < nsite;
  int bc[4];
  const int block = colour_block(a, blockIdx.x, bc);
  // thread t holds the site at parity-sorted position t (see eo_pos)
  const int half = nsite >> 1;
  const int par = (act && t >= half) ? 1 : 0;  // block-local parity
  int l[4], x[4], n;
  {
    const int k = act ? t - par * half : 0;
    n = eo_site(a, k, par, l);
  }
  x[0] = bc[0] * a.bs[0] + l[0];
  x[1] = bc[1] * a.bs[1] + l[1];
  x[2] = bc[2] * a.bs[2] + l[2];
  x[3] = bc[3] * a.bs[3] + l[3];
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;  // lattice parity (the Schur complement's)
  const long i = eo_index(a.g, x);
  const OwnAt own = own_at<BLK>(a, nsite, block, t, p, i);
  const bool ev = act && p == 0, od = act && p == 1;
  const int stride[4] = {a.bs[1] * a.bs[2] * a.bs[3], a.bs[2] * a.bs[3], a.bs[3], 1};
  unsigned up = 0, down = 0;
  int tu[4], td[4];
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    tu[mu] = td[mu] = t;
    if (l[mu] + 1 < a.bs[mu]) {
      up |= 1u << mu;
      tu[mu] = eo_pos(n + stride[mu], par ^ 1, half);
    }
    if (l[mu] > 0) {
      down |= 1u << mu;
      td[mu] = eo_pos(n - stride[mu], par ^ 1, half);
    }
  }
  const int w = t >> 5, nw = (blockDim.x + 31) >> 5;

  eop::Sp6 r, xs;  // r: the residual (odd sites), rhat (even sites)
  eop::sp6_zero(r);
  eop::sp6_zero(xs);
  eop::Link2 u[2];
  // acc += the in-block hops of the published field
  auto dhop = [&](Spinor<float>& acc) {
    eop::sm4_hops<0>(m, tu, td, up, down, u[0], acc);
    eop::sm4_hops<1>(m, tu, td, up, down, u[1], acc);
  };
  char* phi = a.phi + (long)p * a.half_bytes;
  Spinor<float> acc;
  zero_spinor(acc);
  if (act) {
    const float4* q = reinterpret_cast<const float4*>(BLK ? a.blk.clov : p ? a.clov_inv : a.clov) +
                      own.p * 18 * own.V + own.i;
#pragma unroll
    for (int k = 0; k < 18; ++k) cp_async16(m.a + k * nsite + t, q + k * own.V);
    cp_async_commit();
    eop::load_link2<FMT, BLK>(a, own, 0, u[0]);
    eop::load_link2<FMT, BLK>(a, own, 1, u[1]);
    // block residual rho - D phi; the hops from outside the block first
    if (!(a.first && a.colour == 0)) {
      const char* nbf = a.phi + (long)(1 - p) * a.half_bytes;
      outer_hop<FMT, 3>(a, nbf, p, x, up & 8, down & 8, eop::link_of<1>(u[1]), acc);
      outer_hop<FMT, 2>(a, nbf, p, x, up & 4, down & 4, eop::link_of<0>(u[1]), acc);
      outer_hop<FMT, 1>(a, nbf, p, x, up & 2, down & 2, eop::link_of<1>(u[0]), acc);
      outer_hop<FMT, 0>(a, nbf, p, x, up & 1, down & 1, eop::link_of<0>(u[0]), acc);
    }
    Spinor<float> v;
    load_spinor<P_F32>(a.rho + (long)p * a.half_bytes, a.g.Vh, i, v);
    r = eop::pack6(v);
    if (!a.first) {
      load_spinor<P_F32>(phi, a.g.Vh, i, v);
      xs = eop::pack6(v);
    }
    if (!a.first) {
      eop::sm4_publish(m, t, u, xs);
    } else {
      // a dropped hop reads its own position with weight zero: that must hold numbers
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 6; ++k) m.r[k * nsite + t] = z;
#pragma unroll
      for (int k = 0; k < 12; ++k) m.s[k * nsite + t] = z;
    }
    if (!a.first) {
      v = eop::spinor_of(xs);
      Spinor<float> aph;
      clover_apply<float>(a.clov, a.g.Vh, p, i, v, aph);
      eop::sp6_sub(r, eop::pack6(aph));
      eop::sp6_zero(xs);
    }
    cp_async_wait();
    eop::sm4_clover_pairs(m.a, nsite, t);  // read by this thread alone
  }
  if (!a.first) {
    __syncthreads();  // the published phi
    if (act) dhop(acc);
    __syncthreads();  // every read of it is done
  }
  eop::sp6_sub(r, eop::pack6(acc));
  // odd sites publish A^{-1} r_o; even sites: rhat_e = r_e - D_eo A^{-1} r_o
  if (od) {
    eop::Sp6 v;
    eop::sm4_clover(m.a, nsite, t, r, v);
    eop::sm4_publish(m, t, u, v);
  }
  __syncthreads();
  if (ev) {
    zero_spinor(acc);
    dhop(acc);
    eop::sp6_sub(r, eop::pack6(acc));
    eop::sm4_publish(m, t, u, r);  // at even positions, which no one reads in this phase
  }
  double rn_prev = 0.0;
  if (a.adaptive) rn_prev = sqrt(block_sum1(ev ? eop::norm2_of(r) : 0.0, reinterpret_cast<double*>(red)));
  __syncthreads();

  int steps = 0;
  for (int k = 1; k <= a.nmr; ++k) {
    // odd half pass: t_o = A^{-1} D_oe rhat_e
    if (od) {
      zero_spinor(acc);
      dhop(acc);
      eop::Sp6 v;
      eop::sm4_clover(m.a, nsite, t, eop::pack6(acc), v);
      eop::sm4_publish(m, t, u, v);
    }
    __syncthreads();
    // even half pass: q_e = A rhat_e - D_eo t_o, then <q, rhat>, <q, q>
    eop::Sp6 pv;
    float d0 = 0.f, d1 = 0.f, d2 = 0.f;
    if (ev) {
      eop::sm4_clover(m.a, nsite, t, r, pv);
      zero_spinor(acc);
      dhop(acc);
      eop::sp6_sub(pv, eop::pack6(acc));
      eop::mr_dots(pv, r, d0, d1, d2);
    }
    d0 = warp_sum_f(d0);
    d1 = warp_sum_f(d1);
    d2 = warp_sum_f(d2);
    if ((t & 31) == 0) {
      red[3 * w] = d0;
      red[3 * w + 1] = d1;
      red[3 * w + 2] = d2;
    }
    __syncthreads();  // the partial sums
    d0 = d1 = d2 = 0.f;
    for (int j = 0; j < nw; ++j) {
      d0 += red[3 * j];
      d1 += red[3 * j + 1];
      d2 += red[3 * j + 2];
    }
    cx<float> om{0.f, 0.f};
    if (d2 > 0.f) om = cx<float>{d0 / d2, d1 / d2};
    if (ev) {
      eop::mr_update(om, pv, xs, r);
      eop::sm4_publish(m, t, u, r);
    }
    steps = k;
    if (a.adaptive) {
      const double rn_new = sqrt(block_sum1(ev ? eop::norm2_of(r) : 0.0, reinterpret_cast<double*>(red)));
      if ((k >= 4 && rn_new > (double)a.alpha * rn_prev) || rn_new > rn_prev || rn_new < a.tol) break;
      rn_prev = rn_new;
    }
    __syncthreads();  // the odd half pass of the next step reads the even residual
  }
  // delta_e = x_e published; delta_o = A^{-1} (r_o - D_oe delta_e)
  if (ev) eop::sm4_publish(m, t, u, xs);
  __syncthreads();
  if (od) {
    zero_spinor(acc);
    dhop(acc);
    eop::sp6_sub(r, eop::pack6(acc));
    eop::sm4_clover(m.a, nsite, t, r, xs);
  }
  if (act) {
    Spinor<float> v = eop::spinor_of(xs);
    if (!a.first) {
      Spinor<float> ph;
      load_spinor<P_F32>(phi, a.g.Vh, i, ph);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) v.c[s][c] = ph.c[s][c] + v.c[s][c];
    }
    store_spinor<P_F32>(phi, a.g.Vh, i, v);
  }
  if (a.mr_steps && t == 0) atomicAdd(a.mr_steps, (unsigned)steps);
}

// ---------------------------------------------------------------------------
// Block-ordered copies of the links and the clover: [block][chunk][position], the
// order in which the block kernels' threads read them.  In packed order a block of
// 4^4 sites reads runs of 32 bytes (two sites of a parity along x3) whose 64-byte
// DRAM neighbours belong to the other colour: a launch fetched twice its bytes
// (382 MB of DRAM reads for 191 MB on 48x24^3).  EO: A at lattice-even and A^{-1}
// at lattice-odd sites, positions sorted by the block-local parity.
// One CTA per block, one thread per site; 113 us on 48x24^3, where a colour takes
// 204 us from the copies and 228 us from the packed fields.
// ---------------------------------------------------------------------------
template <int EO>
__global__ void __launch_bounds__(256) sap_blocked_kernel(const SapArgs a, int link_chunks, int link_words,
                                                          char* links, float4* clov) {
  const int nsite = a.bs[0] * a.bs[1] * a.bs[2] * a.bs[3];
  const int t = threadIdx.x;
  if (t >= nsite) return;
  int l[4], x[4];
  if (EO) {
    const int half = nsite >> 1, par = t >= half;
    eo_site(a, t - par * half, par, l);
  } else {
    int tt = t;
    l[3] = tt % a.bs[3];
    tt /= a.bs[3];
    l[2] = tt % a.bs[2];
    tt /= a.bs[2];
    l[1] = tt % a.bs[1];
    l[0] = tt / a.bs[1];
  }
  const int block = blockIdx.x;
  int bb = block;
#pragma unroll
  for (int mu = 3; mu >= 0; --mu) {
    x[mu] = (bb % a.nb[mu]) * a.bs[mu] + l[mu];
    bb /= a.nb[mu];
  }
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const long i = eo_index(a.g, x), Vh = a.g.Vh;
  const float4* q = reinterpret_cast<const float4*>(EO && p ? a.clov_inv : a.clov) + (long)p * 18 * Vh + i;
  float4* d = clov + (long)block * 18 * nsite + t;
#pragma unroll 6
  for (int k = 0; k < 18; ++k) d[k * nsite] = q[k * Vh];
  if (link_words == 4) {
    const float4* f = reinterpret_cast<const float4*>(a.links) + (long)p * link_chunks * Vh + i;
    float4* o = reinterpret_cast<float4*>(links) + (long)block * link_chunks * nsite + t;
#pragma unroll 6
    for (int k = 0; k < link_chunks; ++k) o[k * nsite] = f[k * Vh];
  } else {
    const float2* f = reinterpret_cast<const float2*>(a.links) + (long)p * link_chunks * Vh + i;
    float2* o = reinterpret_cast<float2*>(links) + (long)block * link_chunks * nsite + t;
#pragma unroll 6
    for (int k = 0; k < link_chunks; ++k) o[k * nsite] = f[k * Vh];
  }
}

void sap_blocked_bytes(const Geom& g, int fmt, size_t* links, size_t* clov) {
  *links = (size_t)(fmt == LINK_12 ? 12 * sizeof(float4) : 36 * sizeof(float2)) * 2 * g.Vh;
  *clov = 18 * sizeof(float4) * 2 * (size_t)g.Vh;
}

cudaError_t sap_blocked(const Geom& g, const int bs[4], int fmt, const void* links, const void* clov,
                        const void* clov_inv, int eo, void* blinks, void* bclov, cudaStream_t s) {
  SapArgs a = {};
  a.g = g;
  int nblk = 1, nsite = 1;
  for (int mu = 0; mu < 4; ++mu) {
    a.bs[mu] = bs[mu];
    a.nb[mu] = g.L[mu] / bs[mu];
    nblk *= a.nb[mu];
    nsite *= bs[mu];
  }
  a.links = links;
  a.clov = clov;
  a.clov_inv = clov_inv;
  const int chunks = fmt == LINK_12 ? 12 : 36, words = fmt == LINK_12 ? 4 : 2;
  const dim3 block((nsite + 31) / 32 * 32);
  if (eo) sap_blocked_kernel<1><<<nblk, block, 0, s>>>(a, chunks, words, (char*)blinks, (float4*)bclov);
  else sap_blocked_kernel<0><<<nblk, block, 0, s>>>(a, chunks, words, (char*)blinks, (float4*)bclov);
  return cudaGetLastError();
}

// clover, residual and sends of a block in shared memory; at most 147 KB (256 sites)
static size_t sap_smem_bytes(const int bs[4]) {
  const int nsite = bs[0] * bs[1] * bs[2] * bs[3];
  const int threads = (nsite + 31) / 32 * 32;
  return sizeof(float) * (72 + 24 + 48) * (size_t)nsite + sizeof(double) * 3 * (threads / 32);
}

cudaError_t sap_colour(const Geom& g, const int bs[4], int colour, int fmt, const void* links, const void* clov,
                       const void* clov_inv, const void* rho, void* phi, int nmr, int adaptive, float alpha,
                       double tol, unsigned* mr_steps, int kernel, int eo, int cycle, const SapBlocked& blk,
                       cudaStream_t s) {
  SapArgs a;
  a.blk = blk;
  a.first = cycle == 0;
  // every block is written in the first cycle; the kernels that read phi there need zeros
  if (cycle == 0 && colour == 0 && !eo && kernel != 0) {
    const cudaError_t e = cudaMemsetAsync(phi, 0, 2 * spinor_half_bytes(g.Vh, P_F32), s);
    if (e != cudaSuccess) return e;
  }
  a.g = g;
  int nblk = 1;
  for (int mu = 0; mu < 4; ++mu) {
    a.bs[mu] = bs[mu];
    a.nb[mu] = g.L[mu] / bs[mu];
    nblk *= a.nb[mu];
  }
  a.colour = colour;
  a.links = links;
  a.clov = clov;
  a.clov_inv = clov_inv;
  a.rho = (const char*)rho;
  a.phi = (char*)phi;
  a.half_bytes = spinor_half_bytes(g.Vh, P_F32);
  a.nmr = nmr;
  a.adaptive = adaptive;
  a.alpha = alpha;
  a.tol = tol;
  a.mr_steps = mr_steps;
  const int nsite = bs[0] * bs[1] * bs[2] * bs[3];
  const int threads = (nsite + 31) / 32 * 32;
  const size_t smem = sizeof(float) * 24 * nsite + sizeof(double) * 3 * (threads / 32);
  dim3 grid(nblk / 2), block(threads);
  const bool ord = blk.links != nullptr;
  auto launch = [&](void (*k)(SapArgs), size_t bytes) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    k<<<grid, block, bytes, s>>>(a);
  };
  if (eo) {
    // even-odd reduced block solver: one kernel, whatever `kernel` asks for
    const size_t sm2 = sap_smem_bytes(bs);
    if (sm2 > 227 * 1024 || !clov_inv || bs[3] % 2) return cudaErrorInvalidValue;
    launch(fmt == LINK_12 ? (ord ? sap_block_eo_kernel<LINK_12, true> : sap_block_eo_kernel<LINK_12, false>)
                          : (ord ? sap_block_eo_kernel<LINK_18, true> : sap_block_eo_kernel<LINK_18, false>),
           sm2);
    return cudaGetLastError();
  }
  if (kernel == 0) {  // the default
    const size_t sm2 = sap_smem_bytes(bs);
    launch(fmt == LINK_12 ? (ord ? sap_block_kernel<LINK_12, true> : sap_block_kernel<LINK_12, false>)
                          : (ord ? sap_block_kernel<LINK_18, true> : sap_block_kernel<LINK_18, false>),
           sm2);
    return cudaGetLastError();
  }
  if (kernel == 2) {
    if (fmt == LINK_12)
      sap_kernel<LINK_12, 2><<<grid, block, smem, s>>>(a);
    else
      sap_kernel<LINK_18, 2><<<grid, block, smem, s>>>(a);
  } else {
    if (fmt == LINK_12)
      sap_kernel<LINK_12, 1><<<grid, block, smem, s>>>(a);
    else
      sap_kernel<LINK_18, 1><<<grid, block, smem, s>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace oq
