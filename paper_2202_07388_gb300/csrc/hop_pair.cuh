// The one-rhs binary32-arithmetic stencil with two threads per site (F32 /
// BF16 / F16 storage).
//
// hop_kernel gives a site to one thread, which walks its 8 hops one memory
// latency after the other: a small problem takes that long whatever its size,
// and a large one keeps too few loads in flight.  Here the warps of the first
// half of a CTA take the hops along mu = 0, 1 of its 64 sites, those of the
// second half mu = 2, 3; the halves exchange the spins they do not keep through
// shared memory, and the first finishes spins 0, 1 (its chiral clover block and
// half of the epilogue), the second spins 2, 3.  Twice the warps, half the
// latency per thread, the same loads.
// F32 Dhat, 1 rhs: 105 us against 120 us on 48x24^3, 155 against 178 us on 32^4
// (5.4 TB/s of operands), 34 against 43 us on 32x24x16x16, the same on 32x16^3
// (10 us a pass from L2).  Small problems gain in the solver, where a launch may
// start under the one before it (launch_dep) and finds its clover block loaded:
// F32 CGNE on 16^4 6.0 to 4.6 ms, on 32x16^3 8.5 to 7.5 ms.
#pragma once
#include "hop_impl.cuh"

namespace oq {
namespace pairs {

constexpr int SITES = 64, THREADS = 2 * SITES;

// half a packed spinor (spins 2b, 2b+1; 6 complex): 3 float4 (F32), or a
// 16-byte chunk and half of the middle one (BF16 / F16)
template <int P>
__device__ __forceinline__ void load_half_spinor(const char* base, uint32_t Vh, uint32_t i, int b, cx<float> (&v)[6]) {
  if constexpr (P == P_F32) {
    const float4* q = reinterpret_cast<const float4*>(base) + (size_t)(3 * b) * Vh;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float4 w = ld_field(q + (c * Vh + i));
      v[2 * c] = cx<float>{w.x, w.y};
      v[2 * c + 1] = cx<float>{w.z, w.w};
    }
  } else {
    const uint4 f = ld_field(reinterpret_cast<const uint4*>(base) + (size_t)(2 * b) * Vh + i);
    const uint2 m = ld_field(reinterpret_cast<const uint2*>(base) + ((size_t)Vh + i) * 2 + b);
    const uint32_t w[6] = {b ? m.x : f.x, b ? m.y : f.y, b ? f.x : f.z, b ? f.y : f.w, b ? f.z : m.x, b ? f.w : m.y};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float2 z = (P == P_BF16) ? unpack_bf16x2(w[k]) : unpack_f16x2(w[k]);
      v[k] = cx<float>{z.x, z.y};
    }
  }
}

template <int P>
__device__ __forceinline__ void store_half_spinor(char* base, uint32_t Vh, uint32_t i, int b, const cx<float> (&v)[6]) {
  if constexpr (P == P_F32) {
    float4* q = reinterpret_cast<float4*>(base) + (size_t)(3 * b) * Vh;
#pragma unroll
    for (int c = 0; c < 3; ++c) q[c * Vh + i] = make_float4(v[2 * c].re, v[2 * c].im, v[2 * c + 1].re, v[2 * c + 1].im);
  } else {
    uint32_t w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k)
      w[k] = (P == P_BF16) ? pack_bf16x2(v[k].re, v[k].im) : pack_f16x2(v[k].re, v[k].im);
    reinterpret_cast<uint4*>(base)[(size_t)(2 * b) * Vh + i] =
        b ? make_uint4(w[2], w[3], w[4], w[5]) : make_uint4(w[0], w[1], w[2], w[3]);
    reinterpret_cast<uint2*>(base)[((size_t)Vh + i) * 2 + b] = b ? make_uint2(w[0], w[1]) : make_uint2(w[4], w[5]);
  }
}

// round to the storage type and back
template <int P>
__device__ __forceinline__ void round_half(cx<float> (&v)[6]) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if constexpr (P == P_BF16) {
      const float2 z = unpack_bf16x2(pack_bf16x2(v[k].re, v[k].im));
      v[k] = cx<float>{z.x, z.y};
    } else if constexpr (P == P_F16) {
      const float2 z = unpack_f16x2(pack_f16x2(v[k].re, v[k].im));
      v[k] = cx<float>{z.x, z.y};
    }
  }
}

// y = K x for one Hermitian 6x6 block as loaded (clover_apply's order)
__device__ __forceinline__ void block_mul(const float4 (&q)[9], const cx<float> (&x)[6], cx<float> (&y)[6]) {
  float r[36];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    r[4 * k] = q[k].x;
    r[4 * k + 1] = q[k].y;
    r[4 * k + 2] = q[k].z;
    r[4 * k + 3] = q[k].w;
  }
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

// CTA `blk` of the nblk that cover the sites of parity p for right-hand side rhs
// EARLY: launched by launch_dep on a small problem: the site's clover block is
// read before the wait for the previous kernel (36 registers through the hops,
// which cost more than they hide on a large one)
template <int P, int FMT, int MODE, bool DAG, int EPI, bool EARLY>
__device__ __forceinline__ void body(const HopArgs& a, uint32_t blk, int rhs, int p, unsigned nblk) {
  __shared__ float sm[2 * 12 * SITES];
  __shared__ double red_smem[THREADS / 32];
  const int b = threadIdx.x / SITES, s = threadIdx.x % SITES;  // b: the spins 2b, 2b+1 and hops 2b, 2b+1
  const uint32_t Vh = (uint32_t)a.g.Vh;
  const bool live = blk * SITES + s < Vh;
  const uint32_t i = live ? blk * SITES + s : Vh - 1;  // threads past the end repeat the last site, stored by no one
  const long par_in = (MODE == HOP_DW) ? (long)(1 - p) * a.half_bytes : 0;
  const long par_out = (MODE == HOP_DW) ? (long)p * a.half_bytes : 0;
  const char* in = (const char*)a.in + rhs * a.in_stride + par_in;
  int x[4];
  eo_coords(a.g, p, i, x);
  const float4* cl =
      reinterpret_cast<const float4*>(MODE == HOP_P1 ? a.cinv : a.clov) + (size_t)(p * 18 + 9 * b) * Vh + i;
  float4 q[9];  // the site's clover block
  auto load_clover = [&]() {
#pragma unroll
    for (int k = 0; k < 9; ++k) q[k] = ldg_nc(cl + (size_t)k * Vh);
  };
  if constexpr (EARLY) {
    load_clover();
    dep_wait();
  }
  record_live(a);
  if (a.cg && a.cg[rhs].mode != a.gate) return;  // gated off by the solver state: in every CTA of the rhs
  cx<float> res[6];
  if constexpr (MODE != HOP_P1) {
    cx<float> loc[6];
    load_half_spinor<P>((const char*)a.in2 + rhs * a.in2_stride + par_out, Vh, i, b, loc);
    if constexpr (!EARLY) load_clover();
    block_mul(q, loc, res);
  }
  const float w = (MODE == HOP_P2) ? 0.5f : -0.5f;
  Spinor<float> acc;
#pragma unroll
  for (int k = 0; k < 12; ++k) acc.c[k / 3][k % 3] = cx<float>{0.f, 0.f};
  if (b == 0) {
    hop_dir<P, FMT, 0, DAG>(a, in, p, i, x, acc, w);
    hop_dir<P, FMT, 1, DAG>(a, in, p, i, x, acc, w);
  } else {
    hop_dir<P, FMT, 2, DAG>(a, in, p, i, x, acc, w);
    hop_dir<P, FMT, 3, DAG>(a, in, p, i, x, acc, w);
  }
  if constexpr (!EARLY && MODE == HOP_P1) load_clover();
  // operands of the CG update, in flight across the exchange
  cx<float> pv[6], rv[6], xv[6];
  if constexpr (EPI == EPI_CG) {
    load_half_spinor<P>((const char*)a.ep_p + rhs * a.ep_p_stride, Vh, i, b, pv);
    load_half_spinor<P>((const char*)a.ep_r + rhs * a.ep_r_stride, Vh, i, b, rv);
    load_half_spinor<P_F32>((const char*)a.ep_x + rhs * a.ep_x_stride, Vh, i, b, xv);
  }
  float* mine = sm + b * 12 * SITES + s;
  const float* other = sm + (1 - b) * 12 * SITES + s;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const cx<float> z = b ? acc.c[k / 3][k % 3] : acc.c[2 + k / 3][k % 3];
    mine[(2 * k) * SITES] = z.re;
    mine[(2 * k + 1) * SITES] = z.im;
  }
  __syncthreads();
  cx<float> h[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const cx<float> z = b ? acc.c[2 + k / 3][k % 3] : acc.c[k / 3][k % 3];
    h[k] = z + cx<float>{other[(2 * k) * SITES], other[(2 * k + 1) * SITES]};
  }
  if constexpr (MODE == HOP_P1) {
    block_mul(q, h, res);
  } else {
#pragma unroll
    for (int k = 0; k < 6; ++k) res[k] = res[k] + h[k];
  }
  float sq = 0.f;  // the thread's squares (norm epilogues)
  if (live) {
    if constexpr (EPI == EPI_CG) {
      // q = res; x += alpha p; r -= alpha q
      const float al = (float)a.cg[rhs].alpha;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        xv[k].re = fmaf(al, pv[k].re, xv[k].re);
        xv[k].im = fmaf(al, pv[k].im, xv[k].im);
        rv[k].re = fmaf(-al, res[k].re, rv[k].re);
        rv[k].im = fmaf(-al, res[k].im, rv[k].im);
      }
      round_half<P>(rv);  // the norm of what is stored
      store_half_spinor<P_F32>((char*)a.ep_x + rhs * a.ep_x_stride, Vh, i, b, xv);
      store_half_spinor<P>((char*)a.ep_r + rhs * a.ep_r_stride, Vh, i, b, rv);
#pragma unroll
      for (int k = 0; k < 6; ++k) sq += rv[k].re * rv[k].re + rv[k].im * rv[k].im;
    } else {
      store_half_spinor<P>((char*)a.out + rhs * a.out_stride + par_out, Vh, i, b, res);
      if constexpr (EPI == EPI_NORM) {
#pragma unroll
        for (int k = 0; k < 6; ++k) sq += res[k].re * res[k].re + res[k].im * res[k].im;
      }
    }
  }
  if constexpr (EPI != EPI_NONE) grid_reduce(sq, a.red, rhs, a.nrhs, red_smem, blk, nblk);
}

}  // namespace pairs

// grid: rhs fastest, then (HOP_DW) parity, then site blocks
template <int P, int FMT, int MODE, bool DAG, int EPI, bool EARLY>
__global__ void __launch_bounds__(pairs::THREADS, 4) hop_pair_kernel(const HopArgs a) {
  const unsigned rhs = blockIdx.x % (unsigned)a.nrhs, rest = blockIdx.x / (unsigned)a.nrhs;
  const uint32_t blk = (MODE == HOP_DW) ? rest >> 1 : rest;
  const int p = (MODE == HOP_DW) ? (int)(rest & 1) : a.p;
  if constexpr (EARLY) dep_trigger();
  pairs::body<P, FMT, MODE, DAG, EPI, EARLY>(a, blk, (int)rhs, p, gridDim.x / (unsigned)a.nrhs);
}

// several systems (as hop_batch_kernel): CTA = one tile (system, block of 64 sites)
template <int P, int FMT, int MODE, bool DAG, int EPI>
__global__ void __launch_bounds__(pairs::THREADS, 4) hop_pair_batch_kernel(const HopArgs* __restrict__ sys,
                                                                           const int2* __restrict__ tiles) {
  const int2 tl = tiles[blockIdx.x];
  const HopArgs& a = sys[tl.x];
  const uint32_t blk = (MODE == HOP_DW) ? (uint32_t)tl.y >> 1 : (uint32_t)tl.y;
  const int p = (MODE == HOP_DW) ? (tl.y & 1) : a.p;
  pairs::body<P, FMT, MODE, DAG, EPI, false>(a, blk, 0, p, ((uint32_t)a.g.Vh + pairs::SITES - 1) / pairs::SITES);
}

template <int P, int FMT, int MODE, bool DAG, int EPI>
static cudaError_t launch_pair_one(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  if (L.sys) {
    hop_pair_batch_kernel<P, FMT, MODE, DAG, EPI><<<L.ntiles, pairs::THREADS, 0, s>>>(L.sys, L.tiles);
    return cudaGetLastError();
  }
  if (L.bx != pairs::SITES || a.halo_next) return cudaErrorInvalidValue;
  const unsigned nb = (unsigned)((a.g.Vh + pairs::SITES - 1) / pairs::SITES);
  const dim3 grid((MODE == HOP_DW ? 2u * nb : nb) * (unsigned)a.nrhs);
  // early start: 1 rhs, us early against not: F32 Dhat on 8^4 5.5 against 6.2, 32x16^3
  // 17.4 against 17.5 (a CG step 76 against 84), 32x24x20x16 (122,880 sites) 43.4
  // against 41.3 (CG 150 against 152), 32x24^3 73.7 against 69.7 (CG 231 against 225);
  // F16 Dhat 5.2 / 5.9, 16.2 / 16.7, 35.1 / 35.7 and 65.4 / 63.2
  if (a.g.Vh * a.nrhs <= (1L << 17))
    return launch_dep(hop_pair_kernel<P, FMT, MODE, DAG, EPI, true>, grid, dim3(pairs::THREADS), 0, s, a);
  hop_pair_kernel<P, FMT, MODE, DAG, EPI, false><<<grid, pairs::THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

template <int P, int FMT, bool DAG>
static cudaError_t pair_mode_epi(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  switch (L.mode) {
    case HOP_DW:
      if (L.epi == EPI_NONE) return launch_pair_one<P, FMT, HOP_DW, DAG, EPI_NONE>(L, a, s);
      break;
    case HOP_P1:
      if (L.epi == EPI_NONE) return launch_pair_one<P, FMT, HOP_P1, DAG, EPI_NONE>(L, a, s);
      break;
    case HOP_P2:
      if (L.epi == EPI_NONE) return launch_pair_one<P, FMT, HOP_P2, DAG, EPI_NONE>(L, a, s);
      if (L.epi == EPI_NORM) return launch_pair_one<P, FMT, HOP_P2, DAG, EPI_NORM>(L, a, s);
      if (L.epi == EPI_CG) return launch_pair_one<P, FMT, HOP_P2, DAG, EPI_CG>(L, a, s);
      break;
  }
  return cudaErrorInvalidValue;
}

template <int P>
static cudaError_t pair_dispatch(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  if (L.link_fmt == LINK_12)
    return L.dagger ? pair_mode_epi<P, LINK_12, true>(L, a, s) : pair_mode_epi<P, LINK_12, false>(L, a, s);
  return L.dagger ? pair_mode_epi<P, LINK_18, true>(L, a, s) : pair_mode_epi<P, LINK_18, false>(L, a, s);
}

}  // namespace oq
