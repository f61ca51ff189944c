// Layout conversion kernels: canonical binary64 links and spinors (site
// lexicographic, time slowest) to the packed even-odd chunk-major device
// layouts, with rounding to the storage precision (round to nearest even)
// and an optional per-field scale for the 16-bit formats.
#include "oq_internal.h"
#include "oq_kernels.h"

namespace oq {

__device__ __forceinline__ long lex_of(const Geom& g, const int x[4]) {
  return (((long)x[0] * g.L[1] + x[1]) * g.L[2] + x[2]) * g.L[3] + x[3];
}

// one thread per (eo site, parity, mu); u18 (optional) receives an 18-real
// binary32 copy next to a 12-real one; A (optional) multiplies the link by
// exp(i q A_mu(x)) (QCD+QED), uclov / au1 (optional) keep the link before
// the phase and the angle
// cs_l1 > 0 (C* boundaries): canon holds the physical links of L1 = cs_l1
// (half the doubled extent g.L[1]); the sites x1 >= cs_l1 of the doubled
// lattice get the charge-conjugate copy: the complex conjugate link (and the
// U(1) angle negated)
__global__ void pack_links_kernel(Geom g, const double2* __restrict__ canon, double2* __restrict__ u64,
                                  void* __restrict__ u32, int fmt, float2* __restrict__ u18,
                                  const double* __restrict__ A, double q, double2* __restrict__ uclov,
                                  double* __restrict__ au1, int cs_l1) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = blockIdx.y;
  const int mu = blockIdx.z;
  if (i >= g.Vh) return;
  int x[4];
  eo_coords(g, p, i, x);
  bool mirror = false;
  long lex = lex_of(g, x);
  if (cs_l1 > 0) {
    mirror = x[1] >= cs_l1;
    const int x1 = mirror ? x[1] - cs_l1 : x[1];
    lex = (((long)x[0] * cs_l1 + x1) * g.L[2] + x[2]) * g.L[3] + x[3];
  }
  const double2* src = canon + (lex * 4 + mu) * 9;
  double2 m[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) m[k] = mirror ? make_double2(src[k].x, -src[k].y) : src[k];
  if (uclov) {
    double2* d = uclov + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
    for (int k = 0; k < 9; ++k) d[k * g.Vh + i] = m[k];
  }
  if (A) {
    const double a = mirror ? -A[lex * 4 + mu] : A[lex * 4 + mu];
    double sn, cs;
    sincos(q * a, &sn, &cs);
#pragma unroll
    for (int k = 0; k < 9; ++k) m[k] = make_double2(m[k].x * cs - m[k].y * sn, m[k].x * sn + m[k].y * cs);
    au1[(long)(p * 4 + mu) * g.Vh + i] = a;
  }
  double2* d64 = u64 + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
  for (int k = 0; k < 9; ++k) d64[k * g.Vh + i] = m[k];
  if (!u32) return;  // binary64 links only
  if (fmt == LINK_18) {
    float2* d = reinterpret_cast<float2*>(u32) + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
    for (int k = 0; k < 9; ++k) d[k * g.Vh + i] = make_float2(narrow(m[k].x), narrow(m[k].y));
  } else {
    float4* d = reinterpret_cast<float4*>(u32) + ((long)(p * 4 + mu) * 3) * g.Vh;
    d[i] = make_float4(narrow(m[0].x), narrow(m[0].y), narrow(m[1].x), narrow(m[1].y));
    d[g.Vh + i] = make_float4(narrow(m[2].x), narrow(m[2].y), narrow(m[3].x), narrow(m[3].y));
    d[2 * g.Vh + i] = make_float4(narrow(m[4].x), narrow(m[4].y), narrow(m[5].x), narrow(m[5].y));
    if (u18) {
      float2* e = u18 + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
      for (int k = 0; k < 9; ++k) e[k * g.Vh + i] = make_float2(narrow(m[k].x), narrow(m[k].y));
    }
  }
}

cudaError_t pack_links(const Geom& g, const double* canon, double* u64, void* u32, int fmt, void* u18,
                       const double* A, double q, double* uclov, double* au1, cudaStream_t s, int cs_l1) {
  dim3 block(128), grid((unsigned)((g.Vh + 127) / 128), 2, 4);
  pack_links_kernel<<<grid, block, 0, s>>>(g, reinterpret_cast<const double2*>(canon),
                                           reinterpret_cast<double2*>(u64), u32, fmt,
                                           reinterpret_cast<float2*>(u18), A, q,
                                           reinterpret_cast<double2*>(uclov), au1, cs_l1);
  return cudaGetLastError();
}

// one thread per (eo site, parity): the time-like link U_0(x) of the slices
// x0 = 0 (hops 0 <-> 1) and x0 = T-1 (hops T-1 <-> T, i.e. across the
// boundary) becomes zero in every hopping copy, so that no hop reaches the
// x0 = 0 slice, where Schroedinger-functional quark fields vanish
__global__ void sf_mask_links_kernel(Geom g, double2* __restrict__ u64, void* __restrict__ u32, int fmt,
                                     float2* __restrict__ u18) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = blockIdx.y;
  if (i >= g.Vh) return;
  int x[4];
  eo_coords(g, p, i, x);
  if (x[0] != 0 && x[0] != g.L[0] - 1) return;
  const int mu = 0;
  double2* d64 = u64 + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
  for (int k = 0; k < 9; ++k) d64[k * g.Vh + i] = make_double2(0.0, 0.0);
  if (fmt == LINK_18) {
    float2* d = reinterpret_cast<float2*>(u32) + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
    for (int k = 0; k < 9; ++k) d[k * g.Vh + i] = make_float2(0.f, 0.f);
  } else {
    float4* d = reinterpret_cast<float4*>(u32) + ((long)(p * 4 + mu) * 3) * g.Vh;
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k * g.Vh + i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (u18) {
    float2* e = u18 + ((long)(p * 4 + mu) * 9) * g.Vh;
#pragma unroll
    for (int k = 0; k < 9; ++k) e[k * g.Vh + i] = make_float2(0.f, 0.f);
  }
}

cudaError_t sf_mask_links(const Geom& g, double* u64, void* u32, int fmt, void* u18, cudaStream_t s) {
  dim3 block(128), grid((unsigned)((g.Vh + 127) / 128), 2);
  sf_mask_links_kernel<<<grid, block, 0, s>>>(g, reinterpret_cast<double2*>(u64), u32, fmt,
                                              reinterpret_cast<float2*>(u18));
  return cudaGetLastError();
}

// The site's 24 reals in the arithmetic type: at(k) gives complex component k
// (scaled).  Binary32: by integer operations, and over again by the conversion
// instruction if one of them needs it.  One branch a site: with one a value, F32
// fields took 4.5 against 2.9 us on 8^4, and 742 against 395 us for 12 fields of
// zeros on 48x24^3 (418 of other values; by the instruction 693).
template <typename R, typename F>
__device__ __forceinline__ void site_from64(Spinor<R>& s, F at) {
  if constexpr (std::is_same<R, float>::value) {
    bool slow = false;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const double2 v = at(k);
      s.c[k / 3][k % 3] = cx<R>{narrow_bits(v.x, slow), narrow_bits(v.y, slow)};
    }
    if (!slow) return;
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const double2 v = at(k);
    s.c[k / 3][k % 3] = cx<R>{R(v.x), R(v.y)};
  }
}

// four complex values as 16-bit pairs, rounded from binary64 directly (no
// intermediate binary32 rounding)
template <int P, typename F>
__device__ __forceinline__ uint4 chunk16(F at) {
  uint32_t w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double2 v = at(k);
    if constexpr (P == P_BF16) {
      const __nv_bfloat16 a = __double2bfloat16(v.x), b = __double2bfloat16(v.y);
      w[k] = (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
    } else {
      const __half a = __double2half(v.x), b = __double2half(v.y);
      w[k] = (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// one thread per (eo site, parity, rhs).  blockIdx.y = parity index within
// the subset, blockIdx.z = rhs.  UNIT: scale 1 and not a Schroedinger-functional
// lattice (whose field vanishes at x0 = 0: scale 0 there): no multiplications on
// the binary64 pipe.
template <int P, bool UNIT>
__global__ void pack_spinor_kernel(Geom g, const double2* __restrict__ canon, char* __restrict__ out,
                                   int subset, long canon_stride, long out_stride, double scale) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.Vh) return;
  const int p = (subset == 2) ? (int)blockIdx.y : subset;
  const int rhs = blockIdx.z;
  int x[4];
  eo_coords(g, p, i, x);
  const double2* src = canon + rhs * canon_stride + lex_of(g, x) * 12;
  if (!UNIT && g.bc_t == 0.f && x[0] == 0) scale = 0.0;
  auto at = [&](int k) {
    const double2 v = src[k];
    return UNIT ? v : make_double2(v.x * scale, v.y * scale);
  };
  char* dst = out + rhs * out_stride + ((subset == 2) ? (long)p * spinor_half_bytes(g.Vh, P) : 0);
  if constexpr (P == P_BF16 || P == P_F16) {
    uint4* b = reinterpret_cast<uint4*>(dst);
#pragma unroll
    for (int c = 0; c < 3; ++c) b[c * g.Vh + i] = chunk16<P>([&](int k) { return at(4 * c + k); });
  } else {
    Spinor<typename PrecTraits<P>::R> s;
    site_from64(s, at);
    store_spinor<P>(dst, g.Vh, i, s);
  }
}

template <bool UNIT, typename R>
__device__ __forceinline__ double unscaled(R x, double inv_scale) {
  return UNIT ? (double)x : (double)x * inv_scale;
}

// Even-site (or odd-site) canonical fields: the site of eo index i sits at
// position i (lex / 2), so the 128 sites of a CTA are one contiguous run of
// 128 x 12 double2.  The run moves between the canonical field and shared
// memory with consecutive threads on consecutive 16-byte chunks (coalesced,
// which matters when the field is page-locked host memory read or written
// over the host-device link), and each thread converts its own site from
// there.  Shared rows of 13 chunks keep the per-site accesses free of bank
// conflicts.  blockDim.x = 128.
constexpr int HB = 128, HROW = 13;

template <int P, bool UNIT>
__global__ void __launch_bounds__(HB) pack_half_kernel(Geom g, const double2* __restrict__ canon,
                                                       char* __restrict__ out, int p, long canon_stride,
                                                       long out_stride, double scale) {
  __shared__ double2 sm[HB * HROW];
  const int t = threadIdx.x, rhs = blockIdx.z;
  const long i0 = (long)blockIdx.x * HB;
  const int nsite = (int)(g.Vh - i0 < HB ? g.Vh - i0 : HB);
  const double2* src = canon + rhs * canon_stride + i0 * 12;
  for (int e = t; e < nsite * 12; e += HB) sm[(e / 12) * HROW + e % 12] = src[e];
  __syncthreads();
  if (t >= nsite) return;
  const long i = i0 + t;
  if (!UNIT && g.bc_t == 0.f) {  // Schroedinger-functional lattices: the field vanishes at x0 = 0
    int x[4];
    eo_coords(g, p, i, x);
    if (x[0] == 0) scale = 0.0;
  }
  auto at = [&](int k) {
    const double2 v = sm[t * HROW + k];
    return UNIT ? v : make_double2(v.x * scale, v.y * scale);
  };
  char* dst = out + rhs * out_stride;
  if constexpr (P == P_BF16 || P == P_F16) {
    uint4* b = reinterpret_cast<uint4*>(dst);
#pragma unroll
    for (int c = 0; c < 3; ++c) b[c * g.Vh + i] = chunk16<P>([&](int k) { return at(4 * c + k); });
  } else {
    Spinor<typename PrecTraits<P>::R> sp;
    site_from64(sp, at);
    store_spinor<P>(dst, g.Vh, i, sp);
  }
}

// Packed sites to a canonical field of one parity (HALF) or of both (blockIdx.y),
// through shared memory as above: a site's 192 bytes are written by 12
// neighbouring threads.  (Each thread writing its own site's, pieces of 16 bytes
// 384 bytes apart: 12 full fields on 48x24^3 F64 654, F32 1070, F16 1130 us; 560, 446
// and 322 this way.)  UNIT: scale 1, no multiplication on the binary64 pipe (a
// choice per value is a branch before each store: F64 on 8^4 3.5 against 2.0 us).
template <int P, bool UNIT, bool HALF>
__global__ void __launch_bounds__(HB) unpack_kernel(Geom g, const char* __restrict__ in, double2* __restrict__ canon,
                                                    int subset, long in_stride, long canon_stride, double inv_scale) {
  __shared__ double2 sm[HB * HROW];
  __shared__ int at[HB];  // the site's position in the canonical field
  const int t = threadIdx.x, rhs = blockIdx.z, p = subset == 2 ? (int)blockIdx.y : subset;
  const long i0 = (long)blockIdx.x * HB;
  const int nsite = (int)(g.Vh - i0 < HB ? g.Vh - i0 : HB);
  const char* src = in + rhs * in_stride + ((subset == 2) ? (long)p * spinor_half_bytes(g.Vh, P) : 0);
  if (t < nsite) {
    const long i = i0 + t;
    if (!HALF) {
      int x[4];
      eo_coords(g, p, i, x);
      at[t] = (int)(2 * i) + (x[3] & 1);  // lex: the eo index is lex >> 1
    }
    Spinor<typename PrecTraits<P>::R> sp;
    load_spinor<P>(src, g.Vh, i, sp);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const double re = (double)sp.c[k / 3][k % 3].re, im = (double)sp.c[k / 3][k % 3].im;
      sm[t * HROW + k] = UNIT ? make_double2(re, im) : make_double2(re * inv_scale, im * inv_scale);
    }
  }
  __syncthreads();
  double2* dst = canon + rhs * canon_stride;
  for (int e = t; e < nsite * 12; e += HB) {
    const long site = HALF ? i0 + e / 12 : (long)at[e / 12];
    dst[site * 12 + e % 12] = sm[(e / 12) * HROW + e % 12];
  }
}

template <int P, bool UNIT>
static void pack_launch(const Geom& g, int subset, const double2* canon, char* out, double scale, int nrhs,
                        long canon_stride, long out_stride, cudaStream_t s, int half) {
  if (half) {
    const dim3 hb(HB), hg((unsigned)((g.Vh + HB - 1) / HB), 1, nrhs);
    pack_half_kernel<P, UNIT><<<hg, hb, 0, s>>>(g, canon, out, subset, canon_stride, out_stride, scale);
  } else {
    const dim3 block(128), grid((unsigned)((g.Vh + 127) / 128), subset == 2 ? 2 : 1, nrhs);
    pack_spinor_kernel<P, UNIT><<<grid, block, 0, s>>>(g, canon, out, subset, canon_stride, out_stride, scale);
  }
}

cudaError_t pack_spinor(const Geom& g, int prec, int subset, const double* canon, void* out, double scale,
                        int nrhs, long canon_stride_d2, long out_stride_bytes, cudaStream_t s, int half) {
  if (half && subset == 2) return cudaErrorInvalidValue;
  const double2* c = reinterpret_cast<const double2*>(canon);
  char* o = reinterpret_cast<char*>(out);
  auto launch = [&](auto* unit, auto* scaled) {
    (scale == 1.0 && g.bc_t != 0.f ? unit : scaled)(g, subset, c, o, scale, nrhs, canon_stride_d2, out_stride_bytes, s,
                                                    half);
  };
  switch (prec) {
    case P_F64: launch(pack_launch<P_F64, true>, pack_launch<P_F64, false>); break;
    case P_F32: launch(pack_launch<P_F32, true>, pack_launch<P_F32, false>); break;
    case P_BF16: launch(pack_launch<P_BF16, true>, pack_launch<P_BF16, false>); break;
    case P_F16: launch(pack_launch<P_F16, true>, pack_launch<P_F16, false>); break;
    case P_DF64: launch(pack_launch<P_DF64, true>, pack_launch<P_DF64, false>); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int P, bool UNIT>
static void unpack_launch(const Geom& g, int subset, const char* in, double2* canon, double inv_scale, int nrhs,
                          long in_stride, long canon_stride, cudaStream_t s, int half) {
  const dim3 grid((unsigned)((g.Vh + HB - 1) / HB), subset == 2 ? 2 : 1, nrhs);
  auto* k = half ? unpack_kernel<P, UNIT, true> : unpack_kernel<P, UNIT, false>;
  k<<<grid, HB, 0, s>>>(g, in, canon, subset, in_stride, canon_stride, inv_scale);
}

cudaError_t unpack_spinor(const Geom& g, int prec, int subset, const void* in, double* canon, double scale,
                          int nrhs, long in_stride_bytes, long canon_stride_d2, cudaStream_t s, int half) {
  if (half && subset == 2) return cudaErrorInvalidValue;
  double2* c = reinterpret_cast<double2*>(canon);
  const char* i = reinterpret_cast<const char*>(in);
  const double inv = 1.0 / scale;
  auto launch = [&](auto* unit, auto* scaled) {
    (inv == 1.0 ? unit : scaled)(g, subset, i, c, inv, nrhs, in_stride_bytes, canon_stride_d2, s, half);
  };
  switch (prec) {
    case P_F64: launch(unpack_launch<P_F64, true>, unpack_launch<P_F64, false>); break;
    case P_F32: launch(unpack_launch<P_F32, true>, unpack_launch<P_F32, false>); break;
    case P_BF16: launch(unpack_launch<P_BF16, true>, unpack_launch<P_BF16, false>); break;
    case P_F16: launch(unpack_launch<P_F16, true>, unpack_launch<P_F16, false>); break;
    case P_DF64: launch(unpack_launch<P_DF64, true>, unpack_launch<P_DF64, false>); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// binary64 array -> double-float pairs (hi = rn(x), lo = rn(x - hi)), element
// by element: a binary64-layout field or table becomes its DF64 layout
__global__ void split_f64_kernel(const double* __restrict__ in, float2* __restrict__ out, size_t n) {
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    const double x = in[k];
    const float hi = narrow(x);
    out[k] = make_float2(hi, narrow(x - (double)hi));
  }
}

cudaError_t split_f64(const double* in, void* out, size_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  size_t blocks = (n + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  split_f64_kernel<<<(unsigned)blocks, 256, 0, s>>>(in, reinterpret_cast<float2*>(out), n);
  return cudaGetLastError();
}

}  // namespace oq
