// Gauge-equivariant parallel-transport convolution (PTC) layers: the learned
// preconditioner (not in the paper).  A layer maps C_in spinor fields to
// C_out fields,
//
//   out_c'(x) = sum_{q in paths} sum_c W[q][c'][c] (T_q in_c)(x),
//
// paths q = 0 (identity), 1+2mu (+mu: U_mu(x) in(x+mu)), 2+2mu (-mu:
// U_mu(x-mu)^dag in(x-mu)), with the fermion time-boundary factor on hops
// across the time boundary; W[q][c'][c] is a complex 4x4 matrix on spin.
// Weights are used in bfloat16 (rounded from binary32 master weights),
// arithmetic and accumulation binary32, gradient reductions binary64.
//
// The adjoint of a layer (the backward pass for the input) is again a layer:
// W'[reverse(q)][c][c'] = W[q][c'][c]^dag, since T_{+mu}^dag = T_{-mu}.
// Weight gradients: dW[q][c'][c] = sum_x g_c'(x) (T_q in_c)(x)^dag (spin outer
// product, colour summed): per-CTA binary64 partials, summed in a fixed order.
#include <math.h>
#include <string.h>

#include <vector>

#include "../../include/oq.h"
#include "ctx.h"
#include "oq_kernels.h"
#include "reduce.cuh"

namespace oq {

static const int NPATH = 9;
static const int PB = 128;  // threads per CTA

struct PtcArgs {
  Geom g;
  const void* links;  // binary32 packed links
  const char* in;     // C_in packed binary32 full fields
  char* out;          // C_out packed binary32 full fields
  long fbytes;        // bytes of one full field
  long hbytes;        // bytes of one half field
  const __nv_bfloat162* w;  // [NPATH][C_out][C_in][4][4] complex, bfloat16
};

// (T_q psi)(x) for site (p, i, x) of a full field `f`
template <int FMT>
__device__ __forceinline__ void transport(const PtcArgs& a, const char* f, int q, int p, long i, const int x[4],
                                          Spinor<float>& t) {
  if (q == 0) {
    load_spinor<P_F32>(f + (long)p * a.hbytes, a.g.Vh, i, t);
    return;
  }
  const int mu = (q - 1) >> 1;
  const bool fwd = ((q - 1) & 1) == 0;
  bool cr;
  const long j = eo_neighbour_rt(a.g, x, mu, fwd ? +1 : -1, &cr);
  Spinor<float> s;
  load_spinor<P_F32>(f + (long)(1 - p) * a.hbytes, a.g.Vh, j, s);
  Su3<float> u;
  if (fwd)
    load_link<float, FMT>(a.links, a.g.Vh, p, mu, i, u);
  else
    load_link<float, FMT>(a.links, a.g.Vh, 1 - p, mu, j, u);
  const float sg = cr ? a.g.bc_t : 1.0f;
#pragma unroll
  for (int sp = 0; sp < 4; ++sp)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      cx<float> acc{0.f, 0.f};
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (fwd)
          cfma(acc, u.m[c][b], s.c[sp][b]);
        else
          cfmac(acc, u.m[b][c], s.c[sp][b]);
      }
      t.c[sp][c] = sg * acc;
    }
}

// The operands of one path at a site, as loaded: the neighbour's spinors of the
// CIN input fields and the link.
template <int FMT, int CIN>
struct PathIn {
  float4 f[CIN][6];
  Su3<float> u;
  bool cross;  // the hop crosses the time boundary
};

template <int FMT, int CIN, bool FWD>
__device__ __forceinline__ void path_load(const PtcArgs& a, int mu, int p, long i, const int x[4],
                                          PathIn<FMT, CIN>& in) {
  const long j = eo_neighbour_rt(a.g, x, mu, FWD ? +1 : -1, &in.cross);
#pragma unroll
  for (int ci = 0; ci < CIN; ++ci) {
    const float4* f = reinterpret_cast<const float4*>(a.in + ci * a.fbytes + (long)(1 - p) * a.hbytes) + j;
#pragma unroll
    for (int c = 0; c < 6; ++c) in.f[ci][c] = ldg_nc(f + c * a.g.Vh);
  }
  load_link<float, FMT>(a.links, a.g.Vh, FWD ? p : 1 - p, mu, FWD ? i : j, in.u);
}

// component k (= 3 spin + colour) of a field as loaded
__device__ __forceinline__ float2 comp(const float4 (&f)[6], int k) {
  const float4 v = f[k / 2];
  return (k & 1) ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
}
__device__ __forceinline__ float2 swapped(float2 z) { return make_float2(z.y, z.x); }

// acc[s][c] += sum_t W[s][t] f[t][c], lanes (re, im): two packed FMAs per
// complex product, w = (wr, wr, -wi, wi)
__device__ __forceinline__ void spin_mul(const float4* w, const float2 (&f)[12], float2 (&acc)[12]) {
  float2 g[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) g[k] = swapped(f[k]);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float4 v = w[4 * s + t];
      const float2 wr = make_float2(v.x, v.y), wi = make_float2(v.z, v.w);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        acc[3 * s + c] = __ffma2_rn(wr, f[3 * t + c], __ffma2_rn(wi, g[3 * t + c], acc[3 * s + c]));
    }
}

// out = U f (FWD) or U^dag f on colour, times the boundary factor where the hop
// crosses it
template <bool FWD>
__device__ __forceinline__ void colour_mul(const Su3<float>& u, const float2 (&f)[12], bool cross, float bc_t,
                                           float2 (&out)[12]) {
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      cx<float> acc{0.f, 0.f};
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const cx<float> z{f[3 * s + b].x, f[3 * s + b].y};
        if (FWD)
          cfma(acc, u.m[c][b], z);
        else
          cfmac(acc, u.m[b][c], z);
      }
      out[3 * s + c] = make_float2(acc.re, acc.im);
    }
  if (cross) {
#pragma unroll
    for (int k = 0; k < 12; ++k) out[k] = make_float2(bc_t * out[k].x, bc_t * out[k].y);
  }
}

// one path's contribution to the COUT outputs; w: its weights [COUT][CIN][16].
// The spin weights commute with the transport: with more inputs than outputs
// the inputs are contracted at the neighbour and one field is transported.
template <int FMT, int CIN, int COUT, bool FWD>
__device__ __forceinline__ void path_apply(const PathIn<FMT, CIN>& in, float bc_t, const float4* w,
                                           float2 (&acc)[COUT][12]) {
  if constexpr (CIN <= COUT) {
#pragma unroll
    for (int ci = 0; ci < CIN; ++ci) {
      float2 f[12], t[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) f[k] = comp(in.f[ci], k);
      colour_mul<FWD>(in.u, f, in.cross, bc_t, t);
#pragma unroll
      for (int co = 0; co < COUT; ++co) spin_mul(w + (co * CIN + ci) * 16, t, acc[co]);
    }
  } else {
#pragma unroll
    for (int co = 0; co < COUT; ++co) {
      float2 m[12], t[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) m[k] = make_float2(0.f, 0.f);
#pragma unroll
      for (int ci = 0; ci < CIN; ++ci) {
        float2 f[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) f[k] = comp(in.f[ci], k);
        spin_mul(w + (co * CIN + ci) * 16, f, m);
      }
      colour_mul<FWD>(in.u, m, in.cross, bc_t, t);
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[co][k] = __fadd2_rn(acc[co][k], t[k]);
    }
  }
}

// One thread per site.  Bound by the binary32 pipe (4.6k operations per site)
// and by the gather: each direction's operands are loaded while the one before
// is computed, and the spin products run on packed lanes.  48x24^3, both
// layers: 361 us against 435 us scalar with every input transported and no
// operands ahead (12 warps per SM for one 12-real input, 8 otherwise: more
// registers beat more warps by 13 %, 416 us with 8 throughout).
template <int FMT, int CIN, int COUT>
__global__ void __launch_bounds__(PB, CIN == 1 && FMT == LINK_12 ? 3 : 2) ptc_layer_kernel(const PtcArgs a) {
  __shared__ float4 w[NPATH * COUT * CIN * 16];
  for (int k = threadIdx.x; k < NPATH * COUT * CIN * 16; k += blockDim.x) {
    const float2 v = __bfloat1622float2(a.w[k]);
    w[k] = make_float4(v.x, v.x, -v.y, v.y);
  }
  __syncthreads();
  const long j = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= 2 * a.g.Vh) return;
  const int p = j >= a.g.Vh ? 1 : 0;
  const long i = j - p * a.g.Vh;
  int x[4];
  eo_coords(a.g, p, i, x);
  constexpr int NW = COUT * CIN * 16;  // weights per path
  PathIn<FMT, CIN> fw, bw;
  path_load<FMT, CIN, true>(a, 0, p, i, x, fw);
  float2 acc[COUT][12];
#pragma unroll
  for (int co = 0; co < COUT; ++co)
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[co][k] = make_float2(0.f, 0.f);
  // the identity path
#pragma unroll
  for (int ci = 0; ci < CIN; ++ci) {
    const float4* f = reinterpret_cast<const float4*>(a.in + ci * a.fbytes + (long)p * a.hbytes) + i;
    float4 raw[6];
    float2 v[12];
#pragma unroll
    for (int c = 0; c < 6; ++c) raw[c] = ldg_nc(f + c * a.g.Vh);
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = comp(raw, k);
#pragma unroll
    for (int co = 0; co < COUT; ++co) spin_mul(w + (co * CIN + ci) * 16, v, acc[co]);
  }
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    path_load<FMT, CIN, false>(a, mu, p, i, x, bw);
    path_apply<FMT, CIN, COUT, true>(fw, a.g.bc_t, w + (1 + 2 * mu) * NW, acc);
    if (mu < 3) path_load<FMT, CIN, true>(a, mu + 1, p, i, x, fw);
    path_apply<FMT, CIN, COUT, false>(bw, a.g.bc_t, w + (2 + 2 * mu) * NW, acc);
  }
#pragma unroll
  for (int co = 0; co < COUT; ++co) {
    float4* o = reinterpret_cast<float4*>(a.out + co * a.fbytes + (long)p * a.hbytes) + i;
#pragma unroll
    for (int c = 0; c < 6; ++c)
      o[c * a.g.Vh] = make_float4(acc[co][2 * c].x, acc[co][2 * c].y, acc[co][2 * c + 1].x, acc[co][2 * c + 1].y);
  }
}

// The sum over the warp of 32 binary32 values per lane; lane l returns that of
// v[l].  A transposing exchange (each step halves the values a lane holds: 31
// additions per lane instead of 5 per value), in double-float: the first
// additions are exact, the others err by ~2^-47, against the 2^-24 of the
// binary32 sums that come in.  In binary64 (1/64 of the binary32 rate) the warp
// sums were half of the gradient kernels' time; they are taken that way where a
// value of the warp is not finite or above 2^100 (binary32 sums could overflow).
__device__ __forceinline__ double warp_sum32(const float (&v)[32]) {
  const int lane = threadIdx.x & 31;
  bool big = false;
#pragma unroll
  for (int k = 0; k < 32; ++k) big |= !(fabsf(v[k]) <= 1.2676506e30f);
  if (__any_sync(0xffffffffu, big)) {
    double out = 0.0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const double t = warp_sum((double)v[k]);
      if (lane == k) out = t;
    }
    return out;
  }
  dfloat d[16];
  {
    const bool up = lane & 16;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float keep = up ? v[k + 16] : v[k], send = up ? v[k] : v[k + 16];
      d[k] = df_two_sum(keep, __shfl_xor_sync(0xffffffffu, send, 16));
    }
  }
#pragma unroll
  for (int h = 8; h >= 1; h >>= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const dfloat keep = up ? d[k + h] : d[k], send = up ? d[k] : d[k + h];
      const dfloat got(__shfl_xor_sync(0xffffffffu, send.hi, h), __shfl_xor_sync(0xffffffffu, send.lo, h));
      d[k] = keep + got;
    }
  }
  return (double)d[0];
}

// Weight-gradient partials of one path (blockIdx.y) and one pair of channels
// (blockIdx.z = co * CIN + ci): 16 complex per CTA, written in binary64 to
// part[q][cta][32 z ..].  (One CTA for both channel pairs shares the transport
// of a single input but needs 255 registers, 8 warps per SM that wait for their
// gathers: the gradient of 4 pairs on 32x16^3 1.32 against 1.26 ms.)  Bound by
// the gathers from L2, 240 bytes per site and path.
template <int FMT, int CIN>
__global__ void __launch_bounds__(PB, 4) ptc_dw_kernel(const PtcArgs a, const char* grad, double* part) {
  __shared__ double red[PB / 32][32];
  const int q = blockIdx.y, ci = blockIdx.z % CIN, co = blockIdx.z / CIN;
  const char* in = a.in + ci * a.fbytes;
  const char* gf = grad + co * a.fbytes;
  float2 acc[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) acc[k] = make_float2(0.f, 0.f);
  for (long j = (long)blockIdx.x * blockDim.x + threadIdx.x; j < 2 * a.g.Vh; j += (long)gridDim.x * blockDim.x) {
    const int p = j >= a.g.Vh ? 1 : 0;
    const long i = j - p * a.g.Vh;
    int x[4];
    eo_coords(a.g, p, i, x);
    Spinor<float> gv, t;
    load_spinor<P_F32>(gf + (long)p * a.hbytes, a.g.Vh, i, gv);
    transport<FMT>(a, in, q, p, i, x, t);
#pragma unroll
    for (int tt = 0; tt < 4; ++tt)
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        // g[s] conj(t[tt]), lanes (re, im)
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const cx<float> g = gv.c[s][c], z = t.c[tt][c];
          v = __ffma2_rn(make_float2(z.im, z.im), make_float2(g.im, -g.re), v);
          v = __ffma2_rn(make_float2(z.re, z.re), make_float2(g.re, g.im), v);
        }
        acc[s * 4 + tt] = __fadd2_rn(acc[s * 4 + tt], v);
      }
  }
  float v[32];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    v[2 * k] = acc[k].x;
    v[2 * k + 1] = acc[k].y;
  }
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  red[wid][lane] = warp_sum32(v);
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < PB / 32; ++w) s += red[w][lane];
    part[((long)q * gridDim.x + blockIdx.x) * 64 + 32 * blockIdx.z + lane] = s;
  }
}

// sum the per-CTA partials of np pairs in a fixed order:
// dw[layer][q][k] += sum_pair sum_cta part[pair][layer][q][cta][k].  One CTA per
// path (blockIdx.x) and layer (blockIdx.y), thread (k, j) adds the partials j,
// j + FIN, ... of value k, then the FIN sums are added in order (one thread per value, its loads one after the other, took 108
// us for 256 partials on 32x16^3, a fifth of the gradient; this form 9 us for a pair's).
static const int FIN = 16;
__global__ void __launch_bounds__(64 * FIN) ptc_dw_finish(const double* part, int np, int ncta, double* dw) {
  const int layer = blockIdx.y;
  constexpr int NV = 64;
  __shared__ double sum[FIN][NV];
  const int q = blockIdx.x, k = threadIdx.x % NV, j = threadIdx.x / NV;
  double s = 0.0;
  for (int r = 0; r < np; ++r) {
    const double* p = part + (((long)r * 2 + layer) * NPATH + q) * ncta * NV + k;
#pragma unroll 8
    for (int c = j; c < ncta; c += FIN) s += p[(long)c * NV];
  }
  sum[j][k] = s;
  __syncthreads();
  if (j) return;
#pragma unroll
  for (int w = 1; w < FIN; ++w) s += sum[w][k];
  dw[((long)layer * NPATH + q) * NV + k] += s;
}

// bfloat16 forward weights and the adjoint layer's weights from binary32 masters:
// w: [q][co][ci][s][t]; adjoint: [rev(q)][ci][co][t][s] = conj(w[q][co][ci][s][t])
__global__ void ptc_prepare_weights(const float2* master, int cin, int cout, __nv_bfloat162* fwd,
                                    __nv_bfloat162* adj) {
  const int n = NPATH * cout * cin * 16;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    int r = k;
    const int t = r % 4;
    r /= 4;
    const int s = r % 4;
    r /= 4;
    const int ci = r % cin;
    r /= cin;
    const int co = r % cout;
    const int q = r / cout;
    const float2 v = master[k];
    fwd[k] = __floats2bfloat162_rn(v.x, v.y);
    const int qr = q == 0 ? 0 : (((q - 1) & 1) ? q - 1 : q + 1);
    // adjoint layer has C_in' = cout, C_out' = cin
    const int ka = ((qr * cin + ci) * cout + co) * 16 + t * 4 + s;
    adj[ka] = __floats2bfloat162_rn(v.x, -v.y);
  }
}

// g = 2 (y - e) / ||e||^2, loss partial ||y - e||^2 / ||e||^2 -> FIN_STORE slot
__global__ void __launch_bounds__(256) ptc_loss_kernel(const char* y, const char* e, char* g, double inv_en2, long Vh,
                                                       long hb, RedArgs ra) {
  __shared__ double smem[8];
  double acc = 0.0;
  for (long j = (long)blockIdx.x * blockDim.x + threadIdx.x; j < 2 * Vh; j += (long)gridDim.x * blockDim.x) {
    const int p = j >= Vh ? 1 : 0;
    const long i = j - p * Vh;
    Spinor<float> a, b;
    load_spinor<P_F32>(y + p * hb, Vh, i, a);
    load_spinor<P_F32>(e + p * hb, Vh, i, b);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        a.c[s][c] = a.c[s][c] - b.c[s][c];
        const double xr = (double)a.c[s][c].re, xi = (double)a.c[s][c].im;
        acc = fma(xr, xr, fma(xi, xi, acc));
        a.c[s][c] = (float)(2.0 * inv_en2) * a.c[s][c];
      }
    store_spinor<P_F32>(g + p * hb, Vh, i, a);
  }
  grid_reduce(acc * inv_en2, ra, 0, 1, smem, blockIdx.x, gridDim.x);
}

// Adam on binary32 master weights (per real component), gradient in binary64
__global__ void ptc_adam(float* w, float* m, float* v, const double* g, int n, float lr, float b1, float b2,
                         float c1, float c2, float eps) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = (float)g[k];
  const float mk = b1 * m[k] + (1.f - b1) * gk;
  const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  w[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

template <int CIN, int COUT>
static cudaError_t ptc_layer(const PtcArgs& a, int fmt, cudaStream_t s) {
  dim3 grid((unsigned)((2 * a.g.Vh + PB - 1) / PB)), block(PB);
  if (fmt == LINK_12)
    ptc_layer_kernel<LINK_12, CIN, COUT><<<grid, block, 0, s>>>(a);
  else
    ptc_layer_kernel<LINK_18, CIN, COUT><<<grid, block, 0, s>>>(a);
  return cudaGetLastError();
}

template <int CIN, int COUT>
static cudaError_t ptc_dw(const PtcArgs& a, int fmt, const char* grad, double* part, int ncta, cudaStream_t s) {
  static_assert(CIN * COUT == 2, "the partials hold two channel pairs per path");
  dim3 grid(ncta, NPATH, CIN * COUT), block(PB);
  if (fmt == LINK_12)
    ptc_dw_kernel<LINK_12, CIN><<<grid, block, 0, s>>>(a, grad, part);
  else
    ptc_dw_kernel<LINK_18, CIN><<<grid, block, 0, s>>>(a, grad, part);
  return cudaGetLastError();
}

}  // namespace oq

using namespace oq;

namespace {
const int CH = 2;                      // hidden feature fields
const int NW1 = NPATH * CH * 1 * 16;   // complex weights of layer 1 (1 -> CH)
const int NW2 = NPATH * 1 * CH * 16;   // complex weights of layer 2 (CH -> 1)

struct NnBufs {
  __nv_bfloat162 *w1, *w2, *w1a, *w2a;
  char* hid;   // CH fields
  char* ghid;  // CH fields
  char* y;
  char* gy;
};

int nn_bufs(oq_handle h, int lat, NnBufs* b) {
  const long f32 = 2 * spinor_half_bytes(h->lats[lat].g.Vh, P_F32);
  void *wb, *hid, *ghid, *y, *gy;
  int rc = 0;
  rc |= h->workspace(lat, "nn_w", sizeof(__nv_bfloat162) * 2 * (NW1 + NW2), &wb);
  rc |= h->workspace(lat, "nn_hid", f32 * CH, &hid);
  rc |= h->workspace(lat, "nn_ghid", f32 * CH, &ghid);
  rc |= h->workspace(lat, "nn_y", f32, &y);
  rc |= h->workspace(lat, "nn_gy", f32, &gy);
  if (rc) return OQ_ERR_NOMEM;
  b->w1 = (__nv_bfloat162*)wb;
  b->w2 = b->w1 + NW1;
  b->w1a = b->w2 + NW2;
  b->w2a = b->w1a + NW1;
  b->hid = (char*)hid;
  b->ghid = (char*)ghid;
  b->y = (char*)y;
  b->gy = (char*)gy;
  return OQ_OK;
}

int nn_prepare(oq_handle h, const float* master, const NnBufs& b, cudaStream_t s) {
  ptc_prepare_weights<<<4, 256, 0, s>>>((const float2*)master, 1, CH, b.w1, b.w1a);
  ptc_prepare_weights<<<4, 256, 0, s>>>((const float2*)master + NW1, CH, 1, b.w2, b.w2a);
  h->launches += 2;
  return cudaGetLastError() == cudaSuccess ? OQ_OK : OQ_ERR_CUDA;
}

PtcArgs nn_args(oq_handle h, int lat) {
  const LatCtx& L = h->lats[lat];
  PtcArgs a;
  a.g = L.g;
  a.links = L.u32.p;
  a.hbytes = spinor_half_bytes(L.g.Vh, P_F32);
  a.fbytes = 2 * a.hbytes;
  return a;
}

// y = L2(L1(r)) with the prepared bfloat16 weights
int nn_forward(oq_handle h, int lat, const NnBufs& b, const void* r, void* y, cudaStream_t s) {
  const int fmt = h->lats[lat].link_fmt;
  PtcArgs a = nn_args(h, lat);
  a.in = (const char*)r;
  a.out = b.hid;
  a.w = b.w1;
  if (ptc_layer<1, CH>(a, fmt, s) != cudaSuccess) return OQ_ERR_CUDA;
  a.in = b.hid;
  a.out = (char*)y;
  a.w = b.w2;
  if (ptc_layer<CH, 1>(a, fmt, s) != cudaSuccess) return OQ_ERR_CUDA;
  h->launches += 2;
  return OQ_OK;
}

}  // namespace

// internal: the learned preconditioner as used inside flexible GCR
namespace oq {
int nnprec_prepare(oq_handle h, int lat, const float* master, cudaStream_t s) {
  NnBufs b;
  int rc = nn_bufs(h, lat, &b);
  if (rc) return rc;
  return nn_prepare(h, master, b, s);
}
int nnprec_forward(oq_handle h, int lat, const void* r, void* y, cudaStream_t s) {
  NnBufs b;
  int rc = nn_bufs(h, lat, &b);
  if (rc) return rc;
  return nn_forward(h, lat, b, r, y, s);
}
}  // namespace oq

extern "C" int oq_nnprec_apply(oq_handle h, int lat, const float* weights_dev, const void* in_dev, void* out_dev,
                               void* stream) {
  if (!h || lat < 0 || lat >= (int)h->lats.size() || !weights_dev || !in_dev || !out_dev) return OQ_ERR_ARG;
  if (!h->lats[lat].has_gauge || h->lats[lat].halo_t) return OQ_ERR_STATE;  // whole lattices only
  cudaStream_t s = (cudaStream_t)stream;
  int rc = nnprec_prepare(h, lat, weights_dev, s);
  if (rc) return rc;
  return nnprec_forward(h, lat, in_dev, out_dev, s);
}

extern "C" int oq_nnprec_grad(oq_handle h, int lat, const float* weights_dev, const void* r_dev, const void* e_dev,
                              int n, double* grad_dev, double* loss_host, void* stream);

extern "C" int oq_nnprec_train(oq_handle h, int lat, float* weights_dev, const void* r_dev, const void* e_dev, int n,
                               double lr, int steps, double* loss_host, void* stream) {
  if (!h || lat < 0 || lat >= (int)h->lats.size() || !weights_dev || !r_dev || !e_dev || n < 1 || steps < 1 ||
      !(lr > 0.0))
    return OQ_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int nreal = 2 * (NW1 + NW2);
  void *mom, *grad;
  int rc = h->workspace(lat, "nn_adam", sizeof(float) * 2 * nreal, &mom);
  if (!rc) rc = h->workspace(lat, "nn_gradbuf", sizeof(double) * nreal, &grad);
  if (rc) return OQ_ERR_NOMEM;
  if (cudaMemsetAsync(mom, 0, sizeof(float) * 2 * nreal, s) != cudaSuccess) return OQ_ERR_CUDA;
  const float b1 = 0.9f, b2 = 0.999f;
  float p1 = 1.f, p2 = 1.f;
  for (int it = 0; it < steps; ++it) {
    double loss = 0.0;
    rc = oq_nnprec_grad(h, lat, weights_dev, r_dev, e_dev, n, (double*)grad, &loss, stream);
    if (rc) return rc;
    if (loss_host) loss_host[it] = loss;
    p1 *= b1;
    p2 *= b2;
    ptc_adam<<<(nreal + 255) / 256, 256, 0, s>>>(weights_dev, (float*)mom, (float*)mom + nreal, (const double*)grad,
                                                 nreal, (float)lr, b1, b2, 1.f - p1, 1.f - p2, 1e-8f);
    h->launches += 1;
    if (cudaGetLastError() != cudaSuccess) return OQ_ERR_CUDA;
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) return OQ_ERR_CUDA;
  return OQ_OK;
}

extern "C" int oq_nnprec_grad(oq_handle h, int lat, const float* weights_dev, const void* r_dev, const void* e_dev,
                              int n, double* grad_dev, double* loss_host, void* stream) {
  if (!h || lat < 0 || lat >= (int)h->lats.size() || !weights_dev || !r_dev || !e_dev || n < 1 || !grad_dev)
    return OQ_ERR_ARG;
  LatCtx& L = h->lats[lat];
  if (!L.has_gauge || L.halo_t) return OQ_ERR_STATE;  // whole lattices only
  cudaStream_t s = (cudaStream_t)stream;
  NnBufs b;
  int rc = nn_bufs(h, lat, &b);
  if (rc) return rc;
  rc = nn_prepare(h, weights_dev, b, s);
  if (rc) return rc;
  const long Vh = L.g.Vh;
  const long hb = spinor_half_bytes(Vh, P_F32), f32 = 2 * hb;
  const int ncta = reduce_grid(2 * Vh) < 256 ? reduce_grid(2 * Vh) : 256;
  void* part;
  const int GRP = 8;
  const size_t npart = (size_t)NPATH * ncta * 64;  // partials of one pair and layer
  rc = h->workspace(lat, "nn_part", sizeof(double) * 2 * npart * (n < GRP ? n : GRP), &part);
  double en2[GRP];
  if (!rc) rc = h->ensure_reduce(2 * GRP, reduce_grid(2 * Vh));
  if (rc) return rc;
  const int fmt = L.link_fmt;
  const int nreal = 2 * (NW1 + NW2);
  if (cudaMemsetAsync(grad_dev, 0, sizeof(double) * nreal, s) != cudaSuccess) return OQ_ERR_CUDA;
  static_assert(2 * NW1 == NPATH * 64 && NW1 == NW2, "gradients of layer 1, then of layer 2");
  double loss = 0.0;
  // pairs in groups of GRP: the norms of the group's e in one launch per parity
  // (one wait), the losses read back together at the group's end (another) and
  // the weight gradients' partials summed there; a wait for the norm and one for
  // the loss of every pair left the GPU idle between its kernels
  for (int k = 0; k < n; ++k) {
    const int kg = k % GRP, ng = n - (k - kg) < GRP ? n - (k - kg) : GRP;
    const char* r = (const char*)r_dev + (long)k * f32;
    const char* e = (const char*)e_dev + (long)k * f32;
    RedArgs ra = h->red_args(FIN_STORE, 0);
    if (kg == 0) {
      // ||e||^2 of the group: parity halves in results[0 .. ng) and [ng .. 2 ng)
      h->launches += 2;
      if (reduce_norm2(P_F32, e, Vh, f32, ng, ra, s) != cudaSuccess) return OQ_ERR_CUDA;
      ra.result = h->results + ng;
      if (reduce_norm2(P_F32, e + hb, Vh, f32, ng, ra, s) != cudaSuccess) return OQ_ERR_CUDA;
      if (cudaMemcpyAsync(h->results_host, h->results, 2 * ng * sizeof(double), cudaMemcpyDeviceToHost, s) !=
              cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return OQ_ERR_CUDA;
      for (int j = 0; j < ng; ++j) {
        en2[j] = h->results_host[j] + h->results_host[ng + j];
        if (!(en2[j] > 0.0)) return OQ_ERR_ARG;
      }
    }
    rc = nn_forward(h, lat, b, r, b.y, s);
    if (rc) return rc;
    ra = h->red_args(FIN_STORE, 0);
    ra.result = h->results + kg;
    // mean over the n pairs: loss_k / n and its gradient
    ptc_loss_kernel<<<reduce_grid(2 * Vh), 256, 0, s>>>(b.y, e, b.gy, 1.0 / (en2[kg] * n), Vh, hb, ra);
    h->launches += 1;
    // layer 2: dW2 from (hid, gy); g_hid = L2^dag gy
    PtcArgs a = nn_args(h, lat);
    a.in = b.hid;
    a.w = b.w2;
    double* part1 = (double*)part + 2 * npart * kg;
    double* part2 = part1 + npart;
    if (ptc_dw<CH, 1>(a, fmt, b.gy, part2, ncta, s) != cudaSuccess) return OQ_ERR_CUDA;
    a.in = b.gy;
    a.out = b.ghid;
    a.w = b.w2a;
    if (ptc_layer<1, CH>(a, fmt, s) != cudaSuccess) return OQ_ERR_CUDA;
    // layer 1: dW1 from (r, g_hid)
    a = nn_args(h, lat);
    a.in = r;
    a.w = b.w1;
    if (ptc_dw<1, CH>(a, fmt, b.ghid, part1, ncta, s) != cudaSuccess) return OQ_ERR_CUDA;
    h->launches += 3;
    if (cudaGetLastError() != cudaSuccess) return OQ_ERR_CUDA;
    if (kg == ng - 1) {
      ptc_dw_finish<<<dim3(NPATH, 2), 64 * FIN, 0, s>>>((const double*)part, ng, ncta, grad_dev);
      h->launches += 1;
      if (cudaMemcpyAsync(h->results_host, h->results, ng * sizeof(double), cudaMemcpyDeviceToHost, s) !=
              cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return OQ_ERR_CUDA;
      for (int j = 0; j < ng; ++j) loss += h->results_host[j];
    }
  }
  if (loss_host) *loss_host = loss;
  return OQ_OK;
}
