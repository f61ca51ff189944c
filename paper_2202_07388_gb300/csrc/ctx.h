// The handle behind the C ABI: per-lattice packed gauge/clover state, a
// grow-only workspace of named device buffers, the reduction scratch, the
// per-kernel launch shapes chosen by the tuner, and optional CUDA-event
// timing of every stencil launch.
#pragma once
#include <cuda_runtime.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

#include "../../include/oq.h"
#include "oq_internal.h"
#include "oq_kernels.h"

namespace oq {

struct DevBuf {
  void* p = nullptr;
  size_t n = 0;
};

struct LatCtx {
  Geom g;
  int link_fmt = -1;
  bool has_gauge = false, has_clover = false;
  double kappa = 0.0, csw = 0.0;
  DevBuf u64, u32, a64, a32, i64, i32;
  DevBuf u32_18;  // 18-real binary32 copy kept next to 12-real links
  // double-float (hi, lo) splits of the binary64 links, clover and inverse
  // clover, made on the first DF64 use after an upload / clover build
  DevBuf udf, adf, idf;
  bool df_ready = false;
  // Schroedinger-functional lattices (bc_t = 0) and QCD+QED uploads keep the
  // unmasked binary64 links the clover is built from (SU(3) part for QCD+QED)
  // and the packed U(1) angles with their charge
  DevBuf uclov, au1;
  bool uclov_valid = false, has_u1 = false;
  // time-split sub-domain (OQ_BC_HALO): its time hops across x0 = 0 / T-1
  // read faces of the neighbouring sub-domains; uext holds the packed binary64
  // links of the sub-domain extended by one slice on each side (clover build)
  bool halo_t = false, has_uext = false;
  // C* boundaries in this many spatial directions (x1 first): the lattice is
  // doubled in x1 (g.L[1] = 2 L1); 0 = none
  int cstar = 0;
  DevBuf uext;
  double qcharge = 0.0, cF = 1.0, csw_qed = 0.0;
  std::map<std::string, DevBuf> ws;
};

// one timed stencil launch: its algorithmic bytes are fixed (links, clover:
// read once if any right-hand side is live) + per_rhs x (live right-hand
// sides), the live count read back from slot `slot` of the device record
struct ProfRec {
  cudaEvent_t e0, e1;
  int mode, epi, prec, nr, link_fmt, dag;
  double fixed, per_rhs;
  int nrhs;
  long slot;  // -1: no record slot (counted as all right-hand sides live)
};

// tuned CTA shape of one stencil variant; epi = EPI_NONE is the entry for
// every epilogue the tuner did not time separately
struct TuneKey {
  int lat, prec, mode, nrhs, epi;
  bool operator<(const TuneKey& o) const {
    if (lat != o.lat) return lat < o.lat;
    if (prec != o.prec) return prec < o.prec;
    if (mode != o.mode) return mode < o.mode;
    if (nrhs != o.nrhs) return nrhs < o.nrhs;
    return epi < o.epi;
  }
};

// the launch shape chosen for one stencil variant (by the tuner or set)
struct TuneVal {
  int bx = 128, by = 1;  // CTA: bx sites x by groups of nr right-hand sides
  int nr = 1;            // right-hand sides per thread
  int regcap = 0;        // register-capped multi-rhs variant
  int link_fmt = -1;     // binary32 link format (-1: the uploaded one)
  bool pair = false;     // two threads per site (bx = 64, by = nr = 1; reported and pinned as by = 0)
  float ms = 0.f;        // tuner's time per launch (0 if set by hand)
};

}  // namespace oq

struct oq_ctx {
  int device = 0;
  std::vector<oq::LatCtx> lats;
  // reduction scratch
  double* partials = nullptr;
  size_t partials_n = 0;
  unsigned* counters = nullptr;
  size_t counters_n = 0;
  double* results = nullptr;
  double* results_host = nullptr;  // pinned
  size_t results_n = 0;
  int* status_dev = nullptr;
  oq::CgState* cg_dev = nullptr;
  oq::CgState* cg_host = nullptr;  // pinned mirror
  size_t cg_n = 0;
  // launch shapes
  std::map<oq::TuneKey, oq::TuneVal> tuned;
  // kernels launched by this handle so far
  long long launches = 0;
  // CGNE: intermediate reset residuals in double-float arithmetic (default:
  // ~3x faster per pass than binary64 on GB300; every stop decision binary64)
  bool df64_resets = true;   // OQ_OPT_DF64_RESETS
  // test hook: the tensor-core PTC layer issues no MMA, so its bounded wait runs out
  bool hook_tc_skip_commit = false;
  // SAP block kernel: 0 links in registers and clover in shared memory, 1 operands from
  // global memory, 2 the same register-capped for two CTAs per SM
  int sap_kernel = 0;        // OQ_OPT_SAP_KERNEL
  // NN-preconditioned GCR applies the network with the tensor-core layers
  // instead of the (measured faster) binary32 CUDA-core ones
  bool nn_tensor_cores = false;
  // solver diagnostics (OQ_OPT_HISTORY): CGNE's relative recursive residual
  // after every regular step and its relative residual at every reset, per
  // rhs, of the last solve that recorded them
  bool history = false;
  int hist_nrhs = 0;                                    // 0: nothing recorded
  std::vector<std::vector<double>> hist_rec;            // [rhs][step - 1]
  std::vector<std::vector<double>> hist_reset;          // [rhs]: step, residual, step, residual, ...
  // profiling
  bool prof_on = false;
  std::vector<oq::ProfRec> prof;
  std::vector<cudaEvent_t> event_pool;
  // per profiled launch: right-hand sides live in it (written by the kernel)
  unsigned* prof_live = nullptr;
  size_t prof_live_n = 0;

  int alloc(oq::DevBuf* b, size_t n) {
    if (b->n >= n && b->p) return OQ_OK;
    if (b->p) {
      cudaDeviceSynchronize();
      cudaFree(b->p);
      b->p = nullptr;
      b->n = 0;
    }
    if (cudaMalloc(&b->p, n) != cudaSuccess) {
      cudaGetLastError();
      return OQ_ERR_NOMEM;
    }
    b->n = n;
    return OQ_OK;
  }

  int workspace(int lat, const char* name, size_t n, void** out) {
    oq::DevBuf& b = lats[lat].ws[name];
    int rc = alloc(&b, n);
    *out = b.p;
    return rc;
  }

  // library-owned stream for graph capture and replay (the caller's stream
  // may be the legacy default stream, which cannot be captured)
  cudaStream_t work_stream = nullptr;
  int ensure_work_stream() {
    if (!work_stream && cudaStreamCreateWithFlags(&work_stream, cudaStreamNonBlocking) != cudaSuccess)
      return OQ_ERR_CUDA;
    return OQ_OK;
  }

  // pinned host staging for small coefficient uploads (4 KiB)
  void* stage_host = nullptr;
  int ensure_stage() {
    if (!stage_host && cudaMallocHost(&stage_host, 4096) != cudaSuccess) return OQ_ERR_NOMEM;
    return OQ_OK;
  }

  int ensure_scratch() {
    if (!status_dev && cudaMalloc(&status_dev, 64) != cudaSuccess) return OQ_ERR_NOMEM;
    return OQ_OK;
  }

  // room for `slots` reductions of `grid` partials each
  int ensure_reduce(int slots, long grid) {
    int rc = ensure_scratch();
    if (rc) return rc;
    size_t np = (size_t)slots * (size_t)grid;
    if (np > partials_n) {
      cudaDeviceSynchronize();
      cudaFree(partials);
      partials = nullptr;
      if (cudaMalloc(&partials, np * sizeof(double)) != cudaSuccess) return OQ_ERR_NOMEM;
      partials_n = np;
    }
    if ((size_t)slots > counters_n) {
      cudaDeviceSynchronize();
      cudaFree(counters);
      cudaFree(results);
      cudaFreeHost(results_host);
      counters = nullptr;
      results = nullptr;
      results_host = nullptr;
      size_t n = (size_t)slots < 64 ? 64 : (size_t)slots;
      if (cudaMalloc(&counters, n * sizeof(unsigned)) != cudaSuccess) return OQ_ERR_NOMEM;
      if (cudaMemset(counters, 0, n * sizeof(unsigned)) != cudaSuccess) return OQ_ERR_CUDA;
      if (cudaMalloc(&results, 2 * n * sizeof(double)) != cudaSuccess) return OQ_ERR_NOMEM;
      if (cudaMallocHost(&results_host, 2 * n * sizeof(double)) != cudaSuccess) return OQ_ERR_NOMEM;
      counters_n = n;
      results_n = 2 * n;
    }
    return OQ_OK;
  }

  int ensure_cg(int nrhs) {
    if ((size_t)nrhs <= cg_n) return OQ_OK;
    cudaDeviceSynchronize();
    cudaFree(cg_dev);
    cudaFreeHost(cg_host);
    cg_dev = nullptr;
    cg_host = nullptr;
    if (cudaMalloc(&cg_dev, nrhs * sizeof(oq::CgState)) != cudaSuccess) return OQ_ERR_NOMEM;
    if (cudaMallocHost(&cg_host, nrhs * sizeof(oq::CgState)) != cudaSuccess) return OQ_ERR_NOMEM;
    cg_n = nrhs;
    return OQ_OK;
  }

  oq::RedArgs red_args(int fin, int gate) {
    oq::RedArgs r;
    r.partials = partials;
    r.counters = counters;
    r.result = results;
    r.cg = cg_dev;
    r.fin = fin;
    r.gate = gate;
    r.defer = 0;
    return r;
  }

  oq::HopArgs hop_args(int lat, int prec) {
    oq::LatCtx& L = lats[lat];
    oq::HopArgs a;
    memset(&a, 0, sizeof(a));
    a.g = L.g;
    if (prec == oq::P_DF64) {  // ensure_df(lat) has made the splits
      a.links = L.udf.p;
      a.clov = L.adf.p;
      a.cinv = L.idf.p;
    } else {
      const bool f64 = prec == oq::P_F64;
      a.links = f64 ? L.u64.p : L.u32.p;
      a.clov = f64 ? L.a64.p : L.a32.p;
      a.cinv = f64 ? L.i64.p : L.i32.p;
    }
    a.nrhs = 1;
    a.lat = lat;
    return a;
  }

  // the double-float splits of links and clover that DF64 kernels read
  int ensure_df(int lat, cudaStream_t s) {
    oq::LatCtx& L = lats[lat];
    if (L.df_ready) return OQ_OK;
    if (!L.has_clover) return OQ_ERR_STATE;
    const size_t nu = (size_t)2 * 4 * 18 * L.g.Vh, na = (size_t)2 * 72 * L.g.Vh;
    int rc = alloc(&L.udf, nu * sizeof(float2));
    if (!rc) rc = alloc(&L.adf, na * sizeof(float2));
    if (!rc) rc = alloc(&L.idf, na * sizeof(float2));
    if (rc) return rc;
    if (oq::split_f64((const double*)L.u64.p, L.udf.p, nu, s) != cudaSuccess ||
        oq::split_f64((const double*)L.a64.p, L.adf.p, na, s) != cudaSuccess ||
        oq::split_f64((const double*)L.i64.p, L.idf.p, na, s) != cudaSuccess)
      return OQ_ERR_CUDA;
    L.df_ready = true;
    return OQ_OK;
  }

  // Two threads per site by default (hop_pair.cuh; binary32-arithmetic types):
  // every launch with one right-hand side (F32 Dhat on 48x24^3: 105 against
  // 120 us with one thread per site, on 32x24x16x16 34 against 43 us, equal on
  // 32x16^3); with several, while the launch is small enough for its latency to
  // count, against two rhs per thread (work: site-rhs of one parity; Dw launches
  // twice as many, which the limits of the 16-bit types count).  Measured from
  // 8^4 to 32x16^3 with 2 to 12 rhs, us of Dw / Dhat, two threads a site against
  // two rhs a thread:
  //  - passes with a reduction below 2^18 (CG step, F32: 221,184 182 against 196,
  //    262,144 214 against 210; F16: 147,456 141 against 160, 262,144 231 against 209);
  //  - F32 below 2^17 (36,864: 8.2 / 9.5 against 10.0 / 15.8; 98,304: 21.6 / 23.3
  //    against 26.4 / 23.3; 131,072: 31.3 / 33.3 against 33.5 / 30.9);
  //  - 16-bit types on 18-real links below 2^17 launched (Dhat, 73,728: 15.2 against
  //    16.5; 131,072: 24.9 against 24.3; Dw, 55,296: 10.7 against 10.5);
  //  - on 12-real links, staged (below), up to 3 * 2^14 launched (24,576: 6.2 / 8.5
  //    against 6.6 / 10.9; Dw, 36,864: 8.1 against 7.2; Dhat, 41,472: 12.2 against
  //    12.9, 55,296: 14.3 against 13.1).
  static bool pair_pays(int prec, int mode, int epi, long work, int nrhs, int link_fmt) {
    if (prec != oq::P_F32 && prec != oq::P_BF16 && prec != oq::P_F16) return false;
    if (nrhs == 1) return true;
    if (epi != oq::EPI_NONE) return work < (1L << 18);
    if (prec == oq::P_F32) return work < (1L << 17);
    const long launched = mode == oq::HOP_DW ? 2 * work : work;
    return link_fmt == oq::LINK_12 ? launched <= (3L << 14) : launched < (1L << 17);
  }

  oq::HopLaunch hop_launch(int lat, int prec, int mode, int dagger, int epi, int nrhs) {
    oq::HopLaunch l;
    l.prec = prec;
    l.link_fmt = lats[lat].link_fmt;
    l.mode = mode;
    l.dagger = dagger;
    l.epi = epi;
    auto it = tuned.find(oq::TuneKey{lat, prec, mode, nrhs, epi});
    if (it == tuned.end()) it = tuned.find(oq::TuneKey{lat, prec, mode, nrhs, oq::EPI_NONE});
    if (it != tuned.end()) {
      l.bx = it->second.bx;
      l.by = it->second.by;
      l.nr = it->second.nr;
      l.regcap = it->second.regcap;
      l.pair = it->second.pair;
      if (it->second.link_fmt >= 0) l.link_fmt = it->second.link_fmt;
    } else if (pair_pays(prec, mode, epi, lats[lat].g.Vh * nrhs, nrhs, l.link_fmt) && !lats[lat].halo_t) {
      l.bx = 64;
      l.by = 1;
      l.pair = true;
    } else if (prec == oq::P_DF64 && !lats[lat].halo_t) {
      // the double-float site is latency- and issue-bound: 12 warps per SM at
      // 168 registers (Dhat, 12 rhs on 48x24^3: 4.0 ms against 6.5 ms
      // uncapped in 32 x 6 CTAs, 4 rhs on 32x16^3: 304 against 370 us).  The
      // cap of 128 registers (16 warps, some spilling) pays only where it puts
      // a launch of more than 3 CTAs per SM into one wave of 4 (Dhat, 1 rhs on
      // 32x16^3, 512 CTAs: 107 against 116 us; 2 rhs on 16^4: 102 against 103;
      // Dw on 16^4, 512 CTAs: 48.1 against 49.1) and costs elsewhere (Dhat on 8^4:
      // 40.9 against 32.8 us; 16^4, 256 CTAs: 60.8 against 48.8; 4 rhs on
      // 16x12^3, 432 CTAs: 73.7 against 65.0; 2 rhs on 32x16^3: 178 against 173)
      l.bx = 128;
      l.by = 1;
      const long ctas = (lats[lat].g.Vh + 127) / 128 * nrhs * (mode == oq::HOP_DW ? 2 : 1);
      l.regcap = ctas > 3 * 152 && ctas <= 4 * 152 ? 1 : 2;
    } else if (nrhs == 1) {
      l.bx = 128;
      l.by = 1;
    } else if ((prec == oq::P_F32 || prec == oq::P_BF16 || prec == oq::P_F16) && !lats[lat].halo_t) {
      // Several right-hand sides of a binary32-arithmetic type: two per thread,
      // so that links, clover and indices serve both.  64-site CTAs: staged
      // hops at 168 registers for the 16-bit types on 12-real links, else
      // capped at 128 registers; within 10 % of the tuner's choice from 8^4 to
      // 48x24^3 with 2 to 12 rhs, where one rhs per thread in 32 x nrhs CTAs
      // took 1.2 to 1.9 times as long (12 rhs F16 Dhat on 48x24^3: 495 against
      // 814 us; 4 rhs F32 on 32x16^3: 58 against 78 us).
      l.bx = 64;
      l.by = 1;
      l.nr = 2;
      l.regcap = (prec != oq::P_F32 && l.link_fmt == oq::LINK_12) ? 3 : 1;
    } else {
      // several right-hand sides: 32 sites x (largest divisor of nrhs <= 8) rows
      l.bx = 32;
      l.by = 1;
      for (int d = 8; d >= 1; --d)
        if (nrhs % d == 0) {
          l.by = d;
          break;
        }
    }
    if (l.by > nrhs) l.by = nrhs;
    return l;
  }

  // algorithmic bytes of one stencil launch (each operand counted once), as
  // the part read once per launch (links, clover) and the part per live
  // right-hand side (spinors and epilogue vectors)
  void hop_bytes_parts(const oq::HopLaunch& l, const oq::HopArgs& a, double* fixed, double* per_rhs) {
    const double sp = oq::prec_bytes(l.prec);
    const bool wide = l.prec == oq::P_F64 || l.prec == oq::P_DF64;  // binary64 links and clover
    const double su = wide ? 8.0 : 4.0;
    const double ru = (!wide && l.link_fmt == oq::LINK_12) ? 12.0 : 18.0;
    const double sites = (double)a.g.Vh * (l.mode == oq::HOP_DW ? 2.0 : 1.0);
    double spin = 0.0;
    double links = 0.0;
    if (l.mode == oq::HOP_DW) {
      spin = 48.0 * sp;          // in + out
      links = 4.0 * ru * su;     // every link once for the full lattice
    } else {
      spin = (l.mode == oq::HOP_P1 ? 48.0 : 72.0) * sp;
      links = 8.0 * ru * su;     // all links once per half-lattice pass
    }
    if (l.epi == oq::EPI_CG) spin += (24.0 + 24.0 + 48.0 - 24.0) * sp + 48.0 * (l.prec == oq::P_F64 ? 8.0 : 4.0);
    if (l.epi == oq::EPI_RESID64) spin += 24.0 * sp;
    const double clov = 72.0 * su;
    *fixed = sites * (links + clov);
    *per_rhs = sites * spin;
  }

  // the binary32 link copy that matches the launch's link format
  oq::HopArgs with_links(const oq::HopLaunch& l, const oq::HopArgs& a) {
    oq::HopArgs b = a;
    if (l.prec != oq::P_F64 && l.prec != oq::P_DF64 && a.lat >= 0 && a.lat < (int)lats.size()) {
      const oq::LatCtx& L = lats[a.lat];
      if (l.link_fmt == oq::LINK_18 && L.link_fmt == oq::LINK_12 && L.u32_18.p) b.links = L.u32_18.p;
    }
    return b;
  }

  int run_hop(const oq::HopLaunch& l, const oq::HopArgs& a, cudaStream_t s) {
    oq::ProfRec rec;
    rec.slot = -1;
    if (prof_on) {
      if (event_pool.size() < 2) {
        for (int k = 0; k < 64; ++k) {
          cudaEvent_t e;
          if (cudaEventCreate(&e) != cudaSuccess) return OQ_ERR_CUDA;
          event_pool.push_back(e);
        }
      }
      rec.e1 = event_pool.back();
      event_pool.pop_back();
      rec.e0 = event_pool.back();
      event_pool.pop_back();
      rec.mode = l.mode;
      rec.epi = l.epi;
      rec.prec = l.prec;
      rec.nr = l.nr;
      rec.dag = l.dagger;
      rec.link_fmt = (l.prec == oq::P_F64 || l.prec == oq::P_DF64) ? -1 : l.link_fmt;
      hop_bytes_parts(l, a, &rec.fixed, &rec.per_rhs);
      rec.nrhs = a.nrhs;
      rec.slot = prof.size() < prof_live_n ? (long)prof.size() : -1;
      cudaEventRecord(rec.e0, s);
    }
    oq::HopArgs b = with_links(l, a);
    b.live_rec = (prof_on && rec.slot >= 0) ? prof_live + rec.slot : nullptr;
    cudaError_t e = oq::launch_hop_reduced(l, b, s, &launches);
    if (prof_on) {
      cudaEventRecord(rec.e1, s);
      prof.push_back(rec);
    }
    return e == cudaSuccess ? OQ_OK : OQ_ERR_CUDA;
  }

  void release() {
    for (auto& L : lats) {
      oq::DevBuf* bs[] = {&L.u64, &L.u32, &L.a64, &L.a32, &L.i64, &L.i32, &L.u32_18, &L.udf, &L.adf, &L.idf, &L.uclov, &L.au1,
                          &L.uext};
      for (auto* b : bs) cudaFree(b->p);
      for (auto& kv : L.ws) cudaFree(kv.second.p);
    }
    cudaFree(prof_live);
    cudaFree(partials);
    cudaFree(counters);
    cudaFree(results);
    cudaFreeHost(results_host);
    cudaFree(status_dev);
    cudaFree(cg_dev);
    cudaFreeHost(cg_host);
    cudaFreeHost(stage_host);
    if (work_stream) cudaStreamDestroy(work_stream);
    for (auto& r : prof) {
      cudaEventDestroy(r.e0);
      cudaEventDestroy(r.e1);
    }
    for (auto e : event_pool) cudaEventDestroy(e);
  }
};
