// kernels_impl.cuh -- likelihood, waveform and acceptance-walk kernels (sm_103a).
// Included by the kernels_p*.cu units: one per precision (p0, p1, p2) and one per variant of the
// float-float walk (p2w, p2c, p2r; the flow variant is in p2), for parallel builds.
//
// Template parameters of every kernel: PREC (0 FP64, 1 mixed with FP64 phase, 2 mixed with
// float-float phase), NDET (detectors, 1..4) and WF (0 TaylorF2, 1 IMRPhenomD form).
// Per-bin sums per detector: Re and Im of S_det = sum_k a_k z_k exp(-2 pi i Phi_det(f_k)), and
// for the IMRPhenomD form the template power sum_k a_k^2 4 df f^-7/3 / S (TaylorF2 takes it
// from prefix sums).  Threads accumulate disjoint bin subsets (FP64, or FP32 with Kahan
// compensation), then warp-shuffle trees (error-free two-sums in FP32) reduce them.
#pragma once

#include <cooperative_groups.h>
#include <cstdio>
#include <type_traits>

#include "flow.cuh"
#include "gwns_internal.h"
#include "screen.h"
#include "setup_split.cuh"

namespace gwns {

namespace {

// Per-SM arrival counters of walk CTAs.  A CTA's position modulo kThreads/32 picks the warp
// that runs its per-proposal setup, so the CTAs sharing an SM spread that FP64-heavy work
// over different sub-partitions (warp w of a CTA runs on sub-partition w mod 4).
__device__ unsigned int g_walk_sm_arrivals[256];

constexpr int kWarps = kThreads / 32;
constexpr int kMaxVals = 3 * kMaxDet;   // (re, im, hh) per detector

// the hardware base-2 logarithm, for the screens of DE steps (screen.h)
struct FastLog2 {
  __device__ __forceinline__ float operator()(float x) const { return __log2f(x); }
};

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The watchdog of a walk's thread 0: a host-set abort flag (read at the start of a round, so that
// the load's latency overlaps the round) and the task's time budget (nanoseconds since the CTA
// started).
__device__ __forceinline__ int walk_abort_flag(const WalkTask& T) {
  return T.abort ? *(volatile const int32_t*)T.abort : 0;
}
__device__ __forceinline__ bool walk_should_stop(const WalkTask& T, uint64_t t0, int abort_flag) {
  return abort_flag != 0 || (T.budget_ns != 0ull && global_ns() - t0 > T.budget_ns);
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

template <int NDET, int WF>
struct NVals { static constexpr int value = (WF == 1 ? 3 : 2) * NDET; };

// Partial sums of the bins k = start, start + stride, ... of one walker (values laid out
// [det][re, im(, hh)]).  FP64 path: dv; mixed paths: (fv, fc) Kahan pairs, fc the negated error.
template <int PREC, int NDET, int WF>
__device__ inline void partials(const EventDev& ev, const WalkerParams& P, int start, int stride, double* dv,
                                float* fv, float* fc) {
  constexpr int NW = (WF == 1 ? 3 : 2);
  if (WF == 0) {
    if (PREC == 0) {
      AccF64 acc; acc.zero();
      for (int k = start; k < P.k_end; k += stride) bin_accumulate_f64<NDET>(ev, P, k, acc);
#pragma unroll
      for (int d = 0; d < NDET; ++d) { dv[NW * d] = acc.re[d]; dv[NW * d + 1] = acc.im[d]; }
    } else {
      AccF32 acc; acc.zero();
      if (PREC == 1) {
        for (int k = start; k < P.k_end; k += stride) bin_accumulate_mixed<NDET>(ev, P, k, acc);
      } else {
        for (int k = start; k < P.k_end; k += stride) bin_accumulate_ff<NDET>(ev, P, k, acc);
      }
#pragma unroll
      for (int d = 0; d < NDET; ++d) {
        fv[NW * d] = acc.re[d]; fc[NW * d] = -acc.cre[d];
        fv[NW * d + 1] = acc.im[d]; fc[NW * d + 1] = -acc.cim[d];
      }
    }
  } else {
    if (PREC == 0) {
      AccPD64 acc; acc.zero();
      for (int k = start; k < P.k_end; k += stride) pd_accumulate_f64<NDET>(ev, P, P.pd, k, acc);
#pragma unroll
      for (int d = 0; d < NDET; ++d) { dv[NW * d] = acc.re[d]; dv[NW * d + 1] = acc.im[d]; dv[NW * d + 2] = acc.hh[d]; }
    } else {
      AccPD32 acc; acc.zero();
      if (PREC == 1) {
        for (int k = start; k < P.k_end; k += stride) pd_accumulate_mixed<NDET>(ev, P, P.pd, k, acc);
      } else {
        pd_sums_ff<NDET>(ev, P, P.pd, start, P.k_end, stride, acc);
      }
#pragma unroll
      for (int d = 0; d < NDET; ++d) {
        fv[NW * d] = acc.re[d]; fc[NW * d] = -acc.cre[d];
        fv[NW * d + 1] = acc.im[d]; fc[NW * d + 1] = -acc.cim[d];
        fv[NW * d + 2] = acc.hh[d]; fc[NW * d + 2] = -acc.chh[d];
      }
    }
  }
}

// Warp reductions: lane 0 receives the totals.
template <int NV>
__device__ __forceinline__ void warp_reduce_f64(double* dv) {
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    double r = dv[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) r += __shfl_down_sync(0xffffffffu, r, off);
    dv[i] = r;
  }
}

// Compensated all-lane sums of NV values by recursive halving: at the exchange with offset
// S each lane keeps half of the values it still carries (the upper half when bit S of its
// lane is set) and adds its partner's copy of that half, so V = NV rounded up to a power of
// two values need V - 1 pair exchanges before the last value is reduced over the remaining
// lanes (instead of NV * 5).  Every addition is an error-free two-sum whose error joins the
// compensation.  On return lane l holds the total (s, c) of value index
// vbits(l) = bits 4, 3, ... of l read as the binary digits of the index (most significant
// first), for log2 V digits.
template <int V, int S>
__device__ __forceinline__ void halve_step(float* s, float* c, int lane) {
  const bool up = (lane & S) != 0;
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    const float ss = up ? s[i] : s[i + V / 2], sc = up ? c[i] : c[i + V / 2];
    const float ks = up ? s[i + V / 2] : s[i], kc = up ? c[i + V / 2] : c[i];
    const float os = __shfl_xor_sync(0xffffffffu, ss, S), oc = __shfl_xor_sync(0xffffffffu, sc, S);
    float t, e;
    two_sum(ks, os, t, e);
    s[i] = t;
    c[i] = kc + oc + e;
  }
}
template <int S>
__device__ __forceinline__ void fold_step(float& s, float& c) {
  const float os = __shfl_xor_sync(0xffffffffu, s, S), oc = __shfl_xor_sync(0xffffffffu, c, S);
  float t, e;
  two_sum(s, os, t, e);
  s = t;
  c = c + oc + e;
}
template <int NV>
struct Pow2Vals { static constexpr int value = NV <= 2 ? 2 : NV <= 4 ? 4 : NV <= 8 ? 8 : 16; };
// (s, c) of the value this lane ends with; *index receives that value's index.
template <int NV>
__device__ __forceinline__ void warp_halving_sums(const float* fv, const float* fc, int lane, float& s_out,
                                                  float& c_out, int& index) {
  constexpr int V = Pow2Vals<NV>::value;
  float s[V], c[V];
#pragma unroll
  for (int i = 0; i < V; ++i) { s[i] = i < NV ? fv[i] : 0.0f; c[i] = i < NV ? fc[i] : 0.0f; }
  halve_step<V, 16>(s, c, lane);
  if (V >= 4) halve_step<V / 2, 8>(s, c, lane);
  if (V >= 8) halve_step<V / 4, 4>(s, c, lane);
  if (V >= 16) halve_step<V / 8, 2>(s, c, lane);
  float rs = s[0], rc = c[0];
  if (V <= 8) fold_step<2>(rs, rc);
  if (V <= 4) fold_step<4>(rs, rc);
  if (V <= 2) fold_step<8>(rs, rc);
  fold_step<1>(rs, rc);
  int idx = 0;
  idx = (idx << 1) | ((lane >> 4) & 1);
  if (V >= 4) idx = (idx << 1) | ((lane >> 3) & 1);
  if (V >= 8) idx = (idx << 1) | ((lane >> 2) & 1);
  if (V >= 16) idx = (idx << 1) | ((lane >> 1) & 1);
  s_out = rs;
  c_out = rc;
  index = idx;
}

// The same halving in FP64 (plain additions): lane l ends with the total of value index
// vbits(l), as above.
template <int V, int S>
__device__ __forceinline__ void halve_step_f64(double* s, int lane) {
  const bool up = (lane & S) != 0;
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    const double send = up ? s[i] : s[i + V / 2], keep = up ? s[i + V / 2] : s[i];
    s[i] = keep + __shfl_xor_sync(0xffffffffu, send, S);
  }
}
template <int S>
__device__ __forceinline__ void fold_step_f64(double& s) {
  s = s + __shfl_xor_sync(0xffffffffu, s, S);
}
template <int NV>
__device__ __forceinline__ void warp_halving_f64(const double* dv, int lane, double& out, int& index) {
  constexpr int V = Pow2Vals<NV>::value;
  double s[V];
#pragma unroll
  for (int i = 0; i < V; ++i) s[i] = i < NV ? dv[i] : 0.0;
  halve_step_f64<V, 16>(s, lane);
  if (V >= 4) halve_step_f64<V / 2, 8>(s, lane);
  if (V >= 8) halve_step_f64<V / 4, 4>(s, lane);
  if (V >= 16) halve_step_f64<V / 8, 2>(s, lane);
  double r = s[0];
  if (V <= 8) fold_step_f64<2>(r);
  if (V <= 4) fold_step_f64<4>(r);
  if (V <= 2) fold_step_f64<8>(r);
  fold_step_f64<1>(r);
  int idx = (lane >> 4) & 1;
  if (V >= 4) idx = (idx << 1) | ((lane >> 3) & 1);
  if (V >= 8) idx = (idx << 1) | ((lane >> 2) & 1);
  if (V >= 16) idx = (idx << 1) | ((lane >> 1) & 1);
  out = r;
  index = idx;
}

// One proposal's sum has one order whichever threads evaluate it, so that its ln L does not
// depend on the round it was drawn in or on the kernel that evaluates it: chunk w (w = 0..3) is
// the bins 32 w + l + 128 m (m = 0, 1, ...) summed in order on lane l, the lanes' values are
// reduced by the halving tree (compensated in the mixed paths, then converted to FP64), and
// the four chunk totals are added in the order of w in FP64.  The whole CTA forms chunk w on
// warp w; a warp that evaluates a proposal alone forms the four chunks in turn.
//
// chunk_total: this warp's chunk total of every value into out[0 .. NV) (shared memory).
template <int PREC, int NV>
__device__ __forceinline__ void chunk_total(const double* dv, const float* fv, const float* fc, int lane,
                                            double* out) {
  constexpr int group = 32 / Pow2Vals<NV>::value;
  int q;
  if (PREC == 0) {
    double r;
    warp_halving_f64<NV>(dv, lane, r, q);
    if ((lane & (group - 1)) == 0 && q < NV) out[q] = r;
  } else {
    float rs, rc;
    warp_halving_sums<NV>(fv, fc, lane, rs, rc, q);
    if ((lane & (group - 1)) == 0 && q < NV) out[q] = (double)rs + (double)rc;
  }
}
// value q of the four chunk totals ct[w][q], added in chunk order
template <int NV>
__device__ __forceinline__ double chunks_sum(const double (*ct)[NV], int q) {
  double t = 0.0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) t = t + ct[w][q];
  return t;
}
// The four chunks of one proposal on one warp: totals into ct[0 .. kWarps)[0 .. NV).
template <int PREC, int NDET, int WF>
__device__ inline void warp_chunks(const EventDev& ev, const WalkerParams& P, int lane,
                                   double (*ct)[NVals<NDET, WF>::value]) {
  constexpr int NV = NVals<NDET, WF>::value;
#pragma unroll 1
  for (int w = 0; w < kWarps; ++w) {
    double dv[NV];
    float fv[NV], fc[NV];
    partials<PREC, NDET, WF>(ev, P, 32 * w + lane, kThreads, dv, fv, fc);
    chunk_total<PREC, NV>(dv, fv, fc, lane, ct[w]);
  }
  __syncwarp();
}

// Sums of one walker over the whole CTA: totals in `out` (shared), visible to every thread on
// return; `ct` holds the warps' chunk totals.
template <int PREC, int NDET, int WF>
__device__ inline void cta_sums(const EventDev& ev, const WalkerParams& P, double (*ct)[NVals<NDET, WF>::value],
                                double* out) {
  constexpr int NV = NVals<NDET, WF>::value;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double dv[NV];
  float fv[NV], fc[NV];
  partials<PREC, NDET, WF>(ev, P, threadIdx.x, kThreads, dv, fv, fc);
  chunk_total<PREC, NV>(dv, fv, fc, lane, ct[warp]);
  __syncthreads();
  if (threadIdx.x < NV) out[threadIdx.x] = chunks_sum<NV>(ct, threadIdx.x);
  __syncthreads();
}

// ln L from reduced values laid out [det][re, im(, hh)]; the mixed paths' template-power sums
// are in units of the scaled FP32 weights.
template <int PREC, int NDET, int WF>
__device__ inline double lnl_from_vals(const EventDev& ev, const WalkerParams& P, const double* v) {
  constexpr int NW = (WF == 1 ? 3 : 2);
  if (PREC == 2) {   // the float-float path's scaled FP32 amplitudes
    double dh = 0.0, hh = (double)P.hh_f;
#pragma unroll
    for (int d = 0; d < NDET; ++d) {
      dh += (double)P.kpf_re[d] * v[NW * d] - (double)P.kpf_im[d] * v[NW * d + 1];
      if (WF == 1)
        hh += ((double)P.kpf_re[d] * P.kpf_re[d] + (double)P.kpf_im[d] * P.kpf_im[d]) * v[NW * d + 2] *
              (double)ev.hh_unscale_f;
    }
    dh = ldexp(dh, -kKpScaleExp);
    return ev.use_ratio ? dh - 0.5 * hh : -0.5 * (ev.dd_total - 2.0 * dh + hh);
  }
  double sr[kMaxDet], si[kMaxDet], sh[kMaxDet];
  const double hscale = PREC == 0 ? 1.0 : ev.gw32_unscale;
#pragma unroll
  for (int d = 0; d < NDET; ++d) {
    sr[d] = v[NW * d];
    si[d] = v[NW * d + 1];
    sh[d] = (WF == 1) ? v[NW * d + 2] * hscale : 0.0;
  }
  return assemble_lnl(ev, P, sr, si, WF == 1 ? sh : nullptr);
}

// ln L of the float-float TaylorF2 path in float-float arithmetic from the compensated
// per-detector sums ps = [det][re, im] x (sum, compensation): FP64 only converts the result.
template <int NDET, int WF>
__device__ inline double lnl_ff(const EventDev& ev, const WalkerParams& P, const float* ps) {
  constexpr int NS = (WF == 1 ? 6 : 4);   // floats per detector: (re, im(, hh)) x (sum, compensation)
  ff dh = ff_make(0.0f);
  float hh = P.hh_f;
#pragma unroll
  for (int d = 0; d < NDET; ++d) {
    const ff sr = fast_two_sum_ff(ps[NS * d], ps[NS * d + 1]);
    const ff si = fast_two_sum_ff(ps[NS * d + 2], ps[NS * d + 3]);
    dh = ff_add(dh, ff_sub(ff_mul_f(sr, P.kpf_re[d]), ff_mul_f(si, P.kpf_im[d])));
    if (WF == 1)
      hh += (P.kpf_re[d] * P.kpf_re[d] + P.kpf_im[d] * P.kpf_im[d]) * ((ps[NS * d + 4] + ps[NS * d + 5]) * ev.hh_unscale_f);
  }
  dh = ff_ldexp(dh, -kKpScaleExp);
  ff l;
  if (ev.use_ratio) {
    l = ff_add_f(dh, -0.5f * hh);
  } else {
    l = ff_add_f(ff_sub(ff_ldexp(dh, 1), ff{ev.dd_f[0], ev.dd_f[1]}), -hh);
    l = ff_ldexp(l, -1);
  }
  return (double)l.h + (double)l.l;
}

// ---------------------------------------------------------------- relative binning
// The float-float TaylorF2 phase at grid bin k [cycles, reduced to [-1/2, 1/2] plus a small
// low part], as the first half of bin_accumulate_ff computes it.
__device__ __forceinline__ float tf2_ff_r0(const EventDev& ev, const WalkerParams& p, int k) {
  const float2* g = ev.basis_ff + k;
  const size_t gs = (size_t)ev.n_bins;
  float q[kBasis];
  float sl = p.ph0l;
#pragma unroll
  for (int j = 0; j < kBasis; ++j) {
    const float2 gj = g[j * gs];
    q[j] = p.Ch[j] * gj.x;
    float e = fmaf(p.Ch[j], gj.x, -q[j]);
    e = fmaf(p.Ch[j], gj.y, e);
    sl += fmaf(p.Cl[j], gj.x, e);
  }
#pragma unroll
  for (int w = 1; w < kBasis; w <<= 1) {
#pragma unroll
    for (int j = 0; j + w < kBasis; j += 2 * w) {
      const float t = q[j] + q[j + w];
      const float bb = t - q[j];
      sl += (q[j] - (t - bb)) + (q[j + w] - bb);
      q[j] = t;
    }
  }
  const float t = p.ph0h + q[0];
  const float bb = t - p.ph0h;
  sl += (p.ph0h - (t - bb)) + (q[0] - bb);
  return (t - rintf(t)) + sl;
}

// The float-float IMRPhenomD-form phase [cycles] and amplitude shape at grid bin k, as the first
// half of pd_segment_ff computes them.
__device__ __forceinline__ void pd_ff_r0_amp(const EventDev& ev, const WalkerParams& p, const PhenomExtra& e,
                                             int k, float& r0, float& amp) {
  const float2* g = ev.basis_ff + k;
  const size_t gs = (size_t)ev.n_bins;
  const float ff = g[13 * gs].x;
  float sh, sl, extra = 0.f;
  if (k < e.k1) {
    sh = p.ph0h; sl = p.ph0l;
#pragma unroll
    for (int j = 0; j < 8; ++j) ff_term(sh, sl, p.Ch[j], p.Cl[j], g[j * gs]);
    ff_term(sh, sl, e.Cxh[0], e.Cxl[0], g[8 * gs]);
    ff_term(sh, sl, e.Cxh[1], e.Cxl[1], g[9 * gs]);
    ff_term(sh, sl, e.Cxh[2], e.Cxl[2], g[10 * gs]);
  } else if (k < e.k2) {
    sh = e.ph0_int_h; sl = e.ph0_int_l;
    ff_term(sh, sl, e.Cxh[3], e.Cxl[3], g[6 * gs]);
    ff_term(sh, sl, e.Cxh[4], e.Cxl[4], g[11 * gs]);
    ff_term(sh, sl, e.Cxh[5], e.Cxl[5], g[13 * gs]);
  } else {
    sh = e.ph0_mr_h; sl = e.ph0_mr_l;
    ff_term(sh, sl, e.Cxh[6], e.Cxl[6], g[1 * gs]);
    ff_term(sh, sl, e.Cxh[7], e.Cxl[7], g[12 * gs]);
    ff_term(sh, sl, e.Cxh[8], e.Cxl[8], g[13 * gs]);
    extra = e.at_scalef * atanf((e.Mf * ff - e.at_cf) * e.at_invf);
  }
  r0 = (sh - rintf(sh)) + sl + extra;
  amp = pd_amp_f32(e, k, ff, g[4 * gs].x);
}

// ln L of one proposal with the relative-binning likelihood (mode 2), evaluated by one warp
// (every lane returns it).  Coarse bins wholly below the proposal's cutoff whose right edge is
// a grid bin take the linear expansion of r = h / h0 between their edges (31 bins a pass; lane
// l holds edge base + l and reads its right neighbour by a shuffle); from the first other coarse
// bin up to the cutoff the active bins are summed exactly with the per-bin bodies.  *bins
// receives the grid bins the evaluation touched (edges plus the exact range).
template <int NDET, int WF>
__device__ double rb_lnl_warp(const EventDev& ev, const WalkerParams& P, int lane, int* bins = nullptr) {
  const int nb = ev.rb_nb;
  const int32_t* E = ev.rb_edges;
  const int k_end = P.k_end;
  const int kmax = min(k_end, ev.n_bins - 1);
  int lo = 0, hi = nb;   // n_full = the largest n with E[n] <= kmax (E[0] = 0)
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (E[mid] <= kmax) lo = mid;
    else hi = mid - 1;
  }
  const int n_full = lo;
  float dh = 0.f, dhc = 0.f, hh = 0.f, hhc = 0.f;
  const float df = ev.df_f[0];
  for (int base = 0; base < n_full; base += 31) {
    const int ei = base + lane;
    const bool have = ei <= n_full;
    float rre[NDET], rim[NDET];
#pragma unroll
    for (int det = 0; det < NDET; ++det) { rre[det] = 0.f; rim[det] = 0.f; }
    if (have) {
      const int k = E[ei];
      float r0, amp = 1.0f;
      if (WF == 0) r0 = tf2_ff_r0(ev, P, k);
      else pd_ff_r0_amp(ev, P, P.pd, k, r0, amp);
      const float kf = (float)k;
#pragma unroll
      for (int det = 0; det < NDET; ++det) {
        const float kb = kf * P.sbh[det];
        float ph = (r0 + P.sa[det]) + (kb - rintf(kb)) + kf * P.sbl[det];
        ph = ph - rintf(ph);
        float sn, cs;
        sincos_turn_sfu(ph, &sn, &cs);
        // h f^(7/6) 2^70 = amp (K P) exp(-2 pi i ph)
        const float hre = amp * (P.kpf_re[det] * cs + P.kpf_im[det] * sn);
        const float him = amp * (P.kpf_im[det] * cs - P.kpf_re[det] * sn);
        const float2 q = ev.rb_q0[(size_t)det * nb + ei];
        rre[det] = hre * q.x - him * q.y;
        rim[det] = hre * q.y + him * q.x;
      }
    }
    const int b = base + lane;
    const bool bin = lane < 31 && b < n_full;
    const float inv = bin ? 1.0f / ((float)(E[b + 1] - E[b]) * df) : 0.f;
#pragma unroll
    for (int det = 0; det < NDET; ++det) {
      const float nre = __shfl_down_sync(0xffffffffu, rre[det], 1);
      const float nim = __shfl_down_sync(0xffffffffu, rim[det], 1);
      if (bin) {
        const float r1re = (nre - rre[det]) * inv, r1im = (nim - rim[det]) * inv;
        const float2 a0 = ev.rb_a[((size_t)det * nb + b) * 2];
        const float2 a1 = ev.rb_a[((size_t)det * nb + b) * 2 + 1];
        const float4 bq = ev.rb_b[(size_t)det * nb + b];
        kahan_add(dh, dhc, a0.x * rre[det] - a0.y * rim[det] + a1.x * r1re - a1.y * r1im);
        kahan_add(hh, hhc, bq.x * (rre[det] * rre[det] + rim[det] * rim[det]) +
                               2.0f * bq.y * (rre[det] * r1re + rim[det] * r1im) +
                               bq.z * (r1re * r1re + r1im * r1im));
      }
    }
  }
  // exact part: the active bins from the first coarse bin not expanded
  const int kx = E[n_full];
  if (bins) *bins = n_full + 1 + max(k_end - kx, 0);
  double xdh = 0.0, xhh = 0.0;
  if (WF == 0) {
    AccF32 acc;
    acc.zero();
    for (int k = kx + lane; k < k_end; k += 32) bin_accumulate_ff<NDET>(ev, P, k, acc);
    float sdh = 0.f;
#pragma unroll
    for (int det = 0; det < NDET; ++det)
      sdh += P.kpf_re[det] * (acc.re[det] - acc.cre[det]) - P.kpf_im[det] * (acc.im[det] - acc.cim[det]);
    xdh = ldexp((double)sdh, -kKpScaleExp);
    if (lane == 0 && kx < k_end) {
      float hsum = 0.f;
      for (int det = 0; det < NDET; ++det) {
        const float* pre = ev.hhp32 + (size_t)det * ev.n_bins;
        const float seg = pre[k_end - 1] - (kx > 0 ? pre[kx - 1] : 0.f);
        hsum += (P.kpf_re[det] * P.kpf_re[det] + P.kpf_im[det] * P.kpf_im[det]) * seg;
      }
      xhh = (double)hsum;
    }
  } else {
    AccPD32 acc;
    acc.zero();
    pd_sums_ff<NDET>(ev, P, P.pd, kx + lane, k_end, 32, acc);
    float sdh = 0.f, shh = 0.f;
#pragma unroll
    for (int det = 0; det < NDET; ++det) {
      sdh += P.kpf_re[det] * (acc.re[det] - acc.cre[det]) - P.kpf_im[det] * (acc.im[det] - acc.cim[det]);
      shh += (P.kpf_re[det] * P.kpf_re[det] + P.kpf_im[det] * P.kpf_im[det]) * acc.hh[det];
    }
    xdh = ldexp((double)sdh, -kKpScaleExp);
    xhh = (double)shh * (double)ev.hh_unscale_f;
  }
  double tdh = (double)dh - (double)dhc + xdh;
  double thh = (double)hh - (double)hhc + xhh;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    tdh += __shfl_xor_sync(0xffffffffu, tdh, off);
    thh += __shfl_xor_sync(0xffffffffu, thh, off);
  }
  return ev.use_ratio ? tdh - 0.5 * thh : -0.5 * (ev.dd_total - 2.0 * tdh + thh);
}

__device__ inline bool theta_ok(const double* th) {
  for (int i = 0; i < kParams; ++i) if (!isfinite(th[i])) return false;
  return th[0] > 0.0 && th[1] > 0.0 && th[4] > 0.0;
}

// Per-walker constants of one proposal, on one thread: the FP64 path uses the plain FP64 setup, the
// mixed paths the lean one (FP64 only where the phase needs it; in mode 2 for priors that the
// float-float setup of ff_setup.cuh does not transform).
template <int PREC, int WF>
__device__ inline void setup_from_unit(const EventDev& ev, const double* u, WalkerParams& P) {
  if (PREC == 0) {
    double th[kParams], ci, sd, cd;
    unit_to_theta(ev, u, th, &ci, &sd, &cd);
    taylorf2_setup<WF>(ev, th, ci, sd, cd, P);
  } else {
    LeanTheta t;
    unit_to_lean(ev, u, t);
    taylorf2_setup_lean<WF>(ev, t, P);
    if (PREC == 2) make_ff<WF>(ev, P);
  }
}

// ---------------------------------------------------------------- likelihood batch
// ln L of n proposals, in [n][11] physical vectors or (UNIT) [n][D] unit-cube points: one CTA takes a
// tile of `tile` of them.  The four warps form the tile's constants together (setup_tile: a
// proposal a lane), then the likelihoods run in the walks' summation order.  With one proposal a
// CTA, one thread formed its constants while the other 127 waited (barrier stalls 33 of every 48
// warp cycles, the FP64 pipe busy with one lane in 32).  Non-finite vectors: NaN and status; UNIT
// (the initial live points): non-finite results become -inf, so that they die first.
constexpr int kLikTile = 16;

template <int PREC, int NDET, int WF, bool UNIT>
__global__ void __launch_bounds__(kThreads, 4) likelihood_kernel(const EventDev* __restrict__ evp,
                                                                 const double* __restrict__ in, int n, int tile,
                                                                 double* __restrict__ lnl, int32_t* status) {
  constexpr int NV = NVals<NDET, WF>::value;
  __shared__ WalkerParams P[kLikTile];
  __shared__ TilePart<PREC, WF> parts[kLikTile];
  __shared__ double ct[kWarps][kWarps][NV];
  __shared__ double tot[kLikTile][NV];
  __shared__ double rbl[kLikTile];
  __shared__ int ok[kLikTile];
  const EventDev& ev = *evp;
  const int base = blockIdx.x * tile, m = min(tile, n - base);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double* v = in + (size_t)base * (UNIT ? ev.n_dim : kParams);
  if ((int)threadIdx.x < m) ok[threadIdx.x] = UNIT ? 1 : (theta_ok(v + (size_t)threadIdx.x * kParams) ? 1 : 0);
  __syncthreads();
  setup_tile<PREC, WF, UNIT>(ev, v, m, ok, parts, P);
  bool rb = false;
  if constexpr (PREC == 2) rb = ev.rb_nb > 0;
  if (rb) {
    if constexpr (PREC == 2) {   // relative binning: a warp per proposal
      for (int i = warp; i < m; i += kWarps) {
        const double l = ok[i] ? rb_lnl_warp<NDET, WF>(ev, P[i], lane) : 0.0;
        if (lane == 0) rbl[i] = l;
      }
    }
  } else if (WF == 0 && m >= kWarps) {
    // hundreds of bins: a warp per proposal, its four chunks in turn, no barrier between proposals
    for (int i = warp; i < m; i += kWarps) {
      warp_chunks<PREC, NDET, WF>(ev, P[i], lane, ct[warp]);
      if (lane < NV) tot[i][lane] = chunks_sum<NV>(ct[warp], lane);
      __syncwarp();
    }
  } else {
    for (int i = 0; i < m; ++i) cta_sums<PREC, NDET, WF>(ev, P[i], ct[0], tot[i]);
  }
  __syncthreads();
  if ((int)threadIdx.x < m) {
    const int i = threadIdx.x;
    double l = rb ? rbl[i] : lnl_from_vals<PREC, NDET, WF>(ev, P[i], tot[i]);
    if (UNIT) {
      l = isfinite(l) ? l : -INFINITY;
    } else if (!ok[i]) {
      l = __longlong_as_double(0x7ff8000000000000ll);
      atomicOr(status, 1);
    }
    lnl[base + i] = l;
  }
}

// Physical theta [n][11] of unit-cube points u [n][D].
__global__ void unit_to_theta_kernel(const EventDev* __restrict__ evp, const double* __restrict__ u, int64_t n,
                                     double* __restrict__ theta) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const EventDev& ev = *evp;
  double th[kParams], ci, sd, cd;
  unit_to_theta(ev, u + i * ev.n_dim, th, &ci, &sd, &cd);
  for (int k = 0; k < kParams; ++k) theta[i * kParams + k] = th[k];
}

// ---------------------------------------------------------------- waveform (FP64)
// Detector strains of theta blockIdx.y in the bins [span blockIdx.x, span (blockIdx.x + 1)).  The
// CTA forms the constants on its four warps, once for the whole span (a CTA per 256 bins formed
// them on one thread, 64 times a vector at 16,225 bins).
template <int NDET, int WF>
__global__ void __launch_bounds__(kThreads) waveform_kernel(const EventDev* __restrict__ evp,
                                                            const double* __restrict__ theta, int n_bins, int span,
                                                            double* __restrict__ h_re, double* __restrict__ h_im,
                                                            int no_cutoff) {
  __shared__ WalkerParams P;
  __shared__ TilePart<0, WF> part;
  __shared__ int ok;
  const EventDev& ev = *evp;
  const int w = blockIdx.y;
  if (threadIdx.x == 0) ok = 1;
  __syncthreads();
  setup_tile<0, WF, false>(ev, theta + (size_t)w * kParams, 1, &ok, &part, &P);
  const int k_end = no_cutoff ? n_bins : P.k_end;
  const int last = min((int)(blockIdx.x + 1) * span, n_bins);
  for (int k = blockIdx.x * span + threadIdx.x; k < last; k += kThreads) {
    const size_t o0 = (size_t)w * NDET * n_bins + k;
    if (k >= k_end) {
#pragma unroll
      for (int det = 0; det < NDET; ++det) h_re[o0 + (size_t)det * n_bins] = h_im[o0 + (size_t)det * n_bins] = 0.0;
      continue;
    }
    const double f = ev.f_min + ev.df * (double)k;
    const double* g = ev.basis64 + (size_t)k * ev.n_basis;
    double phi, amp;
    if (WF == 0) {
      phi = P.phase0;
#pragma unroll
      for (int j = 0; j < kBasis; ++j) phi = fma(P.C[j], g[j], phi);
      amp = 1.0;
    } else {
      const PhenomExtra& e = P.pd;
      if (k < e.k1) {
        phi = P.phase0;
#pragma unroll
        for (int j = 0; j < kBasis; ++j) phi = fma(P.C[j], g[j], phi);
        phi = fma(e.Cx[0], g[8], fma(e.Cx[1], g[9], fma(e.Cx[2], g[10], phi)));
      } else if (k < e.k2) {
        phi = fma(e.Cx[3], g[6], fma(e.Cx[4], g[11], fma(e.Cx[5], g[13], e.ph0_int)));
      } else {
        phi = fma(e.Cx[6], g[1], fma(e.Cx[7], g[12], fma(e.Cx[8], g[13], e.ph0_mr)));
        phi += e.at_scale * atan((e.M * f - e.at_c) * e.at_inv);
      }
      amp = pd_amp_f64(e, k, f, g[4]);
    }
    const double a7 = ev.a76[k] * amp;
#pragma unroll
    for (int det = 0; det < NDET; ++det) {
      double s, c;
      sincos_phase_f64(fma(P.tau[det], f, phi), &s, &c);
      // a f^-7/6 K P exp(-2 pi i ph)
      h_re[o0 + (size_t)det * n_bins] = a7 * (P.kp_re[det] * c + P.kp_im[det] * s);
      h_im[o0 + (size_t)det * n_bins] = a7 * (P.kp_im[det] * c - P.kp_re[det] * s);
    }
  }
}

// A walker's next round, from its own n_acc acceptances in n_like calls so far: `depth` proposals,
// looking ahead over rejections or (`chain`) over acceptances.
//   A DE move's difference does not depend on the position, so the proposals of later steps follow
// from any guess at the earlier outcomes, and the round holds the likeliest guess:
//   - p below 1/2 acceptances a call: every step from the current position, as if each were
//     rejected; the replay stops at the first acceptance;
//   - p above 1/2: each in-bounds step from the one before it, as if each were accepted; the replay
//     stops at the first rejection.
// The depth is that of the batch retune, about 1.4 expected runs of the guess: 1.4 / p or
// 1.4 / (1 - p), with the task's depth as the first estimate, worth 1.4 outcomes of the other kind.
// A stand-alone walk has no batch before it: a fixed depth of 16 dropped 9 of 10 evaluations at
// p = 0.6.  spec_cap 0 keeps the task's depth, over rejections: a depth fixed by the user, and the
// sampler's walks, whose batch rule knows p (their own estimates, noisier, gained nothing).  Any
// choice gives the same chain.  Asking acceptances to lead by one call before a round looks ahead
// over them spares a walker whose first call was accepted by luck: 4 to 13 % of a 60- or 200-step
// walk at p below 0.2, but it costs 4 to 17 % above 0.75, and against the fixed depth walks of low p
// lose 2 % at most without it (means of four walks each).  pad4: rounds of a warp per proposal,
// padded to a multiple of four.  CH: compiled with the look-ahead over acceptances.
struct Round {
  int depth;
  bool chain;
};
template <bool CH>
__device__ __forceinline__ Round next_round(const WalkTask& T, bool pad4, int n_acc, int n_like) {
  Round r;
  r.depth = T.spec < 1 ? 1 : (T.spec > kSpecMax ? kSpecMax : T.spec);
  r.chain = CH && T.spec_cap > 0 && 2 * n_acc > n_like;
  if (T.spec_cap > 0) {
    const int ends = r.chain ? n_like - n_acc : n_acc;
    r.depth = (int)(1.4f * ((float)n_like + (float)r.depth) / ((float)ends + 1.4f) + 0.5f);
    r.depth = min(max(r.depth, 1), min(T.spec_cap, kSpecMax));
  }
  if (pad4) r.depth = min((r.depth + 3) & ~3, kSpecMax);
  return r;
}

// ---------------------------------------------------------------- acceptance walk
// Modes 0 and 1 (FP64 phase); mode 2 runs walk_kernel_ff below.
// One CTA per walker, persistent over the walk.  A round looks ahead over the next W steps:
//  1. the DE draws of a step depend only on its Philox counter (step, walker, iteration,
//     tag), not on the chain, so every thread screens one candidate step in FP32 from the
//     current position; the candidates that may lie in the cube are compacted into one warp,
//     which redoes their draws and proposals exactly in FP64 and compacts the in-bounds ones,
//     in step order, into at most m slots, m the round's depth (next_round).  A round that looks
//     ahead over acceptances instead chains its moves exactly, each in-bounds one from the last;
//  2. the four warps form the per-proposal constants together (independent chains on different
//     warps, a proposal a lane), and the CTA evaluates the slots' likelihoods, one warp per
//     proposal (the whole CTA per proposal when there are fewer than kWarps of them);
//  3. thread 0 replays the steps in order: out-of-bounds steps reject without a likelihood
//     call, an in-bounds proposal with ln L > ln L* is taken, and the round ends where its guess
//     first fails: at its first acceptance, or, looking ahead over acceptances, its first rejection.
//     Candidates after it were built from a position the chain does not take and are redrawn
//     from the right one in the next round.
// The chain, the accepted and likelihood-call counts and every ln L are those of the walk
// that takes one step at a time.  The setup warp rotates over the CTAs of an SM (an arrival
// counter), so their FP64 work lands on different sub-partitions.
// CL: a cluster of CTAs per walker (launch_walk_f64).  CH: the look-ahead over acceptances.
// Flow steps (task.flow set): a step whose Philox tag-6 draw falls below p_flow proposes the
// precomputed flow sample of the proposal table instead of a DE move, and passes the screen
// iff ln U < ln q(u) - ln q(u') (an independence Metropolis-Hastings test taken before the
// likelihood); ln q of the current point is carried along and re-evaluated on CUDA cores
// after an accepted DE move.
template <int PREC, int NDET, int WF, bool CH, bool CL>
__global__ void __launch_bounds__(kThreads, 4) walk_kernel(const EventDev* __restrict__ evs, WalkTask* tasks,
                                                         const int32_t* __restrict__ blk_task,
                                                         const int32_t* __restrict__ blk_local) {
  constexpr int NV = NVals<NDET, WF>::value;
  __shared__ WalkerParams P[kSpecMax];
  __shared__ union { SetupPart parts[kSpecMax]; double diff[32][kMaxDim]; } sh;
  SetupPart* const parts = sh.parts;
  double (*const diff)[kMaxDim] = sh.diff;
  __shared__ double prop[kSpecMax][kMaxDim];
  __shared__ int cstep[kSpecMax];
  __shared__ int mstep[32];
  __shared__ double lnl_p[kSpecMax];
  __shared__ double tot_p[CL ? 2 : 1][kSpecMax][NV];   // by parity of the round: a rank ahead never overwrites
  __shared__ double ct[kWarps][kWarps][NV];
  __shared__ double u[kMaxDim];
  __shared__ float u32[kMaxDim];
  __shared__ int wcount[kWarps];
  __shared__ int s_next, s_setup_warp, s_nin, s_end, s_needq;
  __shared__ int s_stop[2];
  __shared__ Round s_round;
  __shared__ int s_isflow[kSpecMax];
  __shared__ float s_lqf[kSpecMax];
  __shared__ float s_logq;
  __shared__ FlowScratch fscr;
  // a walker's CTAs (a cluster; one CTA in large launches): every rank runs the same chain
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  const int ranks = CL ? (int)cluster.num_blocks() : 1, rank = CL ? (int)cluster.block_rank() : 0;
  const WalkTask& T = tasks[blk_task[blockIdx.x / ranks]];
  const int j = blk_local[blockIdx.x / ranks];
  const EventDev& ev = evs[T.event];
  if (T.done) return;
  const int D = ev.n_dim;
  const int n_steps = T.n_steps;
  const double lnl_star = T.lnl_star;
  const uint64_t it = (uint64_t)T.iteration;
  const uint64_t wid = (uint64_t)(T.walker_offset + j);
  const uint64_t n_s = (uint64_t)T.n_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < D) {
    u[threadIdx.x] = T.u0[(size_t)j * D + threadIdx.x];
    u32[threadIdx.x] = (float)u[threadIdx.x];
  }
  if (threadIdx.x == 0) {
    unsigned int smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    s_setup_warp = (int)(atomicAdd(&g_walk_sm_arrivals[smid & 255u], 1u) % (unsigned)kWarps);
  }
  double lnl = T.lnl0[j];
  int n_acc = 0, n_acc_flow = 0, n_like = 0;
  int64_t n_bins = 0, n_spec = 0;
  const uint64_t t0 = threadIdx.x == 0 ? global_ns() : 0ull;
  const double de_scale = 2.38 / sqrt(2.0 * (double)D);
  const float de_scale32 = (float)de_scale;
  // a rank stores into the other ranks' shared memory in its first round: not before they run
  if (CL) cluster.sync();
  else __syncthreads();
  const int sw = s_setup_warp;
  const bool use_flow = !CH && T.flow != nullptr && T.p_flow > 0.0;
  const double p_flow = T.p_flow;
  Round rd = next_round<CH>(T, false, 0, 0);
  if (use_flow) {
    const float lq = flow_logq_cta(*T.flow, u, fscr);
    if (threadIdx.x == 0) s_logq = lq;
    __syncthreads();
  }
  int t = 0, par = 0;
  while (t < n_steps) {
    const int abort_flag = threadIdx.x == 0 ? walk_abort_flag(T) : 0;
    const int m = rd.depth;
    if (CH && rd.chain) {
      // 1. the setup warp forms the differences of the next 32 steps (a step a lane), then chains
      //    the in-bounds moves (a coordinate a lane)
      if (warp == sw) {
        const int W = min(32, n_steps - t);
        if (lane < W) {
          const int st = t + lane;
          Philox4 A = philox4x64((uint64_t)st, wid, it, 0ull, T.key0, T.key1);
          const uint64_t a = rand_index(A.v[0], n_s);
          uint64_t b = rand_index(A.v[1], n_s - 1);
          b += (b >= a) ? 1ull : 0ull;
          double sc = 1.0;
          if ((A.v[2] >> 63) == 0ull) {
            Philox4 B = philox4x64((uint64_t)st, wid, it, 1ull, T.key0, T.key1);
            const double prod = __dmul_rn(__dmul_rn(__dmul_rn(rand_open_unit(B.v[0]), rand_open_unit(B.v[1])),
                                                    rand_open_unit(B.v[2])), rand_open_unit(B.v[3]));
            sc = __dmul_rn(de_scale, __dmul_rn(-0.25, log(prod)));
          }
          const double* ua = T.surv + a * D;
          const double* ub = T.surv + b * D;
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d)
            if (d < D) diff[lane][d] = __dmul_rn(sc, __dsub_rn(ua[d], ub[d]));
        }
        __syncwarp();
        const bool wrap = lane < D && ev.prior[ev.dim_param[lane]].periodic;
        double x = lane < D ? u[lane] : 0.0;
        int cnt = 0;
        for (int q = 0; q < W && cnt < m; ++q) {
          double y = 0.0;
          if (lane < D) {
            y = __dadd_rn(x, diff[q][lane]);
            if (wrap) y = __dsub_rn(y, floor(y));
          }
          if (__all_sync(0xffffffffu, (unsigned long long)__double_as_longlong(y) <= 0x3FF0000000000000ull)) {
            x = y;
            if (lane < D) prop[cnt][lane] = y;
            if (lane == 0) cstep[cnt] = t + q;
            ++cnt;
          }
        }
        __syncwarp();
        if (lane == 0) {
          s_nin = cnt;
          s_end = cnt == m ? cstep[m - 1] : t + W - 1;
        }
      }
    } else {
      const int W = min(min(kThreads, max(32, 4 * m)), n_steps - t);
      // 1a. every thread screens one candidate step in FP32
      int maybe = 0;
      const int step = t + (int)threadIdx.x;
      bool fl = false;
      if (use_flow && (int)threadIdx.x < W) {
        Philox4 C = philox4x64((uint64_t)step, wid, it, 6ull, T.key0, T.key1);
        if (rand_open_unit(C.v[0]) < p_flow) {
          fl = true;
          const float lqf = (float)T.flq[(size_t)j * T.f_stride + step];
          maybe = logf((float)rand_open_unit(C.v[1])) < s_logq - lqf;
        }
      }
      if ((int)threadIdx.x < W && !fl) {
        Philox4 A = philox4x64((uint64_t)step, wid, it, 0ull, T.key0, T.key1);
        uint64_t a = rand_index(A.v[0], n_s);
        uint64_t b = rand_index(A.v[1], n_s - 1);
        b += (b >= a) ? 1ull : 0ull;
        float sc = 1.0f;
        if ((A.v[2] >> 63) == 0ull) {
          Philox4 B = philox4x64((uint64_t)step, wid, it, 1ull, T.key0, T.key1);
          sc = screen_scale(B.v, de_scale32, FastLog2{});
        }
        const float margin = screen_margin(sc);
        maybe = 1;
        if (T.survf) {
          const float2* ua = T.survf + a * D;
          const float2* ub = T.survf + b * D;
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d) {
            if (d < D && !ev.prior[ev.dim_param[d]].periodic) {
              float x = u32[d] + sc * (ua[d].x - ub[d].x);
              if (!(x >= -margin && x <= 1.0f + margin)) maybe = 0;
            }
          }
        } else {
          const double* ua = T.surv + a * D;
          const double* ub = T.surv + b * D;
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d) {
            if (d < D && !ev.prior[ev.dim_param[d]].periodic) {
              float x = u32[d] + sc * ((float)ua[d] - (float)ub[d]);
              if (!(x >= -margin && x <= 1.0f + margin)) maybe = 0;
            }
          }
        }
      }
      unsigned mask = __ballot_sync(0xffffffffu, maybe);
      if (lane == 0) wcount[warp] = __popc(mask);
      __syncthreads();
      int before = 0, total = 0;
#pragma unroll
      for (int w2 = 0; w2 < kWarps; ++w2) {
        int cw = wcount[w2];
        before += (w2 < warp) ? cw : 0;
        total += cw;
      }
      const int mslot = before + __popc(mask & ((1u << lane) - 1u));
      if (maybe && mslot < 32) mstep[mslot] = step;
      const int nmaybe = min(total, 32);
      __syncthreads();
      // 1b. the setup warp redoes the maybe-in-bounds steps exactly (FP64, as the walk is
      //     defined) and compacts the in-bounds ones into at most m slots
      if (warp == sw) {
        int in = 0, isf = 0;
        float lqf = 0.0f;
        double pr[kMaxDim];
        const int st = lane < nmaybe ? mstep[lane] : 0;
        if (use_flow && lane < nmaybe) {
          Philox4 C = philox4x64((uint64_t)st, wid, it, 6ull, T.key0, T.key1);
          if (rand_open_unit(C.v[0]) < p_flow) {
            isf = 1;
            lqf = (float)T.flq[(size_t)j * T.f_stride + st];
            in = logf((float)rand_open_unit(C.v[1])) < s_logq - lqf;
            const double* fu = T.fu + ((size_t)j * T.f_stride + st) * D;
#pragma unroll
            for (int d = 0; d < kMaxDim; ++d)
              if (d < D) pr[d] = fu[d];
          }
        }
        if (lane < nmaybe && !isf) {
          Philox4 A = philox4x64((uint64_t)st, wid, it, 0ull, T.key0, T.key1);
          uint64_t a = rand_index(A.v[0], n_s);
          uint64_t b = rand_index(A.v[1], n_s - 1);
          b += (b >= a) ? 1ull : 0ull;
          double sc;
          if ((A.v[2] >> 63) == 1ull) {
            sc = 1.0;
          } else {
            Philox4 B = philox4x64((uint64_t)st, wid, it, 1ull, T.key0, T.key1);
            double prod = __dmul_rn(__dmul_rn(__dmul_rn(rand_open_unit(B.v[0]), rand_open_unit(B.v[1])),
                                              rand_open_unit(B.v[2])), rand_open_unit(B.v[3]));
            sc = __dmul_rn(de_scale, __dmul_rn(-0.25, log(prod)));
          }
          const double* ua = T.surv + a * D;
          const double* ub = T.surv + b * D;
          in = 1;
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d) {
            if (d < D) {
              double x = __dadd_rn(u[d], __dmul_rn(sc, __dsub_rn(ua[d], ub[d])));
              if (ev.prior[ev.dim_param[d]].periodic) x = __dsub_rn(x, floor(x));
              // 0 <= x <= 1 on the bit pattern (integer pipe): +0 .. 1.0 are the patterns up
              // to 0x3FF0000000000000; negative values and NaN compare above.  x is never -0.
              if ((unsigned long long)__double_as_longlong(x) > 0x3FF0000000000000ull) in = 0;
              pr[d] = x;
            }
          }
        }
        const unsigned im = __ballot_sync(0xffffffffu, in);
        const int slot = __popc(im & ((1u << lane) - 1u));
        if (in && slot < m) {
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d)
            if (d < D) prop[slot][d] = pr[d];
          cstep[slot] = st;
          s_isflow[slot] = isf;
          s_lqf[slot] = lqf;
        }
        const int nin_w = min(__popc(im), m);
        // steps covered by this round: up to the m-th in-bounds proposal, else up to the last
        // screened maybe-step, else the whole window
        const unsigned mth = __ballot_sync(0xffffffffu, in && slot == m - 1);
        int end;
        if (__popc(im) > m) end = __shfl_sync(0xffffffffu, st, __ffs(mth) - 1);
        else if (total > 32) end = __shfl_sync(0xffffffffu, st, 31);
        else end = t + W - 1;
        if (lane == 0) { s_nin = nin_w; s_end = end; }
      }
    }
    __syncthreads();
    const int nin = s_nin;
    // 2. proposal constants on all four warps (setup_split.cuh), then the likelihoods: the sums of
    //    proposal i into tot_p[i] (chunk totals in ct), then one lane per proposal assembles ln L (the
    //    FP64 part runs once per proposal, on one warp)
    if (nin > 0) {
      if (lane < nin) f64_split_first<PREC != 0, true>(warp, ev, prop[lane], parts[lane], P[lane]);
      __syncthreads();
      if (lane < nin) f64_split_second<PREC != 0, WF>(warp, ev, parts[lane], P[lane]);
      __syncthreads();
    }
    // proposals rank, rank + ranks, ... of the round; their totals go to every rank
    const int mine = (nin - rank + ranks - 1) / ranks;
    auto store_total = [&](int i, int q, double v) {
      if (!CL) tot_p[par][i][q] = v;
      else
        for (int r = 0; r < ranks; ++r) *cluster.map_shared_rank(&tot_p[par][i][q], r) = v;
    };
    if (mine >= kWarps) {
      // one warp per proposal, its four chunks in turn
      for (int i = rank + ranks * warp; i < nin; i += ranks * kWarps) {
        warp_chunks<PREC, NDET, WF>(ev, P[i], lane, ct[warp]);
        if (lane < NV) store_total(i, lane, chunks_sum<NV>(ct[warp], lane));
        __syncwarp();
      }
    } else {
      // fewer proposals than warps: the whole CTA on each in turn, chunk w on warp w
      for (int i = rank; i < nin; i += ranks) {
        double dv[NV];
        float fv[NV], fc[NV];
        partials<PREC, NDET, WF>(ev, P[i], threadIdx.x, kThreads, dv, fv, fc);
        chunk_total<PREC, NV>(dv, fv, fc, lane, ct[0][warp]);
        __syncthreads();
        if (threadIdx.x < NV) store_total(i, threadIdx.x, chunks_sum<NV>(ct[0], threadIdx.x));
        __syncthreads();
      }
    }
    if (CL) {
      // rank 0 decides on the watchdog for all (each CTA has its own clock and view of the flag)
      if (rank == 0 && threadIdx.x == 0) {
        const int stop = walk_should_stop(T, t0, abort_flag) ? 1 : 0;
        for (int r = 0; r < ranks; ++r) *cluster.map_shared_rank(&s_stop[par], r) = stop;
      }
      cluster.sync();
    } else {
      __syncthreads();
    }
    if (warp == sw && lane < nin) lnl_p[lane] = lnl_from_vals<PREC, NDET, WF>(ev, P[lane], tot_p[par][lane]);
    __syncthreads();
    // 3. the steps in order
    if (threadIdx.x == 0) {
      int nxt = s_end + 1;
      s_needq = 0;
      int take = -1;   // the last accepted proposal
      for (int i = 0; i < nin; ++i) {
        ++n_like;
        n_bins += P[i].k_end;
        const bool up = lnl_p[i] > lnl_star;
        if (up) {
          take = i;
          ++n_acc;
        }
        if (up != (CH && rd.chain)) {   // the guess ends here
          nxt = cstep[i] + 1;
          break;
        }
      }
      if (take >= 0) {
        for (int d = 0; d < D; ++d) { u[d] = prop[take][d]; u32[d] = (float)prop[take][d]; }
        lnl = lnl_p[take];
        if (use_flow) {
          if (s_isflow[take]) {
            s_logq = s_lqf[take];
            ++n_acc_flow;
          } else {
            s_needq = 1;
          }
        }
      }
      n_spec += nin;
      if (CL ? s_stop[par] != 0 : walk_should_stop(T, t0, abort_flag)) {   // watchdog: end the walk after this round
        nxt = n_steps;
        if (T.status && rank == 0) atomicOr(T.status, 1);
      }
      s_next = nxt;
      s_round = next_round<CH>(T, false, n_acc, n_like);
    }
    __syncthreads();
    t = s_next;
    rd = s_round;
    if (CL) par ^= 1;
    if (use_flow && s_needq && t < n_steps) {
      const float lq = flow_logq_cta(*T.flow, u, fscr);
      if (threadIdx.x == 0) s_logq = lq;
      __syncthreads();
    }
  }
  if (rank != 0) return;
  if (threadIdx.x < D) T.u_out[(size_t)j * D + threadIdx.x] = u[threadIdx.x];
  if (threadIdx.x == 0) {
    T.lnl_out[j] = lnl;
    T.n_acc[j] = n_acc;
    if (T.n_acc_flow) T.n_acc_flow[j] = n_acc_flow;
    T.n_like[j] = n_like;
    if (T.n_bins) T.n_bins[j] = n_bins;
    if (T.n_spec) T.n_spec[j] = n_spec;
  }
}

// ---------------------------------------------------------------- float-float walk (mode 2)
__device__ __forceinline__ bool ff_in_unit(ff x) {
  // x normalised (|l| <= ulp(h) / 2, so h = 0 implies l = 0); NaN fails the first test
  return x.h >= 0.0f && (x.h < 1.0f || (x.h == 1.0f && x.l <= 0.0f));
}
// x - floor(x) of a float-float value (the periodic dimensions).
__device__ __forceinline__ ff ff_wrap_unit(ff x) {
  float fl = floorf(x.h);
  if (x.h == fl && x.l < 0.0f) fl -= 1.0f;
  return ff_add_f(x, -fl);
}

// The acceptance walk of mode 2.  The round of walk_kernel, restructured so that its serial
// part is short:
//  1. every thread draws one candidate step of the window and screens its move in FP32; the steps
//     that may stay in the cube (at most 32) are moved exactly, in float-float arithmetic (the DE
//     scale's logarithm, the survivors' float-float difference, the periodic wrap, the bounds test),
//     candidate a lane, coordinates over the warps, and ballots compact the first m in-bounds
//     moves.  Launches with flow proposals, and the sampler's own TaylorF2 walks, form every step's
//     exact move on its thread instead: the sampler's long windows fill the threads, and the
//     screen's draws, compaction and second pass cost more than the exact moves they save (walks
//     of a 4-parameter run to ln Z 15.4 ms screened, 14.6 not; of an 11-parameter one 160.7 and 159.3,
//     6 late batches of it on relative binning 27.1 and 26.5; but 8 batches of the 16,225-bin
//     IMRPhenomD form 354 and 385: its walks screen);
//  2. the proposal constants of the round run on all four warps at once (tf2_split_first /
//     tf2_split_second, pd_split_first / pd_split_second: independent chains, then the
//     products; the IMRPhenomD form's continuity constants and its region boundaries and
//     amplitude shape on different warps);
//  3. the likelihoods: TaylorF2 one warp per proposal, the IMRPhenomD form the whole CTA per
//     proposal;
//  4. warp 0 assembles ln L of every proposal in float-float and finds with one ballot where the
//     round's guess first fails: its first acceptance, or, looking ahead over acceptances, its
//     first rejection (the IMRPhenomD form: every thread assembles ln L after each proposal, and
//     the round ends there, the rest unevaluated).
// Stand-alone walks at 0.4 to 0.9 acceptances a call, against a fixed depth of 16 without look-ahead
// over acceptances, screen, early end and float pairs made once a call (GB300): 500 walkers x 600
// steps on the 4,017-bin TaylorF2 event 9.0 -> 2.2 ms, 1000 x 240 on the 16,225-bin IMRPhenomD-form
// event 151 -> 17.6 ms, on its relative-binning likelihood 13.0 -> 6.6 ms.
// The DE move is the walk's, u' = u + gamma (u_a - u_b), with the position and the survivors as
// float pairs (~48 significant bits): the chain is the FP64 chain up to rounding at ~1e-14.
// A TaylorF2 or relative-binning round is padded to a multiple of four proposals: its
// warp-per-proposal likelihood phase takes as long for 1 or 5 proposals as for 4 or 8, and the
// padding only advances the chain further.  The full grid of the IMRPhenomD form (thousands of bins a
// proposal) runs each proposal on the whole CTA instead.
// Relative binning runs without the flow paths (X 1), with the moves of step 1 and the padding: 1000
// walkers x 240 steps, IMRPhenomD, 122 coarse bins, 7.17 -> 6.57 ms.  Its round is bound by the float-float
// chains of a proposal's constants and moves; the likelihood of the coarse bins is short.
template <int NDET, int WF, int X, bool CH>
__global__ void __launch_bounds__(kThreads, 4) walk_kernel_ff(const EventDev* __restrict__ evs, WalkTask* tasks,
                                                            const int32_t* __restrict__ blk_task,
                                                            const int32_t* __restrict__ blk_local) {
  constexpr bool XF = X == 2;   // flow proposals
  constexpr bool kScreen = !XF && (CH || WF == 1);   // step 1: screened moves
  constexpr int NV = NVals<NDET, WF>::value;
  __shared__ WalkerParams P[kSpecMax];
  __shared__ ff propf[kSpecMax][kMaxDim];
  __shared__ union Parts {
    std::conditional_t<WF == 0, TF2Part, PDPart> p[kSpecMax];
    ff diff[32][kMaxDim];
    __device__ Parts() {}
  } sh;
  auto* const parts = sh.p;
  __shared__ int cstep[kSpecMax];
  __shared__ float part_sums[kSpecMax][2 * kMaxVals];
  __shared__ double s_rbl[kSpecMax];   // relative binning: ln L of each proposal
  __shared__ int s_rbk[kSpecMax];      // and the grid bins it touched
  // IMRPhenomD form: every warp's compensated sums of a proposal (two, so that a warp may write
  // the next proposal's while another still reads this one's)
  __shared__ float wsums[2][kWarps][2 * kMaxVals];
  __shared__ double u[kMaxDim];
  __shared__ ff uf[kMaxDim];
  __shared__ int wcount[kWarps];
  __shared__ unsigned wmask[kWarps];
  // candidates of a round: the step (complemented: unit scale), its survivors, the scale's uniforms
  __shared__ int cand_step[kScreen ? 32 : 1], cand_a[kScreen ? 32 : 1], cand_b[kScreen ? 32 : 1];
  __shared__ uint64_t cand_u[kScreen ? 32 : 1][4];
  __shared__ int s_next, s_setup_warp, s_end, s_needq, s_nin;
  __shared__ Round s_round;
  __shared__ int s_isflow[kSpecMax];
  __shared__ float s_lqf[kSpecMax];
  __shared__ float s_logq;
  __shared__ FlowScratch fscr;
  const WalkTask& T = tasks[blk_task[blockIdx.x]];
  const int j = blk_local[blockIdx.x];
  const EventDev& ev = evs[T.event];
  if (T.done) return;
  const int D = ev.n_dim;
  const int n_steps = T.n_steps;
  const double lnl_star = T.lnl_star;
  const uint64_t it = (uint64_t)T.iteration;
  const uint64_t wid = (uint64_t)(T.walker_offset + j);
  const uint64_t n_s = (uint64_t)T.n_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool split = ev.ff_setup;
  if (threadIdx.x < D) {
    const double v = T.u0[(size_t)j * D + threadIdx.x];
    u[threadIdx.x] = v;
    uf[threadIdx.x] = ff_from_double(v);
  }
  if (threadIdx.x == 0) {
    unsigned int smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    s_setup_warp = (int)(atomicAdd(&g_walk_sm_arrivals[smid & 255u], 1u) % (unsigned)kWarps);
  }
  unsigned periodic = 0u;
#pragma unroll
  for (int d = 0; d < kMaxDim; ++d)
    if (d < D && ev.prior[ev.dim_param[d]].periodic) periodic |= 1u << d;
  double lnl = T.lnl0[j];
  int n_acc = 0, n_acc_flow = 0, n_like = 0;
  int64_t n_bins = 0, n_spec = 0;
  const uint64_t t0 = threadIdx.x == 0 ? global_ns() : 0ull;
  const ff de_scale = ff_from_double(2.38 / sqrt(2.0 * (double)D));
  __syncthreads();
  const int sw = s_setup_warp;
  const bool use_flow = XF && T.flow != nullptr && T.p_flow > 0.0;
  const double p_flow = T.p_flow;
  Round rd = next_round<CH>(T, WF == 0 || (X >= 1 && ev.rb_nb > 0), 0, 0);
  if (use_flow) {
    const float lq = flow_logq_cta(*T.flow, u, fscr);
    if (threadIdx.x == 0) s_logq = lq;
    __syncthreads();
  }
  int t = 0;
  while (t < n_steps) {
    const int abort_flag = threadIdx.x == 0 ? walk_abort_flag(T) : 0;
    const int m = rd.depth;
    int nin;
    if constexpr (kScreen) {
      // 1a. one step a thread: its draws and, looking ahead over rejections, a FP32 screen of its move
      //     (as in walk_kernel; the margin never rejects a step that the exact test accepts: screen.h).  Four
      //     moves of five leave the cube, and the exact move of one is ~700 float-float
      //     instructions: it is formed for the steps that may stay only.  Looking ahead over
      //     acceptances: the next 32 steps, unscreened.
      const bool chain = CH && rd.chain;
      const int W = min(chain ? 32 : min(kThreads, max(32, 4 * m)), n_steps - t);
      const int step = t + (int)threadIdx.x;
      int maybe = 0, ia = 0, ib = 0;
      bool draw_scale = false;
      Philox4 B;
      if ((int)threadIdx.x < W) {
        // tag 0: survivors and scale coin, tag 1: the scale's uniforms -- one inlined generator
        Philox4 A;
#pragma unroll 1
        for (int tag = 0; tag < 2; ++tag) {
          const Philox4 r = philox4x64((uint64_t)step, wid, it, (uint64_t)tag, T.key0, T.key1);
          if (tag == 0) {
            A = r;
            draw_scale = (r.v[2] >> 63) == 0ull;
            if (!draw_scale) break;
          } else {
            B = r;
          }
        }
        ia = (int)rand_index(A.v[0], n_s);
        ib = (int)rand_index(A.v[1], n_s - 1);
        ib += ib >= ia ? 1 : 0;
        maybe = 1;
        if (!chain) {
          float va[kMaxDim], vb[kMaxDim];   // both survivors first: all loads in flight at once
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d) {
            const size_t dd = d < D ? d : D - 1;
            va[d] = T.survf ? T.survf[(size_t)ia * D + dd].x : (float)T.surv[(size_t)ia * D + dd];
            vb[d] = T.survf ? T.survf[(size_t)ib * D + dd].x : (float)T.surv[(size_t)ib * D + dd];
          }
          float sc = 1.0f;
          if (draw_scale) {
            sc = screen_scale(B.v, de_scale.h, FastLog2{});
          }
          const float margin = screen_margin(sc);
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d) {
            const float x = uf[d < D ? d : D - 1].h + sc * (va[d] - vb[d]);
            if (d < D && !((periodic >> d) & 1u) && !(x >= -margin && x <= 1.0f + margin)) maybe = 0;
          }
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, maybe);
      if (lane == 0) wcount[warp] = __popc(mask);
      __syncthreads();
      int before = 0, total = 0;
#pragma unroll
      for (int w2 = 0; w2 < kWarps; ++w2) {
        const int cw = wcount[w2];
        before += (w2 < warp) ? cw : 0;
        total += cw;
      }
      const int cs = before + __popc(mask & ((1u << lane) - 1u));
      if (maybe && cs < 32) {
        cand_step[cs] = draw_scale ? step : ~step;
        cand_a[cs] = ia;
        cand_b[cs] = ib;
        if (draw_scale) {
#pragma unroll
          for (int q = 0; q < 4; ++q) cand_u[cs][q] = B.v[q];
        }
      }
      const int nc = min(total, 32);
      __syncthreads();
      // 1b. the exact moves: candidate `lane`, coordinates warp, warp + 4, ... (float-float)
      constexpr int kQ = (kMaxDim + kWarps - 1) / kWarps;
      ff xq[kQ];
      int in = lane < nc;
      int st = 0;
      if (lane < nc) {
        st = cand_step[lane];
        ff sc = ff_make(1.0f);
        if (st >= 0) sc = ff_mul(ff_mul_f(ff_log_uniform_product(cand_u[lane]), -0.25f), de_scale);
        else st = ~st;
        const size_t oa = (size_t)cand_a[lane] * D, ob = (size_t)cand_b[lane] * D;
        ff ua[kQ], ub[kQ];
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          const int d = min(warp + kWarps * q, D - 1);
          if (T.survf) {
            const float2 pa = T.survf[oa + d], pb = T.survf[ob + d];
            ua[q] = ff{pa.x, pa.y};
            ub[q] = ff{pb.x, pb.y};
          } else {
            ua[q] = ff_from_double(T.surv[oa + d]);
            ub[q] = ff_from_double(T.surv[ob + d]);
          }
        }
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          const int d = warp + kWarps * q;
          if (d < D) {
            const ff df = ff_mul(sc, ff_sub(ua[q], ub[q]));
            if (chain) {
              sh.diff[lane][d] = df;
            } else {
              ff x = ff_add(uf[d], df);
              if ((periodic >> d) & 1u) x = ff_wrap_unit(x);
              if (!ff_in_unit(x)) in = 0;
              xq[q] = x;
            }
          }
        }
      }
      if (!chain) {
        const unsigned mine = __ballot_sync(0xffffffffu, in);
        if (lane == 0) wmask[warp] = mine;
        __syncthreads();
        const unsigned im = wmask[0] & wmask[1] & wmask[2] & wmask[3];
        const int cnt = __popc(im), slot = __popc(im & ((1u << lane) - 1u));
        if (((im >> lane) & 1u) && slot < m) {
#pragma unroll
          for (int q = 0; q < kQ; ++q)
            if (warp + kWarps * q < D) propf[slot][warp + kWarps * q] = xq[q];
          if (warp == 0) {
            cstep[slot] = st;
            // the round covers the steps up to the m-th in-bounds one, else the last candidate if
            // there were more than 32, else the whole window
            if (slot == m - 1 && cnt > m) s_end = st;
          }
        }
        if (threadIdx.x == 31 && cnt <= m) s_end = total > 32 ? st : t + W - 1;
        nin = min(cnt, m);
        __syncthreads();
      } else {
        // warp 0 chains the in-bounds moves, a coordinate a lane
        __syncthreads();
        if (warp == 0) {
          ff x = lane < D ? uf[lane] : ff_make(0.0f);
          int cnt = 0;
          for (int q = 0; q < W && cnt < m; ++q) {
            ff y = ff_make(0.0f);
            if (lane < D) {
              y = ff_add(x, sh.diff[q][lane]);
              if ((periodic >> lane) & 1u) y = ff_wrap_unit(y);
            }
            if (__all_sync(0xffffffffu, ff_in_unit(y))) {
              x = y;
              if (lane < D) propf[cnt][lane] = y;
              if (lane == 0) cstep[cnt] = t + q;
              ++cnt;
            }
          }
          __syncwarp();
          if (lane == 0) {
            s_nin = cnt;
            s_end = cnt == m ? cstep[m - 1] : t + W - 1;
          }
        }
        __syncthreads();
        nin = s_nin;
      }
    } else {
      // 1. the exact move of one candidate step per thread (or its flow proposal)
      const int W = min(min(kThreads, max(32, 4 * m)), n_steps - t);
      const int step = t + (int)threadIdx.x;
      int in = 0, isf = 0;
      float lqf = 0.0f;
      ff xf[kMaxDim];
      if ((int)threadIdx.x < W) {
        // the step's Philox blocks: (tag 6: flow coin,) tag 0: survivors and scale coin,
        // tag 1: the scale's uniforms -- one inlined generator, called up to three times
        Philox4 A, B;
        bool draw_scale = false;
        int tag = use_flow ? 6 : 0;
#pragma unroll 1
        while (tag >= 0) {
          const Philox4 r = philox4x64((uint64_t)step, wid, it, (uint64_t)tag, T.key0, T.key1);
          if (tag == 6) {
            tag = 0;
            if (rand_open_unit(r.v[0]) < p_flow) {
              isf = 1;
              lqf = (float)T.flq[(size_t)j * T.f_stride + step];
              in = logf((float)rand_open_unit(r.v[1])) < s_logq - lqf;
              tag = -1;
            }
          } else if (tag == 0) {
            A = r;
            draw_scale = (r.v[2] >> 63) == 0ull;
            tag = draw_scale ? 1 : -1;
          } else {
            B = r;
            tag = -1;
          }
        }
        if (isf) {
          if (in) {
            const double* fu = T.fu + ((size_t)j * T.f_stride + step) * D;
#pragma unroll
            for (int d = 0; d < kMaxDim; ++d)
              if (d < D) xf[d] = ff_from_double(fu[d]);
          }
        } else {
          const uint64_t a = rand_index(A.v[0], n_s);
          uint64_t b = rand_index(A.v[1], n_s - 1);
          b += (b >= a) ? 1ull : 0ull;
          // both survivors' coordinates first (branch-free, all loads in flight at once)
          ff ua[kMaxDim], ub[kMaxDim];
          if (T.survf) {
#pragma unroll
            for (int d = 0; d < kMaxDim; ++d) {
              const int dd = d < D ? d : D - 1;
              const float2 pa = T.survf[a * D + dd], pb = T.survf[b * D + dd];
              ua[d] = ff{pa.x, pa.y};
              ub[d] = ff{pb.x, pb.y};
            }
          } else {
#pragma unroll
            for (int d = 0; d < kMaxDim; ++d) {
              const int dd = d < D ? d : D - 1;
              ua[d] = ff_from_double(T.surv[a * D + dd]);
              ub[d] = ff_from_double(T.surv[b * D + dd]);
            }
          }
          const ff sc = draw_scale ? ff_mul(ff_mul_f(ff_log_uniform_product(B.v), -0.25f), de_scale) : ff_make(1.0f);
          in = 1;
#pragma unroll
          for (int d = 0; d < kMaxDim; ++d) {
            const ff df = ff_mul(sc, ff_sub(ua[d], ub[d]));
            ff x = ff_add(uf[d < D ? d : D - 1], df);
            const ff xw = ff_wrap_unit(x);
            if ((periodic >> d) & 1u) x = xw;
            if (d < D && !ff_in_unit(x)) in = 0;
            xf[d] = x;
          }
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, in);
      if (lane == 0) wcount[warp] = __popc(mask);
      __syncthreads();
      int before = 0, total = 0;
#pragma unroll
      for (int w2 = 0; w2 < kWarps; ++w2) {
        const int cw = wcount[w2];
        before += (w2 < warp) ? cw : 0;
        total += cw;
      }
      const int slot = before + __popc(mask & ((1u << lane) - 1u));
      if (in && slot < m) {
#pragma unroll
        for (int d = 0; d < kMaxDim; ++d)
          if (d < D) propf[slot][d] = xf[d];
        cstep[slot] = step;
        s_isflow[slot] = isf;
        s_lqf[slot] = lqf;
        // the round covers the steps up to the m-th in-bounds one, else the whole window
        if (slot == m - 1 && total > m) s_end = step;
      }
      if (threadIdx.x == 0 && total <= m) s_end = t + W - 1;
      nin = min(total, m);
      __syncthreads();
    }
    // 2. proposal constants
    if (nin > 0) {
      if (split) {
        if (lane < nin) {
          if constexpr (WF == 0) tf2_split_first(warp, ev, propf[lane], parts[lane], P[lane]);
          else pd_split_first(warp, ev, propf[lane], parts[lane], P[lane]);
        }
        __syncthreads();
        if (lane < nin) {
          if constexpr (WF == 0) tf2_split_second(warp, ev, parts[lane], P[lane]);
          else pd_split_second(warp, ev, parts[lane], P[lane]);
        }
      } else if (warp == sw && lane < nin) {
        double pd[kMaxDim];
#pragma unroll
        for (int d = 0; d < kMaxDim; ++d) pd[d] = d < D ? (double)propf[lane][d].h + (double)propf[lane][d].l : 0.0;
        setup_from_unit<2, WF>(ev, pd, P[lane]);
      }
      __syncthreads();
    }
    // 3. likelihoods
    constexpr int V = Pow2Vals<NV>::value;
    constexpr int group = 32 / V;
    const bool rb = X >= 1 && ev.rb_nb > 0;
    // whole-CTA evaluations: proposals evaluated, the last accepted one and its ln L, the one that
    // ended the round's guess
    int neval = nin, pd_hit = -1, pd_end = -1;
    double pd_l = 0.0, pd_lnl = 0.0;
    if (rb) {
      // relative binning (~10^2 coarse-bin edges a proposal): a warp per proposal
      for (int i = warp; i < nin; i += kWarps) {
        int nk;
        const double v = rb_lnl_warp<NDET, WF>(ev, P[i], lane, &nk);
        if (lane == 0) { s_rbl[i] = v; s_rbk[i] = nk; }
      }
      __syncthreads();
    } else if (WF == 1) {
      // IMRPhenomD form (thousands of bins a proposal): the whole CTA on each proposal in turn,
      // so that proposals of different lengths leave no warp waiting.  Every thread assembles
      // ln L from the four warps' compensated sums, and the round ends at its first acceptance:
      // the proposals after it are never evaluated.  The assembly (~600 cycles, one barrier) is
      // small against an evaluation (~10^5 cycles at four CTAs an SM), so the depth of a round
      // only spreads its fixed costs.
      for (int i = 0; i < nin; ++i) {
        double dv[NV];
        float fv[NV], fc[NV];
        partials<2, NDET, WF>(ev, P[i], threadIdx.x, kThreads, dv, fv, fc);
        float rs, rc;
        int q;
        warp_halving_sums<NV>(fv, fc, lane, rs, rc, q);
        if ((lane & (group - 1)) == 0 && q < NV) { wsums[i & 1][warp][2 * q] = rs; wsums[i & 1][warp][2 * q + 1] = rc; }
        __syncthreads();
        // (s, c) of the four warps, summed with error-free additions
        float ps[2 * NV];
#pragma unroll
        for (int q2 = 0; q2 < NV; ++q2) {
          float sh = wsums[i & 1][0][2 * q2], sl = wsums[i & 1][0][2 * q2 + 1];
#pragma unroll
          for (int w2 = 1; w2 < kWarps; ++w2) {
            float t2, e;
            two_sum(sh, wsums[i & 1][w2][2 * q2], t2, e);
            sh = t2;
            sl += wsums[i & 1][w2][2 * q2 + 1] + e;
          }
          ps[2 * q2] = sh;
          ps[2 * q2 + 1] = sl;
        }
        neval = i + 1;
        pd_l = lnl_ff<NDET, WF>(ev, P[i], ps);
        const bool up = pd_l > lnl_star;
        if (up) {
          pd_hit = i;
          pd_lnl = pd_l;
        }
        if (up != (CH && rd.chain)) {
          pd_end = i;
          break;
        }
      }
    } else {
      for (int i = warp; i < nin; i += kWarps) {
        double dv[NV];
        float fv[NV], fc[NV];
        partials<2, NDET, WF>(ev, P[i], lane, 32, dv, fv, fc);
        float rs, rc;
        int q;
        warp_halving_sums<NV>(fv, fc, lane, rs, rc, q);
        if ((lane & (group - 1)) == 0 && q < NV) { part_sums[i][2 * q] = rs; part_sums[i][2 * q + 1] = rc; }
      }
      __syncthreads();
    }
    // 4. ln L of every proposal, then the steps in order: the first acceptance ends the round
    if (warp == 0) {
      double l = 0.0;
      if (lane < nin) {
        if (rb) {
          l = s_rbl[lane];
        } else if (WF == 1) {
          l = pd_l;
        } else {
          l = lnl_ff<NDET, WF>(ev, P[lane], part_sums[lane]);
        }
      }
      // e: the proposal that ends the round's guess (its first acceptance, or first rejection);
      // c: the last accepted one
      const unsigned am = __ballot_sync(0xffffffffu, lane < nin && l > lnl_star);
      const unsigned live = nin < 32 ? (1u << nin) - 1u : 0xffffffffu;
      const unsigned ends = ((CH && rd.chain) ? ~am : am) & live;
      int e = ends ? __ffs(ends) - 1 : -1;
      int c = (CH && rd.chain) ? (e >= 0 ? e : nin) - 1 : e;
      if (WF == 1 && !rb) {
        e = pd_end;
        c = pd_hit;
      }
      const int used = e >= 0 ? e + 1 : nin;
      const int acc = (CH && rd.chain) ? c + 1 : (c >= 0 ? 1 : 0);
      int kb = lane < used ? (rb ? s_rbk[lane] : P[lane].k_end) : 0;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) kb += __shfl_xor_sync(0xffffffffu, kb, off);
      if (c >= 0) {
        lnl = (WF == 1 && !rb) ? pd_lnl : __shfl_sync(0xffffffffu, l, c);
        if (lane < D) {
          const ff x = propf[c][lane];
          uf[lane] = x;
          u[lane] = (double)x.h + (double)x.l;
        }
      }
      if (lane == 0) {
        n_like += used;
        n_bins += kb;
        n_spec += neval;
        int nxt = e >= 0 ? cstep[e] + 1 : s_end + 1;
        s_needq = 0;
        n_acc += acc;
        if (c >= 0) {
          if (use_flow) {
            if (s_isflow[c]) {
              s_logq = s_lqf[c];
              ++n_acc_flow;
            } else {
              s_needq = 1;
            }
          }
        }
        if (walk_should_stop(T, t0, abort_flag)) {   // watchdog: end the walk after this round
          nxt = n_steps;
          if (T.status) atomicOr(T.status, 1);
        }
        s_next = nxt;
        s_round = next_round<CH>(T, WF == 0 || (X >= 1 && ev.rb_nb > 0), n_acc, n_like);
      }
    }
    __syncthreads();
    t = s_next;
    rd = s_round;
    if (use_flow && s_needq && t < n_steps) {
      const float lq = flow_logq_cta(*T.flow, u, fscr);
      if (threadIdx.x == 0) s_logq = lq;
      __syncthreads();
    }
  }
  if (threadIdx.x < D) T.u_out[(size_t)j * D + threadIdx.x] = u[threadIdx.x];
  if (threadIdx.x == 0) {
    T.lnl_out[j] = lnl;
    T.n_acc[j] = n_acc;
    if (T.n_acc_flow) T.n_acc_flow[j] = n_acc_flow;
    T.n_like[j] = n_like;
    if (T.n_bins) T.n_bins[j] = n_bins;
    if (T.n_spec) T.n_spec[j] = n_spec;
  }
}

// ---------------------------------------------------------------- hit-and-run slice sampling
// Any precision.  One CTA per walker (block b: walker blk_local[b] of task blk_task[b]); thread 0
// runs each move's slice logic and the whole CTA evaluates every in-bounds candidate's ln L (the
// likelihood of the handle's precision; relative binning on warp 0 when the event uses it).  A
// move (Neal 2003, stepping out and shrinkage, along a random line): direction d = C z / |z|
// (z standard normal, C = task.chol, the Cholesky factor of the survivors' covariance), bracket
// [lo, lo + 1] with lo = -U, stepping out by one unit at a time with a budget of kHrssMaxOut - 1
// split as J = floor(kHrssMaxOut V) to the left and the rest to the right while the bracket's
// end is inside the slice, then shrinkage draws until a point inside the slice (at most
// kHrssMaxShrink; then the walker stays).  A candidate outside the cube costs no likelihood
// call; periodic coordinates wrap.  Philox blocks (step, walker, iteration, tag): tags 32 + c
// the normals (Box-Muller on words (0, 1) and (2, 3)), 40 the bracket (U, V), 48 + j / 4 word
// j % 4 the j-th shrinkage uniform.  task.n_steps moves; n_acc receives the moves made,
// n_like the likelihood calls; the watchdog (task.abort, task.budget_ns) is checked before
// every move.
constexpr int kHrssMaxOut = 10;
constexpr int kHrssMaxShrink = 100;

template <int PREC, int NDET, int WF>
__global__ void __launch_bounds__(kThreads) hrss_kernel(const EventDev* __restrict__ evs, WalkTask* tasks,
                                                         const int32_t* __restrict__ blk_task,
                                                         const int32_t* __restrict__ blk_local) {
  __shared__ WalkerParams P;
  __shared__ double red[kWarps][NVals<NDET, WF>::value];
  __shared__ double vals[kMaxVals];
  __shared__ double x[kMaxDim], dvec[kMaxDim], pt[kMaxDim];
  __shared__ double s_rbl;
  __shared__ int s_eval, s_end, s_stop, s_rbk;
  const WalkTask& T = tasks[blk_task[blockIdx.x]];
  const int j = blk_local[blockIdx.x];
  const EventDev& ev = evs[T.event];
  if (T.done) return;
  const int D = ev.n_dim;
  const int n_steps = T.n_steps;
  const double lnl_star = T.lnl_star;
  const uint64_t it = (uint64_t)T.iteration;
  const uint64_t wid = (uint64_t)(T.walker_offset + j);
  const double* chol = T.chol;
  bool rb = false;
  if constexpr (PREC == 2) rb = ev.rb_nb > 0;
  if ((int)threadIdx.x < D) x[threadIdx.x] = T.u0[(size_t)j * D + threadIdx.x];
  double lnl = T.lnl0[j];
  int moves = 0, calls = 0;
  int64_t n_bins = 0;
  const uint64_t t0 = threadIdx.x == 0 ? global_ns() : 0ull;
  // thread 0's state of the current move: phase 0 steps out left, 1 right, 2 shrinks
  double lo = 0.0, hi = 0.0, tc = 0.0;
  int phase = 2, jl = 0, kr = 0, nsh = 0;
  __syncthreads();
  for (int t = 0; t < n_steps; ++t) {
    if (threadIdx.x == 0) {
      s_stop = walk_should_stop(T, t0, walk_abort_flag(T)) ? 1 : 0;
      if (s_stop && T.status) atomicOr(T.status, 1);
      double z[kMaxDim];
      for (int c = 0; 4 * c < D; ++c) {
        const Philox4 b = philox4x64((uint64_t)t, wid, it, 32ull + (uint64_t)c, T.key0, T.key1);
        for (int q = 0; q < 2; ++q) {
          const double r = sqrt(-2.0 * log(rand_open_unit(b.v[2 * q])));
          double sn, cs;
          sincospi(2.0 * rand_open_unit(b.v[2 * q + 1]), &sn, &cs);
          const int i0 = 4 * c + 2 * q;
          if (i0 < D) z[i0] = r * cs;
          if (i0 + 1 < D) z[i0 + 1] = r * sn;
        }
      }
      double nz = 0.0;
      for (int i = 0; i < D; ++i) nz += z[i] * z[i];
      nz = sqrt(nz);
      for (int i = 0; i < D; ++i) {
        double acc = 0.0;
        for (int k = 0; k <= i; ++k) acc += chol[i * D + k] * z[k];
        dvec[i] = acc / nz;
      }
      const Philox4 b = philox4x64((uint64_t)t, wid, it, 40ull, T.key0, T.key1);
      lo = -rand_open_unit(b.v[0]);
      hi = lo + 1.0;
      jl = (int)floor((double)kHrssMaxOut * rand_open_unit(b.v[1]));
      kr = kHrssMaxOut - 1 - jl;
      nsh = 0;
      phase = jl > 0 ? 0 : (kr > 0 ? 1 : 2);
    }
    __syncthreads();
    if (s_stop) break;
    // step-out evaluations <= kHrssMaxOut - 1, shrinkage draws <= kHrssMaxShrink
    for (int iter = 0; iter < kHrssMaxOut + kHrssMaxShrink; ++iter) {
      if (threadIdx.x == 0) {
        if (phase == 0) {
          tc = lo;
        } else if (phase == 1) {
          tc = hi;
        } else {
          const Philox4 b = philox4x64((uint64_t)t, wid, it, 48ull + (uint64_t)(nsh >> 2), T.key0, T.key1);
          tc = lo + (hi - lo) * rand_open_unit(b.v[nsh & 3]);
        }
        int inb = 1;
        for (int i = 0; i < D; ++i) {
          double v = x[i] + tc * dvec[i];
          if (ev.prior[ev.dim_param[i]].periodic) v -= floor(v);
          pt[i] = v;
          if (!(v >= 0.0 && v <= 1.0)) inb = 0;
        }
        s_eval = inb;
        if (inb) setup_from_unit<PREC, WF>(ev, pt, P);
      }
      __syncthreads();
      const int evaluate = s_eval;
      if (evaluate) {
        if (rb) {
          if constexpr (PREC == 2) {
            if (threadIdx.x < 32) {
              int kb = 0;
              const double v = rb_lnl_warp<NDET, WF>(ev, P, threadIdx.x, &kb);
              if (threadIdx.x == 0) { s_rbl = v; s_rbk = kb; }
            }
            __syncthreads();
          }
        } else {
          cta_sums<PREC, NDET, WF>(ev, P, red, vals);
        }
      }
      if (threadIdx.x == 0) {
        bool ins = false;
        double l = 0.0;
        if (evaluate) {
          l = rb ? s_rbl : lnl_from_vals<PREC, NDET, WF>(ev, P, vals);
          ++calls;
          n_bins += rb ? s_rbk : P.k_end;
          ins = l > lnl_star;
        }
        int end = 0;
        if (phase == 0) {
          if (ins) { lo -= 1.0; --jl; }
          if (!ins || jl == 0) phase = kr > 0 ? 1 : 2;
        } else if (phase == 1) {
          if (ins) { hi += 1.0; --kr; }
          if (!ins || kr == 0) phase = 2;
        } else if (ins) {
          for (int i = 0; i < D; ++i) x[i] = pt[i];
          lnl = l;
          ++moves;
          end = 1;
        } else {
          if (tc < 0.0) lo = tc;
          else hi = tc;
          if (++nsh == kHrssMaxShrink) end = 1;
        }
        s_end = end;
      }
      __syncthreads();
      if (s_end) break;
    }
  }
  if ((int)threadIdx.x < D) T.u_out[(size_t)j * D + threadIdx.x] = x[threadIdx.x];
  if (threadIdx.x == 0) {
    T.lnl_out[j] = lnl;
    T.n_acc[j] = moves;
    T.n_like[j] = calls;
    if (T.n_bins) T.n_bins[j] = n_bins;
    if (T.n_spec) T.n_spec[j] = calls;
  }
}

// ---------------------------------------------------------------- speculative HRSS (mode 2)
// The slice-sampling moves of hrss_kernel, with the candidate evaluations of a move batched into
// rounds that run like the float-float walk's: the candidates' points in FP64 on warp 0 (one lane
// each), their constants on the setup warps, their likelihoods one warp per candidate (TaylorF2,
// relative binning) or on the whole CTA in turn (IMRPhenomD form), then thread 0 replays the
// sequential slice logic over them in order.  Which candidates the sequential move evaluates
// next depends on outcomes only through where it stops:
//   stepping out: the left end is tried at lo, lo - 1, lo - 2, ... while it is inside the slice
//     (budget J) and the right end at hi, hi + 1, ... (budget K); a round holds the next ends of
//     both sides, as if every one were inside, and the replay stops each side at its first end
//     outside the slice (the two sides do not interact, so their order does not matter);
//   shrinkage: with the draws U_j fixed by their Philox counters, the j-th candidate is
//     t_j = lo_j + (hi_j - lo_j) U_j, where (lo_j, hi_j) is the bracket left by rejecting
//     t_1 .. t_{j-1}; a round holds the next candidates as if all were rejected, and the replay
//     takes the first inside the slice.
// A stepping-out round holds up to max(1, spec/4) ends a side and fills the rest of the round
// with the first shrinkage candidates of the bracket as it stands: they are the move's next
// candidates exactly when every side still extending stops at its first end in the round, and
// the replay uses them only then -- a move whose bracket does not grow ends in one round.
// The chain, the moves and the likelihood-call counts are those of the one-candidate kernel (calls
// of candidates after the replay's stopping point are counted in n_spec only); per round at most
// task.spec candidates (1 .. kHrssQ).  Directions do not depend on the walker's position: the
// whole CTA forms those of 32 moves at a time (Box-Muller on the Philox blocks of hrss_kernel,
// d = C z / |z| row by row in the same order).
constexpr int kHrssQ = 16;

template <int NDET, int WF>
__global__ void __launch_bounds__(kThreads, 4) hrss_kernel_ff(const EventDev* __restrict__ evs, WalkTask* tasks,
                                                             const int32_t* __restrict__ blk_task,
                                                             const int32_t* __restrict__ blk_local) {
  constexpr int NV = NVals<NDET, WF>::value;
  __shared__ WalkerParams P[kHrssQ];
  __shared__ ff propf[kHrssQ][kMaxDim];
  __shared__ std::conditional_t<WF == 0, TF2Part, PDPart> parts[kHrssQ];
  __shared__ float part_sums[kHrssQ][2 * kMaxVals];
  __shared__ float wsums[WF == 1 ? kHrssQ : 1][kWarps][2 * kMaxVals];
  __shared__ double s_rbl[kHrssQ];
  __shared__ int s_rbk[kHrssQ];
  __shared__ double x[kMaxDim];
  __shared__ double zn_all[32][kMaxDim + 1];     // normals of the next 32 moves
  __shared__ double dir_all[32][kMaxDim];        // their directions d = C z / |z|
  __shared__ double ct[kHrssQ];              // t of each candidate of the round, in evaluation order
  __shared__ double cpt[kHrssQ][kMaxDim];    // its point
  __shared__ ff cf[kHrssQ][kMaxDim];         // the point as float pairs
  __shared__ double s_u[kHrssQ];             // the round's shrinkage draws
  __shared__ int s_oob[kHrssQ];              // the point lies outside the cube
  __shared__ int ins_c[kHrssQ];              // each slot's ln L exceeds ln L*
  __shared__ int cslot[kHrssQ];              // its likelihood slot, -1 for a point outside the cube
  __shared__ double lnl_c[kHrssQ];           // ln L of each slot
  __shared__ int kend_c[kHrssQ];             // grid bins each slot's evaluation touched
  __shared__ int s_nc, s_nin, s_newmove, s_exit, s_t, s_mode, s_nsh;
  const WalkTask& T = tasks[blk_task[blockIdx.x]];
  const int j = blk_local[blockIdx.x];
  const EventDev& ev = evs[T.event];
  if (T.done) return;
  const int D = ev.n_dim;
  const int n_steps = T.n_steps;
  const double lnl_star = T.lnl_star;
  const uint64_t it = (uint64_t)T.iteration;
  const uint64_t wid = (uint64_t)(T.walker_offset + j);
  const double* chol = T.chol;
  const int Q = T.spec < 1 ? 1 : (T.spec > kHrssQ ? kHrssQ : T.spec);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool split = ev.ff_setup;
  const bool rb = ev.rb_nb > 0;
  const int sw = (int)(blockIdx.x % (unsigned)kWarps);   // the setup warp of the non-split setups
  if ((int)threadIdx.x < D) x[threadIdx.x] = T.u0[(size_t)j * D + threadIdx.x];
  double lnl = T.lnl0[j];
  int moves = 0, calls = 0;
  int64_t n_bins = 0, n_spec = 0;
  const uint64_t t0 = threadIdx.x == 0 ? global_ns() : 0ull;
  // thread 0's move state: t the move, stepping (the bracket's ends still extend: jl, kr left),
  // lo, hi the bracket, nsh shrinkage draws used
  int t = 0, jl = 0, kr = 0, nsh = 0;
  bool left_on = false, right_on = false;
  double lo = 0.0, hi = 0.0;
  if (threadIdx.x == 0) {
    s_exit = n_steps <= 0 ? 1 : 0;
    s_newmove = 1;
    s_t = 0;
  }
  __syncthreads();
  while (!s_exit) {
    // A1. the directions of the next 32 moves, on the whole CTA, when a block of moves begins:
    //     a direction depends on its move's Philox counter only, not on the walker's position
    if (s_newmove && (s_t & 31) == 0) {
      const int base = s_t, nm = min(32, n_steps - base), nb = (D + 3) / 4;
      for (int q = threadIdx.x; q < nm * nb; q += kThreads) {
        const int mv = q / nb, c = q - mv * nb;
        const Philox4 b = philox4x64((uint64_t)(base + mv), wid, it, 32ull + (uint64_t)c, T.key0, T.key1);
        for (int h = 0; h < 2; ++h) {
          const double r = sqrt(-2.0 * log(rand_open_unit(b.v[2 * h])));
          double sn, cs;
          sincospi(2.0 * rand_open_unit(b.v[2 * h + 1]), &sn, &cs);
          const int i0 = 4 * c + 2 * h;
          if (i0 < D) zn_all[mv][i0] = r * cs;
          if (i0 + 1 < D) zn_all[mv][i0 + 1] = r * sn;
        }
      }
      __syncthreads();
      for (int q = threadIdx.x; q < nm * D; q += kThreads) {
        const int mv = q / D, i = q - mv * D;
        double nz = 0.0;
        for (int k = 0; k < D; ++k) nz += zn_all[mv][k] * zn_all[mv][k];
        nz = sqrt(nz);
        double acc = 0.0;
        for (int k = 0; k <= i; ++k) acc += chol[i * D + k] * zn_all[mv][k];
        dir_all[mv][i] = acc / nz;
      }
      __syncthreads();
    }
    // A2. warp 0: a new move's bracket; the round's candidates (shrinkage draws on the lanes) and
    //     their points ((candidate, coordinate) pairs over the lanes)
    if (warp == 0) {
      const int tm = s_t;
      const double* dv = dir_all[tm & 31];
      if (lane == 0) {
        if (s_newmove) {
          const Philox4 b = philox4x64((uint64_t)t, wid, it, 40ull, T.key0, T.key1);
          lo = -rand_open_unit(b.v[0]);
          hi = lo + 1.0;
          jl = (int)floor((double)kHrssMaxOut * rand_open_unit(b.v[1]));
          kr = kHrssMaxOut - 1 - jl;
          nsh = 0;
          left_on = jl > 0;
          right_on = kr > 0;
        }
        int ql = 0, qr = 0, S;
        if (left_on || right_on) {
          // stepping out: up to max(1, Q/4) next ends a side, the rest of the round's candidates
          // the shrinkage draws from the current bracket, which hold if every side still extending
          // stops at its first end in this round
          const int qs = max(1, Q / 4);
          ql = left_on ? min(jl, qs) : 0;
          qr = right_on ? min(kr, qs) : 0;
          if (ql + qr > Q) qr = Q - ql;
          S = min(Q - ql - qr, kHrssMaxShrink - nsh);
        } else {
          S = min(Q, kHrssMaxShrink - nsh);
        }
        s_mode = S;
        s_nsh = nsh;
        s_nc = (ql << 8) | (qr << 16);
      }
      __syncwarp();
      const int S = s_mode;
      if (lane < S) {
        const int jj = s_nsh + lane;
        const Philox4 b = philox4x64((uint64_t)tm, wid, it, 48ull + (uint64_t)(jj >> 2), T.key0, T.key1);
        s_u[lane] = rand_open_unit(b.v[jj & 3]);
      }
      __syncwarp();
      if (lane == 0) {
        int nc = 0;
        if (left_on || right_on) {
          // the next ends of both sides, as if every one were inside the slice, then the
          // shrinkage candidates of the bracket as it stands, as if each were rejected
          const int ql = (s_nc >> 8) & 255, qr = (s_nc >> 16) & 255;
          for (int i = 0; i < ql; ++i) ct[nc++] = lo - (double)i;
          for (int i = 0; i < qr; ++i) ct[nc++] = hi + (double)i;
          double l2 = lo, h2 = hi;
          for (int q = 0; q < S; ++q) {
            const double tc = l2 + (h2 - l2) * s_u[q];
            ct[nc++] = tc;
            if (tc < 0.0) l2 = tc;
            else h2 = tc;
          }
          s_nc = nc | (ql << 8) | (qr << 16);
        } else {
          // the next shrinkage candidates, as if every one were rejected
          double l2 = lo, h2 = hi;
          for (int q = 0; q < S; ++q) {
            const double tc = l2 + (h2 - l2) * s_u[q];
            ct[nc++] = tc;
            if (tc < 0.0) l2 = tc;
            else h2 = tc;
          }
          s_nc = nc;
        }
      }
      __syncwarp();
      const int nc = s_nc & 255;
      if (lane < nc) s_oob[lane] = 0;
      __syncwarp();
      for (int q = lane; q < nc * D; q += 32) {
        const int c = q / D, i = q - c * D;
        double v = x[i] + ct[c] * dv[i];
        if (ev.prior[ev.dim_param[i]].periodic) v -= floor(v);
        cpt[c][i] = v;
        cf[c][i] = ff_from_double(v);
        if (!(v >= 0.0 && v <= 1.0)) atomicOr(&s_oob[c], 1);
      }
      __syncwarp();
      const int inb = (lane < nc && s_oob[lane] == 0) ? 1 : 0;
      const unsigned im = __ballot_sync(0xffffffffu, inb);
      if (lane < nc) cslot[lane] = inb ? __popc(im & ((1u << lane) - 1u)) : -1;
      if (lane == 0) s_nin = __popc(im);
      __syncwarp();
      // the in-cube candidates' coordinates in slot order
      for (int q = lane; q < nc * kMaxDim; q += 32) {
        const int c = q / kMaxDim, d = q - c * kMaxDim;
        const int sl = cslot[c];
        if (sl >= 0) propf[sl][d] = d < D ? cf[c][d] : ff_make(0.0f);
      }
    }
    __syncthreads();
    const int nin = s_nin;
    // B. the candidates' constants
    if (nin > 0) {
      if (split) {
        if (lane < nin) {
          if constexpr (WF == 0) tf2_split_first(warp, ev, propf[lane], parts[lane], P[lane]);
          else pd_split_first(warp, ev, propf[lane], parts[lane], P[lane]);
        }
        __syncthreads();
        if (lane < nin) {
          if constexpr (WF == 0) tf2_split_second(warp, ev, parts[lane], P[lane]);
          else pd_split_second(warp, ev, parts[lane], P[lane]);
        }
      } else if (warp == sw && lane < nin) {
        double pd[kMaxDim];
#pragma unroll
        for (int d = 0; d < kMaxDim; ++d) pd[d] = d < D ? (double)propf[lane][d].h + (double)propf[lane][d].l : 0.0;
        setup_from_unit<2, WF>(ev, pd, P[lane]);
      }
      __syncthreads();
    }
    // C. likelihoods
    constexpr int V = Pow2Vals<NV>::value;
    constexpr int group = 32 / V;
    if (nin > 0) {
      if (rb) {
        for (int i = warp; i < nin; i += kWarps) {
          int nk;
          const double v = rb_lnl_warp<NDET, WF>(ev, P[i], lane, &nk);
          if (lane == 0) { s_rbl[i] = v; s_rbk[i] = nk; }
        }
      } else if (WF == 1) {
        for (int i = 0; i < nin; ++i) {
          double dv[NV];
          float fv[NV], fc[NV];
          partials<2, NDET, WF>(ev, P[i], threadIdx.x, kThreads, dv, fv, fc);
          float rs, rc;
          int q;
          warp_halving_sums<NV>(fv, fc, lane, rs, rc, q);
          if ((lane & (group - 1)) == 0 && q < NV) { wsums[i][warp][2 * q] = rs; wsums[i][warp][2 * q + 1] = rc; }
        }
      } else {
        for (int i = warp; i < nin; i += kWarps) {
          double dv[NV];
          float fv[NV], fc[NV];
          partials<2, NDET, WF>(ev, P[i], lane, 32, dv, fv, fc);
          float rs, rc;
          int q;
          warp_halving_sums<NV>(fv, fc, lane, rs, rc, q);
          if ((lane & (group - 1)) == 0 && q < NV) { part_sums[i][2 * q] = rs; part_sums[i][2 * q + 1] = rc; }
        }
      }
      __syncthreads();
    }
    // D. ln L of every slot (warp 0), then thread 0 replays the sequential move over the candidates
    if (warp == 0) {
      if (lane < nin) {
        double l;
        int kb;
        if (rb) {
          l = s_rbl[lane];
          kb = s_rbk[lane];
        } else if (WF == 1) {
          float ps[2 * NV];
#pragma unroll
          for (int q = 0; q < NV; ++q) {
            float sh = wsums[lane][0][2 * q], sl = wsums[lane][0][2 * q + 1];
#pragma unroll
            for (int w2 = 1; w2 < kWarps; ++w2) {
              float tt, e;
              two_sum(sh, wsums[lane][w2][2 * q], tt, e);
              sh = tt;
              sl += wsums[lane][w2][2 * q + 1] + e;
            }
            ps[2 * q] = sh;
            ps[2 * q + 1] = sl;
          }
          l = lnl_ff<NDET, WF>(ev, P[lane], ps);
          kb = P[lane].k_end;
        } else {
          l = lnl_ff<NDET, WF>(ev, P[lane], part_sums[lane]);
          kb = P[lane].k_end;
        }
        lnl_c[lane] = l;
        kend_c[lane] = kb;
        ins_c[lane] = l > lnl_star ? 1 : 0;
      }
      __syncwarp();
      if (lane == 0) {
        const int nc = s_nc & 255;
        n_spec += nin;
        bool move_end = false;
        int sh0 = 0;          // first shrinkage candidate of the round
        bool shrink = true;   // the round's shrinkage candidates are the move's next ones
        if (left_on || right_on) {
          const int ql = (s_nc >> 8) & 255, qr = (s_nc >> 16) & 255;
          // the speculative shrinkage holds iff every side extending at the round's start stops
          // at its first end here (the bracket is then the one the candidates were drawn in)
          if ((left_on && ql == 0) || (right_on && qr == 0)) shrink = false;
          for (int i = 0; i < ql && left_on; ++i) {
            const int sl = cslot[i];
            bool ins = false;
            if (sl >= 0) {
              ++calls;
              n_bins += kend_c[sl];
              ins = ins_c[sl] != 0;
            }
            if (ins) {
              shrink = false;
              lo -= 1.0;
              if (--jl == 0) left_on = false;
            } else {
              left_on = false;
            }
          }
          for (int i = ql; i < ql + qr && right_on; ++i) {
            const int sl = cslot[i];
            bool ins = false;
            if (sl >= 0) {
              ++calls;
              n_bins += kend_c[sl];
              ins = ins_c[sl] != 0;
            }
            if (ins) {
              shrink = false;
              hi += 1.0;
              if (--kr == 0) right_on = false;
            } else {
              right_on = false;
            }
          }
          sh0 = ql + qr;
          if (left_on || right_on) shrink = false;
        }
        if (shrink) {
          for (int i = sh0; i < nc; ++i) {
            const int sl = cslot[i];
            if (sl >= 0) {
              ++calls;
              n_bins += kend_c[sl];
              if (ins_c[sl]) {
                for (int d = 0; d < D; ++d) x[d] = cpt[i][d];
                lnl = lnl_c[sl];
                ++moves;
                move_end = true;
                break;
              }
            }
            if (ct[i] < 0.0) lo = ct[i];
            else hi = ct[i];
            if (++nsh == kHrssMaxShrink) {
              move_end = true;
              break;
            }
          }
        }
        if (move_end) ++t;
        s_newmove = move_end ? 1 : 0;
        s_t = t;
        if (t >= n_steps) s_exit = 1;
        if (!s_exit && walk_should_stop(T, t0, walk_abort_flag(T))) {   // watchdog: the walker stays where it is
          s_exit = 1;
          if (T.status) atomicOr(T.status, 1);
        }
      }
    }
    __syncthreads();
  }
  if ((int)threadIdx.x < D) T.u_out[(size_t)j * D + threadIdx.x] = x[threadIdx.x];
  if (threadIdx.x == 0) {
    T.lnl_out[j] = lnl;
    T.n_acc[j] = moves;
    T.n_like[j] = calls;
    if (T.n_bins) T.n_bins[j] = n_bins;
    if (T.n_spec) T.n_spec[j] = n_spec;
  }
}

}  // namespace

// Launchers of one precision P; each kernels_pP.cu instantiates its own.
#define GWNS_DISPATCH_N(K, P, W)                                                  \
  if (n_det == 1) K(P, 1, W); else if (n_det == 2) K(P, 2, W);                    \
  else if (n_det == 3) K(P, 3, W); else K(P, 4, W);
#define GWNS_DISPATCH_W(K, P)                                                     \
  if (waveform == 0) { GWNS_DISPATCH_N(K, P, 0) } else { GWNS_DISPATCH_N(K, P, 1) }

// Proposals of a CTA: as many as keep each of the 152 SMs at two CTAs (a setup costs its warps the
// same FP64 time for one proposal or for a full tile), up to 16 for TaylorF2; up to 4 for the
// IMRPhenomD form, whose evaluations take ~100 times a setup and balance better in small pieces.
// The result does not depend on the tile; asking the device for its SMs made calls of 1 and 1000
// vectors 2 and 4 us slower (37 and 47 us alone).
inline int lik_tile(int n, int waveform) {
  const int t = (n + 303) / 304, most = waveform == 0 ? kLikTile : 4;
  return t < 1 ? 1 : (t > most ? most : t);
}

template <int P>
cudaError_t launch_likelihood_p(int waveform, int n_det, const EventDev* d_ev, const double* d_theta, int n,
                                double* d_lnl, int32_t* d_status, cudaStream_t s) {
  const int tile = lik_tile(n, waveform), grid = (n + tile - 1) / tile;
#define GWNS_LIK(P_, N, W) \
  likelihood_kernel<P_, N, W, false><<<grid, kThreads, 0, s>>>(d_ev, d_theta, n, tile, d_lnl, d_status)
  GWNS_DISPATCH_W(GWNS_LIK, P)
#undef GWNS_LIK
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_unit_likelihood_p(int waveform, int n_det, const EventDev* d_ev, const double* d_u, int n,
                                     double* d_lnl, cudaStream_t s) {
  const int tile = lik_tile(n, waveform), grid = (n + tile - 1) / tile;
#define GWNS_UL(P_, N, W) \
  likelihood_kernel<P_, N, W, true><<<grid, kThreads, 0, s>>>(d_ev, d_u, n, tile, d_lnl, nullptr)
  GWNS_DISPATCH_W(GWNS_UL, P)
#undef GWNS_UL
  return cudaGetLastError();
}

// Mode 2 runs the float-float walk; modes 0 and 1 the FP64-recheck walk.  extras: 0 no task of the
// launch uses flow proposals or the relative-binning likelihood, 1 relative binning only, 2 flow
// proposals -- each runs the float-float walk compiled without what it does not use (a smaller
// kernel: its round is short and instruction fetch is among its first stalls).  Both properties of
// an event are fixed before its first ns_step (ns_relbin_set is refused after it), so the sampler's
// captured batch graphs keep a valid choice.
// `chain` launches (stand-alone walks) take the kernels that can look ahead over acceptances: their
// acceptance may be anything (500 walkers x 600 steps at 0.87 acceptances a call, 4,017 bins: 4.85 ->
// 2.1 ms).  The sampler's walks accept a few per cent of their calls from the first batches on, and
// there the larger kernel costs 5 % (ten batches: 17.9 -> 19.0 ms of walks), so they take the plain
// one; so do flows.  With relative binning TaylorF2 takes the look-ahead and the IMRPhenomD form does
// not.  It is the acceptance p that decides between the two kernels, and alike for both forms, us
// without -> with (500 x 240 TaylorF2; 1000 x 240 IMRPhenomD):
//   p 0.93   1057 ->  458;  3807 -> 1585      p 0.35   708 -> 782;  2772 -> 3071
//   p 0.78    957 ->  644;  3439 -> 2315      p 0.24   648 -> 693;  2220 -> 2347
//   p 0.58    876 ->  835;  3199 -> 3234      p 0.15   535 -> 560;  1547 -> 1658
// so the IMRPhenomD form's line is not a property of the form: its walks lose 1 to 10 % below p = 0.6
// and would gain above 0.7; a launch does not know p.
// The float-float walk's variants are compiled in units of their own (GWNS_FF_WALK: parallel builds).
#define GWNS_WALK_ARGS \
  int waveform, int n_det, const EventDev *d_evs, WalkTask *d_tasks, const int32_t *d_blk_task, \
      const int32_t *d_blk_local, int n_blocks, cudaStream_t s
cudaError_t launch_walk_ff_plain(GWNS_WALK_ARGS);         // kernels_p2w.cu
cudaError_t launch_walk_ff_chain(GWNS_WALK_ARGS);         // kernels_p2c.cu
cudaError_t launch_walk_ff_relbin(GWNS_WALK_ARGS);        // kernels_p2r.cu
cudaError_t launch_walk_ff_relbin_chain(GWNS_WALK_ARGS);  // kernels_p2r.cu, TaylorF2
cudaError_t launch_walk_ff_flow(GWNS_WALK_ARGS);          // kernels_p2.cu
#define GWNS_FF_WALK(NAME, X, CH)                                                                                    \
  cudaError_t NAME(GWNS_WALK_ARGS) {                                                                                 \
    GWNS_DISPATCH_W(GWNS_FF_WALK_ONE_##X##CH, 2)                                                                     \
    return cudaGetLastError();                                                                                       \
  }
#define GWNS_FF_WALK_RUN(N, W, X, CH) \
  walk_kernel_ff<N, W, X, CH><<<n_blocks, kThreads, 0, s>>>(d_evs, d_tasks, d_blk_task, d_blk_local)
#define GWNS_FF_WALK_ONE_00(P_, N, W) GWNS_FF_WALK_RUN(N, W, 0, false)
#define GWNS_FF_WALK_ONE_01(P_, N, W) GWNS_FF_WALK_RUN(N, W, 0, true)
#define GWNS_FF_WALK_ONE_10(P_, N, W) GWNS_FF_WALK_RUN(N, W, 1, false)
#define GWNS_FF_WALK_ONE_11(P_, N, W) GWNS_FF_WALK_RUN(N, W, 1, true)
#define GWNS_FF_WALK_ONE_20(P_, N, W) GWNS_FF_WALK_RUN(N, W, 2, false)

// Modes 0 and 1 are bound by the FP64 pipe of a walker's SM (half of a round of eight proposals),
// so a launch of few walkers spreads each over a cluster of CTAs: every rank runs the moves, the
// constants and the replay, and evaluates its share of the round's proposals.
template <int P, int N, int W>
void launch_walk_f64(bool chain, int ranks, int n_blocks, cudaStream_t s, const EventDev* d_evs, WalkTask* d_tasks,
                     const int32_t* d_blk_task, const int32_t* d_blk_local) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)ranks;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_blocks * ranks));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = ranks > 1 ? 1 : 0;
  // the error, if any, is read by the caller
  const auto k = ranks > 1 ? (chain ? walk_kernel<P, N, W, true, true> : walk_kernel<P, N, W, false, true>)
                           : (chain ? walk_kernel<P, N, W, true, false> : walk_kernel<P, N, W, false, false>);
  cudaLaunchKernelEx(&cfg, k, d_evs, d_tasks, d_blk_task, d_blk_local);
}

template <int P>
cudaError_t launch_walk_p(int waveform, int n_det, const EventDev* d_evs, WalkTask* d_tasks,
                          const int32_t* d_blk_task, const int32_t* d_blk_local, int n_blocks, cudaStream_t s,
                          int extras, bool chain) {
  if constexpr (P == 2) {
    const auto f = extras == 2 ? launch_walk_ff_flow
                               : extras == 1 ? (chain && waveform == 0 ? launch_walk_ff_relbin_chain : launch_walk_ff_relbin)
                                             : (chain ? launch_walk_ff_chain : launch_walk_ff_plain);
    return f(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s);
  } else {
    // the largest of 4, 2 and 1 ranks that gives every CTA an SM of its own (50 walkers of 1,969 bins,
    // 26 batches to the evidence: 76 ms on one CTA each, 63 on two, 69 on three)
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int ranks = extras == 2 ? 1 : 4 * n_blocks <= sms ? 4 : 2 * n_blocks <= sms ? 2 : 1;
#define GWNS_WALK(P_, N, W) \
  launch_walk_f64<P_, N, W>(chain && extras != 2, ranks, n_blocks, s, d_evs, d_tasks, d_blk_task, d_blk_local)
    GWNS_DISPATCH_W(GWNS_WALK, P)
#undef GWNS_WALK
    return cudaGetLastError();
  }
}

// Mode 2 runs the speculative float-float HRSS kernel; modes 0 and 1 one candidate at a time.
template <int P, int N, int W>
void launch_hrss_one(int n_blocks, cudaStream_t s, const EventDev* d_evs, WalkTask* d_tasks,
                     const int32_t* d_blk_task, const int32_t* d_blk_local) {
  if constexpr (P == 2) hrss_kernel_ff<N, W><<<n_blocks, kThreads, 0, s>>>(d_evs, d_tasks, d_blk_task, d_blk_local);
  else hrss_kernel<P, N, W><<<n_blocks, kThreads, 0, s>>>(d_evs, d_tasks, d_blk_task, d_blk_local);
}

template <int P>
cudaError_t launch_hrss_p(int waveform, int n_det, const EventDev* d_evs, WalkTask* d_tasks,
                          const int32_t* d_blk_task, const int32_t* d_blk_local, int n_blocks, cudaStream_t s) {
#define GWNS_HRSS(P_, N, W) launch_hrss_one<P_, N, W>(n_blocks, s, d_evs, d_tasks, d_blk_task, d_blk_local)
  GWNS_DISPATCH_W(GWNS_HRSS, P)
#undef GWNS_HRSS
  return cudaGetLastError();
}

}  // namespace gwns
