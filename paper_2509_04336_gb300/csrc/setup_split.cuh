// setup_split.cuh -- the per-proposal constants of modes 0 and 1 (taylorf2_setup,
// taylorf2_setup_lean, phenomd_extra) formed by the four warps of a CTA at once, lane i on proposal
// i, and the tile setup of the likelihood kernels.
//
// A setup is one dependent chain after another on the FP64 pipe (64 cycles an operation, 16 cycles a
// warp instruction however many lanes are active), so a lone thread took ~25 us for one proposal.
// Here its independent chains run on different warps -- first pass: (0) mass scales, logarithm,
// prefactor; (1) PN coefficients; (2) sky, antenna patterns, delays; (3) the amplitude scale;
// second pass: (0, 1) basis coefficients, (2) phase constant and projection factors, (3) the cutoff
// and <h|h>, or the IMRPhenomD-form regions -- for up to 32 proposals at once.  A part transforms
// only the parameters it reads (the one-thread setup also formed arccosines and arcsines that
// nothing read).  The expressions are the one-thread setup's.
#pragma once

#include <type_traits>

#include "gwns_internal.h"

namespace gwns {

// Parameters of one proposal from its unit-cube point (UNIT) or its physical vector; LEAN: the
// mixed paths' transform (a power law in FP32).
template <bool LEAN, bool UNIT>
struct ParamSource {
  const EventDev& ev;
  const double* v;
  __device__ double x(int i) const {
    if (!UNIT) return v[i];
    const PriorDev& p = ev.prior[i];
    if (p.kind == kFixed) return p.value;
    const double w = v[ev.param_dim[i]];
    if (p.kind == kUniform) return __dadd_rn(p.lo, __dmul_rn(w, p.w));
    if (p.kind == kPowerLaw) {
      const double y = __dadd_rn(p.A, __dmul_rn(w, p.B));
      if (LEAN) return (double)powf((float)y, (float)(1.0 / p.e));
      return (p.e == 3.0) ? cbrt(y) : pow(y, 1.0 / p.e);
    }
    if (p.kind == kSine) return acos(fmin(1.0, fmax(-1.0, __dsub_rn(p.A, __dmul_rn(w, p.B)))));
    return asin(fmin(1.0, fmax(-1.0, __dadd_rn(p.A, __dmul_rn(w, p.B)))));
  }
  __device__ double cos_iota() const {
    if (!UNIT) return cos(v[5]);
    const PriorDev& p = ev.prior[5];
    if (p.kind == kFixed) return p.cosv;
    if (p.kind == kSine) return fmin(1.0, fmax(-1.0, __dsub_rn(p.A, __dmul_rn(v[ev.param_dim[5]], p.B))));
    return cos(x(5));
  }
  __device__ void dec(double* sd, double* cd) const {
    if (UNIT) {
      const PriorDev& p = ev.prior[10];
      if (p.kind == kFixed) {
        *sd = p.sinv;
        *cd = p.cosv;
        return;
      }
      if (p.kind == kCosine) {
        const double s = fmin(1.0, fmax(-1.0, __dadd_rn(p.A, __dmul_rn(v[ev.param_dim[10]], p.B))));
        *sd = s;
        *cd = sqrt(fmax(0.0, (1.0 - s) * (1.0 + s)));
        return;
      }
    }
    sincos(x(10), sd, cd);
  }
};

// What the first pass hands to the second.
struct SetupPart {
  double q, eta, delta, chis, chia, chi1, chi2, phic;
  double c1, ci1, ci2, ci3, ci5, lpm, pre, fcut;
  double a[8];
  double K, pr[kMaxDet], pi[kMaxDet];
};

template <bool LEAN>
__device__ __forceinline__ void mass_ratio_f64(double q, double* eta, double* delta) {
  if (LEAN) {
    const double opq = 1.0 + q;
    const double r_opq = 1.0 / opq;
    *eta = q * r_opq * r_opq;
    *delta = (1.0 - q) * r_opq;
  } else {
    *eta = q / ((1.0 + q) * (1.0 + q));
    *delta = (1.0 - q) / (1.0 + q);
  }
}

template <bool LEAN, bool UNIT>
__device__ __noinline__ void f64_split_first(int part, const EventDev& ev, const double* v, SetupPart& s,
                                             WalkerParams& p) {
  const ParamSource<LEAN, UNIT> src{ev, v};
  if (part == 0) {
    const double mc = src.x(0), q = src.x(1);
    double eta, delta;
    mass_ratio_f64<LEAN>(q, &eta, &delta);
    if (LEAN) {
      const double opq = 1.0 + q;
      const double pmc = kPi * kMsunS * mc;              // pi Mc [s]
      const double w = rcbrt_newton(pmc);                // (pi Mc)^(-1/3)
      const double z = rfifth_newton(eta);               // eta^(-1/5)
      s.c1 = pmc * w * w * z;                            // (pi M)^(1/3) = (pi Mc)^(1/3) eta^(-1/5)
      const double z2 = z * z;
      s.ci1 = w * eta * z2 * z2;                         // (pi M)^(-1/3)
      s.ci2 = s.ci1 * s.ci1;
      s.ci3 = s.ci1 * s.ci1 * s.ci1;                     // 1/(pi M)
      s.fcut = (1.0 / kSix15) * s.ci3;
      s.lpm = 3.0 * log(s.c1);
      s.pre = (3.0 / (256.0 * kPi)) * opq * opq / q;     // 3/(256 pi eta)
    } else {
      const double mtot = mc * pow(eta, -0.6);
      const double piM = kPi * (mtot * kMsunS);
      s.fcut = 1.0 / (kSix15 * piM);
      s.lpm = log(piM);
      s.c1 = cbrt(piM);
      s.ci1 = 1.0 / s.c1;
      s.ci2 = s.ci1 * s.ci1;
      s.ci3 = s.ci2 * s.ci1;
      s.pre = 3.0 / (256.0 * kPi * eta);                 // 3/(128 eta) / (2 pi): cycles
    }
    s.ci5 = s.ci3 * s.ci2;
  } else if (part == 1) {
    s.q = src.x(1);
    s.chi1 = src.x(2);
    s.chi2 = src.x(3);
    s.phic = src.x(7);
    mass_ratio_f64<LEAN>(s.q, &s.eta, &s.delta);
    s.chis = 0.5 * (s.chi1 + s.chi2);
    s.chia = 0.5 * (s.chi1 - s.chi2);
    double a[8], al[8];
    taylorf2_pn_coeffs(s.eta, s.delta, s.chis, s.chia, a, al);
#pragma unroll
    for (int k = 0; k < 8; ++k) s.a[k] = a[k];
  } else if (part == 2) {
    double sd, cd, sp, cp;
    const double ci = src.cos_iota(), tc = src.x(8), psi = src.x(6);
    src.dec(&sd, &cd);
    sincos(src.x(9) - ev.gmst, &sp, &cp);
    if (LEAN) {
      // sky direction in FP64 (it sets the arrival delays), the rest in FP32
      const double n0 = cd * cp, n1 = cd * sp, n2 = sd;
      const float spf = (float)sp, cpf = (float)cp, ctf = (float)sd, stf = (float)cd, cif = (float)ci;
      float ssf, csf;
      sincosf((float)psi, &ssf, &csf);
      const float X0 = spf * csf - ssf * cpf * ctf, X1 = -(cpf * csf + ssf * spf * ctf), X2 = ssf * stf;
      const float Y0 = -spf * ssf - csf * cpf * ctf, Y1 = cpf * ssf - csf * spf * ctf, Y2 = stf * csf;
      const float mcs = (float)(src.x(0) * kMsunS);
      const float K = (float)kAmp0 * sqrtf(mcs) * cbrtf(mcs) * (float)(kC / kMpcM) / (float)src.x(4);
      const float ap = 0.5f * (1.0f + cif * cif);
      for (int det = 0; det < ev.n_det; ++det) {
        const float* xa = ev.xarm32[det];
        const float* ya = ev.yarm32[det];
        float xX = xa[0] * X0 + xa[1] * X1 + xa[2] * X2, xY = xa[0] * Y0 + xa[1] * Y1 + xa[2] * Y2;
        float yX = ya[0] * X0 + ya[1] * X1 + ya[2] * X2, yY = ya[0] * Y0 + ya[1] * Y1 + ya[2] * Y2;
        float fp = 0.5f * (xX * xX - xY * xY - yX * yX + yY * yY);
        float fc = xX * xY - yX * yY;
        float pr = fp * ap, pi_ = -fc * cif;
        p.kp_re[det] = (double)(K * pr);
        p.kp_im[det] = (double)(K * pi_);
        const double* r = ev.vertex[det];
        p.tau[det] = tc - (r[0] * n0 + r[1] * n1 + r[2] * n2) * (1.0 / kC);
      }
    } else {
      double ss, cs;
      sincos(psi, &ss, &cs);
      const double ap = 0.5 * (1.0 + ci * ci);
      for (int det = 0; det < ev.n_det; ++det) {
        double fp, fc, dt;
        detector_response(ev, det, sp, cp, sd, cd, ss, cs, &fp, &fc, &dt);
        s.pr[det] = fp * ap;
        s.pi[det] = -fc * ci;
        p.tau[det] = tc + dt;
      }
    }
  } else if (!LEAN) {
    // restricted amplitude K = sqrt(5/24) pi^(-2/3) (G Mc/c^3)^(5/6) / (d_L/c)
    const double mcs = src.x(0) * kMsunS;
    s.K = kAmp0 * sqrt(mcs) * cbrt(mcs) * kC / (src.x(4) * kMpcM);
  }
}

template <bool LEAN, int WF>
__device__ __noinline__ void f64_split_second(int part, const EventDev& ev, const SetupPart& s, WalkerParams& p) {
  const double al5 = 3.0 * s.a[5], al6 = -6848.0 / 21.0;
  if (part == 0) {
    p.C[0] = s.pre * s.ci5 * s.a[0];
    p.C[1] = s.pre * s.ci3 * s.a[2];
    p.C[2] = s.pre * s.ci2 * s.a[3];
    p.C[3] = s.pre * s.ci1 * s.a[4];
    p.C[5] = s.pre * s.c1 * s.c1 * s.a[7];
  } else if (part == 1) {
    p.C[4] = s.pre * s.c1 * (s.a[6] + al6 * s.lpm / 3.0);
    p.C[6] = s.pre * al5 / 3.0;
    p.C[7] = s.pre * s.c1 * al6 / 3.0;
  } else if (part == 2) {
    p.phase0 = s.pre * (s.a[5] + al5 * s.lpm / 3.0) - s.phic / kPi - 0.125;
    if (!LEAN) {
      for (int det = 0; det < ev.n_det; ++det) {
        p.kp_re[det] = s.K * s.pr[det];
        p.kp_im[det] = s.K * s.pi[det];
      }
    }
  } else {
    double hh = 0.0;
    if (WF == 0) {
      const int k_end = bins_below(ev.f_min, ev.df, ev.n_bins, s.fcut);
      p.k_end = k_end;
      for (int det = 0; det < ev.n_det; ++det) {
        const double psum = k_end > 0 ? ev.hh_prefix[(size_t)det * ev.n_bins + k_end - 1] : 0.0;
        // K ~ 1e-21: its square underflows FP32, so |K P|^2 is formed in FP64
        if (LEAN) hh += (p.kp_re[det] * p.kp_re[det] + p.kp_im[det] * p.kp_im[det]) * psum;
        else hh += s.K * s.K * (s.pr[det] * s.pr[det] + s.pi[det] * s.pi[det]) * psum;
      }
    } else {
      double a[8], al[8] = {0.0, 0.0, 0.0, 0.0, 0.0, al5, al6, 0.0};
      for (int k = 0; k < 8; ++k) a[k] = s.a[k];
      phenomd_extra<LEAN>(ev, p, p.pd, s.eta, s.delta, s.chis, s.chia, a, al, s.c1, s.lpm, s.q, s.chi1, s.chi2,
                          s.phic);
    }
    p.hh = hh;
  }
}

// Shared memory of a tile's first pass.
template <int PREC, int WF>
union TilePart {
  SetupPart d;
  std::conditional_t<PREC == 2, std::conditional_t<WF == 0, TF2Part, PDPart>, char> f;
  __device__ TilePart() {}
};

// The constants of the m <= 32 proposals v (UNIT: unit-cube points [m][D]; else physical vectors
// [m][11]) into P[0 .. m), by a CTA of 128 threads.  ok[i] = 0 leaves proposal i out (k_end 0).
// Ends with a barrier.
template <int PREC, int WF, bool UNIT>
__device__ void setup_tile(const EventDev& ev, const double* v, int m, const int* ok, TilePart<PREC, WF>* parts,
                           WalkerParams* P) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool mine = lane < m && ok[lane];
  const double* x = v + (size_t)lane * (UNIT ? ev.n_dim : kParams);
  if constexpr (PREC == 2 && UNIT) {
    if (ev.ff_setup) {
      if (mine) {
        ff xf[kMaxDim];
#pragma unroll
        for (int d = 0; d < kMaxDim; ++d) xf[d] = d < ev.n_dim ? ff_from_double(x[d]) : ff_make(0.0f);
        if constexpr (WF == 0) tf2_split_first(warp, ev, xf, parts[lane].f, P[lane]);
        else pd_split_first(warp, ev, xf, parts[lane].f, P[lane]);
      }
      __syncthreads();
      if (mine) {
        if constexpr (WF == 0) tf2_split_second(warp, ev, parts[lane].f, P[lane]);
        else pd_split_second(warp, ev, parts[lane].f, P[lane]);
      }
      if (warp == 0 && lane < m && !ok[lane]) P[lane].k_end = 0;
      __syncthreads();
      return;
    }
  }
  if (mine) f64_split_first<PREC != 0, UNIT>(warp, ev, x, parts[lane].d, P[lane]);
  __syncthreads();
  if (mine) f64_split_second<PREC != 0, WF>(warp, ev, parts[lane].d, P[lane]);
  if (warp == 0 && lane < m && !ok[lane]) P[lane].k_end = 0;
  __syncthreads();
  if (PREC == 2) {
    if (mine && warp == 0) make_ff<WF>(ev, P[lane]);
    __syncthreads();
  }
}

}  // namespace gwns
