// Reverse (adjoint) of one recombination step, FP64, tallies held fixed.
//
// Forward substep per cell (see rec_step.cu): T' from Eq. (Tb-evolution),
// alpha = alpha_e(T'), A = dt alpha n_H, s = dt w, and x' the backward-Euler
// root of A x'^2 + (1 + sG) x' - (x + sG) = 0 with G = (1-C) lambda + C beta e_a;
// lambda solves F(lambda) = sum alpha n^2 x'^2 - lambda sum n (1 - x') = 0;
// C depends on S_1s = sum Delta (1 - x) through R_alpha^mix; U' = U exp(-(kd x' + H) dt).
//
// Reverse, by the implicit-function theorem for lambda (no differentiation
// through Newton iterations):
//   mu  = -(sum_i xbar'_i dx'_i/dlambda) / (dF/dlambda)
//   y_i = xbar'_i + mu (2 alpha n^2 x' + lambda n)        (effective adjoint of x'_i)
//   then the chain through A, s, w, alpha(T'), T', Delta, x and the global sums.
// Passes (all on the context stream):
//   k_adj_prep      sums of the pre-step state (S_1s, tally total, lambda guess)
//   k_substep       recomputes lambda as the forward step does; its first
//                   evaluation keeps the cells' coefficients
//   k_adj_r1        mu numerator/denominator and X_e of the end state; keeps x'
//   k_adj_r2        per-cell adjoints; sums for the C and S_1s paths
//   k_adj_r3        the S_1s term applied to xbar and g_delta
// Every pass but the last is bound by the binary64 pipe (two operations per
// cycle and SM), so coefficients are computed once and read back (40 bytes per
// cell), and quotients by sums are taken of the sums.  256^3: 50.2 -> 18.7 ms per
// reversed step.  (Reciprocals shared between a cell's quotients: 14.5 ms, at 1 to 2 % more
// error in the gradients.)

#include <cmath>

#include "rec_internal.cuh"
#include "rec_reduce.cuh"

namespace rec {

namespace adj {

constexpr int NT = kPassThreads;

struct AdjArgs {
  int64_t n3;
  const double* delta;
  const double* x;
  const double* T;
  const double4_32a* U;
  const uint32_t* tally;
  double* xbar;
  double* Tbar;
  double4_32a* Ubar;
  double* g_delta;
  double* g_a;
  double Xe_bar;
  DevScalars* sc;
  double* part;
  StepCoef k;
  const double4_32a* cc;  // {alpha(T'), w, T', t^pd} kept by the first evaluation (NULL: recompute)
  double* xr;             // x' kept by R1 (with cc)
};

struct Fwd {
  double Tn, al, n, A, w, s, tpd, xr, D;
  bool wt;  // w from the tallies
};

// The forward step of a cell: coefficients (read back with KEPT), root x' and D = 2 A x' + B.
// ROOT: x' is computed (and kept with KEPT), otherwise read back.
template <bool KEPT, bool ROOT>
__device__ __forceinline__ Fwd forward_cell(const AdjArgs& a, int64_t i, double d, double x, double tot, double S1s,
                                            double G) {
  const StepCoef& k = a.k;
  Fwd f;
  const double n1s_rel = d * (1.0 - x);
  f.wt = k.mixing == REC_MIX_TALLY && tot > 0.0 && S1s > 0.0 && n1s_rel > 0.0;
  if (KEPT) {
    const double4_32a q = a.cc[i];
    f.al = q.x; f.w = q.y; f.Tn = q.z; f.tpd = q.w;
  } else {
    const double T = a.T[i];
    const double opx = 1.0 + k.fHe + x, g = k.kc * x / opx;
    f.Tn = (T + k.dt * (g * k.Tg + k.hq / (d * opx))) / (1.0 + k.dt * (2.0 * k.H + g));
    const double lt = log(f.Tn * 1.0e-4);
    f.tpd = exp(k.pd * lt);
    f.al = k.fa * exp(k.pb * lt) / (1.0 + k.pc * f.tpd);
    f.w = f.wt ? (double)(a.tally ? a.tally[i] : 0u) / tot * S1s / n1s_rel : 1.0;
  }
  f.n = k.nH * d;
  f.A = k.dt * f.al * f.n;
  f.s = k.dt * f.w;
  const double B = 1.0 + f.s * G;
  if (KEPT && !ROOT) {
    f.xr = a.xr[i];
  } else {
    const double cc = x + f.s * G;
    const double sq = sqrt(B * B + 4.0 * f.A * cc);
    f.xr = 2.0 * cc / (B + sq);
    if (KEPT) a.xr[i] = f.xr;
  }
  f.D = 2.0 * f.A * f.xr + B;
  return f;
}

// Incoming adjoint of x' with the X_e seed and the drag term folded in.
__device__ __forceinline__ double xbar_out(const AdjArgs& a, int64_t i, const Fwd& f, double d, double XeSd) {
  double xb = a.xbar[i] + XeSd * d;
  if (a.Ubar) {
    double4_32a ub = a.Ubar[i], u = a.U[i];
    double E = exp(-(a.k.kd * f.xr + a.k.H) * a.k.dt);
    double dot = (ub.x * u.x + ub.y * u.y + ub.z * u.z) * E;  // Ubar' . U'
    xb += -a.k.kd * a.k.dt * dot;
  }
  return xb;
}

// Sums of the pre-step state: S_1s, sum delta, tally total, and a lambda guess with
// alpha at the mean temperature (the evaluations converge from it as they do
// from the step before; a logarithm and two exponentials per cell are saved).
__global__ void __launch_bounds__(NT) k_adj_prep(AdjArgs a) {
  double v[5] = {0, 0, 0, 0, 0};
  unsigned long long tot = 0;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < a.n3; i += (int64_t)gridDim.x * NT) {
    const double d = a.delta[i], x = a.x[i];
    const double n1s = d * (1.0 - x), ne = d * x;
    v[0] += n1s;
    v[1] += d;
    tot += a.tally ? a.tally[i] : 0u;
    v[3] += ne * ne;
    v[4] += a.T[i];
  }
  v[2] = (double)tot;
  block_sum<5, NT>(v);
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; ++k) a.part[(size_t)blockIdx.x * kMaxSums + k] = v[k];
  if (!last_block_done(&a.sc->counter)) return;
  double S[5];
  combine_partials<5, NT>(a.part, gridDim.x, kMaxSums, S);
  if (threadIdx.x == 0) {
    const double lt = log(S[4] / (double)a.n3 * 1.0e-4);
    const double al = a.k.fa * exp(a.k.pb * lt) / (1.0 + a.k.pc * exp(a.k.pd * lt));
    a.sc->S1s = S[0];
    a.sc->Sd = S[1];
    a.sc->tally_total = (unsigned long long)(S[2] + 0.5);
    a.sc->lam_state = S[0] > 0.0 ? al * a.k.nH * S[3] / S[0] : 0.0;
    a.sc->lam_prev = -1.0;
    a.sc->flags &= 8;  // an expired wait stays until it is reported
    a.sc->counter = 0;
  }
}

// R1: numerator and denominator of mu, X_e of the end state.
template <bool KEPT>
__global__ void __launch_bounds__(NT) k_adj_r1(AdjArgs a) {
  DevScalars* sc = a.sc;
  const double lam = sc->lam, omC = sc->omC, G = omC * lam + sc->G0;
  const double tot = (double)sc->tally_total, S1s = sc->S1s, XeSd = a.Xe_bar / sc->Sd;
  double v[3] = {0, 0, 0};  // sum xbar' dx'/dlambda, dF/dlambda, sum delta x'
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < a.n3; i += (int64_t)gridDim.x * NT) {
    double d = a.delta[i];
    const Fwd f = forward_cell<KEPT, true>(a, i, d, a.x[i], tot, S1s, G);
    const double xb = xbar_out(a, i, f, d, XeSd);
    const double dxdl = f.s * (1.0 - f.xr) / f.D * omC;
    v[0] += xb * dxdl;
    v[1] += (2.0 * f.al * f.n * f.n * f.xr + lam * f.n) * dxdl - f.n * (1.0 - f.xr);
    v[2] += d * f.xr;
  }
  block_sum<3, NT>(v);
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; ++k) a.part[(size_t)blockIdx.x * kMaxSums + k] = v[k];
  if (!last_block_done(&sc->counter)) return;
  double S[3];
  combine_partials<3, NT>(a.part, gridDim.x, kMaxSums, S);
  if (threadIdx.x == 0) {
    sc->last_step = -S[0] / S[1];  // mu
    sc->Sdx = S[2];
    sc->counter = 0;
  }
}

// R2: per-cell adjoints (before the S_1s term); sums for the C and S_1s paths.
template <bool KEPT>
__global__ void __launch_bounds__(NT) k_adj_r2(AdjArgs a) {
  DevScalars* sc = a.sc;
  const double lam = sc->lam, omC = sc->omC, G = omC * lam + sc->G0;
  const double tot = (double)sc->tally_total, S1s = sc->S1s, XeSd = a.Xe_bar / sc->Sd;
  const double mu = sc->last_step, Xe1 = sc->Sdx / sc->Sd;
  const StepCoef& k = a.k;
  const double dGdC = k.beta * k.ea - lam;
  double v[2] = {0, 0};  // Cbar / dG/dC, S_1s times its direct adjoint through w
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < a.n3; i += (int64_t)gridDim.x * NT) {
    const double d = a.delta[i], x = a.x[i], y1 = 1.0 - x;
    const Fwd f = forward_cell<KEPT, false>(a, i, d, x, tot, S1s, G);
    const double xb1 = xbar_out(a, i, f, d, XeSd);
    const double an2 = f.al * f.n * f.n, yr = 1.0 - f.xr;
    const double y = xb1 + mu * (2.0 * an2 * f.xr + lam * f.n);
    // partials of x': the common factor y / D
    const double yD = y / f.D;
    const double Ab = -yD * f.xr * f.xr;
    const double sb = yD * G * yr;
    double xbar = yD;
    v[0] += yD * f.s * yr;
    // explicit dependence of F on alpha and n, then A = dt alpha n
    const double alb = mu * f.n * f.n * f.xr * f.xr + Ab * k.dt * f.n;
    const double nb = mu * (2.0 * f.al * f.n * f.xr * f.xr - lam * yr) + Ab * k.dt * f.al;
    // s = dt w
    const double wb = sb * k.dt;
    double db = nb * k.nH;
    double ab = 0.0;
    if (f.wt) {
      const double ww = wb * f.w;
      ab = wb * S1s / (d * y1);
      v[1] += ww;
      db -= ww / d;
      xbar += ww / y1;
    }
    // alpha(T'): d alpha/dT' = (alpha/T') (pb - pc pd t^pd / (1 + pc t^pd))
    const double dal = f.al / f.Tn * (k.pb - k.pc * k.pd * f.tpd / (1.0 + k.pc * f.tpd));
    const double Tnb = a.Tbar[i] + alb * dal;
    // T' = (T + dt (g Tg + hh)) / den
    const double opx = 1.0 + k.fHe + x;
    const double g = k.kc * x / opx;
    const double Tb = Tnb / (1.0 + k.dt * (2.0 * k.H + g));
    const double hhb = Tb * k.dt;
    const double gb = hhb * (k.Tg - f.Tn);
    xbar += gb * k.kc * (1.0 + k.fHe) / (opx * opx);
    if (k.hq != 0.0) {
      const double hh = k.hq / (d * opx);
      db -= hhb * hh / d;
      xbar -= hhb * hh / opx;
    }
    // X_e of the end state: d/d delta_i of sum(delta x')/sum(delta)
    db += XeSd * (f.xr - Xe1);
    if (a.Ubar) {
      double E = exp(-(k.kd * f.xr + k.H) * k.dt);
      double4_32a ub = a.Ubar[i];
      ub.x *= E; ub.y *= E; ub.z *= E;
      a.Ubar[i] = ub;
    }
    a.xbar[i] = xbar;
    a.Tbar[i] = Tb;
    a.g_delta[i] += db;
    if (a.g_a) a.g_a[i] += ab;
  }
  block_sum<2, NT>(v);
  if (threadIdx.x == 0)
    for (int q = 0; q < 2; ++q) a.part[(size_t)blockIdx.x * kMaxSums + q] = v[q];
  if (!last_block_done(&sc->counter)) return;
  double S[2];
  combine_partials<2, NT>(a.part, gridDim.x, kMaxSums, S);
  if (threadIdx.x == 0) {
    // C = (L + R)/(beta + L + R), R = KR n3 / (nH S_1s): dC/dS = beta/(beta+L+R)^2 * (-R/S)
    double R = k.KR * (double)a.n3 / (k.nH * S1s);
    double den = k.beta + k.L2g + R;
    double dCdS = k.beta / (den * den) * (-R / S1s);
    sc->Sdx = S[0] * dGdC * dCdS + (S[1] != 0.0 ? S[1] / S1s : 0.0);  // adjoint of S_1s
    sc->counter = 0;
  }
}

// R3: S_1s = sum delta (1 - x) pulls the S_1s adjoint back to x and delta.
__global__ void __launch_bounds__(NT) k_adj_r3(AdjArgs a) {
  const double Sb = a.sc->Sdx;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < a.n3; i += (int64_t)gridDim.x * NT) {
    double d = a.delta[i], x = a.x[i];
    a.xbar[i] += -Sb * d;
    a.g_delta[i] += Sb * (1.0 - x);
  }
}

// X_e adjoint at a node: X_e = sum(delta x)/sum(delta).
__global__ void __launch_bounds__(NT) k_xe_sum(const double* delta, const double* x, int64_t n3, DevScalars* sc,
                                               double* part) {
  double v[2] = {0, 0};
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n3; i += (int64_t)gridDim.x * NT) {
    v[0] += delta[i] * x[i];
    v[1] += delta[i];
  }
  block_sum<2, NT>(v);
  if (threadIdx.x == 0)
    for (int q = 0; q < 2; ++q) part[(size_t)blockIdx.x * kMaxSums + q] = v[q];
  if (!last_block_done(&sc->counter)) return;
  double S[2];
  combine_partials<2, NT>(part, gridDim.x, kMaxSums, S);
  if (threadIdx.x == 0) {
    sc->Sdx = S[0];
    sc->Sd = S[1];
    sc->counter = 0;
  }
}

__global__ void __launch_bounds__(NT) k_xe_apply(const double* delta, const double* x, int64_t n3, DevScalars* sc,
                                                 double Xe_bar, double* xbar, double* g_delta) {
  const double Sd = sc->Sd, Xe = sc->Sdx / Sd;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n3; i += (int64_t)gridDim.x * NT) {
    xbar[i] += Xe_bar * delta[i] / Sd;
    g_delta[i] += Xe_bar * (x[i] - Xe) / Sd;
  }
}

}  // namespace adj

cudaError_t launch_rec_step_adjoint(rec_ctx* c, double z_from, double z_to, const double* x_in, const double* T_in,
                                    const double* vel4_in, const uint32_t* tally_in, double* xbar, double* Tbar,
                                    double* Ubar, double* g_delta, double* g_a, double Xe_bar_out) {
  StepCoef k = step_coef(c->cosmo, c->params, z_from, z_to, 1);
  adj::AdjArgs a;
  a.n3 = c->n3;
  a.delta = (const double*)c->box.delta;
  a.x = x_in;
  a.T = T_in;
  a.U = (const double4_32a*)vel4_in;
  a.tally = tally_in;
  a.xbar = xbar;
  a.Tbar = Tbar;
  a.Ubar = (double4_32a*)Ubar;
  a.g_delta = g_delta;
  a.g_a = g_a;
  a.Xe_bar = Xe_bar_out;
  a.sc = c->sc_adj;
  a.part = c->part;
  a.k = k;
  a.cc = (const double4_32a*)c->cellcache;
  a.xr = a.cc ? (double*)c->cellcache + 4 * c->n3 : nullptr;
  GroupTimer t(c, kTAdj, 5);
  adj::k_adj_prep<<<c->grid, adj::NT, 0, c->stream>>>(a);
  cudaError_t e = enqueue_newton_passes(c, c->sc_adj, k, x_in, T_in, tally_in);
  if (e != cudaSuccess) return e;
  if (a.cc) {
    adj::k_adj_r1<true><<<c->grid, adj::NT, 0, c->stream>>>(a);
    adj::k_adj_r2<true><<<c->grid, adj::NT, 0, c->stream>>>(a);
  } else {
    adj::k_adj_r1<false><<<c->grid, adj::NT, 0, c->stream>>>(a);
    adj::k_adj_r2<false><<<c->grid, adj::NT, 0, c->stream>>>(a);
  }
  adj::k_adj_r3<<<c->grid, adj::NT, 0, c->stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_xe_adjoint(rec_ctx* c, const double* x, double Xe_bar, double* xbar, double* g_delta) {
  const double* delta = (const double*)c->box.delta;
  GroupTimer t(c, kTOther, 2);
  adj::k_xe_sum<<<c->grid, adj::NT, 0, c->stream>>>(delta, x, c->n3, c->sc_adj, c->part);
  adj::k_xe_apply<<<c->grid, adj::NT, 0, c->stream>>>(delta, x, c->n3, c->sc_adj, Xe_bar, xbar, g_delta);
  return cudaGetLastError();
}

}  // namespace rec
