// Per-cell proximal map of tau*phi (Sec. 3), fused with the dual lift
// x = C^T z, the primal step y - tau x, the extrapolation
// ybar = y_new + theta (y_new - y) and the step-size update of Sec. 5.
//
// The paper takes prox_{tau phi_ij} from its reference (BAKS, Cor. 3.1) without
// printing it.  For q' = 2 the first-order conditions give, with
// P = P_K(w_bar) (projection onto the cone K of Sec. 2):
//   w = m/(m + tau) P,
//   h(m) = m - m_bar + tau f_eff(m) - tau |P|^2 / (2 (m + tau)^2) = 0,
// h strictly increasing (f_eff nondecreasing); m = 0, w = 0 when h(0) >= 0,
// otherwise the root lies in (0, m_hi], m_hi = max(0, m_bar - tau f_eff(0)) +
// |P|^2/(2 tau).  f_eff(m) = f_a m + f_b m^2 + V(x), plus (g_a m + W(x))/dt on
// the last plane (G weighted by 1/dt in calF, Sec. 2).
//
// Root finder: Newton from m = 0 with the bracket [lo, hi] kept by the sign of
// h and a bisection step whenever Newton leaves it (for f_b = 0, h is concave
// and Newton from the left never does); see prox_cell for the precision split.
#include <algorithm>

#include "df64.cuh"
#include "mfg_internal.cuh"
#include "reduce.cuh"

namespace mfg {

// Safeguarded Newton on h in FP32, from x = 0 with the bracket [0, hi].
__device__ __forceinline__ float newton_h32(float hi, float B, float hP, float tau, float a1, float tb) {
  float x = 0.0f, lo = 0.0f;
  for (int it = 0; it < 24; ++it) {
    const float it1 = 1.0f / (x + tau);
    const float it2 = it1 * it1;
    const float hx = fmaf(tb, x * x, a1 * x) - B - hP * it2;
    if (hx < 0.0f) lo = x; else hi = x;
    if (hx == 0.0f) break;
    const float dh = fmaf(2.0f * tb, x, a1) + 2.0f * hP * it2 * it1;
    float xn = x - hx / dh;
    if (!(xn >= lo && xn <= hi)) xn = 0.5f * (lo + hi);
    const float dxv = fabsf(xn - x);
    x = xn;
    if (dxv <= 2e-7f * x || hi - lo <= 2e-7f * hi) break;
  }
  return x;
}

// FP64 Newton on h from x = 0 with bisection safeguard: the path for inputs
// outside the FP32 range of the fast path.
// A NaN in the cell's data (m_bar, the fluxes, V, W or the dual) comes out as
// NaN rather than as a bracketed root, so the CP step norm reports it.
__device__ __noinline__ double newton_h64(double B, double hP, double tau, double a1, double tb, double hi) {
  if (isnan(B) || isnan(hP)) return __longlong_as_double(0x7ff8000000000000LL);
  double x = 0.0, lo = 0.0;
  for (int it = 0; it < 200; ++it) {
    const double it1 = 1.0 / (x + tau);
    const double it2 = it1 * it1;
    const double hx = fma(tb, x * x, a1 * x) - B - hP * it2;
    if (hx < 0.0) lo = x; else hi = x;
    if (hx == 0.0) break;
    const double dh = fma(2.0 * tb, x, a1) + 2.0 * hP * it2 * it1;
    double xn = x - hx / dh;
    if (!(xn >= lo && xn <= hi)) xn = 0.5 * (lo + hi);
    const double dxv = fabs(xn - x);
    x = xn;
    if (dxv <= 1e-16 * x || hi - lo <= 4e-16 * hi) break;
  }
  return x;
}

// A whole cell on that path, zero test included (out of line, so that its divisions
// are no predicated instructions of the fast path): the root and w = (.).y P.
__device__ __noinline__ double2 cell_h64(double B, double P2, double tau, double half_itau, double a1, double tb) {
  if (B + P2 * half_itau <= 0.0) return make_double2(0.0, 0.0);
  const double x = newton_h64(B, 0.5 * tau * P2, tau, a1, tb, fmax(B, 0.0) + P2 * half_itau);
  return make_double2(x, x / (x + tau));
}

// Prox for the general power Hamiltonian |p|^{q'}/q', q = q'/(q'-1), b_hat =
// |w|^q/(q m^{q-1}) (Sec. 2).  For fixed m > 0 the minimising flux is
// w = m t P/|P| with t >= 0 the root of g(t) = m t + tau t^{q-1} - |P|, and m
// is the root of the increasing function
//   h_q(m) = a1 m + tau b m^2 - B - (tau/q') t(m)^q,
// h_q'(m) = a1 + 2 tau b m + tau (q-1) t^q / (m + tau (q-1) t^{q-2}),
// with (0, 0) the prox when h_q(0) = -B - (tau/q') (|P|/tau)^{q'} >= 0 and the
// root in (0, max(0, B) + (tau/q') (|P|/tau)^{q'}] otherwise.  velocity_q: t(m)
// by safeguarded FP64 Newton (the bracket kept by the sign, a bisection step
// whenever Newton leaves it).  q' = 2 never takes this path.
__device__ double velocity_q(double m, double Pn, double tau, double q) {
  double lo = 0.0, hi = fmin(Pn / m, pow(Pn / tau, 1.0 / (q - 1.0)));
  double t = hi;
  for (int it = 0; it < 200; ++it) {
    const double tq2 = pow(t, q - 2.0);
    const double gt = m * t + tau * tq2 * t - Pn;
    if (gt < 0.0) lo = t; else hi = t;
    if (gt == 0.0 || hi - lo <= 4e-16 * hi) break;
    const double dg = m + tau * (q - 1.0) * tq2;
    double tn = t - gt / dg;
    if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);
    const double step = fabs(tn - t);
    t = tn;
    if (step <= 1e-16 * t) break;
  }
  return t;
}

// Root of the two equations above by nested FP64 Newton: m outside, t(m) inside
// (tens of FP64 pow per cell).  Only for inputs the paired iteration below
// gives up on.  Returns m and t; lim = (tau/q') (|P|/tau)^{q'}.
__device__ __noinline__ double2 root_q64(double B, double Pn, double tau, double qp, double a1, double tb, double lim) {
  const double q = qp / (qp - 1.0);
  double lo = 0.0, hi = fmax(B, 0.0) + lim;
  double x = 0.5 * hi, t = 0.0;
  for (int it = 0; it < 200; ++it) {
    t = Pn > 0.0 ? velocity_q(x, Pn, tau, q) : 0.0;
    const double tq = pow(t, q);
    const double hx = fma(tb, x * x, a1 * x) - B - (tau / qp) * tq;
    if (hx < 0.0) lo = x; else hi = x;
    if (hx == 0.0 || hi - lo <= 4e-16 * hi) break;
    const double dh = fma(2.0 * tb, x, a1) + (Pn > 0.0 ? tau * (q - 1.0) * tq / (x + tau * (q - 1.0) * pow(t, q - 2.0)) : 0.0);
    double xn = x - hx / dh;
    if (!(xn > lo && xn < hi)) xn = 0.5 * (lo + hi);
    const double step = fabs(xn - x);
    x = xn;
    if (step <= 1e-16 * x) break;
  }
  t = Pn > 0.0 ? velocity_q(x, Pn, tau, q) : 0.0;
  return make_double2(x, t);
}

// t^e for the exponent e = q - 2 shared by all cells: multiples of 1/2 up to 4
// by products and one square root, others by pow.
__device__ __forceinline__ double pow_q2(double t, double e) {
  const double e2 = 2.0 * fabs(e);
  const int k = (int)e2;
  if (e2 != (double)k || k > 8) return pow(t, e);
  double r = (k & 1) ? sqrt(t) : 1.0;
  for (int i = 0; i < (k >> 1); ++i) r *= t;
  return e < 0.0 ? 1.0 / r : r;
}

// FP32 root of the pair in the single unknown s = 1/t: from g = 0, m(s) = |P| s -
// tau s^{2-q}, and F(s) = h_q(m(s)) increases from F(1/t0) < 0 (m = 0).  s lies
// below max(2 m_hi/|P|, s0 2^{1/(q-1)}): one of the two terms of s = m/|P| + (tau/|P|)
// s^{2-q} is at least s/2.  Safeguarded Newton, one powf per step.
__device__ __forceinline__ float2 root_q32(float B, float Pn, float tau, float q, float a1, float tb, float lim,
                                           float s0) {
  const float cq = tau * (q - 1.0f) / q;  // tau / q'
  float lo = s0, hi = fmaxf(2.0f * (fmaxf(B, 0.0f) + lim) / Pn, s0 * exp2f(1.0f / (q - 1.0f)));
  float s = lo, m = 0.0f;
  for (int it = 0; it < 40; ++it) {
    const float u = powf(s, 2.0f - q), is = 1.0f / s;
    m = fmaf(Pn, s, -tau * u);
    const float sq = u * is * is;  // s^{-q}
    const float F = fmaf(fmaf(tb, m, a1), m, -B) - cq * sq;
    if (F < 0.0f) lo = s; else hi = s;
    if (F == 0.0f) break;
    const float dF = fmaf(2.0f * tb, m, a1) * fmaf(tau * (q - 2.0f), u * is, Pn) + tau * (q - 1.0f) * sq * is;
    float sn = s - F / dF;
    if (!(sn >= lo && sn <= hi)) sn = 0.5f * (lo + hi);
    const float ds = fabsf(sn - s);
    s = sn;
    if (ds <= 3e-7f * s) break;
  }
  return make_float2(fmaxf(m, 0.0f), 1.0f / s);
}

// One cell of the general map.  What bounds it is FP64 pow: nested Newton on m
// and t takes ~100 of them per cell.  Here the pair (m, t) is found in FP32 and
// then corrected together by Newton steps on
//   m t + tau t^{q-1} = |P|,   a1 m + tau b m^2 - B = (tau/q') t^q,
// residuals in FP64 (one t^{q-2} each), the 2 x 2 system in FP32: a step leaves
// ~1e-6 of the error, so two or three steps reach FP64 round-off (the same
// residuals vanish as in the nested iteration).  Steps that do not settle, and
// data outside the FP32 range, take root_q64.  mfg_prox, q' = 1.5, 120 x 96 x 40:
// 110.1 ms -> 0.133 ms (error against 64-bit bisection 1.7e-16 -> 1.4e-16).
template <int NW>
__device__ void prox_cell_q(double mbar, const double (&wbar)[NW], double tau, double qp, double a1, double tb,
                            double c, double& m, double (&w)[NW]) {
  const double q = qp / (qp - 1.0);
  double P[NW];
  double P2 = 0.0;
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    const bool neg = __double_as_longlong(wbar[k]) < 0;
    P[k] = ((k & 1) ? neg : !neg) ? wbar[k] : 0.0;
    P2 = fma(P[k], P[k], P2);
  }
  const double Pn = sqrt(P2);
  const double B = fma(-tau, c, mbar);
  if (isnan(B) || isnan(Pn)) {  // NaN in, NaN out (the CP step norm reports it)
    m = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
    for (int k = 0; k < NW; ++k) w[k] = m;
    return;
  }
  // h_q(0) = -B - lim decides between (0, 0) and a root; FP32 settles it unless
  // the two are within 1e-4 of each other
  const float Pf = (float)Pn, Bf = (float)B, tauf = (float)tau, qf = (float)q;
  const float r0 = Pf / tauf, limf = tauf / (float)qp * powf(r0, (float)qp);
  const float s0 = powf(r0, -1.0f / (qf - 1.0f));
  const bool f32 = Pf > 1e-12f && Pf < 1e12f && tauf > 1e-9f && tauf < 1e9f && fabsf(Bf) < 1e12f && limf > 1e-20f &&
                   limf < 1e15f && s0 > 1e-12f && s0 < 1e12f;
  double lim = 0.0;
  bool zero;
  if (!(Pn > 0.0)) {
    zero = B <= 0.0;
  } else if (f32 && fabsf(Bf + limf) > 1e-4f * limf) {
    zero = Bf + limf < 0.0f;
  } else {
    lim = (tau / qp) * pow(Pn / tau, qp);
    zero = -B - lim >= 0.0;
  }
  if (zero) {
    m = 0.0;
#pragma unroll
    for (int k = 0; k < NW; ++k) w[k] = 0.0;
    return;
  }
  double x, t;
  bool ok = false;
  if (!(Pn > 0.0)) {  // a1 m + tau b m^2 = B, t = 0
    t = 0.0;
    x = tb > 0.0 ? 2.0 * B / (a1 + sqrt(fma(4.0 * tb, B, a1 * a1))) : B / a1;
    ok = isfinite(x);
  } else if (f32) {
    const float2 g0 = root_q32(Bf, Pf, tauf, qf, (float)a1, (float)tb, limf, s0);
    x = g0.x;
    t = g0.y;
    const double cq = tau / qp;
    const float eq = (float)(tau * (q - 1.0)), a1f = (float)a1, tb2f = (float)(2.0 * tb);
    for (int it = 0; it < 8 && !ok; ++it) {
      const double tq2 = pow_q2(t, q - 2.0), tq1 = tq2 * t;
      const float rg = (float)(fma(x, t, fma(tau, tq1, -Pn)));
      const float rh = (float)(fma(fma(tb, x, a1), x, -B) - cq * tq1 * t);
      const float xf = (float)x, tf = (float)t, D = fmaf(eq, (float)tq2, xf), H = fmaf(tb2f, xf, a1f),
                  E = eq * (float)tq1;
      const float id = -1.0f / fmaf(tf, E, D * H);
      const float dx = fmaf(rg, E, D * rh) * id, dt = fmaf(H, rg, -tf * rh) * id;
      x += (double)dx;
      t += (double)dt;
      if (!(x > 0.0 && t > 0.0)) break;
      ok = fabsf(dx) <= 1e-9f * (float)x && fabsf(dt) <= 1e-9f * (float)t;
    }
  }
  if (!ok) {
    if (lim == 0.0) lim = (tau / qp) * pow(Pn / tau, qp);
    const double2 g = root_q64(B, Pn, tau, qp, a1, tb, lim);
    x = g.x;
    t = g.y;
  }
  m = x;
  const double s = Pn > 0.0 ? x * t / Pn : 0.0;
#pragma unroll
  for (int k = 0; k < NW; ++k) w[k] = s * P[k];
}

// Per-step constants of the prox (tau is the CP primal step).
struct ProxK {
  double tau, tau2, half_tau, half_itau, tb;  // tau, tau^2, tau/2, 1/(2 tau), tau f_b
  float tauf, tbf, itau2f;                    // itau2f = 1/tau^2
  df taud, tbd;                         // tau, tau f_b as double-float pairs
  bool tau_ok;                          // tau inside the FP32 fast-path range
};

__device__ __forceinline__ ProxK prox_consts(double tau, double half_itau, double f_b) {
  ProxK k;
  k.tau = tau;
  k.tau2 = tau * tau;
  k.half_tau = 0.5 * tau;
  k.half_itau = half_itau;
  k.tb = tau * f_b;
  k.tauf = (float)tau;
  k.tbf = (float)k.tb;
  k.itau2f = (float)(4.0 * half_itau * half_itau);
  k.taud = df_from_double(tau);
  k.tbd = df_from_double(k.tb);
  k.tau_ok = tau > 1e-15 && tau < 1e15;
  return k;
}

// Root of h(m) = a1 m + tau b m^2 - B - hP/(m + tau)^2 with a1 = 1 + tau a,
// B = m_bar - tau c and hP = tau |P|^2 / 2 (the scalar equation above, with
// the FP64 constants combined before any rounding), then w = m/(m + tau) P.
// FP64 issues at 1/64 of the FP32 rate on GB300, so the root is found in FP32
// and polished in double-float arithmetic (df64.cuh, ~48 bits) by Newton
// steps on
//   g(m) = h(m) (m + tau)^2 = (a1 m + tau b m^2 - B) (m + tau)^2 - hP,
// which has the sign of h (the bracket stays valid) and needs no reciprocal;
// g' = (a1 + 2 tau b m)(m + tau)^2 + 2 (a1 m + tau b m^2 - B)(m + tau) > 0 near
// the root (there a1 m + tau b m^2 - B = hP/(m + tau)^2 >= 0) and is taken in
// FP32, so each step shrinks the error by ~1e-7 (plus the quadratic term):
// from an FP32 root two steps reach the double-float resolution.  The polish
// stops after a step below 1e-9 relative and keeps the bracket, bisecting if
// a step leaves it.  Inputs outside the FP32 range take an FP64 Newton.
// (FP64 issue bounds the prox, so the set-up takes as few FP64 instructions as it
// can: sign and zero tests on bit patterns, the bracket in FP32, all FP32 values
// from the double-float splits.)
template <int NW>
__device__ __forceinline__ void prox_cell(double mbar, const double (&wbar)[NW], const ProxK& K, double a1,
                                          float a1f, const df& a1d, double c, double& m, double (&w)[NW]) {
  // projection onto K by sign tests on the bit patterns (no FP64 min/max)
  double P[NW];
  double P2 = 0.0;
#pragma unroll
  for (int q = 0; q < NW; ++q) {
    const bool neg = __double_as_longlong(wbar[q]) < 0;
    P[q] = ((q & 1) ? neg : !neg) ? wbar[q] : 0.0;
    P2 = fma(P[q], P[q], P2);
  }
  const double B = fma(-K.tau, c, mbar);
  const double hP = K.half_tau * P2;
  // h(0) = -B - |P|^2/(2 tau) >= 0, as the sign of tau^2 B + hP; a NaN is not a zero
  // cell (a tau whose square leaves the range takes cell_h64 below)
  const double zt = fma(B, K.tau2, hP);
  const unsigned zh = (unsigned)__double2hiint(zt), zl = (unsigned)__double2loint(zt), za = zh & 0x7FFFFFFFu;
  const bool znan = za > 0x7FF00000u || (za == 0x7FF00000u && zl != 0u);
  if (K.tau_ok && (((zh >> 31) && !znan) || (za | zl) == 0u)) {
    m = 0.0;
#pragma unroll
    for (int q = 0; q < NW; ++q) w[q] = 0.0;
    return;
  }
  const df Bd = df_from_double(B), hPd = df_from_double(hP);
  const float Bf = Bd.hi, hPf = hPd.hi;
  // upper end of the bracket, max(0, B) + |P|^2/(2 tau), a little above its FP32 value
  const float hif = (fmaxf(Bf, 0.0f) + hPf * K.itau2f) * 1.000001f;
  const bool fp32_ok = K.tau_ok && hif < 1e15f && hPf < 1e30f && fabsf(Bf) < 1e30f;
  if (!fp32_ok) {
    const double2 xs = cell_h64(B, P2, K.tau, K.half_itau, a1, K.tb);
    m = xs.x;
#pragma unroll
    for (int q = 0; q < NW; ++q) w[q] = xs.y * P[q];
    return;
  }
  df lo{0.0f, 0.0f}, hi{hif, 0.0f};
  df x{newton_h32(hif, Bf, hPf, K.tauf, a1f, K.tbf), 0.0f};
  for (int it = 0; it < 100; ++it) {
    const df t = df_add_same(x, K.taud);
    const df t2 = df_mul(t, t);
    const df u = df_add_same(df_mul(K.tbd, x), a1d);  // a1 + tau b x
    const df v = df_sub(df_mul(u, x), Bd);            // a1 x + tau b x^2 - B
    const df gx = df_sub(df_mul(v, t2), hPd);
    if (gx.hi < 0.0f) lo = x; else hi = x;
    if (gx.hi == 0.0f) break;
    const float dg = fmaf(fmaf(2.0f * K.tbf, x.hi, a1f), t2.hi, 2.0f * v.hi * t.hi);
    const float dx = __fdiv_rn(gx.hi, dg);
    const df xn = df_add_f(x, -dx);
    if (df_le(lo, xn) && df_le(xn, hi)) {
      x = xn;
      if (fabsf(dx) <= 1e-9f * x.hi) break;
    } else {
      const df mid = df_add_same(lo, hi);
      x = df{0.5f * mid.hi, 0.5f * mid.lo};
      if (df_sub(hi, lo).hi <= 1e-14f * hi.hi) break;
    }
  }
  // s = x / (x + tau): FP32 reciprocal refined once in double-float
  const df t = df_add_same(x, K.taud);
  const float r0 = __frcp_rn(t.hi);
  const df e = df_sub(df{1.0f, 0.0f}, df_mul(t, df{r0, 0.0f}));  // 1 - t r0, ~1e-7
  const df r = df_add_f(df{r0 * e.hi, 0.0f}, r0);                // r0 (1 + e)
  m = df_to_double(x);
  const double s = df_to_double(df_mul(x, r));
#pragma unroll
  for (int q = 0; q < NW; ++q) w[q] = s * P[q];
}

// End of a CP step: acc = this thread's share of ||m_{l+1} - m_l||^2; the last
// block updates the step sizes and decides whether the loop goes on.
__device__ __forceinline__ void prox_tail(double acc, double tau, double theta, double gamma, double* partials,
                                          DevScalars* sc, cudaGraphConditionalHandle h, int use_handle) {
  double part[1] = {acc};
  block_sum<1>(part);
  if (!publish_and_check_last<1>(part, partials, &sc->counter)) return;
  double tot[1];
  gather_partials<1>(partials, tot);
  if (flat_tid() == 0) {
    const double r = sqrt(tot[0]);
    sc->dm2 = tot[0];
    sc->r_last = r;
    const double tau_next = theta * tau;
    sc->tau = tau_next;
    sc->sigma = sc->sigma / theta;
    sc->theta = 1.0 / sqrt(1.0 + 2.0 * gamma * tau_next);
    sc->half_itau = 0.5 / tau_next;
    sc->ell += 1;
    sc->cp_iters += 1;
    sc->cg_total += sc->cg_it;
    if (sc->cg_it > sc->cg_max) sc->cg_max = sc->cg_it;
    sc->cp_left -= 1;
    if (!isfinite(r)) {
      sc->status = MFG_ERR_NONFINITE;
      sc->cp_done = 1;
    }
    // a non-finite value or a timed-out device wait ends the instance's solve
    if (sc->status == MFG_ERR_NONFINITE || sc->status == MFG_ERR_TIMEOUT) sc->cp_done = 1;
    if (sc->cp_tol > 0.0 && r <= sc->cp_tol) sc->cp_done = 1;
    if (use_handle) cudaGraphSetConditional(h, (sc->cp_left > 0 && !sc->cp_done) ? 1u : 0u);
    sc->counter = 0;
  }
}

// y, ybar hold c planes; z one plane set.  Cell e pairs (m^{k+1}, w^k).
// The lift x = C^T z is formed from the four one-sided differences of z, which
// serve both the fluxes (x_w = D^T-type differences / dx) and
//   K z = ax ((z - zE) - (zW - z)) + ay ((z - zN) - (zS - z));
// on a Neumann axis the neighbour index of an end point is the point itself,
// so the difference across the end (a flux slot of Sec. 4.3 that does not
// exist) is zero and K takes its one-sided form.  VN (viscosity field): nu K z
// becomes K_nu z = kf_yp dyp - kf_ym dym (+ x terms), the face coefficients of
// Geom::kfx / kfy.  Point by point: a walk in warp strips forms each difference of z
// once, but issues a row's loads only behind the previous row's roots, and was slower
// at every width and occupation (256^2 x 128 755 us point by point, 934 us in strips;
// 512 x 20 x 200 202, 373 us; 4000 x 250 in 1-D 77, 136 us).
template <int ACTX, bool GENQ, bool VN>
__global__ void __launch_bounds__(kThreads) k_prox_cp(Geom g, Coef cf, const double* __restrict__ z,
                                                      double* __restrict__ y, double* __restrict__ ybar,
                                                      const double* __restrict__ V,
                                                      const double* __restrict__ W, double* partials,
                                                      DevScalars* sc, cudaGraphConditionalHandle h,
                                                      int use_handle, double* __restrict__ Az,
                                                      const double* __restrict__ rfin) {
  dep_sync();
  constexpr int NW = ACTX ? 4 : 2;
  const long long n = g.n;
  const double tau = sc->tau, theta = sc->theta;
  const ProxK K = prox_consts(tau, sc->half_itau, cf.f_b);
  const double t_nu = tau * g.nu, t_idt = tau * g.idt, t_idx = tau * g.idx, t_idy = tau * g.idy;
  const double a1_in = fma(tau, cf.f_a, 1.0), a1_last = fma(tau, fma(cf.g_a, g.idt, cf.f_a), 1.0);
  const float a1f_in = (float)a1_in, a1f_last = (float)a1_last;
  const df a1d_in = df_from_double(a1_in), a1d_last = df_from_double(a1_last);
  double acc = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e % g.ny);
    const long long t = e / g.ny;
    const int i = (int)(t % g.nx);
    const int k = (int)(t / g.nx);
    const long long base = (long long)k * g.S;
    const long long rowi = base + (long long)i * g.ny;
    const int jm = j == 0 ? (g.pery ? g.ny - 1 : 0) : j - 1;
    const int jp = j == g.ny - 1 ? (g.pery ? 0 : g.ny - 1) : j + 1;
    const double zc = z[e];
    if (Az != nullptr) Az[e] -= rfin[e];  // AAt z_{l+1} = b - r_final (stop reference)
    const double dyp = zc - z[rowi + jp], dym = z[rowi + jm] - zc;
    const long long f0 = (long long)i * g.ny;
    double Kz = VN ? fma(g.kfy[f0 + j], dyp, -g.kfy[f0 + jm] * dym) : g.ay * (dyp - dym);
    double d[NW];
    if (ACTX) {
      const int im = i == 0 ? (g.perx ? g.nx - 1 : 0) : i - 1;
      const int ip = i == g.nx - 1 ? (g.perx ? 0 : g.nx - 1) : i + 1;
      const double dxp = zc - z[base + (long long)ip * g.ny + j], dxm = z[base + (long long)im * g.ny + j] - zc;
      if (VN)
        Kz = fma(g.kfx[f0 + j], dxp, fma(-g.kfx[(long long)im * g.ny + j], dxm, Kz));
      else
        Kz = fma(g.ax, dxp - dxm, Kz);
      d[0] = dxp; d[1] = dxm; d[2] = dyp; d[3] = dym;
    } else {
      d[0] = dyp; d[1] = dym;
    }
    const double zn = (k + 1 < g.nt) ? z[e + g.S] : 0.0;
    // primal step y - tau x, x_m = nu K z + (z - z_next)/dt, x_w = d / dx
    const double m_old = y[e];
    const double mbar = fma(VN ? -tau : -t_nu, Kz, fma(-t_idt, zc - zn, m_old));
    double w_old[NW], wbar[NW], w_new[NW];
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      w_old[q] = y[e + (q + 1) * n];
      wbar[q] = fma(-((ACTX && q < 2) ? t_idx : t_idy), d[q], w_old[q]);
    }
    const bool last = (k == g.nt - 1);
    const long long f = (long long)i * g.ny + j;
    const double cc = last ? fma(W[f], g.idt, V[f]) : V[f];
    double m_new;
    if constexpr (GENQ)
      prox_cell_q<NW>(mbar, wbar, tau, cf.qprime, last ? a1_last : a1_in, K.tb, cc, m_new, w_new);
    else
      prox_cell<NW>(mbar, wbar, K, last ? a1_last : a1_in, last ? a1f_last : a1f_in, last ? a1d_last : a1d_in, cc,
                    m_new, w_new);
    const double dm = m_new - m_old;
    y[e] = m_new;
    ybar[e] = fma(theta, dm, m_new);
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      y[e + (q + 1) * n] = w_new[q];
      ybar[e + (q + 1) * n] = fma(theta, w_new[q] - w_old[q], w_new[q]);
    }
    acc = fma(dm, dm, acc);
  }
  prox_tail(acc, tau, theta, cf.gamma, partials, sc, h, use_handle);
}

template <int ACTX, bool GENQ>
__global__ void __launch_bounds__(kThreads) k_prox_plain(Geom g, Coef cf, double tau,
                                                         const double* v, double* y,
                                                         const double* __restrict__ V,
                                                         const double* __restrict__ W) {
  dep_sync();
  constexpr int NW = ACTX ? 4 : 2;
  const long long n = g.n;
  const ProxK K = prox_consts(tau, 0.5 / tau, cf.f_b);
  const double a1_in = fma(tau, cf.f_a, 1.0), a1_last = fma(tau, fma(cf.g_a, g.idt, cf.f_a), 1.0);
  const float a1f_in = (float)a1_in, a1f_last = (float)a1_last;
  const df a1d_in = df_from_double(a1_in), a1d_last = df_from_double(a1_last);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e / g.S);
    const long long f = e % g.S;
    double wbar[NW], w_new[NW];
#pragma unroll
    for (int q = 0; q < NW; ++q) wbar[q] = v[e + (q + 1) * n];
    const bool last = (k == g.nt - 1);
    const double cc = last ? fma(W[f], g.idt, V[f]) : V[f];
    double m_new;
    if constexpr (GENQ)
      prox_cell_q<NW>(v[e], wbar, tau, cf.qprime, last ? a1_last : a1_in, K.tb, cc, m_new, w_new);
    else
      prox_cell<NW>(v[e], wbar, K, last ? a1_last : a1_in, last ? a1f_last : a1f_in, last ? a1d_last : a1d_in, cc,
                    m_new, w_new);
    y[e] = m_new;
#pragma unroll
    for (int q = 0; q < NW; ++q) y[e + (q + 1) * n] = w_new[q];
  }
}

// One wave of resident blocks per instantiation (SMs x blocks per SM from the
// occupancy calculator), set by prox_configure: the prox step is FP64-bound
// with ~100 registers a thread, so a grid past one wave only adds a tail.
int g_prox_wave[8] = {kRedBlocks, kRedBlocks, kRedBlocks, kRedBlocks, kRedBlocks, kRedBlocks, kRedBlocks,
                      kRedBlocks};

int prox_configure() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return MFG_ERR_CUDA;
  const void* fns[8] = {(const void*)k_prox_cp<0, false, false>, (const void*)k_prox_cp<0, false, true>,
                        (const void*)k_prox_cp<0, true, false>,  (const void*)k_prox_cp<0, true, true>,
                        (const void*)k_prox_cp<1, false, false>, (const void*)k_prox_cp<1, false, true>,
                        (const void*)k_prox_cp<1, true, false>,  (const void*)k_prox_cp<1, true, true>};
  for (int i = 0; i < 8; ++i) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fns[i], kThreads, 0) != cudaSuccess) return MFG_ERR_CUDA;
    g_prox_wave[i] = std::max(1, std::min(kVecBlocksMax, sms * std::max(occ, 1)));
  }
  return MFG_OK;
}

void launch_prox_cp(const Geom& g, const Coef& cf, const double* z, double* y, double* ybar,
                    const double* V, const double* W, double* partials, DevScalars* sc,
                    cudaGraphConditionalHandle h, int use_handle, cudaStream_t s, double* Az,
                    const double* rfin) {
  const int idx = (g.actx ? 4 : 0) + (cf.qprime != 2.0 ? 2 : 0) + (g.kfy != nullptr ? 1 : 0);
  const int nb = red_blocks(g.n, g_prox_wave[idx]);
  // the general-q' root finder and the viscosity field are their own
  // instantiations, so the q' = 2, constant-nu kernel keeps its registers
#define MFG_PROX_CP(A, Q, N) \
  launch_k(k_prox_cp<A, Q, N>, nb, kThreads, 0, s, g, cf, z, y, ybar, V, W, partials, sc, h, use_handle, Az, rfin)
  const bool gq = cf.qprime != 2.0, vn = g.kfy != nullptr;
  if (g.actx) {
    if (gq) { if (vn) MFG_PROX_CP(1, true, true); else MFG_PROX_CP(1, true, false); }
    else    { if (vn) MFG_PROX_CP(1, false, true); else MFG_PROX_CP(1, false, false); }
  } else {
    if (gq) { if (vn) MFG_PROX_CP(0, true, true); else MFG_PROX_CP(0, true, false); }
    else    { if (vn) MFG_PROX_CP(0, false, true); else MFG_PROX_CP(0, false, false); }
  }
#undef MFG_PROX_CP
}

void launch_prox_plain(const Geom& g, const Coef& cf, double tau, const double* v, double* y,
                       const double* V, const double* W, cudaStream_t s) {
  const int nb = red_blocks(g.n, g.vec_blocks);
  if (cf.qprime != 2.0) {
    if (g.actx)
      launch_k(k_prox_plain<1, true>, nb, kThreads, 0, s, g, cf, tau, v, y, V, W);
    else
      launch_k(k_prox_plain<0, true>, nb, kThreads, 0, s, g, cf, tau, v, y, V, W);
  } else if (g.actx) {
    launch_k(k_prox_plain<1, false>, nb, kThreads, 0, s, g, cf, tau, v, y, V, W);
  } else {
    launch_k(k_prox_plain<0, false>, nb, kThreads, 0, s, g, cf, tau, v, y, V, W);
  }
}

}  // namespace mfg
