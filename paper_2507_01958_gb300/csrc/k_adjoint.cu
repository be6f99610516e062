// Adjoint of the converged equilibrium by implicit differentiation of the KKT
// conditions of (VMFG_h) (Sec. 2-3).  At a CP solution (y, z):
//   R1 = grad phi_A(y) + (C^T z)_A = 0   (active set A: m > 0, w_c != 0),
//   R2 = C y - d(m0) = 0.
// The adjoint system [[H, C_A^T], [C_A, 0]] [mu; eta] = [g; 0], with H the
// per-cell Hessian of phi = b_hat + F on A, is solved through its Schur
// complement (C_A H^{-1} C_A^T) eta = C_A H^{-1} g by the same PCG kernels
// and the same preconditioner P as the forward solve, then
// mu = H^{-1} (g - C^T eta).  Gradients (dloss/dtheta = -[mu; eta].dR/dtheta):
//   dm0(x) = eta(0, x)/dt,  dV(x) = -sum_k mu_m(k, x),  dW(x) = -mu_m(N_t-1, x)/dt,
//   dnu = -sum mu_m (K z) - sum eta (K m);
// with a viscosity field, K_nu in C and, per node a (dK_nu/dnu_a = sum over
// the faces f of a of g_f g_f^T / (2 dx^2), g_f the face difference),
//   dnu(a) = -(1/2) sum_k sum_{f of a} [(g_f.mu_m)(g_f.z) + (g_f.eta)(g_f.m)] / dx^2.
//
// H^{-1} per cell in closed form.  With a' = f_eff'(m) (f_a + 2 f_b m, plus
// g_a/dt on the last plane), H = [[|w|^2/m^3 + a', -w^T/m^2], [-w/m^2, I/m]]
// on the active components; its Schur complement in m is exactly a' because
// the inactive w components are zero, so
//   (H^{-1} u)_m = (u_m + w.u_w / m) / a',  (H^{-1} u)_w = m u_w + (w/m) (H^{-1} u)_m,
// and 0 on inactive components.
//
// y is fixed over the whole adjoint solve, so the velocities v = w/m and 1/a' are
// formed once (k_hinv, which also applies H^{-1} to the right-hand side) and each
// PCG iteration has no division left: 23 FP64 instructions and 5 comparisons per point
// instead of 54 in all, FP64 issue being what bounds it (128^2 x 64, cold: 114 -> 70 us; the whole
// adjoint 7.9 -> 5.6 ms).
#include "mfg_internal.cuh"
#include "reduce.cuh"
#include "strip.cuh"

namespace mfg {

// om, ow = H^{-1} (um, uw) with the cell's m, velocities v (0 on inactive
// components, and all 0 with iap = 0 where m <= 0) and iap = 1/a'.
template <int NW>
__device__ __forceinline__ void hinv_cell(double m, const double (&v)[NW], double iap, double um,
                                          const double (&uw)[NW], double& om, double (&ow)[NW]) {
  if (!(m > 0.0)) {
    om = 0.0;
#pragma unroll
    for (int q = 0; q < NW; ++q) ow[q] = 0.0;
    return;
  }
#pragma unroll
  for (int q = 0; q < NW; ++q) um = fma(v[q], uw[q], um);
  om = um * iap;
#pragma unroll
  for (int q = 0; q < NW; ++q) ow[q] = v[q] != 0.0 ? fma(m, uw[q], v[q] * om) : 0.0;
}

// v = w/m and 1/a' of a cell, 0 where m <= 0.
template <int NW>
__device__ __forceinline__ void cell_data(const Geom& g, const Coef& cf, double m, bool last, const double (&w)[NW],
                                          double (&v)[NW], double& iap) {
  const bool on = m > 0.0;
  const double im = on ? 1.0 / m : 0.0;
  iap = on ? 1.0 / (cf.f_a + 2.0 * cf.f_b * m + (last ? cf.g_a * g.idt : 0.0)) : 0.0;
#pragma unroll
  for (int q = 0; q < NW; ++q) {
    v[q] = on ? w[q] * im : 0.0;
    // w != 0 marks an active component: a quotient that underflows keeps the mark
    if (on && w[q] != 0.0 && v[q] == 0.0) v[q] = __longlong_as_double(1);
  }
}

// out = H^{-1} u, and the cell data of y that later applies read: vel (v, then
// 1/a', NW + 1 planes; null where the device had no room for them).
template <int ACTX>
__global__ void __launch_bounds__(kThreads) k_hinv(Geom g, Coef cf, const double* __restrict__ y,
                                                   const double* __restrict__ u, double* __restrict__ out,
                                                   double* __restrict__ vel) {
  dep_sync();
  constexpr int NW = ACTX ? 4 : 2;
  const long long n = g.n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e / g.S);
    const double m = y[e];
    double w[NW], v[NW], uw[NW], ow[NW], om, iap;
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      uw[q] = u[e + (q + 1) * n];
      w[q] = y[e + (q + 1) * n];
    }
    cell_data<NW>(g, cf, m, k == g.nt - 1, w, v, iap);
    if (vel != nullptr) {
#pragma unroll
      for (int q = 0; q < NW; ++q) vel[e + q * n] = v[q];
      vel[e + NW * n] = iap;
    }
    hinv_cell<NW>(m, v, iap, u[e], uw, om, ow);
    out[e] = om;
#pragma unroll
    for (int q = 0; q < NW; ++q) out[e + (q + 1) * n] = ow[q];
  }
}

constexpr int kCtHinvPerSm = 2;  // 256-thread blocks per SM

// out = H^{-1} (C^T p)  or, with GSUB, out = H^{-1} (gsub - C^T p), in warp strips
// (strip.cuh): 13 reads and writes of 8 bytes, 23 FP64 instructions and 5 comparisons per point.
template <int ACTX, bool GSUB>
__global__ void __launch_bounds__(256, kCtHinvPerSm) k_ct_hinv(Geom g, StripGrid sg, const double* __restrict__ m,
                                                              const double* __restrict__ vel,
                                                              const double* __restrict__ p,
                                                              const double* __restrict__ gsub,
                                                              double* __restrict__ out, const DevScalars* sc) {
  dep_sync();
  if (sc != nullptr && sc->cg_done) return;
  constexpr int NW = ACTX ? 4 : 2;
  int j0, i0, i1, k;
  if (!strip_item(sg, g, j0, i0, i1, k)) return;
  const long long n = g.n, base = (long long)k * g.S;
  const double* pk = p + base;
  const int j = j0 + (threadIdx.x & 31), jc = j < g.ny ? j : g.ny - 1;
  const bool last = k + 1 >= g.nt;
  const double nx = g.nu * g.ax, ny = g.nu * g.ay;
  struct Row {
    double pn, m, iap, v[NW], um, uw[NW];
  };
  diff_march<ACTX, 2>(
      g, i0, i1, j0, [&](int i, int jj) { return pk[i * g.ny + jj]; },
      [&](int i) {
        const long long e = base + i * g.ny + jc;
        Row w;
        w.pn = last ? 0.0 : p[e + g.S];
        w.m = m[e];
        w.iap = vel[e + NW * n];
        w.um = GSUB ? gsub[e] : 0.0;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
          w.v[q] = vel[e + q * n];
          w.uw[q] = GSUB ? gsub[e + (q + 1) * n] : 0.0;
        }
        return w;
      },
      [&](int i, double pc, const Diff& d, const Row& w) {
        if (j >= g.ny) return;
        double xm = fma(ny, d.yy, (pc - w.pn) * g.idt), om, ow[NW];
        double xw[NW];
        if (ACTX) {
          xm = fma(nx, d.xx, xm);
          xw[0] = d.xp; xw[1] = d.xm; xw[NW - 2] = d.yp; xw[NW - 1] = d.ym;
        } else {
          xw[0] = d.yp; xw[1] = d.ym;
        }
        if (GSUB) {
          xm = w.um - xm;
#pragma unroll
          for (int q = 0; q < NW; ++q) xw[q] = w.uw[q] - xw[q];
        }
        hinv_cell<NW>(w.m, w.v, w.iap, xm, xw, om, ow);
        const long long e = base + i * g.ny + j;
        out[e] = om;
#pragma unroll
        for (int q = 0; q < NW; ++q) out[e + (q + 1) * n] = ow[q];
      });
}

// The same point by point, for viscosity fields (VN: L = K_nu + I/dt with the face
// coefficients of Geom::kfx / kfy) and for rows too short for strips.  DATA = false:
// the cell data formed from y again in every apply, for a device without room for vel.
template <int ACTX, bool VN, bool DATA>
__global__ void __launch_bounds__(kThreads) k_ct_hinv_flat(Geom g, Coef cf, const double* __restrict__ y,
                                                           const double* __restrict__ vel,
                                                           const double* __restrict__ p,
                                                           const double* __restrict__ gsub,
                                                           double* __restrict__ out, const DevScalars* sc) {
  dep_sync();
  if (sc != nullptr && sc->cg_done) return;
  constexpr int NW = ACTX ? 4 : 2;
  const long long n = g.n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e % g.ny);
    const long long t = e / g.ny;
    const int i = (int)(t % g.nx);
    const int k = (int)(t / g.nx);
    const long long base = (long long)k * g.S;
    const long long rowi = base + (long long)i * g.ny;
    const double pc = p[e];
    const bool hmy = g.pery || j >= 1, hpy = g.pery || j <= g.ny - 2;
    const int jm = hmy ? (j == 0 ? g.ny - 1 : j - 1) : j;
    const int jp = hpy ? (j == g.ny - 1 ? 0 : j + 1) : j;
    const double pjm = p[rowi + jm], pjp = p[rowi + jp];
    const long long f0 = (long long)i * g.ny;
    // K_nu p: a missing face has its neighbour index at the node itself (difference 0)
    double Kp = VN ? fma(g.kfy[f0 + j], pc - pjp, g.kfy[f0 + jm] * (pc - pjm))
                   : g.ay * ((hmy ? pc - pjm : 0.0) + (hpy ? pc - pjp : 0.0));
    double xw[NW];
    if (ACTX) {
      const bool hmx = g.perx || i >= 1, hpx = g.perx || i <= g.nx - 2;
      const int im = hmx ? (i == 0 ? g.nx - 1 : i - 1) : i;
      const int ip = hpx ? (i == g.nx - 1 ? 0 : i + 1) : i;
      const double pim = p[base + (long long)im * g.ny + j], pip = p[base + (long long)ip * g.ny + j];
      if (VN)
        Kp = fma(g.kfx[f0 + j], pc - pip, fma(g.kfx[(long long)im * g.ny + j], pc - pim, Kp));
      else
        Kp += g.ax * ((hmx ? pc - pim : 0.0) + (hpx ? pc - pip : 0.0));
      xw[0] = hpx ? (pc - pip) * g.idx : 0.0;
      xw[1] = hmx ? (pim - pc) * g.idx : 0.0;
      xw[2] = hpy ? (pc - pjp) * g.idy : 0.0;
      xw[3] = hmy ? (pjm - pc) * g.idy : 0.0;
    } else {
      xw[0] = hpy ? (pc - pjp) * g.idy : 0.0;
      xw[1] = hmy ? (pjm - pc) * g.idy : 0.0;
    }
    const double pn = (k + 1 < g.nt) ? p[e + g.S] : 0.0;
    double xm = (VN ? Kp : g.nu * Kp) + (pc - pn) * g.idt;
    if (gsub != nullptr) {
      xm = gsub[e] - xm;
#pragma unroll
      for (int q = 0; q < NW; ++q) xw[q] = gsub[e + (q + 1) * n] - xw[q];
    }
    double v[NW], ow[NW], om, iap;
    const double m = y[e];
    if constexpr (DATA) {
#pragma unroll
      for (int q = 0; q < NW; ++q) v[q] = vel[e + q * n];
      iap = vel[e + NW * n];
    } else {
      double w[NW];
#pragma unroll
      for (int q = 0; q < NW; ++q) w[q] = y[e + (q + 1) * n];
      cell_data<NW>(g, cf, m, k == g.nt - 1, w, v, iap);
    }
    hinv_cell<NW>(m, v, iap, xm, xw, om, ow);
    out[e] = om;
#pragma unroll
    for (int q = 0; q < NW; ++q) out[e + (q + 1) * n] = ow[q];
  }
}

// A block takes 32 spatial points and splits their time planes over 8 warps (one
// thread per point left 64 blocks of serial loops at 128^2: 119 us); the warps'
// sums are added in order.  dnu by reduction, or (VN) the node derivative dnu(f)
// written per point.
template <bool VN>
__global__ void __launch_bounds__(kThreads) k_adj_grads(Geom g, const double* __restrict__ y,
                                                        const double* __restrict__ z,
                                                        const double* __restrict__ eta,
                                                        const double* __restrict__ mu, double* dm0,
                                                        double* dV, double* dW, double* dnu,
                                                        double* partials, DevScalars* sc) {
  dep_sync();
  __shared__ double part_s[2][8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double acc = 0.0, sv = 0.0, node = 0.0;
  const int f = blockIdx.x * 32 + lane;
  if (f < g.S) {
    const int j = f % g.ny, i = f / g.ny;
    const bool hmy = g.pery || j >= 1, hpy = g.pery || j <= g.ny - 2;
    const int jm = hmy ? (j == 0 ? g.ny - 1 : j - 1) : j;
    const int jp = hpy ? (j == g.ny - 1 ? 0 : j + 1) : j;
    const bool hmx = g.actx && (g.perx || i >= 1), hpx = g.actx && (g.perx || i <= g.nx - 2);
    const int im = hmx ? (i == 0 ? g.nx - 1 : i - 1) : i;
    const int ip = hpx ? (i == g.nx - 1 ? 0 : i + 1) : i;
    for (int k = warp; k < g.nt; k += 8) {
      const long long base = (long long)k * g.S;
      const long long e = base + f;
      const double mum = mu[e];
      sv += mum;
      if (VN) {
        // the node's faces: (g.mu)(g.z) + (g.eta)(g.m) per face, times 1/dx^2
        auto face = [&](long long nb, double c) {
          const double a = (mum - mu[nb]) * (z[e] - z[nb]) + (eta[e] - eta[nb]) * (y[e] - y[nb]);
          return c * a;
        };
        double t = 0.0;
        if (hmy) t += face(base + (long long)i * g.ny + jm, g.ay);
        if (hpy) t += face(base + (long long)i * g.ny + jp, g.ay);
        if (hmx) t += face(base + (long long)im * g.ny + j, g.ax);
        if (hpx) t += face(base + (long long)ip * g.ny + j, g.ax);
        node += t;
      } else {
        auto K5 = [&](const double* a) {
          const double c = a[e];
          return g.ay * ((hmy ? c - a[base + (long long)i * g.ny + jm] : 0.0) +
                         (hpy ? c - a[base + (long long)i * g.ny + jp] : 0.0)) +
                 g.ax * ((hmx ? c - a[base + (long long)im * g.ny + j] : 0.0) +
                         (hpx ? c - a[base + (long long)ip * g.ny + j] : 0.0));
        };
        acc -= mum * K5(z) + eta[e] * K5(y);
      }
    }
  }
  part_s[0][warp][lane] = sv;
  part_s[1][warp][lane] = node;
  __syncthreads();
  if (warp == 0 && f < g.S) {
    for (int w = 1; w < 8; ++w) {
      sv += part_s[0][w][lane];
      node += part_s[1][w][lane];
    }
    if (VN) dnu[f] = -0.5 * node;
    dm0[f] = eta[f] * g.idt;
    dV[f] = -sv;
    if (dW != nullptr) dW[f] = -mu[(long long)(g.nt - 1) * g.S + f] * g.idt;
  }
  if (VN) return;
  double part[1] = {acc};
  block_sum<1>(part);
  if (!publish_and_check_last<1>(part, partials, &sc->counter)) return;
  double tot[1];
  gather_partials<1>(partials, tot);
  if (flat_tid() == 0) {
    *dnu = tot[0];
    sc->counter = 0;
  }
}

void launch_hinv(const Geom& g, const Coef& cf, const double* y, const double* u, double* out, double* vel,
                 cudaStream_t s) {
  const int nb = red_blocks(g.n, kVecBlocksMax);
  if (g.actx)
    launch_k(k_hinv<1>, nb, kThreads, 0, s, g, cf, y, u, out, vel);
  else
    launch_k(k_hinv<0>, nb, kThreads, 0, s, g, cf, y, u, out, vel);
}

void launch_ct_hinv(const Geom& g, const Coef& cf, const double* y, const double* vel, const double* p,
                    const double* gsub, double* out, cudaStream_t s, const DevScalars* sc) {
  // an iteration of the adjoint with H^-1 C^T in strips against point by point: 300 x 45 x 60
  // 203 / 194 us, 300 x 50 x 60 214 / 206, 512 x 26 x 60 189 / 189, 300 x 56 x 60 216 / 219,
  // 300 x 64 x 60 204 / 217
  if (vel == nullptr || !strips_filled(g, 7, 8)) {
    const int nb = red_blocks(g.n, kVecBlocksMax);
#define MFG_CT_HINV(A, N, D) launch_k(k_ct_hinv_flat<A, N, D>, nb, kThreads, 0, s, g, cf, y, vel, p, gsub, out, sc)
#define MFG_CT_HINV_D(D)                                                                                  \
  if (g.kfy != nullptr) { if (g.actx) MFG_CT_HINV(1, true, D); else MFG_CT_HINV(0, true, D); }            \
  else                  { if (g.actx) MFG_CT_HINV(1, false, D); else MFG_CT_HINV(0, false, D); }
    if (vel != nullptr) { MFG_CT_HINV_D(true) } else { MFG_CT_HINV_D(false) }
#undef MFG_CT_HINV_D
#undef MFG_CT_HINV
    return;
  }
  const StripGrid sg = strip_grid(g, kCtHinvPerSm);
#define MFG_CT_HINV(A, G) launch_k(k_ct_hinv<A, G>, sg.blocks, 32 * sg.warps, 0, s, g, sg, y, vel, p, gsub, out, sc)
  if (gsub != nullptr) { if (g.actx) MFG_CT_HINV(1, true); else MFG_CT_HINV(0, true); }
  else                 { if (g.actx) MFG_CT_HINV(1, false); else MFG_CT_HINV(0, false); }
#undef MFG_CT_HINV
}

int adj_grads_blocks(const Geom& g) { return (g.S + 31) / 32; }

void launch_adj_grads(const Geom& g, const double* y, const double* z, const double* eta,
                      const double* mu, double* dm0, double* dV, double* dW, double* dnu,
                      double* partials, DevScalars* sc, cudaStream_t s) {
  const int nb = adj_grads_blocks(g);
  if (g.kfy != nullptr)
    launch_k(k_adj_grads<true>, nb, kThreads, 0, s, g, y, z, eta, mu, dm0, dV, dW, dnu, partials, sc);
  else
    launch_k(k_adj_grads<false>, nb, kThreads, 0, s, g, y, z, eta, mu, dm0, dV, dW, dnu, partials, sc);
}

}  // namespace mfg
