// Space-time stencils of the discrete Fokker-Planck constraint:
//   C v      (eq. ABC, reduced), the CP right-hand side sigma (C ybar - d),
//   C^T p    (its transpose),
//   C C^T p  (eq. largeA), in two halo-free passes over p.
//
// Row k of C (plane k, time level k+1) reads
//   L m^{k+1} - m^k/dt + div_h w^k,  L = nu K + I/dt   (Sec. 3, matrices A, B)
// with K the negative 5-point Laplacian and div_h the divergence of Sec. 2,
// D^1/D^2 blocks of Sec. 4.3 per axis.  On a Neumann axis the blocks have no
// entries past the ends; on a periodic axis indices wrap.  Both cases use one
// rule: a point has a "minus" neighbour (hm) and a "plus" neighbour (hp) unless
// it sits at the matching end of a Neumann axis.
#include "df64.cuh"
#include "mfg_internal.cuh"
#include "pcg_tail.cuh"
#include "reduce.cuh"
#include "strip.cuh"

namespace mfg {

// 256-thread blocks per SM that the launch bounds of the strip kernels admit
constexpr int kCPerSm = 2, kCtPerSm = 3, kUPerSm = 4, kQPerSm = 3;

// C^T in strips from 2/3 of the lanes filled on: 512 x ny x 100, in strips against point by
// point 39.3 / 36.2 us at ny = 20, 39.3 / 40.0 at 22, 74.7 / 77.3 at 43, 75.7 / 92.2 at 52;
// 2000 x 250 in 1-D 11.1 / 12.5.
static bool ct_strips_fit(const Geom& g) { return strips_filled(g, 2, 3); }
// C in 2-D from 7/8 on: 512 x ny x 100, 51.4 / 39.6 us at ny = 20, 51.6 / 46.8 at 24, 102.0 / 88.8
// at 45, 102.5 / 101.3 at 52, 103.1 / 108.8 at 56; 512^2 x 64 489 / 602.  Not in 1-D, where a
// strip is one row and its borders a load each: 2000 x 250 17.9 / 15.3.
static bool c_strips_fit(const Geom& g) { return g.actx && strips_filled(g, 7, 8); }

struct Nb {
  int im, ip;
  bool hm, hp;
};

__device__ __forceinline__ Nb nbr(int i, int N, int per) {
  Nb b;
  if (per) {
    b.im = (i == 0) ? N - 1 : i - 1;
    b.ip = (i == N - 1) ? 0 : i + 1;
    b.hm = b.hp = true;
  } else {
    b.hm = i >= 1;
    b.hp = i <= N - 2;
    b.im = b.hm ? i - 1 : i;
    b.ip = b.hp ? i + 1 : i;
  }
  return b;
}

// ------------------------------------------------------------------- C v --
// mode 0: r = alpha * (C v - d), d = m0/dt on plane 0 when m0 != nullptr.
// mode 1: CP right-hand side r = sigma (C v - d) with sigma from the device
//         scalars; reduces ||r||^2, resets the PCG state for the new solve.
//         With Az != nullptr (the MFG_CG_REF_RHS stop reference) Az holds
//         AAt z_l on entry and b = AAt z_l + r, the right-hand side of the
//         system of eq. CC*, on exit; ||b||^2 becomes the reference of the
//         relative tolerance, and a warm start already inside it stops the
//         solve before its first iteration.
// mode 2: PCG step of the adjoint Schur system: r = C v, reduces pdot.r,
//         alpha = rz/(pdot.r).
// mode 3: adjoint right-hand side r = C v; reduces ||r||^2, resets the PCG
//         state with the fixed tolerance.
//
// Terms of a point: nu K m by neighbour sums (strip.cuh), and per axis
// ((w1_i - w1_{i-1}) + (w2_{i+1} - w2_i)) / dx, 0 past a Neumann end.  Each flux by its own
// difference, exact where it varies slowly: sums w1_i + w2_{i+1} per face, formed once,
// take two FP64 instructions less but round at the size of the flux (128^2 torus, nu = 0,
// both fluxes smooth: up to 1e-16 -> 5e-15 off 64 bits).  FP64 issue bounds the kernel: 15
// instructions per point (17 with oblong cells; 2 more with Az), ~28 point by point.
__device__ __forceinline__ void rhs_tail(double acc, double accb, bool have_b, double* partials, DevScalars* sc) {
  double part[2] = {acc, accb};
  block_sum<2>(part);
  if (!publish_and_check_last<2>(part, partials, &sc->counter)) return;
  double tot[2];
  gather_partials<2>(partials, tot);
  if (flat_tid() == 0) {
    const double rr0 = tot[0], b2 = have_b ? tot[1] : tot[0];
    sc->bnorm2 = b2;  // reference of the relative tolerance: ||b||^2 or ||r_0||^2
    sc->rr = rr0;
    sc->cg_it = 0;
    // The paper's adaptive rule, min{1e-4, max{1e-6, 1e-4 r}} (Sec. 5).
    double tol = sc->cg_tol_fixed;
    if (sc->cg_rule == MFG_CG_ADAPTIVE) tol = fmin(1e-4, fmax(1e-6, 1e-4 * sc->r_last));
    sc->cg_tol = tol;
    // no iteration when r_0 = 0 or r_0 is already inside the tolerance (NaN: flagged below)
    sc->cg_done = !(rr0 > 0.0) || rr0 <= tol * tol * b2;
    if (!isfinite(rr0) || !isfinite(b2)) {
      sc->cg_done = 1;
      sc->status = MFG_ERR_NONFINITE;
    }
    sc->counter = 0;
  }
}

template <bool ISO, int MODE>
__global__ void __launch_bounds__(256, kCPerSm) k_apply_C(Geom g, StripGrid sg, const double* __restrict__ v,
                                                    double* __restrict__ r, double alpha,
                                                    const double* __restrict__ m0, const double* __restrict__ pdot,
                                                    double* partials, DevScalars* sc, double* __restrict__ Az) {
  dep_sync();
  if (MODE == 2 && sc->cg_done) return;
  if (MODE == 1) alpha = sc->sigma;
  double acc = 0.0, accb = 0.0;
  int j0, i0, i1, k;
  if (strip_item(sg, g, j0, i0, i1, k)) {
    const long long n = g.n, base = (long long)k * g.S;
    const double* m = v + base;
    const double* wx1 = v + n + base;
    const double* wx2 = v + 2 * n + base;
    const double* wy1 = v + 3 * n + base;
    const double* wy2 = v + 4 * n + base;
    const StripCols c = strip_cols(g, j0);
    const int lane = threadIdx.x & 31, j = j0 + lane;
    const bool end_y = !g.pery && j == g.ny - 1, first_y = !g.pery && j == 0;  // no face beyond
    auto at = [&](int i, int jj) { return i * g.ny + jj; };  // < S, an int
    const int ir = min(i0 + lane, i1 - 1);
    const double w2r = wy2[at(ir, c.right)];
    const double w1l = (!g.pery && j0 == 0) ? 0.0 : wy1[at(ir, c.left)];
    double x1m = 0.0, x2c = 0.0;  // w1_{i-1}, w2_i
    if (g.perx || i0 > 0) {
      x1m = wx1[at(ghost(i0 - 1, g.nx, g.perx), c.j)];
      x2c = wx2[at(i0, c.j)];
    }
    const double ky = alpha * g.nu * g.ay, rho = g.ax / g.ay, kc = 2.0 * (1.0 + rho) * ky;
    const double aix = alpha * g.idx, aiy = alpha * g.idy, aidt = alpha * g.idt;
    const double* mp = k >= 1 ? m - g.S : m0;  // m of the previous level (plane 0: m0, or 0)
    struct Row {
      double wy1, wy2, wx1, wx2, mp, extra;
    };
    const bool have_mp = mp != nullptr, have_az = MODE == 1 && Az != nullptr;
    sum_march<ISO, 2>(
        g, rho, i0, i1, j0, [&](int i, int jj) { return m[at(i, jj)]; },
        [&](int i) {
          const int e = at(i, c.j);
          Row w{wy1[e], wy2[e], 0.0, 0.0, 0.0, 0.0};
          w.wx1 = wx1[e];
          w.wx2 = wx2[at(ghost(i + 1, g.nx, g.perx), c.j)];
          if (have_mp) w.mp = mp[e];
          if (MODE == 2) w.extra = pdot[base + e];
          if (have_az) w.extra = Az[base + e];
          return w;
        },
        [&](int i, double mc, double sum, const Row& w) {
          const double y1 = end_y ? 0.0 : w.wy1, y2 = first_y ? 0.0 : w.wy2;
          double y2r = from_right(y2, w2r, i - i0);
          if (end_y) y2r = 0.0;
          const double sy = (y1 - from_left(y1, w1l, i - i0)) + (y2r - y2);
          double val = fma(kc, mc, -ky * sum);
          const bool end_x = !g.perx && i == g.nx - 1;
          const double x1 = end_x ? 0.0 : w.wx1, x2 = end_x ? 0.0 : w.wx2;
          const double sx = (x1 - x1m) + (x2 - x2c);
          x1m = x1;
          x2c = x2;
          val = ISO ? fma(aiy, sx + sy, val) : fma(aix, sx, fma(aiy, sy, val));
          if (j >= g.ny) return;
          val = fma(aidt, mc - w.mp, val);
          const int e = at(i, j);
          r[base + e] = val;
          if constexpr (MODE == 2) acc = fma(w.extra, val, acc);
          if constexpr (MODE == 1 || MODE == 3) acc = fma(val, val, acc);
          if constexpr (MODE == 1) {
            if (have_az) {
              const double b = w.extra + val;
              Az[base + e] = b;
              accb = fma(b, b, accb);
            }
          }
        });
  }
  if constexpr (MODE == 2) aat_tail(acc, partials, sc);
  if constexpr (MODE == 1 || MODE == 3) rhs_tail(acc, accb, Az != nullptr, partials, sc);
}

// The same terms point by point, for 1-D grids, viscosity fields and grids whose rows
// would leave too much of a 32-column strip empty (c_strips_fit).  Two blocks per SM in
// the launch bounds: with the compiler's own choice of 64 registers a grid of two
// blocks per SM took 99.4 us for 512 x 45 x 100, with 100 registers 88.8.  VN (viscosity field):
// nu K m becomes K_nu m = sum over the node's faces of kf (m - m_nb), kf the face
// coefficient of Geom::kfx / kfy; at a Neumann end the neighbour index is the node
// itself, so the missing face adds nothing.
template <int ACTX, bool VN>
__global__ void __launch_bounds__(kThreads, 2) k_apply_C_flat(Geom g, const double* __restrict__ v,
                                                      double* __restrict__ r, double alpha,
                                                      const double* __restrict__ m0,
                                                      const double* __restrict__ pdot,
                                                      double* partials, DevScalars* sc, int mode,
                                                      double* __restrict__ Az) {
  dep_sync();
  if (mode == 2 && sc->cg_done) return;
  if (mode == 1) alpha = sc->sigma;
  const long long n = g.n;
  const double* m = v;
  const double* wx1 = v + n;
  const double* wx2 = v + 2 * n;
  const double* wy1 = ACTX ? v + 3 * n : v + n;
  const double* wy2 = ACTX ? v + 4 * n : v + 2 * n;
  // alpha folded into the coefficients: r = alpha nu K m + alpha div_h w + alpha (m^k - m^{k-1})/dt
  const double anu = alpha * g.nu, ax = ACTX ? g.ax : 0.0;
  const double kc = anu * 2.0 * (ax + g.ay), kx = anu * ax, ky = anu * g.ay;
  const double aix = alpha * g.idx, aiy = alpha * g.idy, aidt = alpha * g.idt;
  double acc = 0.0, accb = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e % g.ny);
    const long long t = e / g.ny;
    const int i = (int)(t % g.nx);
    const int k = (int)(t / g.nx);
    const long long base = (long long)k * g.S;
    const long long rowi = base + (long long)i * g.ny;
    // K m with the point itself as the missing neighbour at a Neumann end (one-sided rows)
    const Nb by = nbr(j, g.ny, g.pery);
    const double mc = m[e];
    double t1 = ky * (m[rowi + by.im] + m[rowi + by.ip]);
    // div_h w: flux slots past a Neumann end do not exist and read as zero
    const double sy = ((by.hp ? wy1[e] : 0.0) - (by.hm ? wy1[rowi + by.im] : 0.0)) +
                      ((by.hp ? wy2[rowi + by.ip] : 0.0) - (by.hm ? wy2[e] : 0.0));
    double val;
    double kvm = 0.0;  // K_nu m (VN)
    if (VN) {
      const long long f = (long long)i * g.ny;
      kvm = fma(g.kfy[f + j], mc - m[rowi + by.ip], g.kfy[f + by.im] * (mc - m[rowi + by.im]));
    }
    if (ACTX) {
      const Nb bx = nbr(i, g.nx, g.perx);
      const long long em = base + (long long)bx.im * g.ny + j, ep = base + (long long)bx.ip * g.ny + j;
      t1 = fma(kx, m[em] + m[ep], t1);
      const double sx = ((bx.hp ? wx1[e] : 0.0) - (bx.hm ? wx1[em] : 0.0)) +
                        ((bx.hp ? wx2[ep] : 0.0) - (bx.hm ? wx2[e] : 0.0));
      if (VN) {
        kvm = fma(g.kfx[(long long)i * g.ny + j], mc - m[ep], kvm);
        kvm = fma(g.kfx[(long long)bx.im * g.ny + j], mc - m[em], kvm);
        val = fma(aix, sx, fma(aiy, sy, alpha * kvm));
      } else {
        val = fma(aix, sx, fma(aiy, sy, fma(kc, mc, -t1)));
      }
    } else {
      val = VN ? fma(aiy, sy, alpha * kvm) : fma(aiy, sy, fma(kc, mc, -t1));
    }
    const double mprev = k >= 1 ? m[e - g.S] : (m0 != nullptr ? m0[(long long)i * g.ny + j] : 0.0);
    val = fma(aidt, mc - mprev, val);
    r[e] = val;
    acc = (mode == 2) ? fma(pdot[e], val, acc) : fma(val, val, acc);
    if (Az != nullptr) {
      const double b = Az[e] + val;
      Az[e] = b;
      accb = fma(b, b, accb);
    }
  }
  if (mode == 0) return;
  if (mode == 2)
    aat_tail(acc, partials, sc);
  else
    rhs_tail(acc, accb, Az != nullptr, partials, sc);
}

void launch_apply_C(const Geom& g, const double* v, double* r, double alpha, const double* m0,
                    double* partials, DevScalars* sc, int mode, cudaStream_t s, const double* pdot,
                    double* Az) {
  if (!c_strips_fit(g)) {
    const int nb = red_blocks(g.n, g.vec_blocks);
#define MFG_C_FLAT(A, N) launch_k(k_apply_C_flat<A, N>, nb, kThreads, 0, s, g, v, r, alpha, m0, pdot, partials, sc, mode, Az)
    if (g.kfy != nullptr) { if (g.actx) MFG_C_FLAT(1, true); else MFG_C_FLAT(0, true); }
    else                  { if (g.actx) MFG_C_FLAT(1, false); else MFG_C_FLAT(0, false); }
#undef MFG_C_FLAT
    return;
  }
  const StripGrid sg = strip_grid(g, kCPerSm);
#define MFG_C(I, M) \
  launch_k(k_apply_C<I, M>, sg.blocks, 32 * sg.warps, 0, s, g, sg, v, r, alpha, m0, pdot, partials, sc, Az)
#define MFG_C_MODE(I)       \
  switch (mode) {              \
    case 0: MFG_C(I, 0); break; \
    case 1: MFG_C(I, 1); break; \
    case 2: MFG_C(I, 2); break; \
    default: MFG_C(I, 3); break; \
  }
  if (g.ax == g.ay)
    MFG_C_MODE(true)
  else
    MFG_C_MODE(false)
#undef MFG_C_MODE
#undef MFG_C
}

// ----------------------------------------------------------------- C^T p --
// x_m^k = L p^k - p^{k+1}/dt (p^{N_t} := 0),  x_w^k = B^T p^k = -D_h p^k.
// Face form: the two flux rows of an axis are the same face differences, one
// node apart, so each is formed and scaled once (10 FP64 instructions per point
// instead of ~23; 48 bytes written and 8 read).
template <int ACTX>
__global__ void __launch_bounds__(256, kCtPerSm) k_apply_Ct(Geom g, StripGrid sg, const double* __restrict__ p,
                                                     double* __restrict__ x) {
  dep_sync();
  int j0, i0, i1, k;
  if (!strip_item(sg, g, j0, i0, i1, k)) return;
  const long long n = g.n, base = (long long)k * g.S;
  const double* pk = p + base;
  double* xm = x + base;
  double* xx1 = x + n + base;
  double* xx2 = x + 2 * n + base;
  double* xy1 = x + (ACTX ? 3 : 1) * n + base;
  double* xy2 = x + (ACTX ? 4 : 2) * n + base;
  const int j = j0 + (threadIdx.x & 31);
  const bool last = k + 1 >= g.nt;
  const double nx = g.nu * g.ax, ny = g.nu * g.ay;
  const int jc = j < g.ny ? j : g.ny - 1;
  const double* pn1 = pk + (last ? 0 : g.S);  // not i * ny + jc + S, which passes 2^31 from S = 2^30 on
  diff_march<ACTX, 4>(
      g, i0, i1, j0, [&](int i, int jj) { return pk[i * g.ny + jj]; },
      [&](int i) { return last ? 0.0 : pn1[i * g.ny + jc]; },
      [&](int i, double pc, const Diff& d, double pn) {
        if (j >= g.ny) return;
        const int e = i * g.ny + j;
        double m = fma(ny, d.yy, (pc - pn) * g.idt);
        xy1[e] = d.yp;
        xy2[e] = d.ym;
        if (ACTX) {
          m = fma(nx, d.xx, m);
          xx1[e] = d.xp;
          xx2[e] = d.xm;
        }
        xm[e] = m;
      });
}

// Point by point (see k_apply_C_flat).  VN: L = K_nu + I/dt with the face
// coefficients of Geom::kfx / kfy.
template <int ACTX, bool VN>
__global__ void __launch_bounds__(kThreads) k_apply_Ct_flat(Geom g, const double* __restrict__ p,
                                                       double* __restrict__ x) {
  dep_sync();
  const long long n = g.n;
  double* xm = x;
  double* xx1 = x + n;
  double* xx2 = x + 2 * n;
  double* xy1 = ACTX ? x + 3 * n : x + n;
  double* xy2 = ACTX ? x + 4 * n : x + 2 * n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e % g.ny);
    const long long t = e / g.ny;
    const int i = (int)(t % g.nx);
    const int k = (int)(t / g.nx);
    const long long base = (long long)k * g.S;
    const long long rowi = base + (long long)i * g.ny;
    const Nb by = nbr(j, g.ny, g.pery);
    const double pc = p[e];
    const double pjm = p[rowi + by.im], pjp = p[rowi + by.ip];
    const long long f = (long long)i * g.ny;
    double Kp = VN ? fma(g.kfy[f + j], pc - pjp, g.kfy[f + by.im] * (pc - pjm))
                   : g.ay * ((by.hm ? pc - pjm : 0.0) + (by.hp ? pc - pjp : 0.0));
    xy1[e] = by.hp ? (pc - pjp) * g.idy : 0.0;
    xy2[e] = by.hm ? (pjm - pc) * g.idy : 0.0;
    if (ACTX) {
      const Nb bx = nbr(i, g.nx, g.perx);
      const double pim = p[base + (long long)bx.im * g.ny + j], pip = p[base + (long long)bx.ip * g.ny + j];
      if (VN)
        Kp = fma(g.kfx[f + j], pc - pip, fma(g.kfx[(long long)bx.im * g.ny + j], pc - pim, Kp));
      else
        Kp += g.ax * ((bx.hm ? pc - pim : 0.0) + (bx.hp ? pc - pip : 0.0));
      xx1[e] = bx.hp ? (pc - pip) * g.idx : 0.0;
      xx2[e] = bx.hm ? (pim - pc) * g.idx : 0.0;
    }
    const double pn = (k + 1 < g.nt) ? p[e + g.S] : 0.0;
    xm[e] = (VN ? Kp : g.nu * Kp) + (pc - pn) * g.idt;
  }
}

void launch_apply_Ct(const Geom& g, const double* p, double* x, cudaStream_t s) {
  if (!ct_strips_fit(g)) {
    const int nb = red_blocks(g.n, g.vec_blocks);
#define MFG_CT_FLAT(A, N) launch_k(k_apply_Ct_flat<A, N>, nb, kThreads, 0, s, g, p, x)
    if (g.kfy != nullptr) { if (g.actx) MFG_CT_FLAT(1, true); else MFG_CT_FLAT(0, true); }
    else                  { if (g.actx) MFG_CT_FLAT(1, false); else MFG_CT_FLAT(0, false); }
#undef MFG_CT_FLAT
    return;
  }
  const StripGrid sg = strip_grid(g, kCtPerSm);
  if (g.actx)
    launch_k(k_apply_Ct<1>, sg.blocks, 32 * sg.warps, 0, s, g, sg, p, x);
  else
    launch_k(k_apply_Ct<0>, sg.blocks, 32 * sg.warps, 0, s, g, sg, p, x);
}

// ---------------------------------------------------------------- C C^T p --
// FP64 issue is the limit on GB300 (a warp's FP64 instruction takes 16 SM
// clocks; the bytes moved take a third of that time), so the operator is
// arranged for the fewest FP64 instructions per point.  Factored form
// q = C (C^T p): with x^k = L p^k - p^{k+1}/dt (the m rows of C^T p, p^{N_t} := 0)
// and BB^T = 2K (eq. precstead),
//   q^k = L x^k - x^{k-1}/dt + 2 K p^k        (x^{-1} := 0),
// in two passes over the grid, each point computed once.  With K p = -ay u,
//   u = (p_S + p_N) + rho (p_W + p_E) - 2 (1 + rho) p,   rho = ax / ay:
//   pass 1:  u,  X = dt x = (p^k - p^{k+1}) - nu ay dt u
//   pass 2:  q = c4 X - (X^{k-1}/dt^2 + c1 sum(X) + 2 ay u),   c1 = nu ay/dt,
//            c4 = 2 (1 + rho) c1 + 1/dt^2, sum the neighbour sum of u's formula.
// The time differences are formed from neighbouring planes of p, exactly where p
// varies slowly; a second difference of p - nu ay dt u (the same number of
// instructions) rounds at the size of p/dt^2, 10 to 35 times as far off for fields
// smooth in time on grids with 1/dt^2 >> ay (8^2 x 200: 2e-16 against 8e-15).
// Square cells (rho = 1) share the diagonal pair sums A(i, j) = p(i, j+1) + p(i+1, j):
//   p_N + p_S + p_W + p_E = A(i, j) + A(i-1, j-1),
// one addition less per point and pass.  FP64 instructions per point: 5 + 7
// with p.q (6 + 8 when rho != 1).
// On a Neumann axis the neighbour index of an end point is the point itself
// (u_{-1} = u_0, u_N = u_{N-1}), which turns the same formula into the
// one-sided D^1 (D^1)^T rows of Sec. 4.3, for p and for X alike.
//
// Both passes walk the grid in warp strips (strip.cuh).  512^2 x 128: 748 us, 12 FP64
// instructions per point (949 us one column per thread, 15 instructions).
struct AatCoef {
  double rho, m2r;        // ax / ay, -2 (1 + rho)
  double alpha;           // nu ay dt
  double ay2, c1, idt2, c4r;  // 2 ay, nu ay/dt, 1/dt^2, 2 (1 + rho) c1 + 1/dt^2
  double ax, ay, cK;      // viscosity field and double-float passes
  double ndt, c2, c4;
  double dt, idt;
};

AatCoef aat_coef(const Geom& g) {
  const double ax = g.actx ? g.ax : 0.0, ay = g.ay, cK = 2.0 * (ax + ay);
  const double dt = 1.0 / g.idt, idt2 = g.idt * g.idt, rho = ax / ay, c1 = g.nu * ay * g.idt;
  return AatCoef{rho, -2.0 * (1.0 + rho), g.nu * ay * dt, 2.0 * ay, c1, idt2, 2.0 * (1.0 + rho) * c1 + idt2, ax, ay, cK,
                 g.nu * dt, g.nu * ax * g.idt, g.nu * cK * g.idt + idt2, dt, g.idt};
}

template <bool ISO>
__global__ void __launch_bounds__(256, kUPerSm) k_aat_u(Geom g, AatCoef a, StripGrid ag, const double* __restrict__ p,
                                                        double* __restrict__ U, double* __restrict__ X,
                                                        const DevScalars* sc, int mode) {
  dep_sync();
  if (mode != 0 && sc->cg_done) return;
  int j0, i0, i1, k;
  if (!strip_item(ag, g, j0, i0, i1, k)) return;
  const long long base = (long long)k * g.S;
  const int j = j0 + (threadIdx.x & 31), jc = j < g.ny ? j : g.ny - 1;
  const bool last = k + 1 >= g.nt;
  const double* pk = p + base;
  const double* pkn = pk + (last ? 0 : g.S);
  sum_march<ISO, 4>(g, a.rho, i0, i1, j0, [&](int i, int jj) { return pk[i * g.ny + jj]; },
                    [&](int i) { return last ? 0.0 : pkn[i * g.ny + jc]; },
                    [&](int i, double c, double sum, double next) {
                      if (j >= g.ny) return;
                      const double u = fma(a.m2r, c, sum);
                      const int f = i * g.ny + j;
                      U[base + f] = u;
                      X[base + f] = fma(-a.alpha, u, c - next);
                    });
}

// q = AAt p; STEP (PCG step): also reduces p.q and sets alpha = rz/(p.q) in the
// device scalars.
template <bool ISO, bool STEP>
__global__ void __launch_bounds__(256, kQPerSm) k_aat_q2(Geom g, AatCoef a, StripGrid ag, const double* __restrict__ U,
                                                   const double* __restrict__ X, const double* __restrict__ p,
                                                   double* __restrict__ q, double* partials, DevScalars* sc) {
  dep_sync();
  if (STEP && sc->cg_done) return;
  double acc = 0.0;
  int j0, i0, i1, k;
  if (strip_item(ag, g, j0, i0, i1, k)) {
    const long long base = (long long)k * g.S;
    const double* xk = X + base;
    const int j = j0 + (threadIdx.x & 31);
    struct Row {
      double u, xp, p;
    };
    const int jc = j < g.ny ? j : g.ny - 1;
    sum_march<ISO, 4>(g, a.rho, i0, i1, j0, [&](int i, int jj) { return xk[i * g.ny + jj]; },
                      [&](int i) {
                        const long long e = base + i * g.ny + jc;
                        return Row{U[e], k > 0 ? X[e - g.S] : 0.0, STEP ? p[e] : 0.0};
                      },
                      [&](int i, double c, double sum, const Row& w) {
                        if (j >= g.ny) return;
                        const double t = fma(a.ay2, w.u, fma(a.c1, sum, a.idt2 * w.xp));
                        const double qv = fma(a.c4r, c, -t);
                        q[base + i * g.ny + j] = qv;
                        if constexpr (STEP) acc = fma(qv, w.p, acc);
                      });
  }
  if constexpr (STEP) aat_tail(acc, partials, sc);
}

// Viscosity field (VN) and double-float passes: threads own one (i, j) column
// and march over a chunk of time planes, so p^{k+1} and X^{k-1} stay in registers.
constexpr int AJ = 32, AI = 8;  // block = AJ x AI columns

int aat2_chunk(const Geom& g) {
  const long long cols = (long long)((g.ny + AJ - 1) / AJ) * ((g.nx + AI - 1) / AI);
  const long long want = g.aat_want;  // default 152 * 8: 256-thread blocks, 8 per SM fill it
  long long chunks = (want + cols - 1) / cols;
  if (chunks < 1) chunks = 1;
  if (chunks > g.nt) chunks = g.nt;
  return (int)((g.nt + chunks - 1) / chunks);
}

dim3 aat2_grid(const Geom& g, int kc) {
  return dim3((g.ny + AJ - 1) / AJ, (g.nx + AI - 1) / AI, (g.nt + kc - 1) / kc);
}

struct Cols {
  int jm, jp, im, ip;
};

// Neighbour columns: wrapped on a periodic axis, the point itself at the end
// of a Neumann axis (and on an axis of length 1).
__device__ __forceinline__ Cols aat_cols(const Geom& g, int i, int j) {
  Cols c;
  c.jm = j == 0 ? (g.pery ? g.ny - 1 : 0) : j - 1;
  c.jp = j == g.ny - 1 ? (g.pery ? 0 : g.ny - 1) : j + 1;
  c.im = i == 0 ? (g.perx ? g.nx - 1 : 0) : i - 1;
  c.ip = i == g.nx - 1 ? (g.perx ? 0 : g.nx - 1) : i + 1;
  return c;
}

// Viscosity field (VN): with L = K_nu + I/dt the two passes read
//   pass 1:  kp = K p,  X = dt K_nu p + p^k - p^{k+1}
//   pass 2:  q = (K_nu X)/dt + (X - X^{k-1})/dt^2 + 2 kp,
// K_nu u = sum over the node's faces of kf (u - u_nb); the four face
// coefficients of a column are loaded once, before its march over the planes.
struct FaceCoef {
  double yp, ym, xp, xm;
};

__device__ __forceinline__ FaceCoef face_coef(const Geom& g, int i, int j, const Cols& nb, double scale) {
  FaceCoef f;
  const long long row = (long long)i * g.ny;
  f.yp = g.kfy[row + j] * scale;
  f.ym = g.kfy[row + nb.jm] * scale;
  f.xp = g.actx ? g.kfx[row + j] * scale : 0.0;
  f.xm = g.actx ? g.kfx[(long long)nb.im * g.ny + j] * scale : 0.0;
  return f;
}

template <int ACTX>
__global__ void __launch_bounds__(AJ * AI) k_aat_x(Geom g, AatCoef a, int kc, const double* __restrict__ p,
                                                   double* __restrict__ X, double* __restrict__ KP,
                                                   const DevScalars* sc, int mode) {
  dep_sync();
  if (mode != 0 && sc->cg_done) return;
  const int j = blockIdx.x * AJ + threadIdx.x, i = blockIdx.y * AI + threadIdx.y;
  if (i >= g.nx || j >= g.ny) return;
  const int k0 = blockIdx.z * kc, k1 = min(g.nt, k0 + kc);
  const Cols nb = aat_cols(g, i, j);
  const long long row = (long long)i * g.ny;
  const FaceCoef fc = face_coef(g, i, j, nb, a.dt);
  long long base = (long long)k0 * g.S;
  double c = p[base + row + j];
  for (int k = k0; k < k1; ++k) {
    const double pn = (k + 1 < g.nt) ? p[base + g.S + row + j] : 0.0;
    const double pS = p[base + row + nb.jm], pN = p[base + row + nb.jp];
    double t = a.ay * (pS + pN);
    double pW = 0.0, pE = 0.0;
    if (ACTX) {
      pW = p[base + (long long)nb.im * g.ny + j];
      pE = p[base + (long long)nb.ip * g.ny + j];
      t = fma(a.ax, pW + pE, t);
    }
    const double kp = fma(a.cK, c, -t);
    double kv = fma(fc.yp, c - pN, fc.ym * (c - pS));  // dt K_nu p
    if (ACTX) kv = fma(fc.xp, c - pE, fma(fc.xm, c - pW, kv));
    X[base + row + j] = kv + (c - pn);
    KP[base + row + j] = kp;
    c = pn;
    base += g.S;
  }
}

template <int ACTX>
__global__ void __launch_bounds__(AJ * AI, 3) k_aat_q(Geom g, AatCoef a, int kc, const double* __restrict__ X,
                                                   const double* __restrict__ KP, const double* __restrict__ p,
                                                   double* __restrict__ q, double* partials, DevScalars* sc,
                                                   int mode) {
  dep_sync();
  if (mode != 0 && sc->cg_done) return;
  const int j = blockIdx.x * AJ + threadIdx.x, i = blockIdx.y * AI + threadIdx.y;
  double acc = 0.0;
  if (i < g.nx && j < g.ny) {
    const int k0 = blockIdx.z * kc, k1 = min(g.nt, k0 + kc);
    const Cols nb = aat_cols(g, i, j);
    const long long row = (long long)i * g.ny;
    const FaceCoef fc = face_coef(g, i, j, nb, a.idt);
    long long base = (long long)k0 * g.S;
    double xprev = k0 > 0 ? X[base - g.S + row + j] : 0.0;
    for (int k = k0; k < k1; ++k) {
      const double xc = X[base + row + j];
      const double xS = X[base + row + nb.jm], xN = X[base + row + nb.jp];
      double kv = fma(fc.yp, xc - xN, fc.ym * (xc - xS));  // K_nu X / dt
      if (ACTX) {
        const double xW = X[base + (long long)nb.im * g.ny + j], xE = X[base + (long long)nb.ip * g.ny + j];
        kv = fma(fc.xp, xc - xE, fma(fc.xm, xc - xW, kv));
      }
      const double qv = fma(2.0, KP[base + row + j], fma(a.idt2, xc - xprev, kv));
      q[base + row + j] = qv;
      if (mode == 1) acc = fma(qv, p[base + row + j], acc);
      xprev = xc;
      base += g.S;
    }
  }
  if (mode == 0) return;
  aat_tail(acc, partials, sc);
}

// Blocks of the AAt launch, the larger of its two passes.
int aat_blocks(const Geom& g, int df64) {
  if (g.kfy != nullptr || df64) {
    const dim3 g2 = aat2_grid(g, aat2_chunk(g));
    return (int)((long long)g2.x * g2.y * g2.z);
  }
  return std::max(strip_grid(g, kUPerSm, g.aat_want).blocks, strip_grid(g, kQPerSm, g.aat_want).blocks);
}

// At least the blocks of any reducing launch over the grid, in strips (for any
// blocks per SM) or in columns (viscosity fields, the double-float stencil).
int stencil_blocks_max(const Geom& g) {
  const dim3 g2 = aat2_grid(g, aat2_chunk(g));
  int most = (int)((long long)g2.x * g2.y * g2.z);
  for (int per_sm = 1; per_sm <= 6; ++per_sm) most = std::max({most, strip_grid(g, per_sm).blocks, strip_grid(g, per_sm, g.aat_want).blocks});
  return most;
}

// The same two passes in double-float arithmetic (df64.cuh, the MFG_MIXED_DF
// precision): p is split into FP32 pairs as it is loaded, every stencil
// operation runs on FP32 pairs, X and Kp are stored as pairs (8 bytes, like a
// double), and q is joined back to FP64 (one FP64 add) together with the FP64
// p.q.  About 48 significant bits; ~2 FP64 instructions per point instead of
// 15, the rest on the FP32 pipes.
__device__ __forceinline__ df df_scale2(df a) { return df{2.0f * a.hi, 2.0f * a.lo}; }

template <int ACTX>
__global__ void __launch_bounds__(AJ * AI) k_aat_x_df(Geom g, AatCoef ad, int kc, const double* __restrict__ p,
                                                      df* __restrict__ X, df* __restrict__ KP,
                                                      const DevScalars* sc, int mode) {
  dep_sync();
  if (mode != 0 && sc->cg_done) return;
  const int j = blockIdx.x * AJ + threadIdx.x, i = blockIdx.y * AI + threadIdx.y;
  if (i >= g.nx || j >= g.ny) return;
  const df ax = df_from_double(ad.ax), ay = df_from_double(ad.ay), cK = df_from_double(ad.cK),
           ndt = df_from_double(ad.ndt);
  const int k0 = blockIdx.z * kc, k1 = min(g.nt, k0 + kc);
  const Cols nb = aat_cols(g, i, j);
  const long long row = (long long)i * g.ny;
  long long base = (long long)k0 * g.S;
  df c = df_from_double(p[base + row + j]);
  for (int k = k0; k < k1; ++k) {
    const df pn = (k + 1 < g.nt) ? df_from_double(p[base + g.S + row + j]) : df{0.0f, 0.0f};
    df t = df_mul(ay, df_add(df_from_double(p[base + row + nb.jm]), df_from_double(p[base + row + nb.jp])));
    if (ACTX)
      t = df_add(t, df_mul(ax, df_add(df_from_double(p[base + (long long)nb.im * g.ny + j]),
                                      df_from_double(p[base + (long long)nb.ip * g.ny + j]))));
    const df kp = df_sub(df_mul(cK, c), t);
    X[base + row + j] = df_add(df_mul(ndt, kp), df_sub(c, pn));
    KP[base + row + j] = kp;
    c = pn;
    base += g.S;
  }
}

template <int ACTX>
__global__ void __launch_bounds__(AJ * AI) k_aat_q_df(Geom g, AatCoef ad, int kc, const df* __restrict__ X,
                                                      const df* __restrict__ KP, const double* __restrict__ p,
                                                      double* __restrict__ q, double* partials, DevScalars* sc,
                                                      int mode) {
  dep_sync();
  if (mode != 0 && sc->cg_done) return;
  const int j = blockIdx.x * AJ + threadIdx.x, i = blockIdx.y * AI + threadIdx.y;
  double acc = 0.0;
  if (i < g.nx && j < g.ny) {
    const df c1 = df_from_double(ad.c1), c2 = df_from_double(ad.c2), c4 = df_from_double(ad.c4),
             idt2 = df_from_double(ad.idt2);
    const int k0 = blockIdx.z * kc, k1 = min(g.nt, k0 + kc);
    const Cols nb = aat_cols(g, i, j);
    const long long row = (long long)i * g.ny;
    long long base = (long long)k0 * g.S;
    df xprev = k0 > 0 ? X[base - g.S + row + j] : df{0.0f, 0.0f};
    for (int k = k0; k < k1; ++k) {
      const df xc = X[base + row + j];
      df t = df_mul(c1, df_add(X[base + row + nb.jm], X[base + row + nb.jp]));
      if (ACTX)
        t = df_add(t, df_mul(c2, df_add(X[base + (long long)nb.im * g.ny + j], X[base + (long long)nb.ip * g.ny + j])));
      t = df_add(t, df_mul(idt2, xprev));
      t = df_sub(t, df_scale2(KP[base + row + j]));
      const double qv = df_to_double(df_sub(df_mul(c4, xc), t));
      q[base + row + j] = qv;
      if (mode == 1) acc = fma(qv, p[base + row + j], acc);
      xprev = xc;
      base += g.S;
    }
  }
  if (mode == 0) return;
  aat_tail(acc, partials, sc);
}

void launch_AAt(const Geom& g, const double* p, double* q, double* scratch, double* partials,
                DevScalars* sc, int mode, cudaStream_t s, int df64) {
  const AatCoef a = aat_coef(g);
  const int kc = aat2_chunk(g);
  const dim3 grid = aat2_grid(g, kc), block(AJ, AI);
  if (df64 && g.kfy == nullptr) {  // a viscosity field takes the FP64 stencil
    df* X = reinterpret_cast<df*>(scratch);
    df* KP = X + g.n;
    if (g.actx) {
      launch_k(k_aat_x_df<1>, grid, block, 0, s, g, a, kc, p, X, KP, sc, mode);
      launch_k(k_aat_q_df<1>, grid, block, 0, s, g, a, kc, X, KP, p, q, partials, sc, mode);
    } else {
      launch_k(k_aat_x_df<0>, grid, block, 0, s, g, a, kc, p, X, KP, sc, mode);
      launch_k(k_aat_q_df<0>, grid, block, 0, s, g, a, kc, X, KP, p, q, partials, sc, mode);
    }
    return;
  }
  double* X = scratch;
  double* KP = scratch + g.n;  // K p of a viscosity field, else u
  if (g.kfy != nullptr) {
    if (g.actx) {
      launch_k(k_aat_x<1>, grid, block, 0, s, g, a, kc, p, X, KP, sc, mode);
      launch_k(k_aat_q<1>, grid, block, 0, s, g, a, kc, X, KP, p, q, partials, sc, mode);
    } else {
      launch_k(k_aat_x<0>, grid, block, 0, s, g, a, kc, p, X, KP, sc, mode);
      launch_k(k_aat_q<0>, grid, block, 0, s, g, a, kc, X, KP, p, q, partials, sc, mode);
    }
    return;
  }
  const StripGrid ug = strip_grid(g, kUPerSm, g.aat_want), ag = strip_grid(g, kQPerSm, g.aat_want);
  const int nth = 32 * ag.warps;
  const bool iso = g.actx && g.ax == g.ay, step = mode != 0;
#define MFG_AAT(I, ST) launch_k(k_aat_q2<I, ST>, ag.blocks, nth, 0, s, g, a, ag, KP, X, p, q, partials, sc)
  if (iso)
    launch_k(k_aat_u<true>, ug.blocks, 32 * ug.warps, 0, s, g, a, ug, p, KP, X, sc, mode);
  else
    launch_k(k_aat_u<false>, ug.blocks, 32 * ug.warps, 0, s, g, a, ug, p, KP, X, sc, mode);
  if (iso) { if (step) MFG_AAT(true, true); else MFG_AAT(true, false); }
  else     { if (step) MFG_AAT(false, true); else MFG_AAT(false, false); }
#undef MFG_AAT
}

int aat_kernel_count(int) { return 2; }

}  // namespace mfg
