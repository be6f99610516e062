// The parallel-in-time preconditioner P of Sec. 4 (eq. prec), applied through
// its fully diagonalised form eq. pstrec:
//   P = (V^T (x) H^T (x) G^T) (I (x) Lambda_1 + Lambda_t (x) Lambda_2) (V (x) H (x) G),
// i.e. Alg. 1 with Alg. 2 in place of its per-time-step solve.
//
// Transforms (all real and orthonormal, so the inverse is the transpose):
//   time  V: DCT-VIII for l = 1, DST-I for l = 2 (Sec. 4.1, eigenvalues eq. eigs)
//   space H, G: periodic axis -> discrete Hartley transform, a real orthonormal
//         eigenbasis of the circulant Laplacian (same eigenvalues
//         2 - 2cos(2 pi v/N) as the DFT of Alg. 2); Neumann axis -> DCT-II
//         (eigenvalues 2 - 2cos(pi v/N), Alg. 2).
//   Lambda_1 = nu^2 D^2 + 2 D, Lambda_2 = (nu D + 1/dt)/dt (eq. lambda1, lambda2)
//   with D the tiled spatial eigenvalues of Alg. 2; the per-frequency
//   divisor S = Lambda_1 + lambda_k Lambda_2 (Alg. 2) is formed on
//   the fly, never stored as an n-sized table.
//
// Passes over the data (ping-pong work buffers, 10n words in total):
//   y-forward, x-forward, [time forward, divide by S, time inverse] fused,
//   x-inverse, y-inverse.  A spatial pass is an FFT (k_fft.cu, k_fft_mixed.cu)
//   when the axis length has no prime factor above 13, otherwise a small dense
//   matrix applied along the axis (a SIMT GEMM with the transform matrix on
//   the left); the time pass is a tridiagonal elimination per spatial mode, or the
//   two dense products on the tensor cores (k_time_tc.cu).
#include <algorithm>
#include <cmath>
#include <vector>

#include "mfg_internal.cuh"

namespace mfg {

// ---------------------------------------------------------------- tables --
static void axis_basis(int N, int periodic, std::vector<double>& H, std::vector<double>& lam) {
  H.assign((size_t)N * N, 0.0);
  lam.assign(N, 0.0);
  const double pi = 3.14159265358979323846;
  if (N == 1) {
    H[0] = 1.0;
    return;
  }
  for (int a = 0; a < N; ++a) {
    if (periodic) {
      lam[a] = 2.0 - 2.0 * std::cos(2.0 * pi * a / N);
      for (int b = 0; b < N; ++b) {
        const double th = 2.0 * pi * (double)((long long)a * b % N) / N;
        H[(size_t)a * N + b] = (std::cos(th) + std::sin(th)) / std::sqrt((double)N);
      }
    } else {
      lam[a] = 2.0 - 2.0 * std::cos(pi * a / N);
      const double ca = a == 0 ? std::sqrt(1.0 / N) : std::sqrt(2.0 / N);
      for (int b = 0; b < N; ++b) H[(size_t)a * N + b] = ca * std::cos(pi * a * (2.0 * b + 1.0) / (2.0 * N));
    }
  }
}

static void time_basis(int N, int l, std::vector<double>& V, std::vector<double>& lam) {
  V.assign((size_t)N * N, 0.0);
  lam.assign(N, 0.0);
  const double pi = 3.14159265358979323846;
  for (int k = 0; k < N; ++k) {
    if (l == 1) {
      lam[k] = 2.0 - 2.0 * std::cos(pi * (k + 0.5) / (N + 0.5));
      for (int j = 0; j < N; ++j)
        V[(size_t)k * N + j] = 2.0 / std::sqrt(2.0 * N + 1.0) *
                               std::cos(pi * (2.0 * k + 1.0) * (2.0 * j + 1.0) / (2.0 * (2.0 * N + 1.0)));
    } else {
      lam[k] = 2.0 - 2.0 * std::cos(pi * (k + 1.0) / (N + 1.0));
      for (int j = 0; j < N; ++j)
        V[(size_t)k * N + j] = std::sqrt(2.0 / (N + 1.0)) * std::sin(pi * (j + 1.0) * (k + 1.0) / (N + 1.0));
    }
  }
}

// max |M M^T - I|: orthonormality guard on the host tables.
static double ortho_defect(const std::vector<double>& M, int N) {
  double worst = 0.0;
  for (int a = 0; a < N; ++a)
    for (int b = 0; b < N; ++b) {
      double s = 0.0;
      for (int t = 0; t < N; ++t) s += M[(size_t)a * N + t] * M[(size_t)b * N + t];
      worst = std::fmax(worst, std::fabs(s - (a == b ? 1.0 : 0.0)));
    }
  return worst;
}

template <typename T>
static T* upload(const std::vector<double>& h, std::string* err) {
  std::vector<T> tmp(h.begin(), h.end());
  T* d = nullptr;
  if (cudaMalloc(&d, sizeof(T) * tmp.size()) != cudaSuccess) {
    *err = "cudaMalloc failed for preconditioner tables";
    return nullptr;
  }
  if (cudaMemcpy(d, tmp.data(), sizeof(T) * tmp.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    *err = "cudaMemcpy failed for preconditioner tables";
    cudaFree(d);
    return nullptr;
  }
  return d;
}

__global__ void k_tri_table(double* G, const double* L1, const double* L2, int l, int nt, int S);

int build_prec_tables(const mfg_problem& p, const Geom& g, PrecTables* t, std::string* err) {
  *t = PrecTables{};
  t->nx = g.nx;
  t->ny = g.ny;
  t->nt = g.nt;
  t->l = p.l;
  std::vector<double> Hx, lx, Hy, ly, V, lt;
  axis_basis(g.nx, g.perx, Hx, lx);
  axis_basis(g.ny, g.pery, Hy, ly);
  time_basis(g.nt, p.l == 0 ? 2 : p.l, V, lt);  // l = 0 has no time transform (unused table)
  const double dx_defect = std::fmax(ortho_defect(Hx, g.nx), ortho_defect(Hy, g.ny));
  const double dt_defect = ortho_defect(V, g.nt);
  if (dx_defect > 1e-10 || dt_defect > 1e-10) {
    *err = "transform tables failed the orthonormality check";
    return MFG_ERR_INVALID_ARG;
  }
  double asym = 0.0;
  for (int a = 0; a < g.nt; ++a)
    for (int b = 0; b < g.nt; ++b) asym = std::fmax(asym, std::fabs(V[(size_t)a * g.nt + b] - V[(size_t)b * g.nt + a]));
  if (asym > 1e-12) {
    *err = "time transform table is not symmetric";
    return MFG_ERR_INVALID_ARG;
  }
  std::vector<double> L1((size_t)g.S), L2((size_t)g.S);
  if (p.l == 0) {
    // Exact variant (P = AAt): per spatial mode with Laplacian eigenvalue kappa,
    // the block of eq. largeA is the SPD tridiagonal matrix with diagonal
    // (C, C + 1/dt^2, ...), C = L^2 + 2 kappa, L = nu kappa + 1/dt, and
    // off-diagonal -L/dt.  Its Thomas factors depend only on the mode, so they
    // are formed once here: c_k = off/den_k and 1/den_k, den_k = diag_k - off c_{k-1}.
    std::vector<double> cf((size_t)g.n), idn((size_t)g.n), off((size_t)g.S);
    const double dtv = 1.0 / g.idt;
    for (int a = 0; a < g.nx; ++a)
      for (int b = 0; b < g.ny; ++b) {
        const size_t sidx = (size_t)a * g.ny + b;
        const double kap = lx[a] * g.ax + ly[b] * g.ay;
        const double Ls = g.nu * kap + 1.0 / dtv;
        const double Cs = Ls * Ls + 2.0 * kap;
        const double o = -Ls / dtv;
        off[sidx] = o;
        double cprev = 0.0;
        for (int k = 0; k < g.nt; ++k) {
          const double diag = Cs + (k >= 1 ? 1.0 / (dtv * dtv) : 0.0);
          const double den = diag - (k >= 1 ? o * cprev : 0.0);
          const size_t e = (size_t)k * g.S + sidx;
          idn[e] = 1.0 / den;
          cprev = o / den;
          cf[e] = cprev;
        }
      }
    t->thc64 = upload<double>(cf, err);
    t->thd64 = upload<double>(idn, err);
    t->tho64 = upload<double>(off, err);
    t->thc32 = upload<float>(cf, err);
    t->thd32 = upload<float>(idn, err);
    t->tho32 = upload<float>(off, err);
    if (!t->thc64 || !t->thd64 || !t->tho64 || !t->thc32 || !t->thd32 || !t->tho32) {
      free_prec_tables(t);
      return MFG_ERR_CUDA;
    }
  }
  const double dtv = 1.0 / g.idt, nu = g.nu;
  for (int a = 0; a < g.nx; ++a)
    for (int b = 0; b < g.ny; ++b) {
      const double D = lx[a] * g.ax + ly[b] * g.ay;
      L1[(size_t)a * g.ny + b] = nu * nu * D * D + 2.0 * D;
      L2[(size_t)a * g.ny + b] = (nu * D + 1.0 / dtv) / dtv;
    }
  t->Hx64 = upload<double>(Hx, err);
  t->Hy64 = upload<double>(Hy, err);
  t->Vt64 = upload<double>(V, err);
  t->lamt64 = upload<double>(lt, err);
  t->L1_64 = upload<double>(L1, err);
  t->L2_64 = upload<double>(L2, err);
  t->Hx32 = upload<float>(Hx, err);
  t->Hy32 = upload<float>(Hy, err);
  t->Vt32 = upload<float>(V, err);
  t->lamt32 = upload<float>(lt, err);
  t->L1_32 = upload<float>(L1, err);
  t->L2_32 = upload<float>(L2, err);
  // FFT twiddles: tw[m] = (cos, sin)(2 pi m/N), dct[k] = (cos, sin)(pi k/(2N)).
  auto fft_tables = [&](int N, double** tw64, float** tw32, double** dc64, float** dc32) {
    if (!fft_supported(N)) return true;
    const double pi = 3.14159265358979323846;
    std::vector<double> tw((size_t)2 * N), dc((size_t)2 * N);
    for (int m = 0; m < N; ++m) {
      tw[2 * m] = std::cos(2.0 * pi * m / N);
      tw[2 * m + 1] = std::sin(2.0 * pi * m / N);
    }
    for (int k = 0; k < N; ++k) {
      dc[2 * k] = std::cos(pi * k / (2.0 * N));
      dc[2 * k + 1] = std::sin(pi * k / (2.0 * N));
    }
    *tw64 = upload<double>(tw, err);
    *tw32 = upload<float>(tw, err);
    *dc64 = upload<double>(dc, err);
    *dc32 = upload<float>(dc, err);
    return *tw64 && *tw32 && *dc64 && *dc32;
  };
  const bool fft_ok = (g.nx == 1 || fft_tables(g.nx, &t->twx64, &t->twx32, &t->dctx64, &t->dctx32)) &&
                      fft_tables(g.ny, &t->twy64, &t->twy32, &t->dcty64, &t->dcty32);
  if (!fft_ok || !t->Hx64 || !t->Hy64 || !t->Vt64 || !t->lamt64 || !t->L1_64 || !t->L2_64 || !t->Hx32 ||
      !t->Hy32 || !t->Vt32 || !t->lamt32 || !t->L1_32 || !t->L2_32) {
    free_prec_tables(t);
    return MFG_ERR_CUDA;
  }
  if (p.nu_field != nullptr) {
    const int rc = build_band_tables(p, g, lt.data(), t, err);
    if (rc != MFG_OK) {
      free_prec_tables(t);
      return rc;
    }
  }
  return MFG_OK;
}

// The factors are n doubles that the elimination can do without (it then forms them
// per apply), so a plan takes them last, and only where `reserve` bytes stay free.
int build_time_factors(const mfg_problem& p, const Geom& g, size_t reserve, PrecTables* t, std::string* err) {
  if (p.precision != MFG_FP64 || p.l == 0 || t->band_w > 0) return MFG_OK;
  const size_t vec = sizeof(double) * (size_t)g.n;
  size_t avail = 0, total = 0;
  if (cudaMemGetInfo(&avail, &total) != cudaSuccess || avail < vec + reserve ||
      cudaMalloc(&t->tri64, vec) != cudaSuccess) {
    t->tri64 = nullptr;
    cudaGetLastError();
    return MFG_OK;
  }
  launch_k(k_tri_table, (g.S + 127) / 128, 128, 0, (cudaStream_t) nullptr, t->tri64, t->L1_64, t->L2_64, p.l, g.nt, g.S);
  if (cudaStreamSynchronize(nullptr) != cudaSuccess) {
    *err = "building the time elimination's factors failed";
    return MFG_ERR_CUDA;
  }
  return MFG_OK;
}

void free_prec_tables(PrecTables* t) {
  void* ptrs[] = {t->Hx64, t->Hy64, t->Vt64, t->lamt64, t->L1_64, t->L2_64, t->Hx32, t->Hy32,
                  t->Vt32, t->lamt32, t->L1_32, t->L2_32, t->twx64, t->twx32, t->dctx64, t->dctx32,
                  t->twy64, t->twy32, t->dcty64, t->dcty32, t->thc64, t->thd64, t->tho64,
                  t->thc32, t->thd32, t->tho32, t->tri64, t->kfx, t->kfy, t->band_perm, t->bandc64,
                  t->bandr64, t->bandc32, t->bandr32};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  *t = PrecTables{};
}

// ------------------------------------------------------- axis transform --
// out(a, col) = sum_b M(a, b) in(b, col), M(a, b) = trans ? M[b*N + a] : M[a*N + b],
// where column col = (o, i) addresses in[(o*N + b)*inner + i].  CONTIG: the
// transformed axis is the contiguous one (inner == 1).
constexpr int BM = 64, BN = 64, BK = 16;

template <typename TI, typename T, typename TO, bool CONTIG>
__global__ void __launch_bounds__(256) k_axis(const TI* __restrict__ in, TO* __restrict__ out,
                                              const T* __restrict__ M, int N, long long inner,
                                              long long ncols, int trans, const DevScalars* sc) {
  dep_sync();
  if (sc != nullptr && sc->cg_done) return;
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  const int tid = threadIdx.x;
  const int tr = CONTIG ? (tid & 15) : (tid >> 4);
  const int tc = CONTIG ? (tid >> 4) : (tid & 15);
  const int a0 = blockIdx.y * BM;
  const long long c0 = (long long)blockIdx.x * BN;
  T acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = T(0);

  for (int b0 = 0; b0 < N; b0 += BK) {
    // A tile: As[bb][aa] = M(a0+aa, b0+bb)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int s = tid + 256 * q;
      int aa, bb;
      if (trans) { aa = s % BM; bb = s / BM; } else { bb = s % BK; aa = s / BK; }
      const int a = a0 + aa, b = b0 + bb;
      T val = T(0);
      if (a < N && b < N) val = trans ? M[(long long)b * N + a] : M[(long long)a * N + b];
      As[bb][aa] = val;
    }
    // B tile: Bs[bb][cc] = in(b0+bb, c0+cc)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int s = tid + 256 * q;
      int bb, cc;
      if (CONTIG) { bb = s % BK; cc = s / BK; } else { cc = s % BN; bb = s / BN; }
      const int b = b0 + bb;
      const long long col = c0 + cc;
      T val = T(0);
      if (b < N && col < ncols) {
        const long long o = col / inner, i = col - o * inner;
        val = (T)in[(o * N + b) * inner + i];
      }
      Bs[bb][cc] = val;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T av[4], bv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) av[u] = As[kk][tr + 16 * u];
#pragma unroll
      for (int v = 0; v < 4; ++v) bv[v] = Bs[kk][tc + 16 * v];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int a = a0 + tr + 16 * u;
    if (a >= N) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const long long col = c0 + tc + 16 * v;
      if (col >= ncols) continue;
      const long long o = col / inner, i = col - o * inner;
      out[(o * N + a) * inner + i] = (TO)acc[u][v];
    }
  }
}

template <typename TI, typename T, typename TO>
static void axis_pass(const TI* in, TO* out, const T* M, int N, long long inner, long long outer,
                      int trans, const DevScalars* sc, cudaStream_t s) {
  const long long ncols = inner * outer;
  dim3 grid((unsigned)((ncols + BN - 1) / BN), (N + BM - 1) / BM);
  if (inner == 1)
    launch_k(k_axis<TI, T, TO, true>, grid, 256, 0, s, in, out, M, N, inner, ncols, trans, sc);
  else
    launch_k(k_axis<TI, T, TO, false>, grid, 256, 0, s, in, out, M, N, inner, ncols, trans, sc);
}

// ------------------------------------------------------------ time pass --
// Time forward, division by S(k, s) and time inverse of Alg. 1 in one
// elimination.  V diagonalises the second difference D of Sec. 4.1 (tridiagonal
// -1, 2, -1, first diagonal entry l), so per spatial mode s
//   V^T diag_k(1 / (Lambda_1 + lambda_k Lambda_2)) V = (Lambda_1 I + Lambda_2 D)^{-1},
// a symmetric positive definite tridiagonal system: O(N_t) operations per mode
// where the two dense products take O(N_t^2).  With rho = Lambda_1 / Lambda_2 >= 0
// the pivots of the elimination are 1 + delta_k,
//   delta_0 = l - 1 + rho,  delta_k = rho + delta_{k-1} / (1 + delta_{k-1}),
// sums and quotients of non-negative numbers only, so neither a small rho (the
// low modes) nor a large one loses digits; g_k = 1 / (1 + delta_k),
//   e_k = b_k + g_{k-1} e_{k-1},   x_k = g_k (e_k / Lambda_2 + x_{k+1}).
//
// One thread per mode.  The pass is bound by memory (one read and one write of
// the data) in FP32 and by ~9 FP64 instructions per element in FP64, if enough
// bytes are in flight: a thread issues its whole column of N_t loads as
// cp.async into its own column of shared memory, forms the g_k (which need no
// data) while they land, and then runs the two recurrences in place.  No
// thread reads another's column, so nothing synchronises.  512^2 x 128 FP32:
// 169 us (dense products on the tensor cores) -> 64 us, with a tenth of the
// apply's error (3e-6 -> 3e-7 against 64 bits); 256^2 x 64 FP64: 973 us (dense
// products on the CUDA cores) -> 41 us with the plan's g_k.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* smem, const T* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"((int)sizeof(T)) : "memory");
}

// 1/x to one unit in the last place
__device__ __forceinline__ float recip(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

// The g_k of every mode, [nt][S]: FP64 plans keep them (8 bytes per element read
// instead of 6 of the 9 FP64 instructions; in FP32 they cost less than their bytes).
// P^{-1} 256^2 x 64 740 -> 678 us; the 64-point 1-D solve 7.9 -> 6.9 ms, where the g_k
// were a serial chain in front of every pass.
__global__ void __launch_bounds__(128) k_tri_table(double* __restrict__ G, const double* __restrict__ L1,
                                                   const double* __restrict__ L2, int l, int nt, int S) {
  dep_sync();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const double rho = L1[s] / L2[s];
  double d = (double)(l - 1) + rho;
  for (int k = 0;; ++k) {
    const double g = recip(1.0 + d);
    G[(long long)k * S + s] = g;
    if (k + 1 == nt) break;
    d = fma(d, g, rho);
  }
}

template <typename T, bool TAB>
__global__ void __launch_bounds__(128) k_time_tri(const T* __restrict__ in, T* __restrict__ out,
                                                  const T* __restrict__ L1, const T* __restrict__ L2,
                                                  const T* __restrict__ tab, int l, int nt, int S,
                                                  const DevScalars* sc) {
  dep_sync();
  if (sc != nullptr && sc->cg_done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int bd = blockDim.x, s = blockIdx.x * bd + threadIdx.x;
  T* E = reinterpret_cast<T*>(smem_raw) + threadIdx.x;  // [nt][bd], this thread's column
  T* G = E + (size_t)nt * bd;
  if (s >= S) return;
  const T* src = in + s;
#pragma unroll 8
  for (int k = 0; k < nt; ++k) {
    cp_async_elem(E + k * bd, src + (long long)k * S);
    if constexpr (TAB) cp_async_elem(G + k * bd, tab + (long long)k * S + s);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  const T l2 = L2[s], il2 = T(1) / l2;
  T g;
  if constexpr (!TAB) {
    const T rho = L1[s] / l2;
    T d = T(l - 1) + rho;
    g = recip(T(1) + d);
    G[0] = g;
#pragma unroll 4
    for (int k = 1; k < nt; ++k) {
      d = fma(d, g, rho);
      g = recip(T(1) + d);
      G[k * bd] = g;
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  // eight steps at a time: their shared loads are issued together, ahead of
  // the chain and of the stores they cannot be moved across
  T e = T(0);
  g = T(0);
  int k = 0;
  for (; k + 8 <= nt; k += 8) {
    T ev[8], gv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) { ev[u] = E[(k + u) * bd]; gv[u] = G[(k + u) * bd]; }
#pragma unroll
    for (int u = 0; u < 8; ++u) { e = fma(u ? gv[u - 1] : g, e, ev[u]); ev[u] = e; }
    g = gv[7];
#pragma unroll
    for (int u = 0; u < 8; ++u) E[(k + u) * bd] = ev[u];
  }
  for (; k < nt; ++k) {
    e = fma(g, e, E[k * bd]);
    E[k * bd] = e;
    g = G[k * bd];
  }
  T* dst = out + s;
  T x = T(0);
  for (k = nt; k % 8 != 0; --k) {
    x = G[(k - 1) * bd] * fma(E[(k - 1) * bd], il2, x);
    dst[(long long)(k - 1) * S] = x;
  }
  for (; k > 0; k -= 8) {
    T ev[8], gv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) { ev[u] = E[(k - 1 - u) * bd]; gv[u] = G[(k - 1 - u) * bd]; }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      x = gv[u] * fma(ev[u], il2, x);
      dst[(long long)(k - 1 - u) * S] = x;
    }
  }
}

// Threads per block: 128, 64 or 32, the largest whose two columns per thread
// fit in 64 KB (three blocks per SM) and whose grid still has a block per SM.
template <typename T>
static int tri_threads(int nt, int S) {
  int bd = 128;
  while (bd > 32 && (2 * sizeof(T) * (size_t)nt * bd > 65536 || (S + bd - 1) / bd < 152)) bd >>= 1;
  return bd;
}

template <typename T>
static void time_pass(const T* in, T* out, const T* L1, const T* L2, const T* tab, int l, int nt, int S,
                      const DevScalars* sc, cudaStream_t s) {
  const int bd = tri_threads<T>(nt, S), nb = (S + bd - 1) / bd;
  const size_t sm = 2 * sizeof(T) * (size_t)nt * bd;
  if (tab != nullptr)
    launch_k(k_time_tri<T, true>, nb, bd, sm, s, in, out, L1, L2, tab, l, nt, S, sc);
  else
    launch_k(k_time_tri<T, false>, nb, bd, sm, s, in, out, L1, L2, tab, l, nt, S, sc);
}

// Exact time solve of the l = 0 variant: per spatial mode s, the tridiagonal
// system of eq. largeA in time by Thomas elimination with the precomputed
// factors (forward sweep into `out`, then back substitution in place).  One
// thread per mode; loads at a fixed k are contiguous across the threads.
template <typename T>
__global__ void __launch_bounds__(256) k_thomas(const T* __restrict__ in, T* __restrict__ out,
                                                const T* __restrict__ cf, const T* __restrict__ idn,
                                                const T* __restrict__ off, int nt, int S,
                                                const DevScalars* sc) {
  dep_sync();
  if (sc != nullptr && sc->cg_done) return;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
    const T o = off[s];
    T d = T(0);
#pragma unroll 8
    for (int k = 0; k < nt; ++k) {
      const long long e = (long long)k * S + s;
      d = (in[e] - o * d) * idn[e];
      out[e] = d;
    }
    T x = d;
#pragma unroll 8
    for (int k = nt - 2; k >= 0; --k) {
      const long long e = (long long)k * S + s;
      x = out[e] - cf[e] * x;
      out[e] = x;
    }
  }
}

template <typename T>
static void precond_typed(const Geom& g, const T* Hx, const T* Hy, const T* V, const T* lamt,
                          const T* L1, const T* L2, const T* twx, const T* dctx, const T* twy,
                          const T* dcty, const T* thc, const T* thd, const T* tho, const T* tri, int l,
                          const double* r, double* z, T* w0, T* w1,
                          const DevScalars* sc, cudaStream_t s, const PcgDot* dot,
                          const PcgZr* zr, bool tc = false) {
  const long long S = g.S, n = g.n;
  const bool fy = g.fft_y && twy != nullptr && fft_supported(g.ny);
  const bool fx = g.fft_x && twx != nullptr && fft_supported(g.nx);
  // y forward: axis length ny, contiguous
  if (fy) {
    fft_y_forward<T>(g.ny, g.pery, r, w0, twy, dcty, n / g.ny, sc, s, zr);
  } else {
    if (zr) launch_update_zr(n, zr->z, zr->r, zr->p, zr->q, zr->partials, zr->sc, s, g.vec_blocks);
    axis_pass<double, T, T>(r, w0, Hy, g.ny, 1, n / g.ny, 0, sc, s);
  }
  T* a = w0;
  T* b = w1;
  if (g.nx > 1) {
    if (fx)
      fft_x<T>(g.nx, g.perx, 0, a, b, twx, dctx, g.ny, (long long)g.nt, sc, s);
    else
      axis_pass<T, T, T>(a, b, Hx, g.nx, g.ny, (long long)g.nt, 0, sc, s);
    T* t = a; a = b; b = t;
  }
  if (thc != nullptr) {
    launch_k(k_thomas<T>, (int)((S + 255) / 256), 256, 0, s, a, b, thc, thd, tho, g.nt, (int)S, sc);
  } else if constexpr (sizeof(T) == 4) {
    if (tc && !g.time_simt && time_tc_supported(g.nt))
      launch_time_tc(a, b, V, lamt, L1, L2, g.nt, (int)S, sc, s);
    else
      time_pass<T>(a, b, L1, L2, tri, l, g.nt, (int)S, sc, s);
  } else {
    time_pass<T>(a, b, L1, L2, tri, l, g.nt, (int)S, sc, s);
  }
  { T* t = a; a = b; b = t; }
  if (g.nx > 1) {
    if (fx)
      fft_x<T>(g.nx, g.perx, 1, a, b, twx, dctx, g.ny, (long long)g.nt, sc, s);
    else
      axis_pass<T, T, T>(a, b, Hx, g.nx, g.ny, (long long)g.nt, 1, sc, s);
    T* t = a; a = b; b = t;
  }
  if (fy) {
    fft_y_inverse<T>(g.ny, g.pery, a, z, twy, dcty, n / g.ny, sc, s, dot);
  } else {
    axis_pass<T, T, double>(a, z, Hy, g.ny, 1, n / g.ny, 1, sc, s);
    if (dot) launch_dot_beta(n, dot->r, z, dot->q, dot->flex, dot->partials, dot->sc, s, g.vec_blocks);
  }
}

void launch_precond(const Geom& g, const PrecTables& t, int precision, const double* r, double* z,
                    double* work64, float* work32, const DevScalars* sc, cudaStream_t s,
                    const PcgDot* dot, const PcgZr* zr) {
  if (t.band_w > 0) {  // viscosity field: time transforms around banded per-frequency solves
    if (zr) launch_update_zr(g.n, zr->z, zr->r, zr->p, zr->q, zr->partials, zr->sc, s, g.vec_blocks);
    launch_precond_band(g, t, precision, r, z, work64, work32, sc, s);
    if (dot) launch_dot_beta(g.n, dot->r, z, dot->q, dot->flex, dot->partials, dot->sc, s, g.vec_blocks);
    return;
  }
  if (precision == MFG_MIXED || precision == MFG_MIXED_DF || precision == MFG_MIXED_TC)
    precond_typed<float>(g, t.Hx32, t.Hy32, t.Vt32, t.lamt32, t.L1_32, t.L2_32, t.twx32, t.dctx32,
                         t.twy32, t.dcty32, t.thc32, t.thd32, t.tho32, nullptr, t.l, r, z, work32, work32 + g.n,
                         sc, s, dot, zr, precision == MFG_MIXED_TC);
  else
    precond_typed<double>(g, t.Hx64, t.Hy64, t.Vt64, t.lamt64, t.L1_64, t.L2_64, t.twx64, t.dctx64,
                          t.twy64, t.dcty64, t.thc64, t.thd64, t.tho64, t.tri64, t.l, r, z, work64, work64 + g.n,
                          sc, s, dot, zr);
}

int precond_kernel_count(const Geom& g) { return g.kfy != nullptr ? 4 : (g.nx > 1 ? 5 : 3); }

// Kernels of a preconditioner apply that also runs the PCG update and dot products.
int precond_step_kernel_count(const Geom& g, const PrecTables& t) {
  if (t.band_w > 0) return 4 + 2;
  const bool fused = g.fft_y && t.twy32 != nullptr && fft_supported(g.ny);
  return precond_kernel_count(g) + (fused ? 0 : 2);
}

// Opt-in shared memory for the time pass; called once per device before any
// launch or stream capture.
int precond_configure() {
  // one warp's columns of the longest time axis
  const int tri = 2 * kMaxNt * 32;
  int bad = cudaFuncSetAttribute(k_time_tri<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 std::max(65536, tri * (int)sizeof(double))) != cudaSuccess;
  bad |= cudaFuncSetAttribute(k_time_tri<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 std::max(65536, tri * (int)sizeof(double))) != cudaSuccess;
  bad |= cudaFuncSetAttribute(k_time_tri<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              std::max(65536, tri * (int)sizeof(float))) != cudaSuccess;
  bad |= fft_configure() != MFG_OK;
  bad |= band_configure() != MFG_OK;
  bad |= prox_configure() != MFG_OK;
  bad |= time_tc_configure() != MFG_OK;
  return bad ? MFG_ERR_CUDA : MFG_OK;
}

}  // namespace mfg
