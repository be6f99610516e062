// Spatial passes by FFT for axis lengths up to 2048 whose prime factors are at
// most 13 (the lengths k_fft.cu does not take; longer factors stay with the
// dense transform).
//
// Same transforms as k_fft.cu: real lines packed in pairs, a Stockham FFT in
// shared memory (mixed radix, Govindaraju et al., SC 2008), Hermitian split;
// DCT-II and DCT-III through Makhoul's reordering, whose identity holds for odd
// N as well.  What differs is that N is a run-time value: a length is factored
// into radices 2..8, 10, 11, 13 on the host, and a stage's butterflies of all of the
// block's lines are spread over all its threads (a line of 150 points has 25
// or 30 butterflies per stage: one warp per line would idle).  Index divisions
// are multiplications by a precomputed reciprocal.
//
// The dense transform costs 2N flops per element; this costs ~5 log2 N and
// leaves the pass bound by its shared-memory stages.  200 x 150 x 60, FP32: four
// dense passes 300 us -> ~75 us together (P^{-1} 307 -> 87 us, its error against
// 64 bits 4.8e-7 -> 1.7e-7); 8 is the shortest line that fills a stage.
#include <cmath>

#include "fft_common.cuh"
#include "pcg_tail.cuh"
#include "reduce.cuh"

namespace mfg {
namespace {

constexpr int kMaxN = 2048, kMaxStages = 10, kBlock = 256;  // kBlock: most threads per block

// x / d for x * d < 2^32 (m = ceil(2^32 / d); d = 1 has m = 0).
struct Div {
  unsigned m;
};
__device__ __forceinline__ int quot(int x, Div d) { return d.m ? (int)__umulhi((unsigned)x, d.m) : x; }
Div make_div(int d) { return Div{d == 1 ? 0u : (unsigned)(((1ull << 32) + d - 1) / (unsigned)d)}; }

struct FftPlan {
  int N, stages, lines;  // lines: complex lines per block
  Div dN;
  double r1, r2, rh;  // 1/sqrt(N), sqrt(2/N), 1/sqrt(2N): formed on the host, an FP64 root per thread is not free
  int radix[kMaxStages];
  Div dB[kMaxStages];   // by N / R, the butterflies of a line
  int Ns[kMaxStages];
  Div dNs[kMaxStages];
};

// Radices of N, odd ones first: the early stages store with strides of R, which
// an odd R spreads over all banks.  0 stages if a prime factor exceeds 13.
int factor(int N, int* radix) {
  int e[14] = {0};
  for (int p : {2, 3, 5, 7, 11, 13})
    while (N % p == 0) { N /= p; ++e[p]; }
  if (N != 1) return 0;
  int n = 0, tail[kMaxStages], nt = 0;
  if (e[2] % 3 == 1) {  // a single 2 joins a 5 or a 3
    if (e[5] > 0) { tail[nt++] = 10; --e[5]; --e[2]; }
    else if (e[3] > 0) { tail[nt++] = 6; --e[3]; --e[2]; }
  }
  for (int p : {13, 11, 7, 5, 3})
    while (e[p]-- > 0) { if (n == kMaxStages) return 0; radix[n++] = p; }
  while (e[2] >= 3) { tail[nt++] = 8; e[2] -= 3; }
  if (e[2]) tail[nt++] = 1 << e[2];
  if (n + nt > kMaxStages) return 0;
  for (int i = 0; i < nt; ++i) radix[n++] = tail[i];
  return n;
}

template <typename T>
size_t smem_bytes(int N, int lines) {
  return ((size_t)2 * lines * (N + 1) + 2 * (size_t)N) * sizeof(cx<T>);
}

template <typename T>
__device__ __forceinline__ cx<T> cadd(cx<T> a, cx<T> b) { return cx<T>{a.x + b.x, a.y + b.y}; }
template <typename T>
__device__ __forceinline__ cx<T> csub(cx<T> a, cx<T> b) { return cx<T>{a.x - b.x, a.y - b.y}; }

// DFT of R values in place, sign sgn; w[j * nb] = exp(2 pi i j / R) in the line's table.
template <typename T, int R>
__device__ __forceinline__ void dft(cx<T> (&a)[R], const cx<T>* w, int nb, T sgn) {
  auto rot = [&](cx<T> v) { return cx<T>{-sgn * v.y, sgn * v.x}; };  // times sgn i
  if constexpr (R == 2) {
    const cx<T> t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  } else if constexpr (R == 4) {
    const cx<T> s0 = cadd(a[0], a[2]), d0 = csub(a[0], a[2]), s1 = cadd(a[1], a[3]), d1 = rot(csub(a[1], a[3]));
    a[0] = cadd(s0, s1);
    a[1] = cadd(d0, d1);
    a[2] = csub(s0, s1);
    a[3] = csub(d0, d1);
  } else if constexpr (R == 8) {
    cx<T> e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
    dft<T, 4>(e, w, nb, sgn);
    dft<T, 4>(o, w, nb, sgn);
    const T h = T(0.70710678118654752440);  // cos(pi/4)
    o[1] = cx<T>{h * (o[1].x - sgn * o[1].y), h * (o[1].y + sgn * o[1].x)};
    o[2] = rot(o[2]);
    o[3] = cx<T>{h * (-o[3].x - sgn * o[3].y), h * (-o[3].y + sgn * o[3].x)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = cadd(e[k], o[k]);
      a[k + 4] = csub(e[k], o[k]);
    }
  } else if constexpr (R % 2 == 0) {
    // R = 2 P, P odd: the prime-factor map n = P n1 + 2 n2, k = P k1 + (P + 1) k2
    // (mod R) splits it into P-point DFTs of sums and differences, no twiddles
    constexpr int P = R / 2;
    cx<T> u[P], v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
      u[i] = cadd(a[(2 * i) % R], a[(2 * i + P) % R]);
      v[i] = csub(a[(2 * i) % R], a[(2 * i + P) % R]);
    }
    dft<T, P>(u, w, 2 * nb, sgn);
    dft<T, P>(v, w, 2 * nb, sgn);
#pragma unroll
    for (int k = 0; k < P; ++k) {
      a[((P + 1) * k) % R] = u[k];
      a[((P + 1) * k + P) % R] = v[k];
    }
  } else {
    // odd R: X_k, X_{R-k} = a_0 + sum_j cos(2 pi j k/R) (a_j + a_{R-j})
    //                       +- i sgn sum_j sin(2 pi j k/R) (a_j - a_{R-j})
    constexpr int H = (R - 1) / 2;
    cx<T> s[H], d[H];
    T c[H], n[H];
    cx<T> x0 = a[0];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      s[j] = cadd(a[j + 1], a[R - 1 - j]);
      d[j] = csub(a[j + 1], a[R - 1 - j]);
      const cx<T> t = w[(j + 1) * nb];
      c[j] = t.x;
      n[j] = t.y;
      x0 = cadd(x0, s[j]);
    }
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      cx<T> p = a[0], q{T(0), T(0)};
#pragma unroll
      for (int j = 1; j <= H; ++j) {
        const int jk = (j * k) % R, f = jk <= H ? jk : R - jk;  // folded: sin changes sign
        p.x = fma(c[f - 1], s[j - 1].x, p.x);
        p.y = fma(c[f - 1], s[j - 1].y, p.y);
        const T sn = jk <= H ? n[f - 1] : -n[f - 1];
        q.x = fma(sn, d[j - 1].x, q.x);
        q.y = fma(sn, d[j - 1].y, q.y);
      }
      q = rot(q);
      a[k] = cadd(p, q);
      a[R - k] = csub(p, q);
    }
    a[0] = x0;
  }
}

// One Stockham stage of all lines of the block: v_r = src[j + r N/R] twiddled by
// exp(sgn 2 pi i r (j mod Ns) / (R Ns)), dst[(j - j mod Ns) R + j mod Ns + r Ns].
template <typename T, int R>
__device__ void stage(const cx<T>* src, cx<T>* dst, const cx<T>* tw, int N, int lines, int Ns, Div dB, Div dNs, T sgn) {
  const int nb = N / R, step = quot(nb, dNs);
  for (int idx = threadIdx.x; idx < lines * nb; idx += blockDim.x) {
    const int q = quot(idx, dB), j = idx - q * nb, b = quot(j, dNs), k = j - b * Ns;
    const cx<T>* sp = src + q * (N + 1) + j;
    cx<T> a[R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = sp[r * nb];
    if (Ns > 1) {
      const int ks = k * step;
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const cx<T> t = tw[r * ks];
        const T wy = sgn * t.y, x = a[r].x;
        a[r].x = x * t.x - a[r].y * wy;
        a[r].y = x * wy + a[r].y * t.x;
      }
    }
    dft<T, R>(a, tw, nb, sgn);
    cx<T>* dp = dst + q * (N + 1) + b * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dp[r * Ns] = a[r];
  }
}

// All stages; the result's buffer (0: the first, 1: the second) is returned.
// One copy per type, shared by the kernels.
template <typename T>
__device__ __noinline__ int fft_stages(const FftPlan& P, T sgn) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* b0 = reinterpret_cast<cx<T>*>(smem_raw);
  cx<T>* b1 = b0 + P.lines * (P.N + 1);
  const cx<T>* tw = b1 + P.lines * (P.N + 1);
  for (int i = 0; i < P.stages; ++i) {
    const cx<T>* src = (i & 1) ? b1 : b0;
    cx<T>* dst = (i & 1) ? b0 : b1;
    switch (P.radix[i]) {
#define MFG_STAGE(R) case R: stage<T, R>(src, dst, tw, P.N, P.lines, P.Ns[i], P.dB[i], P.dNs[i], sgn); break;
      MFG_STAGE(2) MFG_STAGE(3) MFG_STAGE(4) MFG_STAGE(5) MFG_STAGE(6) MFG_STAGE(7) MFG_STAGE(8) MFG_STAGE(10)
      MFG_STAGE(11) MFG_STAGE(13)
#undef MFG_STAGE
      default: break;
    }
    __syncthreads();
  }
  return P.stages & 1;
}

// One block: 2 P.lines real lines (rows when inner = 1, else columns of the
// strided axis; blockIdx.y the plane).  DOT, ZR as in k_fft.cu.
template <typename T, typename TI, typename TO, bool CONTIG, bool DOT, bool ZR>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 8 ? 2 : 3) k_fft_mixed(const TI* __restrict__ in, TO* __restrict__ out,
                                                      const T* __restrict__ tw, const T* __restrict__ dct,
                                                      const __grid_constant__ FftPlan P, int mode, int llb,
                                                      long long inner, long long nlines, const DevScalars* sc,
                                                      DotFuse df, ZrFuse zf) {
  dep_sync();
  if (sc != nullptr && sc->cg_done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = P.N, NP = N + 1, CL = P.lines, LB = 2 * CL, tid = threadIdx.x, nth = blockDim.x;
  cx<T>* buf0 = reinterpret_cast<cx<T>*>(smem_raw);
  cx<T>* buf1 = buf0 + CL * NP;
  T* real1 = reinterpret_cast<T*>(buf1);  // [LB][NP] real staging
  cx<T>* tws = buf1 + CL * NP;
  cx<T>* dcs = tws + N;
  for (int q = tid; q < N; q += nth) {
    tws[q] = cx<T>{tw[2 * q], tw[2 * q + 1]};
    if (mode != FFT_DHT) {  // phases with the transform's scale, as in k_fft.cu
      const T f = mode == FFT_DCT2 ? T(0.5) * (q == 0 ? (T)P.r1 : (T)P.r2) : (q == 0 ? (T)P.r1 : (T)P.rh);
      dcs[q] = cx<T>{f * dct[2 * q], f * dct[2 * q + 1]};
    }
  }
  const long long line0 = (long long)blockIdx.x * LB, o = blockIdx.y;
  const int total = LB * N;
  auto element = [&](int idx, int& l, int& i, long long& addr) -> bool {
    if (CONTIG) { l = quot(idx, P.dN); i = idx - l * N; } else { i = idx >> llb; l = idx & (LB - 1); }
    const long long line = line0 + l;
    addr = CONTIG ? line * N + i : (o * N + i) * inner + line;
    return idx < total && line < nlines;
  };
  auto put = [&](int l, int i, T v) {
    if (mode == FFT_DCT3) {
      real1[l * NP + i] = v;
    } else {
      const int p = mode == FFT_DCT2 ? ((i & 1) ? N - 1 - (i >> 1) : (i >> 1)) : i;
      reinterpret_cast<T*>(&buf0[(l >> 1) * NP + p])[l & 1] = v;
    }
  };
  double rr = 0.0;
  const double alpha = ZR ? zf.sc->alpha : 0.0;
  // loads in batches, all of a batch issued before the first is used
  constexpr int BL = ZR ? 4 : 8;
  for (int e0 = tid; e0 < total; e0 += nth * BL) {
    int ls[BL], is[BL];
    long long ad[BL];
    bool lv[BL];
#pragma unroll
    for (int u = 0; u < BL; ++u) lv[u] = element(e0 + nth * u, ls[u], is[u], ad[u]);
    if constexpr (ZR) {
      double zv[BL], pv[BL], rv[BL], qv[BL];
#pragma unroll
      for (int u = 0; u < BL; ++u) {
        zv[u] = lv[u] ? zf.z[ad[u]] : 0.0;
        pv[u] = lv[u] ? zf.p[ad[u]] : 0.0;
        rv[u] = lv[u] ? zf.r[ad[u]] : 0.0;
        qv[u] = lv[u] ? zf.q[ad[u]] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < BL; ++u) {
        const double rn = fma(-alpha, qv[u], rv[u]);
        if (lv[u]) {
          zf.z[ad[u]] = fma(alpha, pv[u], zv[u]);
          zf.r[ad[u]] = rn;
        }
        rr = fma(rn, rn, rr);
        if (e0 + nth * u < total) put(ls[u], is[u], (T)rn);
      }
    } else {
      T v[BL];
#pragma unroll
      for (int u = 0; u < BL; ++u) v[u] = lv[u] ? (T)in[ad[u]] : T(0);
#pragma unroll
      for (int u = 0; u < BL; ++u)
        if (e0 + nth * u < total) put(ls[u], is[u], v[u]);
    }
  }
  __syncthreads();
  if (mode == FFT_DCT3) {
    // exp(i th_k) (X_k - i X_{N-k}) with X = C/c, times 1/N of the inverse FFT
    for (int idx = tid; idx < CL * N; idx += nth) {
      const int q = quot(idx, P.dN), k = idx - q * N;
      const T* xa = real1 + (2 * q) * NP;
      const T* xb = xa + NP;
      const T ak = xa[k], bk = xb[k];
      const T am = k == 0 ? T(0) : xa[N - k], bm = k == 0 ? T(0) : xb[N - k];
      const T c = dcs[k].x, s = dcs[k].y;
      buf0[q * NP + k] = cx<T>{(c * ak + s * am) - (s * bk - c * bm), (s * ak - c * am) + (c * bk + s * bm)};
    }
    __syncthreads();
  }
  const int odd = fft_stages<T>(P, mode == FFT_DCT3 ? T(1) : T(-1));
  const cx<T>* Z = odd ? buf1 : buf0;
  T* R = reinterpret_cast<T*>(odd ? buf0 : buf1);  // real outputs [LB][NP]
  const T hrs = T(0.5) * (T)P.r1;
  for (int idx = tid; idx < CL * N; idx += nth) {
    const int q = quot(idx, P.dN), k = idx - q * N;
    T* ra = R + (2 * q) * NP + k;
    if (mode == FFT_DCT3) {
      const cx<T> v = Z[q * NP + ((k & 1) ? N - 1 - (k >> 1) : (k >> 1))];
      ra[0] = v.x;
      ra[NP] = v.y;
    } else {
      const cx<T> zk = Z[q * NP + k], zm = Z[q * NP + (k == 0 ? 0 : N - k)];
      const T sr = zk.x + zm.x, si = zk.y - zm.y;  // 2 X_a
      const T dr = zk.y + zm.y, di = zm.x - zk.x;  // 2 X_b
      if (mode == FFT_DHT) {
        ra[0] = (sr - si) * hrs;
        ra[NP] = (dr - di) * hrs;
      } else {
        const T c = dcs[k].x, s = dcs[k].y;
        ra[0] = c * sr + s * si;
        ra[NP] = c * dr + s * di;
      }
    }
  }
  __syncthreads();
  double a0 = 0.0, a1 = 0.0;
  constexpr int BS = DOT ? 4 : 8;
  for (int e0 = tid; e0 < total; e0 += nth * BS) {
    int ls[BS], is[BS];
    long long ad[BS];
    bool lv[BS];
    double dr[DOT ? BS : 1], dq[DOT ? BS : 1];
#pragma unroll
    for (int u = 0; u < BS; ++u) {
      lv[u] = element(e0 + nth * u, ls[u], is[u], ad[u]);
      if constexpr (DOT) {
        dr[u] = lv[u] ? df.r[ad[u]] : 0.0;
        dq[u] = (lv[u] && df.flex) ? df.q[ad[u]] : 0.0;
      }
    }
#pragma unroll
    for (int u = 0; u < BS; ++u)
      if (lv[u]) {
        const TO v = (TO)R[ls[u] * NP + is[u]];
        out[ad[u]] = v;
        if constexpr (DOT) {
          a0 = fma(dr[u], (double)v, a0);
          a1 = fma(dq[u], (double)v, a1);
        }
      }
  }
  if constexpr (ZR) zr_tail(rr, zf.partials, zf.sc);
  if constexpr (DOT) dot_tail(a0, a1, df.flex, df.partials, df.sc);
}

constexpr int kSmemCap = 200 * 1024;

template <typename T, typename TI, typename TO, bool CONTIG, bool DOT = false, bool ZR = false>
void launch_mixed(int N, int mode, const TI* in, TO* out, const T* tw, const T* dct, long long inner, long long outer,
                  long long nlines, const DevScalars* sc, cudaStream_t s, DotFuse df = DotFuse{}, ZrFuse zf = ZrFuse{}) {
  FftPlan P{};
  P.N = N;
  P.stages = factor(N, P.radix);
  P.dN = make_div(N);
  P.r1 = 1.0 / std::sqrt((double)N);
  P.r2 = std::sqrt(2.0 / N);
  P.rh = 1.0 / std::sqrt(2.0 * N);
  for (int i = 0, Ns = 1; i < P.stages; Ns *= P.radix[i], ++i) {
    P.dB[i] = make_div(N / P.radix[i]);
    P.Ns[i] = Ns;
    P.dNs[i] = make_div(Ns);
  }
  // 8 complex lines per block (16 neighbouring columns of the strided axis);
  // fewer where three blocks would not share an SM, or the grid would leave SMs idle
  int lines = 8, llb = 4;
  while (lines > 1 && (smem_bytes<T>(N, lines) > 72 * 1024 || (nlines + 2 * lines - 1) / (2 * lines) * outer < 152)) {
    lines >>= 1;
    --llb;
  }
  P.lines = lines;
  int nth = kBlock;  // four elements of the complex lines per thread, at least two warps
  while (nth > 64 && lines * N <= 2 * nth) nth >>= 1;
  const dim3 grid((unsigned)((nlines + 2 * lines - 1) / (2 * lines)), (unsigned)outer);
  launch_k(k_fft_mixed<T, TI, TO, CONTIG, DOT, ZR>, grid, nth, smem_bytes<T>(N, lines), s, in, out, tw, dct, P, mode, llb, inner, nlines, sc, df, zf);
}

template <typename T>
int set_attrs() {
  int bad = 0;
#define MFG_MIX_ATTR(...)                                                                                     \
  bad |= cudaFuncSetAttribute(k_fft_mixed<T, __VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap) != \
         cudaSuccess;
  MFG_MIX_ATTR(double, T, true, false, false)
  MFG_MIX_ATTR(double, T, true, false, true)
  MFG_MIX_ATTR(T, double, true, false, false)
  MFG_MIX_ATTR(T, double, true, true, false)
  MFG_MIX_ATTR(T, T, false, false, false)
#undef MFG_MIX_ATTR
  return bad;
}

}  // namespace

bool fft_mixed_supported(int N) {
  int radix[kMaxStages];
  return N >= 8 && N <= kMaxN && factor(N, radix) > 0 && smem_bytes<double>(N, 1) <= (size_t)kSmemCap;
}

int fft_mixed_configure() { return set_attrs<float>() | set_attrs<double>() ? MFG_ERR_CUDA : MFG_OK; }

template <typename T>
void fft_mixed_y_forward(int N, int periodic, const double* in, T* out, const T* tw, const T* dct, long long nlines,
                         const DevScalars* sc, cudaStream_t s, const PcgZr* zr) {
  const int mode = periodic ? FFT_DHT : FFT_DCT2;
  if (zr)
    launch_mixed<T, double, T, true, false, true>(N, mode, in, out, tw, dct, 1, 1, nlines, sc, s, DotFuse{},
                                                  ZrFuse{zr->z, zr->r, zr->p, zr->q, zr->partials, zr->sc});
  else
    launch_mixed<T, double, T, true>(N, mode, in, out, tw, dct, 1, 1, nlines, sc, s);
}
template <typename T>
void fft_mixed_y_inverse(int N, int periodic, const T* in, double* out, const T* tw, const T* dct, long long nlines,
                         const DevScalars* sc, cudaStream_t s, const PcgDot* dot) {
  const int mode = periodic ? FFT_DHT : FFT_DCT3;
  if (dot)
    launch_mixed<T, T, double, true, true>(N, mode, in, out, tw, dct, 1, 1, nlines, sc, s,
                                           DotFuse{dot->r, dot->q, dot->partials, dot->sc, dot->flex});
  else
    launch_mixed<T, T, double, true>(N, mode, in, out, tw, dct, 1, 1, nlines, sc, s);
}
template <typename T>
void fft_mixed_x(int N, int periodic, int inverse, const T* in, T* out, const T* tw, const T* dct, long long inner,
                 long long outer, const DevScalars* sc, cudaStream_t s) {
  launch_mixed<T, T, T, false>(N, periodic ? FFT_DHT : (inverse ? FFT_DCT3 : FFT_DCT2), in, out, tw, dct, inner, outer,
                               inner, sc, s);
}

#define MFG_MIX_INST(T)                                                                                               \
  template void fft_mixed_y_forward<T>(int, int, const double*, T*, const T*, const T*, long long, const DevScalars*, \
                                       cudaStream_t, const PcgZr*);                                                   \
  template void fft_mixed_y_inverse<T>(int, int, const T*, double*, const T*, const T*, long long, const DevScalars*, \
                                       cudaStream_t, const PcgDot*);                                                  \
  template void fft_mixed_x<T>(int, int, int, const T*, T*, const T*, const T*, long long, long long,                 \
                               const DevScalars*, cudaStream_t);
MFG_MIX_INST(float)
MFG_MIX_INST(double)
#undef MFG_MIX_INST

}  // namespace mfg
