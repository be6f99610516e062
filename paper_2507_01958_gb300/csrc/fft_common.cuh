// What the two FFT translation units share: complex values, modes, and the PCG
// work a pass can carry.
#pragma once

#include "mfg_internal.cuh"

namespace mfg {

template <typename T>
struct __align__(2 * sizeof(T)) cx {
  T x, y;
};

enum { FFT_DHT = 0, FFT_DCT2 = 1, FFT_DCT3 = 2 };

// Dot products fused into the last pass of a PCG preconditioner apply: while
// zp = P^{-1} r is stored, r.zp (and q.zp for the flexible variant) are
// accumulated and the last block forms beta (dot_tail).
struct DotFuse {
  const double* r;
  const double* q;
  double* partials;
  DevScalars* sc;
  int flex;
};

// The PCG update fused into the first pass: z += alpha p, r -= alpha q for the
// elements this block transforms, ||r||^2 accumulated, and the last block runs
// the convergence test (zr_tail).  The pass then transforms the new r.
struct ZrFuse {
  double* z;
  double* r;
  const double* p;
  const double* q;
  double* partials;
  DevScalars* sc;
};

// Lengths that are no power of two up to 512 (k_fft_mixed.cu).
bool fft_mixed_supported(int N);
int fft_mixed_configure();
template <typename T>
void fft_mixed_y_forward(int N, int periodic, const double* in, T* out, const T* tw, const T* dct, long long nlines,
                         const DevScalars* sc, cudaStream_t s, const PcgZr* zr);
template <typename T>
void fft_mixed_y_inverse(int N, int periodic, const T* in, double* out, const T* tw, const T* dct, long long nlines,
                         const DevScalars* sc, cudaStream_t s, const PcgDot* dot);
template <typename T>
void fft_mixed_x(int N, int periodic, int inverse, const T* in, T* out, const T* tw, const T* dct, long long inner,
                 long long outer, const DevScalars* sc, cudaStream_t s);

}  // namespace mfg
