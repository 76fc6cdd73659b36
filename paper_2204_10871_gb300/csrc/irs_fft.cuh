// irs_fft.cuh -- complex FFTs of length 2^a 3^b (a >= 1) in shared memory
// (irs_fft.cu), in double-float arithmetic on float4 values (re.hi, im.hi,
// re.lo, im.lo; irs_df.cuh) or in FP32 on float2 values (re, im).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace irs {

constexpr int FFT_MAX_LEN = 9216;  // longest line (3^2 2^10): 144 KB of double-float complex values
                                   // and an 81 KB twiddle table

// One batched pass of 1-D FFTs over `n_lines` lines of length L.
struct FftLines {
  int L, n3, n2, B;         // line length L = 3^n3 2^n2, lines per CTA
  int in_len, out_len;      // valid input elements (rest zero), outputs written
  int64_t n_lines;
  int64_t in_line_stride, in_elem_stride, out_line_stride, out_elem_stride;
  int64_t in_grid_stride, out_grid_stride;  // between grids of a batch
};

// A padded Nx x Ny spectrum layout with its twiddle tables.
struct Fft2d {
  int Nx, Ny;        // 3^n3 2^n2 each
  int n3x, n2x, n3y, n2y;
  float4* tw_x;  // W_N^t, t < N/2, as double-float complex
  float4* tw_y;
  int num_sms;  // of the device that runs it
};

// Smallest length 2^a 3^b >= n_min with a >= 1 and at most FFT_MAX_LEN, or -1;
// its radix-3 and radix-2 stage counts.
int fft_good_size(int64_t n_min, int* n3, int* n2);
cudaError_t fft_twiddles(int L, float4** d_tw);
cudaError_t fft_setup_attributes();
// kernel launches of one 2-D transform, either way
int fft2d_launches(const Fft2d& f);
// compact [ngrids][ny][nx] -> padded spectra [ngrids][Ny][Nx], double-float planes
// (4) and FP32 planes (2) together, each axis in the forward transform's own
// order (the mixed-radix digit reversal of the frequency index): only pointwise
// products and sums of spectra made by these transforms are meaningful before
// fft2d_inverse, which expects that order
cudaError_t fft2d_forward(const float4* compact4, float4* spec4, int ngrids4, const float2* compact2, float2* spec2,
                          int ngrids2, int64_t nx, int64_t ny, int64_t in_grid_stride, const Fft2d& f,
                          cudaStream_t s);
// padded spectra (overwritten) -> compact [ngrids][ny][nx], unnormalised (the
// 1/(Nx Ny) is the caller's)
cudaError_t fft2d_inverse(float4* spec4, float4* compact4, int ngrids4, float2* spec2, float2* compact2, int ngrids2,
                          const Fft2d& f, int64_t nx, int64_t ny, int64_t out_grid_stride, cudaStream_t s);

}  // namespace irs
