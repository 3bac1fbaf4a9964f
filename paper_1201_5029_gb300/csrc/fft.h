// Real 3-D transforms of the library's own (fft.cu), for the sides they take;
// other sides go through cuFFT.  Layouts are cuFFT's: real [z][y][x], half
// spectrum [z][y][n/2 + 1], unnormalised, forward exponent -1.
#pragma once

#include <cuda_runtime.h>

namespace pycool {

// n a power of two, 64 .. 256 (smaller ones are faster through cuFFT)
inline bool fft_takes(int n) { return n == 64 || n == 128 || n == 256; }
// `batch` real arrays of n^3 values, one after another, into as many half spectra
cudaError_t fft_forward(const double* in, double2* out, int n, int batch, cudaStream_t s);
// the inverse; the spectra are overwritten
cudaError_t fft_inverse(double2* spec, double* out, int n, int batch, cudaStream_t s);

}  // namespace pycool
