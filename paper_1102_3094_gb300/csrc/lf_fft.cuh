// lf_fft.cuh -- FP64 transforms of the real fields of a lattice, for S(k)
// (lf_diag.cu) and the implicit temperature step (lf_timplicit.cu).
//
// A real [nz][ny][nx] field is held in Fourier space as its half spectrum
// along x: [nz][ny][nx / 2 + 1] complex doubles (the rest is the conjugate),
// times two (the transform along x leaves the factor 1/2 of the split of two
// packed rows to the caller, who has a scale to apply anyway).
#pragma once

#include "lf_internal.cuh"

namespace lf {

// Complex doubles per row of the half spectrum.
__host__ __device__ inline int half_nx(int nx) { return nx / 2 + 1; }

// Whether a line of length n is within reach (prime factors up to 31, n <= 4096).
bool fft_supported(int n);

// out = 2 x forward DFT along x (kernel e^{-2 pi i j k / nx}) of the rows of
// the state field `f` (rows of g.pitch).
template <typename R>
cudaError_t rfft_x(const Geom& g, const R* f, double2* out, cudaStream_t s);

// Forward DFT along axis 1 (y) or 2 (z) of a half spectrum, in place.
cudaError_t fft_axis(const Geom& g, double2* data, int axis, cudaStream_t s);

// f = DFT along x of the half spectrum `in`, whose rows are the DFTs of real
// rows up to a conjugation (so the result is real).  Sets *flag when a value is
// not finite.
template <typename R>
cudaError_t irfft_x(const Geom& g, const double2* in, R* f, int* flag, cudaStream_t s);

}  // namespace lf
