// lf_cvt.h -- double to float with integer operations (where the result is a
// normal number; the caller converts the rest with a cast), and the block size of
// the layout conversion (lf_util.cu).
//
// The cast runs on the FP64 pipe, 1.8 results per clock and SM on this GPU; the
// integer form takes eight of the 128 lanes' operations instead.  The
// values are those of the cast, rounded to the nearest even.  (Widening in the
// same way gained nothing where it was tried, the transform along x of a real
// field: 412 us with the cast, 419 with integers at 256^3.)
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define LF_CVT_FN __host__ __device__ __forceinline__
#else
#define LF_CVT_FN inline
#endif

namespace lf {

// Bits of the float nearest to the double with bits `u` (infinity beyond the
// largest); false unless its exponent is that of a normal float.
LF_CVT_FN bool narrow_bits(uint64_t u, uint32_t* out)
{
    const uint64_t r = (u & 0x7fffffffffffffffull) + 0x0fffffffull + ((u >> 29) & 1u);
    *out = ((uint32_t)(r >> 29) - (896u << 23)) | ((uint32_t)(u >> 32) & 0x80000000u);
    return ((uint32_t)(u >> 52) & 0x7ffu) - 897u < 254u;
}

// Threads per block of the conversion of `planes` planes of `groups` groups of
// elements, `per_thread` of them a thread's: 256, fewer while there are not four
// blocks for every SM (a conversion between FP32 and FP64 takes its SM's FP64
// pipe): FP64 phi of 1024^2 to device memory 14.6 -> 14.1 us.
inline unsigned convert_threads(unsigned groups, unsigned per_thread, int planes, int sms)
{
    unsigned nt = 256;
    while (nt > 32 && (uint64_t)((groups + nt * per_thread - 1) / (nt * per_thread)) * planes < 4 * (uint64_t)sms) nt /= 2;
    return nt;
}

}  // namespace lf
