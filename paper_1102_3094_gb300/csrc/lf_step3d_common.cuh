// lf_step3d_common.cuh -- index maps and copy helpers shared by the passes of
// the three-pass D3Q19 step (lf_step3d_split.cu, lf_step3d_iso.cu).
#pragma once

#include "lf_internal.cuh"

namespace lf {
namespace {

__device__ __forceinline__ int wrap_s(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// Storage plane of an unwrapped z (periodic, or mirrored about the half-way
// walls with period 2n); the division only for v outside [-n, 2n).
__device__ __forceinline__ int map_z(int v, int n, int walls)
{
    if (v >= 0 && v < n) return v;
    const int d = walls ? (v < 0 ? -1 - v : 2 * n - 1 - v) : (v < 0 ? v + n : v - n);
    if (d >= 0 && d < n) return d;
    if (!walls) return wrap_s(v, n);
    const int m = wrap_s(v, 2 * n);
    return m < n ? m : 2 * n - 1 - m;
}

template <typename R>
__device__ __forceinline__ R rcp_s(R x) { return R(1) / x; }
template <>
__device__ __forceinline__ float rcp_s<float>(float x) { return __frcp_rn(x); }

template <int B>
__device__ __forceinline__ void cp_async_s(void* dst, const void* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (B == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}

// Planes per segment (or per lane of a two-lane segment: `lanes` = 2) of a
// column march over `tiles` columns of a CTA, `lag` planes longer than its
// segment, `res` CTAs resident per SM.  The march of a CTA takes about as
// long as it has planes, so the time is the number of rounds of resident CTAs
// times (planes + lag); a last round that leaves every SM at most one of two
// places runs at 0.6 of a full one (an SM's issue rate is then shared by half
// the CTAs).  The number of segments with the least of that wins; few planes
// per segment on small lattices, where everything fits in one round and only
// the length of the march counts.  The planes before a segment's first skip their
// later stages, so `lag` is less than their number: 3 for the one-lane forms.
// Pass times against the best of all heights, on average and at worst: FP64 0.2 %
// and 5 % (18 lattices from 24^3 to 256^3, both stencils, with and without
// hydrodynamics), FP32 on one lane 1 to 4 % and 14 % (11 lattices from 24^3 to
// 384^3), packed 5 % and 15 % (compact, lag 6), 2 % and 6 % (isotropic, lag 8).
// Segments of at least 16 planes, the rule before, cost 64^3 29.5 us instead of
// 15.0 (compact) and 32 x 32 x 256 29.2 instead of 18.2.
inline int march3_planes(int64_t tiles, int nz, int lanes, int lag, int res, int sms)
{
    int best = nz;
    double best_cost = 1e300;
    for (int k = 1; k * lanes <= 2 * nz && k <= 4096; ++k) {
        const int H = (nz + k * lanes - 1) / (k * lanes);
        const int64_t ctas = tiles * ((nz + H * lanes - 1) / (H * lanes));
        const int64_t full = ctas / (res * (int64_t)sms), left = ctas - full * res * sms;
        const double rounds = (double)full + (left == 0 ? 0.0 : (res == 2 && left <= sms ? 0.6 : 1.0));
        const double cost = rounds * (H + lag);
        if (cost < best_cost) { best_cost = cost; best = H; }
        if (H == 1) break;
    }
    return best;
}

}  // namespace
}  // namespace lf
