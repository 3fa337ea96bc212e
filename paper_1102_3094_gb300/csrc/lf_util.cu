// lf_util.cu -- initial state and layout conversion kernels.
#include "lf_cvt.h"
#include "lf_internal.cuh"

namespace lf {

namespace {

// SplitMix64 (Steele, Lea & Flood 2014): the k-th output of the generator
// whose state starts at `seed`.  Counter-based, so every site draws its own
// value independently of the launch shape.
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t k)
{
    uint64_t z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Initial state (arXiv:1102.3094 Sec. 3: disordered phi around zero, T above
// Tc with the walls at T_w).  phi = amp (2u - 1), u the top 53 bits of the
// generator output; the products are rounded explicitly so the FP64 value is
// the same on every compiler and machine.
template <typename R>
__global__ void k_init(Geom g, uint64_t seed, double amp, double T0, double T_w, int quench,
                       R* __restrict__ phi, R* __restrict__ T)
{
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    const int wall_len = (g.d == 2) ? g.ny : g.nz;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < N;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(k % g.nx);
        const int64_t row = k / g.nx;                   // y + ny z
        const int y = (int)(row % g.ny);
        const int z = (int)(row / g.ny);
        const int h = (g.d == 2) ? y : z;               // position along the wall axis
        const uint64_t r = splitmix64_at(seed, (uint64_t)k);
        const double u = (double)(r >> 11) * 0x1.0p-53;
        const double v = __dadd_rn(__dmul_rn(2.0, u), -1.0);
        const int64_t site = row * g.pitch + x;
        phi[site] = (R)__dmul_rn(amp, v);
        double t = T0;
        if (quench) t = T_w;
        else if (g.walls && g.t_mode == LF_TWALL_LAYERS && (h == 0 || h == wall_len - 1)) t = T_w;
        T[site] = (R)t;
    }
}

// Layout conversion between the padded state ([rows][pitch], deviations for
// the populations) and a packed caller array ([rows][nx]), one plane per
// blockIdx.y.  A thread moves kGroups groups of V consecutive elements of one
// row, blockDim.x groups apart: V = 4 (one vector access on each side; fewer
// requests when the caller array is host memory reached through the device
// mapping) when every row of both arrays starts on a 16-byte boundary, else
// V = 1.  Groups are counted over the whole plane, not per row, so that short
// rows fill their warps too.
//
// The offset w_i n0 is added in the arithmetic of the caller's type.  The
// FP64 pipe of this GPU issues 1.8 operations per clock and SM (FP32: 118), and
// converting FP32 state through it made this kernel three FP64 operations per
// element, 0.16 G elements/ms whatever the bandwidth.  FP32 to FP32 therefore
// adds the offset as three floats (24 + 24 + 5 bits hold the double exactly)
// with error-free sums: the result is the sum rounded once, to within 2^-46
// relative, as (float)((double)v + a) is.  19 populations at 384^3: 6.6 ms
// before, 1.23 ms now (7.0 TB/s).
constexpr int kGroups = 2;

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
    using type = float4;
};
template <>
struct Vec4<double> {
    using type = double4_16a;
};

template <typename T, int V>
__device__ __forceinline__ void load_v(const T* p, T v[V])
{
    if constexpr (V == 4) {
        const typename Vec4<T>::type w = *reinterpret_cast<const typename Vec4<T>::type*>(p);
        v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
    } else {
        v[0] = *p;
    }
}

template <typename T, int V>
__device__ __forceinline__ void store_v(T* p, const T v[V])
{
    if constexpr (V == 4) {
        typename Vec4<T>::type w;
        w.x = v[0]; w.y = v[1]; w.z = v[2]; w.w = v[3];
        *reinterpret_cast<typename Vec4<T>::type*>(p) = w;
    } else {
        *p = v[0];
    }
}

// The offsets of the planes: as doubles, and each split into three floats.
struct Offsets {
    double d[19];
    float h[19], m[19], l[19];
};

Offsets split_offsets(const PlaneAdd& a, double sign, int nplanes)
{
    Offsets o{};
    for (int q = 0; q < nplanes; ++q) {
        const double v = sign * a.v[q];
        o.d[q] = v;
        o.h[q] = (float)v;
        o.m[q] = (float)(v - (double)o.h[q]);
        o.l[q] = (float)(v - (double)o.h[q] - (double)o.m[q]);
    }
    return o;
}

// s + e = a + b exactly (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float b, float& e)
{
    const float s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// (D)(v + offset of plane q), rounded once.
template <typename S, typename D>
__device__ __forceinline__ D add_offset(S v, const Offsets& o, int q)
{
    if constexpr (sizeof(S) == 4 && sizeof(D) == 4) {
        if (o.h[q] == 0.f) return v + o.h[q];            // phi, T, checkpoints: (+-0) as the double sum has it
        float e, f;
        const float s = two_sum(v, o.h[q], e);
        const float t = two_sum(s, o.m[q], f);
        const float r = t + (f + (e + o.l[q]));
        return fabsf(s) <= 3.402823466e38f ? r : s;      // NaN and Inf pass through
    } else {
        return (D)((double)v + o.d[q]);
    }
}

// SRC, DST: row strides in elements; `sp`, `dp`: plane strides.
template <typename S, typename D, int V>
__global__ void __launch_bounds__(256) k_convert(const S* __restrict__ src, D* __restrict__ dst, unsigned groups,
                                                 unsigned row_groups, int64_t srow, int64_t drow, int64_t sp, int64_t dp,
                                                 Offsets off)
{
    const int q = blockIdx.y;
    src += q * sp;
    dst += q * dp;
    const unsigned nt = blockDim.x, g0 = blockIdx.x * (nt * kGroups) + threadIdx.x;
    S v[kGroups][V];
    int64_t to[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const unsigned k = g0 + nt * u;
        if (k < groups) {
            const unsigned row = k / row_groups, x = (k - row * row_groups) * V;
            to[u] = row * drow + x;
            load_v<S, V>(src + row * srow + x, v[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if (g0 + nt * u < groups) {
            D o[V];
#pragma unroll
            for (int i = 0; i < V; ++i) o[i] = add_offset<S, D>(v[u][i], off, q);
            store_v<D, V>(dst + to[u], o);
        }
}

// Vector accesses need every row and plane start of both arrays 16-byte
// aligned (a: the padded state in R, b: the packed array in D).
template <typename R, typename D>
bool vec_ok(const Geom& g, const void* a, const void* b)
{
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    const bool rows = g.nx % 4 == 0 && ((size_t)g.nx * sizeof(D)) % 16 == 0 && ((size_t)g.pitch * sizeof(R)) % 16 == 0 &&
                      ((size_t)N * sizeof(D)) % 16 == 0 && ((size_t)g.plane * sizeof(R)) % 16 == 0;
    return rows && ((uintptr_t)a % 16 == 0) && ((uintptr_t)b % 16 == 0);
}

template <typename S, typename D>
cudaError_t convert(const Geom& g, const S* src, D* dst, int nplanes, int64_t srow, int64_t drow, int64_t sp, int64_t dp,
                    bool vec, const Offsets& off, cudaStream_t s)
{
    // sites < 2^31 / Q (checked at creation), so groups fit 32 bits
    int sms = 0;
    const cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    // Small planes: one element per group and small blocks, because a thread that converts four between FP32 and FP64
    // is a chain on the FP64 pipe of one SM.  64 x 64 populations and a host array of the other type, one plane at a
    // time: read 138 -> 128 us, written 68.5 -> 64.5.
    if ((uint64_t)g.nx * g.ny * g.nz * nplanes < 256ull * sms) vec = false;
    const unsigned row_groups = vec ? g.nx / 4 : g.nx;
    const unsigned groups = row_groups * (unsigned)(g.ny * g.nz);
    const unsigned nt = convert_threads(groups, kGroups, nplanes, sms), per = nt * kGroups;
    const dim3 grid((groups + per - 1) / per, nplanes);
    if (vec) k_convert<S, D, 4><<<grid, nt, 0, s>>>(src, dst, groups, row_groups, srow, drow, sp, dp, off);
    else k_convert<S, D, 1><<<grid, nt, 0, s>>>(src, dst, groups, row_groups, srow, drow, sp, dp, off);
    return cudaGetLastError();
}

inline unsigned grid_for(const Geom& g)
{
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    int64_t b = (N + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

template <typename R>
cudaError_t launch_init(const Geom& g, uint64_t seed, double amp, double T0, double T_w, int quench,
                        R* phi, R* T, cudaStream_t s)
{
    k_init<R><<<grid_for(g), 256, 0, s>>>(g, seed, amp, T0, T_w, quench, phi, T);
    return cudaGetLastError();
}

template <typename R, typename D>
cudaError_t launch_pack(const Geom& g, const R* src, D* dst, int nplanes, const PlaneAdd& add, cudaStream_t s)
{
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    return convert<R, D>(g, src, dst, nplanes, g.pitch, g.nx, g.plane, N, vec_ok<R, D>(g, src, dst),
                         split_offsets(add, 1.0, nplanes), s);
}

template <typename R, typename D>
cudaError_t launch_unpack(const Geom& g, const D* src, R* dst, int nplanes, const PlaneAdd& sub, cudaStream_t s)
{
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    return convert<D, R>(g, src, dst, nplanes, g.nx, g.pitch, N, g.plane, vec_ok<R, D>(g, dst, src),
                         split_offsets(sub, -1.0, nplanes), s);
}

template cudaError_t launch_init<float>(const Geom&, uint64_t, double, double, double, int, float*, float*, cudaStream_t);
template cudaError_t launch_init<double>(const Geom&, uint64_t, double, double, double, int, double*, double*, cudaStream_t);
template cudaError_t launch_pack<float, float>(const Geom&, const float*, float*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_pack<float, double>(const Geom&, const float*, double*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_pack<double, float>(const Geom&, const double*, float*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_pack<double, double>(const Geom&, const double*, double*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_unpack<float, float>(const Geom&, const float*, float*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_unpack<float, double>(const Geom&, const double*, float*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_unpack<double, float>(const Geom&, const float*, double*, int, const PlaneAdd&, cudaStream_t);
template cudaError_t launch_unpack<double, double>(const Geom&, const double*, double*, int, const PlaneAdd&, cudaStream_t);

}  // namespace lf
