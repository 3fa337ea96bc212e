// lf_fft.cu -- FP64 transforms of real fields (lf_fft.cuh): line by line along
// each axis, each line in shared memory by a mixed-radix Cooley-Tukey
// (decimation in time).
//
// What bounds it: the FP64 pipe, 1.8 operations per clock and SM on this GPU
// (a 256^3 complex transform along one axis took 985 us, 0.08 ms of it memory
// time).  So the work is cut in FP64 operations:
//   - fields are real: along x two rows are packed into one complex line, and
//     only the half spectrum is transformed along the other axes;
//   - a radix-4 butterfly is two levels of radix-2 ones written
//       s = a + w b,  d = 2 a - s
//     (four fused operations and two), 24 operations for 4 points against 28
//     with separate products; the first stage has no twiddles and runs in
//     registers on the way into shared memory;
//   - one quadrant of the twiddles is evaluated, the rest are its rotations,
//     and a CTA keeps them (and the digit reversal) over all its lines.
// 256^3, one axis: 985 us before; now 360 us along y (the pipe's time for 22
// operations per point of the half spectrum: 354 us), 412 us along x from the
// field, 448 us back to it (528 with the scaling, the test for finite values and
// the narrowing on the FP64 pipe).
#include <algorithm>
#include <cmath>

#include "lf_cvt.h"
#include "lf_fft.cuh"

namespace lf {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxRadix = 32;
constexpr int kMaxStages = 40;

struct FftPlan {
    int n;
    int nst;
    int log2n;                 // of a power of two, else -1
    int radix[kMaxStages];
};

bool make_plan(int n, FftPlan* p)
{
    p->n = n;
    p->nst = 0;
    p->log2n = -1;
    if ((n & (n - 1)) == 0)
        for (p->log2n = 0; (1 << p->log2n) < n;) ++p->log2n;
    int m = n;
    while (m % 4 == 0) { p->radix[p->nst++] = 4; m /= 4; }
    for (int r = 2; r <= kMaxRadix && m > 1; ++r)
        while (m % r == 0) {
            if (p->nst >= kMaxStages) return false;
            p->radix[p->nst++] = r;
            m /= r;
        }
    return m == 1;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
// multiply by -i
__device__ __forceinline__ double2 cmul_mi(double2 a) { return make_double2(a.y, -a.x); }

// a + w b and a - w b
__device__ __forceinline__ void bfly2(double2 a, double2 b, double2 w, double2& s, double2& d)
{
    s.x = fma(-b.y, w.y, fma(b.x, w.x, a.x));
    s.y = fma(b.y, w.x, fma(b.x, w.y, a.y));
    d.x = fma(2.0, a.x, -s.x);
    d.y = fma(2.0, a.y, -s.y);
}

// y[0 .. r-1] = r-point DFT of x[0 .. r-1] (already multiplied by their
// twiddles) for r = 2, 3, 4, 5.
__device__ __forceinline__ void dft2(double2* x)
{
    const double2 a = x[0];
    x[0] = cadd(a, x[1]);
    x[1] = csub(a, x[1]);
}
__device__ __forceinline__ void dft3(double2* x)
{
    const double h = 0.86602540378443864676;     // sin(2 pi / 3)
    const double2 t = cadd(x[1], x[2]), u = csub(x[1], x[2]);
    const double2 m = make_double2(fma(-0.5, t.x, x[0].x), fma(-0.5, t.y, x[0].y));
    x[0] = cadd(x[0], t);
    x[1] = make_double2(fma(h, u.y, m.x), fma(-h, u.x, m.y));
    x[2] = make_double2(fma(-h, u.y, m.x), fma(h, u.x, m.y));
}
__device__ __forceinline__ void dft4(double2* x)
{
    const double2 a0 = cadd(x[0], x[2]), a1 = csub(x[0], x[2]);
    const double2 b0 = cadd(x[1], x[3]), b1 = cmul_mi(csub(x[1], x[3]));
    x[0] = cadd(a0, b0);
    x[1] = cadd(a1, b1);
    x[2] = csub(a0, b0);
    x[3] = csub(a1, b1);
}
__device__ __forceinline__ void dft5(double2* x)
{
    const double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;   // cos(2 pi / 5), cos(4 pi / 5)
    const double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;    // sin(2 pi / 5), sin(4 pi / 5)
    const double2 t1 = cadd(x[1], x[4]), t2 = cadd(x[2], x[3]), u1 = csub(x[1], x[4]), u2 = csub(x[2], x[3]);
    const double2 a = x[0];
    const double2 m1 = make_double2(fma(c2, t2.x, fma(c1, t1.x, a.x)), fma(c2, t2.y, fma(c1, t1.y, a.y)));
    const double2 m2 = make_double2(fma(c1, t2.x, fma(c2, t1.x, a.x)), fma(c1, t2.y, fma(c2, t1.y, a.y)));
    const double2 v1 = make_double2(fma(s2, u2.x, s1 * u1.x), fma(s2, u2.y, s1 * u1.y));
    const double2 v2 = make_double2(fma(-s1, u2.x, s2 * u1.x), fma(-s1, u2.y, s2 * u1.y));
    x[0] = cadd(a, cadd(t1, t2));
    x[1] = make_double2(m1.x + v1.y, m1.y - v1.x);
    x[4] = make_double2(m1.x - v1.y, m1.y + v1.x);
    x[2] = make_double2(m2.x + v2.y, m2.y - v2.x);
    x[3] = make_double2(m2.x - v2.y, m2.y + v2.x);
}
// any radix, by its definition; tw: the table of the whole line, wr = n / r
__device__ __noinline__ void dft_any(double2* x, int r, const double2* tw, int wr)
{
    double2 y[kMaxRadix];
    for (int q = 0; q < r; ++q) {
        double2 acc = x[0];
        for (int s = 1; s < r; ++s) acc = cadd(acc, cmul(x[s], tw[((q * s) % r) * wr]));
        y[q] = acc;
    }
    for (int q = 0; q < r; ++q) x[q] = y[q];
}

// Stores off the FP64 pipe (lf_cvt.h): no conversion, no comparison on it.
__device__ __forceinline__ void narrow(double v, float* p)
{
    uint32_t b;
    *p = narrow_bits((uint64_t)__double_as_longlong(v), &b) ? __uint_as_float(b) : (float)v;
}
__device__ __forceinline__ void narrow(double v, double* p) { *p = v; }
__device__ __forceinline__ bool finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// Quotient and remainder by d: shifts when the line length is a power of two
// (then d is one too), else a division.
template <bool POW2>
__device__ __forceinline__ void divmod(int v, int d, int sh, int& q, int& r)
{
    if constexpr (POW2) { q = v >> sh; r = v & (d - 1); }
    else { q = (int)((unsigned)v / (unsigned)d); r = v - q * d; }
}

// The lines of one axis of a half spectrum: line l starts at (l / inner) *
// outer + l % inner and has element stride es.
struct AxisIO {
    double2* data;
    int inner;
    int64_t outer, es;
    static constexpr bool kAlongLine = false;    // consecutive lines are neighbours in memory
    static constexpr bool kHalfOut = false;
    __device__ __forceinline__ int64_t base(unsigned l) const
    {
        const unsigned o = l / (unsigned)inner;
        return o * outer + (l - o * (unsigned)inner);
    }
    __device__ __forceinline__ double2 load(int64_t base, int64_t, int j, int) const { return data[base + j * es]; }
    __device__ __forceinline__ bool store(int64_t base, int64_t, int j, int, const double2* buf) const
    {
        data[base + j * es] = buf[j];
        return true;
    }
};

// Two rows of a real field packed into one complex line, out to the half
// spectrum of both: with Z the transform of a + i b,
//   2 A_k = Z_k + conj Z_{n-k},  2 B_k = -i (Z_k - conj Z_{n-k}).
template <typename R>
struct RealIn {
    const R* f;
    double2* out;
    int64_t rows;
    int pitch;
    static constexpr bool kAlongLine = true;
    static constexpr bool kHalfOut = true;
    __device__ __forceinline__ int64_t base(unsigned) const { return 0; }
    __device__ __forceinline__ double2 load(int64_t, int64_t l, int j, int) const
    {
        const R* p = f + 2 * l * pitch + j;
        return make_double2((double)p[0], 2 * l + 1 < rows ? (double)p[pitch] : 0.0);
    }
    __device__ __forceinline__ bool store(int64_t, int64_t l, int k, int n, const double2* buf) const
    {
        const double2 a = buf[k], b = buf[k == 0 ? 0 : n - k];
        double2* o = out + 2 * l * half_nx(n) + k;
        o[0] = make_double2(a.x + b.x, a.y - b.y);
        if (2 * l + 1 < rows) o[half_nx(n)] = make_double2(a.y + b.y, b.x - a.x);
        return true;
    }
};

// The way back: the lines A_k + i B_k of two rows' half spectra, whose
// transform is a + i b with a, b real.
template <typename R>
struct RealOut {
    const double2* in;
    R* f;
    int64_t rows;
    int pitch;
    static constexpr bool kAlongLine = true;
    static constexpr bool kHalfOut = false;
    __device__ __forceinline__ int64_t base(unsigned) const { return 0; }
    __device__ __forceinline__ double2 load(int64_t, int64_t l, int j, int n) const
    {
        const bool up = 2 * j > n;               // conjugate half
        const int k = up ? n - j : j;
        const double2* p = in + 2 * l * half_nx(n) + k;
        const double2 a = p[0], b = 2 * l + 1 < rows ? p[half_nx(n)] : make_double2(0.0, 0.0);
        return up ? make_double2(a.x + b.y, b.x - a.y) : make_double2(a.x - b.y, a.y + b.x);
    }
    __device__ __forceinline__ bool store(int64_t, int64_t l, int j, int, const double2* buf) const
    {
        const double2 v = buf[j];
        R* p = f + 2 * l * pitch + j;
        narrow(v.x, p);
        if (2 * l + 1 >= rows) return finite(v.x);
        narrow(v.y, p + pitch);
        return finite(v.x) && finite(v.y);
    }
};

// C lines of length n at a time per CTA.  Shared memory: the twiddles tw[j] =
// e^{-2 pi i j / n}, the C lines, the digit reversal of the index inside the
// first stage's groups.
template <class IO, bool POW2>
__global__ void __launch_bounds__(kThreads) k_fft_lines(IO io, FftPlan plan, int64_t nlines, int C, int* flag)
{
    extern __shared__ double2 smem_fft[];
    __shared__ int64_t lbase[16];
    const int n = plan.n;
    double2* tw = smem_fft;
    double2* buf = smem_fft + n;
    unsigned short* rev = reinterpret_cast<unsigned short*>(buf + (size_t)C * n);
    const int r0 = plan.nst > 0 ? plan.radix[0] : 1, g0 = n / r0;
    if (n % 4 == 0) {
        for (int j = threadIdx.x; j < n / 4; j += kThreads) {
            double sn, cs;
            sincospi(-2.0 * (double)j / (double)n, &sn, &cs);
            const double2 w = make_double2(cs, sn);
            tw[j] = w;
            tw[j + n / 4] = cmul_mi(w);
            tw[j + n / 2] = make_double2(-cs, -sn);
            tw[j + 3 * (n / 4)] = make_double2(-sn, cs);
        }
    } else {
        for (int j = threadIdx.x; j < n; j += kThreads) {
            double sn, cs;
            sincospi(-2.0 * (double)j / (double)n, &sn, &cs);
            tw[j] = make_double2(cs, sn);
        }
    }
    // the element j = jl + s g0 (s < r0) goes to position rev[jl] + s
    for (int j = threadIdx.x; j < g0; j += kThreads) {
        int pos = 0, rem = j, size = n;
        for (int st = plan.nst - 1; st > 0; --st) {
            const int r = plan.radix[st];
            size /= r;
            pos += (rem % r) * size;
            rem /= r;
        }
        rev[j] = (unsigned short)pos;
    }
    bool ok = true;
    const int sh0 = POW2 ? __popc(g0 - 1) : 0, shn = POW2 ? plan.log2n : 0;
    for (int64_t l0 = (int64_t)blockIdx.x * C; l0 < nlines; l0 += (int64_t)gridDim.x * C) {
        const int nl = (int)(nlines - l0 < C ? nlines - l0 : C);
        __syncthreads();                         // tables ready; the previous lines stored
        if ((int)threadIdx.x < nl) lbase[threadIdx.x] = io.base((unsigned)(l0 + threadIdx.x));
        __syncthreads();
        // element t of the batch along the lines, or across them when those are neighbours in memory
        auto across = [&](int t, int& c, int& j) {
            if (nl == 16) { j = t >> 4; c = t & 15; }
            else { j = (int)((unsigned)t / (unsigned)nl); c = t - j * nl; }
        };
        // first stage on the way in: no twiddles
        for (int t = threadIdx.x; t < nl * g0; t += kThreads) {
            int c, jl;
            if (IO::kAlongLine) divmod<POW2>(t, g0, sh0, c, jl);
            else across(t, c, jl);
            double2* b = buf + c * n + rev[jl];
            const int64_t lb = lbase[c], l = l0 + c;
            if (r0 == 4) {
                double2 x[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) x[s] = io.load(lb, l, jl + s * g0, n);
                dft4(x);
#pragma unroll
                for (int s = 0; s < 4; ++s) b[s] = x[s];
            } else if (r0 == 2) {
                double2 x[2] = {io.load(lb, l, jl, n), io.load(lb, l, jl + g0, n)};
                dft2(x);
                b[0] = x[0];
                b[1] = x[1];
            } else if (POW2 || r0 == 1) {
                b[0] = io.load(lb, l, jl, n);
            } else {
                double2 x[kMaxRadix];
                for (int s = 0; s < r0; ++s) x[s] = io.load(lb, l, jl + s * g0, n);
                if (r0 == 3) dft3(x);
                else if (r0 == 5) dft5(x);
                else dft_any(x, r0, tw, g0);
                for (int s = 0; s < r0; ++s) b[s] = x[s];
            }
        }
        __syncthreads();
        int m = r0, shm = POW2 ? __popc(r0 - 1) : 0;
        for (int st = 1; st < plan.nst; ++st) {
            const int r = plan.radix[st];
            const int nb = n / r;
            const int stride = n / (m * r);      // tw index step of W_{m r}
            const int shb = POW2 ? __popc(nb - 1) : 0;
            for (int t = threadIdx.x; t < nl * nb; t += kThreads) {
                int c, bi, grp, k;
                divmod<POW2>(t, nb, shb, c, bi);
                divmod<POW2>(bi, m, shm, grp, k);
                double2* b = buf + c * n + grp * m * r + k;
                if (r == 4) {
                    const double2 w1 = tw[k * stride], w2 = tw[2 * k * stride];
                    double2 a0, a1, u, v, s, d;
                    bfly2(b[0], b[2 * m], w2, a0, a1);
                    bfly2(b[m], b[3 * m], w2, u, v);
                    bfly2(a0, u, w1, s, d);
                    b[0] = s;
                    b[2 * m] = d;
                    bfly2(a1, v, cmul_mi(w1), s, d);
                    b[m] = s;
                    b[3 * m] = d;
                } else if (r == 2) {
                    double2 s, d;
                    bfly2(b[0], b[m], tw[k * stride], s, d);
                    b[0] = s;
                    b[m] = d;
                } else if (!POW2 && r == 3) {
                    double2 x[3] = {b[0], cmul(b[m], tw[k * stride]), cmul(b[2 * m], tw[2 * k * stride])};
                    dft3(x);
                    b[0] = x[0]; b[m] = x[1]; b[2 * m] = x[2];
                } else if (!POW2 && r == 5) {
                    double2 x[5];
                    x[0] = b[0];
#pragma unroll
                    for (int s = 1; s < 5; ++s) x[s] = cmul(b[s * m], tw[s * k * stride]);
                    dft5(x);
#pragma unroll
                    for (int s = 0; s < 5; ++s) b[s * m] = x[s];
                } else if (!POW2) {
                    double2 x[kMaxRadix];
                    x[0] = b[0];
                    for (int s = 1; s < r; ++s) x[s] = cmul(b[s * m], tw[s * k * stride]);
                    dft_any(x, r, tw, n / r);
                    for (int s = 0; s < r; ++s) b[s * m] = x[s];
                }
            }
            __syncthreads();
            m *= r;
            if (POW2) shm += __popc(r - 1);
        }
        const int no = IO::kHalfOut ? half_nx(n) : n;
        for (int t = threadIdx.x; t < nl * no; t += kThreads) {
            int c, j;
            if (!IO::kAlongLine) across(t, c, j);
            else if (IO::kHalfOut) { c = (int)((unsigned)t / (unsigned)no); j = t - c * no; }
            else divmod<POW2>(t, n, shn, c, j);
            ok &= io.store(lbase[c], l0 + c, j, n, buf + c * n);
        }
    }
    if (!ok && flag) *reinterpret_cast<volatile int*>(flag) = 1;
}

template <class IO, bool POW2>
cudaError_t launch_lines(const IO& io, const FftPlan& plan, int64_t nlines, int* flag, cudaStream_t s)
{
    const int n = plan.n;
    const int C = std::max(1, std::min(16, 4096 / n));
    const int g0 = n / (plan.nst > 0 ? plan.radix[0] : 1);
    const size_t smem = sizeof(double2) * (size_t)(C + 1) * n + sizeof(unsigned short) * ((g0 + 7) / 8 * 8);
    auto kern = k_fft_lines<IO, POW2>;
    // the largest a line of 4096 needs, once per instantiation and device
    static unsigned long long attr_done = 0;
    cudaError_t e = raise_smem_limit(kern, (int)(sizeof(double2) * 2 * 4096 + sizeof(unsigned short) * 4096), &attr_done);
    int sms = 0;
    if (e == cudaSuccess) e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    // resident CTAs (bounded by shared memory), each over its share of the lines
    const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(4, (int64_t)(220 * 1024 / smem)));
    const int64_t blocks = std::min<int64_t>((nlines + C - 1) / C, per_sm * sms);
    kern<<<(unsigned)blocks, kThreads, smem, s>>>(io, plan, nlines, C, flag);
    return cudaGetLastError();
}

template <class IO>
cudaError_t run_lines(const IO& io, int n, int64_t nlines, int* flag, cudaStream_t s)
{
    FftPlan plan;
    if (!make_plan(n, &plan) || n > 4096) return cudaErrorInvalidValue;
    return plan.log2n >= 0 ? launch_lines<IO, true>(io, plan, nlines, flag, s)
                           : launch_lines<IO, false>(io, plan, nlines, flag, s);
}

}  // namespace

bool fft_supported(int n)
{
    FftPlan p;
    return n <= 4096 && make_plan(n, &p);
}

template <typename R>
cudaError_t rfft_x(const Geom& g, const R* f, double2* out, cudaStream_t s)
{
    const int64_t rows = (int64_t)g.ny * g.nz;
    return run_lines(RealIn<R>{f, out, rows, g.pitch}, g.nx, (rows + 1) / 2, nullptr, s);
}

cudaError_t fft_axis(const Geom& g, double2* data, int axis, cudaStream_t s)
{
    const int H = half_nx(g.nx);
    const int64_t plane = (int64_t)H * g.ny;
    if (axis == 1) return run_lines(AxisIO{data, H, plane, H}, g.ny, (int64_t)H * g.nz, nullptr, s);
    if (axis == 2) return run_lines(AxisIO{data, (int)plane, 0, plane}, g.nz, plane, nullptr, s);
    return cudaErrorInvalidValue;
}

template <typename R>
cudaError_t irfft_x(const Geom& g, const double2* in, R* f, int* flag, cudaStream_t s)
{
    const int64_t rows = (int64_t)g.ny * g.nz;
    return run_lines(RealOut<R>{in, f, rows, g.pitch}, g.nx, (rows + 1) / 2, flag, s);
}

#define LF_INST(R)                                                                       \
    template cudaError_t rfft_x<R>(const Geom&, const R*, double2*, cudaStream_t);       \
    template cudaError_t irfft_x<R>(const Geom&, const double2*, R*, int*, cudaStream_t);
LF_INST(float)
LF_INST(double)
#undef LF_INST

}  // namespace lf
