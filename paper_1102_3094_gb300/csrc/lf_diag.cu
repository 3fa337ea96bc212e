// lf_diag.cu -- diagnostics kernels.
//
// Sums are FP64 whatever the state precision: every site's contribution is
// converted to double, reduced within a CTA by warp shuffles, written as one
// partial per CTA, and the partials are reduced in a fixed order by a single
// CTA, so the result does not depend on scheduling.
//
// S(k) = |sum_r (phi - mean) e^{-i k.r}|^2 / N: the FFT runs in FP64 on the
// GPU on the half spectrum of the real field (lf_fft.cu).
// The k = 0 coefficient, the only one the mean affects, is left out of the
// shells.  Shells have width dk = 2 pi / L_min; bin b = floor(|k|/dk + 1/2),
// b = 1 .. L_min/2.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "lf_diag.cuh"
#include "lf_fft.cuh"

namespace lf {

namespace {

constexpr int kBlocks = 152 * 8;   // partial sums there is room for
constexpr int kResident = 152 * 3; // CTAs of k_diag_partial that run at once
constexpr int kThreads = 256;
constexpr int kMaxBins = 2048;     // of S(k): half the longest line the FFT takes

struct Scratch {
    double* part;    // kBlocks * DQ_N
    double* res;     // DQ_N
    double* layers;  // L * 2
    double* bins;    // (B + 1) * 2: sum, count
    double2* fft;    // half spectrum (nx / 2 + 1) ny nz <= N
};

size_t a256(size_t v) { return (v + 255) / 256 * 256; }

Scratch carve(const Geom& g, void* base)
{
    Scratch s;
    unsigned char* p = (unsigned char*)base;
    const int64_t L = g.d == 2 ? g.ny : g.nz;
    int64_t lmin = g.nx < g.ny ? g.nx : g.ny;
    if (g.d == 3 && g.nz < lmin) lmin = g.nz;
    const int64_t B = lmin / 2;
    s.part = (double*)p; p += a256(sizeof(double) * kBlocks * DQ_N);
    s.res = (double*)p; p += a256(sizeof(double) * DQ_N);
    s.layers = (double*)p; p += a256(sizeof(double) * 2 * L);
    s.bins = (double*)p; p += a256(sizeof(double) * 2 * (B + 1));
    s.fft = (double2*)p;
    return s;
}

__device__ __forceinline__ int nb_index(int v, int step, int n, int mirror)
{
    int t = v + step;
    if (t < 0) return mirror ? 0 : n - 1;
    if (t >= n) return mirror ? n - 1 : 0;
    return t;
}

template <typename R>
__device__ __forceinline__ double at(const R* f, const Geom& g, int x, int y, int z)
{
    return (double)f[((int64_t)z * g.ny + y) * g.pitch + x];
}

// Central differences of phi at (x, y, z); along the wall axis the neighbour
// beyond the last layer is the layer itself (even mirror).
template <typename R>
__device__ void phi_grad(const R* phi, const Geom& g, int x, int y, int z, double* grad)
{
    const int wy = g.walls && g.d == 2, wz = g.walls && g.d == 3;
    grad[0] = 0.5 * (at(phi, g, nb_index(x, 1, g.nx, 0), y, z) - at(phi, g, nb_index(x, -1, g.nx, 0), y, z));
    grad[1] = 0.5 * (at(phi, g, x, nb_index(y, 1, g.ny, wy), z) - at(phi, g, x, nb_index(y, -1, g.ny, wy), z));
    grad[2] = 0.0;
    if (g.d == 3)
        grad[2] = 0.5 * (at(phi, g, x, y, nb_index(z, 1, g.nz, wz)) - at(phi, g, x, y, nb_index(z, -1, g.nz, wz)));
}

// Sums (slot max_slot: maximum) of v over the CTA, in a fixed order.  The
// values go through shared memory and 16 threads per slot add 16 of them each:
// a fifth of the FP64 operations of a shuffle tree in every warp.
template <int NQ>
__device__ void block_reduce_store(double (&v)[NQ], double* out, int max_slot)
{
    static_assert(NQ % 2 == 0 && NQ * 16 <= kThreads && kThreads == 256, "whole warps of 16-thread groups");
    __shared__ double red[NQ][kThreads];
    const int tid = threadIdx.x;
#pragma unroll
    for (int q = 0; q < NQ; ++q) red[q][tid] = v[q];
    __syncthreads();
    if (tid < NQ * 16) {
        const int q = tid >> 4, l = tid & 15;
        const bool mx = q == max_slot;
        double x = red[q][l];
#pragma unroll
        for (int i = 1; i < 16; ++i) {
            const double y = red[q][l + 16 * i];
            x = mx ? fmax(x, y) : x + y;
        }
        for (int o = 8; o > 0; o >>= 1) {
            const double y = __shfl_down_sync(0xffffffffu, x, o, 16);
            x = mx ? fmax(x, y) : x + y;
        }
        if (l == 0) out[q] = x;
    }
}

// Bound by the FP64 pipe, so counted in its operations: about 30 per site.  The
// halves and the coefficients of the free energy multiply a thread's sums once
// (a site's division by Tc and its products were 75 operations): 155 -> 85 us
// at 1024^2.
template <typename R>
__global__ void __launch_bounds__(kThreads, 3) k_diag_partial(Geom g, const R* __restrict__ phi, const R* __restrict__ T,
                                                              const R* __restrict__ aux, double b, double kappa, double c,
                                                              double Tc, double* part)
{
    double v[DQ_N], links = 0.0, lap2 = 0.0;
#pragma unroll
    for (int q = 0; q < DQ_N; ++q) v[q] = 0.0;
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    const int64_t P = g.plane;
    const int wy = g.walls && g.d == 2, wz = g.walls && g.d == 3;
    const double ha = 0.5 / Tc, hb = 0.25 * b;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x) {
        int64_t row;
        int x, y, z;
        if (N <= INT32_MAX) {
            const unsigned r = (unsigned)k / (unsigned)g.nx;
            x = (int)((unsigned)k - r * (unsigned)g.nx);
            z = (int)(r / (unsigned)g.ny);
            y = (int)(r - (unsigned)z * (unsigned)g.ny);
            row = r;
        } else {
            row = k / g.nx;
            x = (int)(k - row * g.nx);
            z = (int)(row / g.ny);
            y = (int)(row - (int64_t)z * g.ny);
        }
        const int64_t site = row * g.pitch + x;
        const double ph = (double)phi[site];
        // differences to the neighbours; beyond a wall the layer itself (even mirror)
        const double xp = at(phi, g, nb_index(x, 1, g.nx, 0), y, z) - ph, xm = at(phi, g, nb_index(x, -1, g.nx, 0), y, z) - ph;
        const double yp = at(phi, g, x, nb_index(y, 1, g.ny, wy), z) - ph, ym = at(phi, g, x, nb_index(y, -1, g.ny, wy), z) - ph;
        const double gx = xp - xm, gy = yp - ym;             // twice the central difference
        double lap = (xp + xm) + (yp + ym);
        v[DQ_GX] = fma(gx, gx, v[DQ_GX]);
        v[DQ_GY] = fma(gy, gy, v[DQ_GY]);
        links = fma(xp, xp, fma(yp, yp, links));             // forward links; the one out of the last layer is zero
        if (g.d == 3) {
            const double zp = at(phi, g, x, y, nb_index(z, 1, g.nz, wz)) - ph, zm = at(phi, g, x, y, nb_index(z, -1, g.nz, wz)) - ph;
            const double gz = zp - zm;
            lap += zp + zm;
            v[DQ_GZ] = fma(gz, gz, v[DQ_GZ]);
            links = fma(zp, zp, links);
        }
        lap2 = fma(lap, lap, lap2);
        const double n = (double)aux[4 * P + site];
        const double ux = (double)aux[5 * P + site], uy = (double)aux[6 * P + site], uz = (double)aux[7 * P + site];
        v[DQ_MASS] += n;
        v[DQ_PHI] += ph;
        v[DQ_MX] = fma(n, ux, v[DQ_MX]);
        v[DQ_MY] = fma(n, uy, v[DQ_MY]);
        v[DQ_MZ] = fma(n, uz, v[DQ_MZ]);
        const double p2 = ph * ph;                           // a phi^2 / 2 + b phi^4 / 4, a = (T - Tc) / Tc
        v[DQ_FE] = fma(fma((double)T[site] - Tc, ha, hb * p2), p2, v[DQ_FE]);
        v[DQ_U2MAX] = fmax(v[DQ_U2MAX], fma(ux, ux, fma(uy, uy, uz * uz)));
    }
    v[DQ_GX] *= 0.25;
    v[DQ_GY] *= 0.25;
    v[DQ_GZ] *= 0.25;
    v[DQ_FE] = fma(0.5 * kappa, links, fma(0.5 * c, lap2, v[DQ_FE]));
    block_reduce_store<DQ_N>(v, part + (int64_t)blockIdx.x * DQ_N, DQ_U2MAX);
}

__global__ void __launch_bounds__(kThreads) k_diag_final(const double* __restrict__ part, int nblk, double* res)
{
    double v[DQ_N];
#pragma unroll
    for (int q = 0; q < DQ_N; ++q) v[q] = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x)
#pragma unroll
        for (int q = 0; q < DQ_N; ++q)
            v[q] = (q == DQ_U2MAX) ? fmax(v[q], part[(int64_t)i * DQ_N + q]) : v[q] + part[(int64_t)i * DQ_N + q];
    block_reduce_store<DQ_N>(v, res, DQ_U2MAX);
}

// One CTA per layer along the wall normal: sum (d_perp phi)^2, |grad phi|^2.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_layers(Geom g, const R* __restrict__ phi, double* out)
{
    const int h = blockIdx.x;
    const int64_t per = g.d == 2 ? g.nx : (int64_t)g.nx * g.ny;
    double v[2] = {0.0, 0.0};
    for (int64_t k = threadIdx.x; k < per; k += blockDim.x) {
        int x, y, z;
        if (g.d == 2) { x = (int)k; y = h; z = 0; }
        else { x = (int)(k % g.nx); y = (int)(k / g.nx); z = h; }
        double gr[3];
        phi_grad(phi, g, x, y, z, gr);
        const double gp = g.d == 2 ? gr[1] : gr[2];
        v[0] += gp * gp;
        v[1] += gr[0] * gr[0] + gr[1] * gr[1] + gr[2] * gr[2];
    }
    block_reduce_store<2>(v, out + 2 * h, -1);
}

// ---- structure factor --------------------------------------------------------
__device__ __forceinline__ double kfreq2(int i, int n, int64_t lmin)
{
    const int f = (2 * i <= n) ? i : i - n;
    const double r = (double)f * (double)lmin / (double)n;   // |k| / dk along this axis
    return r * r;
}

// Shell sums of |X|^2 over the half spectrum X (2 x the transform, rows of H =
// nx / 2 + 1): a mode with a conjugate partner counts twice.  A warp takes a
// row at a time, so its (ky, kz) part is formed once per row, the kx parts come
// from a table, and the shell b = floor(sqrt(r2) + 1/2) from an FP32 root
// corrected against (b - 1/2)^2 <= r2 < (b + 1/2)^2 in FP64: about ten FP64
// operations per mode (the divisions and the FP64 root made it sixty): 114 ->
// 32 us at 1024^2.  A lattice of few rows is cut into `parts` parts of a row, a
// multiple of 32 modes each: 4096 x 64 had eight CTAs, whose lanes add to the same
// shell one after the other (298 us; 40 with parts on every SM).
__global__ void __launch_bounds__(kThreads) k_shells(Geom g, const double2* __restrict__ X, int64_t lmin, int B, int parts,
                                                     double* __restrict__ bins)
{
    extern __shared__ double sm[];
    const int H = half_nx(g.nx);
    double* sum = sm;                            // B + 1
    double* kx2 = sum + B + 1;                   // H
    unsigned* cnt = reinterpret_cast<unsigned*>(kx2 + H);   // B + 1
    for (int i = threadIdx.x; i <= B; i += kThreads) { sum[i] = 0.0; cnt[i] = 0u; }
    for (int i = threadIdx.x; i < H; i += kThreads) kx2[i] = kfreq2(i, g.nx, lmin);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int items = g.ny * g.nz * parts, step = gridDim.x * (kThreads / 32);
    const int span = ((H + 31) / 32 + parts - 1) / parts * 32;
    const double top = ((double)B + 0.5) * ((double)B + 0.5);
    for (int it = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); it < items; it += step) {
        const int row = it / parts, beg = (it - row * parts) * span, end = min(beg + span, H);
        const int iz = row / g.ny, iy = row - iz * g.ny;
        double rr = kfreq2(iy, g.ny, lmin);
        if (g.d == 3) rr += kfreq2(iz, g.nz, lmin);
        if (rr >= top) continue;
        const double2* x = X + (int64_t)row * H;
        for (int ix = beg + lane; ix < end; ix += 32) {
            const double r2 = kx2[ix] + rr;
            if (r2 >= top) break;
            int b = (int)(sqrtf((float)r2) + 0.5f);
            const double e = r2 - 0.25;          // b (b - 1) <= e < b (b + 1)
            if (e < (double)(b * (b - 1))) --b;
            else if (e >= (double)(b * (b + 1))) ++b;
            if (b < 1) continue;
            const double2 v = x[ix];
            const bool two = ix > 0 && 2 * ix < g.nx;
            double p = v.x * v.x + v.y * v.y;
            if (two) p += p;
            atomicAdd(&sum[b], p);
            atomicAdd(&cnt[b], two ? 2u : 1u);
        }
    }
    __syncthreads();
    const double inv = 0.25 / ((double)g.nx * g.ny * g.nz);
    for (int i = threadIdx.x; i <= B; i += kThreads)
        if (cnt[i]) {
            atomicAdd(&bins[2 * i], sum[i] * inv);
            atomicAdd(&bins[2 * i + 1], (double)cnt[i]);
        }
}

unsigned grid_n(int64_t N)
{
    int64_t b = (N + kThreads - 1) / kThreads;
    if (b > kResident) b = kResident;
    return (unsigned)(b < 1 ? 1 : b);
}

int64_t lmin_of(const Geom& g)
{
    int64_t l = g.nx < g.ny ? g.nx : g.ny;
    if (g.d == 3 && g.nz < l) l = g.nz;
    return l;
}

// FFT of phi into sc.fft and the shell sums into sc.bins (device).  Returns
// false when a lattice size has a prime factor above 31 or a line does not
// fit in shared memory.
bool enqueue_sk(const DiagInput& in, const Scratch& sc, cudaStream_t s, cudaError_t* err)
{
    const Geom& g = in.g;
    const int64_t lmin = lmin_of(g), B = lmin / 2;
    const int sizes[3] = {g.nx, g.ny, g.nz};
    for (int a = 0; a < g.d; ++a)
        if (!fft_supported(sizes[a])) return false;
    static_assert(kMaxBins * 2 == 4096, "B <= kMaxBins for every supported line");
    *err = in.prec == LF_FP64 ? rfft_x<double>(g, (const double*)in.phi, sc.fft, s)
                              : rfft_x<float>(g, (const float*)in.phi, sc.fft, s);
    for (int a = 1; a < g.d && *err == cudaSuccess; ++a) *err = fft_axis(g, sc.fft, a, s);
    if (*err != cudaSuccess) return true;
    cudaMemsetAsync(sc.bins, 0, sizeof(double) * 2 * (B + 1), s);
    const size_t hs = (sizeof(double) + sizeof(unsigned)) * (B + 1) + sizeof(double) * half_nx(g.nx);
    static unsigned long long attr_done = 0;
    const int most = (int)((sizeof(double) + sizeof(unsigned)) * (kMaxBins + 1) + sizeof(double) * (kMaxBins + 1));
    if ((*err = raise_smem_limit(k_shells, most, &attr_done)) != cudaSuccess) return true;
    // about one CTA for every SM where whole rows give fewer, as far as parts of 32 modes go
    const int64_t rows = (int64_t)g.ny * g.nz, cta = kThreads / 32;
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>(152 * cta / rows, (half_nx(g.nx) + 31) / 32));
    const unsigned nblk = (unsigned)std::min<int64_t>(152 * 4, (rows * parts + cta - 1) / cta);
    k_shells<<<nblk, kThreads, hs, s>>>(g, sc.fft, lmin, (int)B, parts, sc.bins);
    *err = cudaGetLastError();
    return true;
}

void peak_from_bins(const std::vector<double>& bins, int64_t B, int64_t lmin, double* k_peak, double* s_peak)
{
    const double dk = 2.0 * M_PI / (double)lmin;
    std::vector<double> S(B + 1, 0.0);
    double smax = 0.0;
    for (int64_t b = 1; b <= B; ++b) {
        S[b] = bins[2 * b + 1] > 0 ? bins[2 * b] / bins[2 * b + 1] : 0.0;
        if (S[b] > smax) smax = S[b];
    }
    double num = 0.0, den = 0.0;
    for (int64_t b = 1; b <= B; ++b)
        if (S[b] > 0.5 * smax) { num += b * dk * S[b]; den += S[b]; }
    *s_peak = smax;
    *k_peak = den > 0 ? num / den : 0.0;
}

}  // namespace

size_t diag_scratch_bytes(int d, int64_t nx, int64_t ny, int64_t nz)
{
    const int64_t L = d == 2 ? ny : nz;
    int64_t lmin = nx < ny ? nx : ny;
    if (d == 3 && nz < lmin) lmin = nz;
    const int64_t B = lmin / 2;
    return a256(sizeof(double) * kBlocks * DQ_N) + a256(sizeof(double) * DQ_N) + a256(sizeof(double) * 2 * L) +
           a256(sizeof(double) * 2 * (B + 1)) + a256(sizeof(double2) * (size_t)(nx * ny * nz));
}

double2* fft_buffer(const Geom& g, void* scratch) { return carve(g, scratch).fft; }

int run_diag(const DiagInput& in, DiagResult* r, cudaStream_t s)
{
    const Geom& g = in.g;
    const Scratch sc = carve(g, in.scratch);
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    const unsigned nblk = grid_n(N);
    if (in.prec == LF_FP64)
        k_diag_partial<double><<<nblk, kThreads, 0, s>>>(g, (const double*)in.phi, (const double*)in.T,
                                                         (const double*)in.aux, in.b, in.kappa, in.c, in.Tc, sc.part);
    else
        k_diag_partial<float><<<nblk, kThreads, 0, s>>>(g, (const float*)in.phi, (const float*)in.T,
                                                        (const float*)in.aux, in.b, in.kappa, in.c, in.Tc, sc.part);
    k_diag_final<<<1, kThreads, 0, s>>>(sc.part, (int)nblk, sc.res);
    if (cudaGetLastError() != cudaSuccess) return LF_ECUDA;
    cudaError_t e = cudaSuccess;
    const bool have_sk = enqueue_sk(in, sc, s, &e);
    if (e != cudaSuccess) return LF_ECUDA;
    const int64_t lmin = lmin_of(g), B = lmin / 2;
    std::vector<double> host(DQ_N + 2 * (B + 1));
    if (cudaMemcpyAsync(host.data(), sc.res, sizeof(double) * DQ_N, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return LF_ECUDA;
    if (have_sk && cudaMemcpyAsync(host.data() + DQ_N, sc.bins, sizeof(double) * 2 * (B + 1), cudaMemcpyDeviceToHost,
                                   s) != cudaSuccess)
        return LF_ECUDA;
    int rc = wait_stream(s);
    if (rc != LF_OK) return rc;
    std::memcpy(r->sums, host.data(), sizeof(double) * DQ_N);
    if (have_sk) {
        std::vector<double> bins(host.begin() + DQ_N, host.end());
        peak_from_bins(bins, B, lmin, &r->k_peak, &r->s_peak);
    } else {
        r->k_peak = r->s_peak = NAN;
    }
    return LF_OK;
}

int run_layers(const DiagInput& in, double* out_host, cudaStream_t s)
{
    const Geom& g = in.g;
    const Scratch sc = carve(g, in.scratch);
    const int L = g.d == 2 ? g.ny : g.nz;
    if (in.prec == LF_FP64) k_layers<double><<<L, kThreads, 0, s>>>(g, (const double*)in.phi, sc.layers);
    else k_layers<float><<<L, kThreads, 0, s>>>(g, (const float*)in.phi, sc.layers);
    if (cudaGetLastError() != cudaSuccess) return LF_ECUDA;
    std::vector<double> h(2 * (size_t)L);
    if (cudaMemcpyAsync(h.data(), sc.layers, sizeof(double) * 2 * L, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return LF_ECUDA;
    int rc = wait_stream(s);
    if (rc != LF_OK) return rc;
    const int d = g.d;
    for (int i = 0; i < L; ++i)
        out_host[i] = h[2 * i + 1] > 0 ? (d * h[2 * i] / h[2 * i + 1] - 1.0) / (d - 1) : 0.0;
    return LF_OK;
}

int run_sk_shells(const DiagInput& in, double* out_host, int64_t nb, cudaStream_t s)
{
    const Geom& g = in.g;
    const int64_t lmin = lmin_of(g), B = lmin / 2;
    if (nb != B + 1) return LF_EINVAL;
    const Scratch sc = carve(g, in.scratch);
    cudaError_t e = cudaSuccess;
    if (!enqueue_sk(in, sc, s, &e)) return LF_EINVAL;
    if (e != cudaSuccess) return LF_ECUDA;
    std::vector<double> bins(2 * (B + 1));
    if (cudaMemcpyAsync(bins.data(), sc.bins, sizeof(double) * 2 * (B + 1), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return LF_ECUDA;
    int rc = wait_stream(s);
    if (rc != LF_OK) return rc;
    out_host[0] = 0.0;
    for (int64_t b = 1; b <= B; ++b) out_host[b] = bins[2 * b + 1] > 0 ? bins[2 * b] / bins[2 * b + 1] : 0.0;
    return LF_OK;
}

}  // namespace lf

// ===========================================================================
// Diagnostics without allocation (lf_diag_sums_noalloc in include/lf.h).
//
// For callers that cannot allocate device memory on the way: a reduction
// started while a CUDA graph is being captured, a real-time loop that must
// not stall on cudaMalloc's implicit synchronisation, or a host framework
// that owns every byte of device memory.  Same kernels as lf_diag's sums and
// layer sums; their scratch (per-CTA partial sums and per-layer sums) lives in
// the file-scope array below instead of a context's workspace.  Every GPU that
// loads this library holds the array (kNoAllocScratchBytes) until exit.
// ===========================================================================
namespace lf {
namespace {

constexpr int kNoAllocMaxLayers = 4096;
constexpr size_t kNoAllocPartDoubles = (size_t)kBlocks * DQ_N;
constexpr size_t kNoAllocScratchDoubles = kNoAllocPartDoubles + 2 * (size_t)kNoAllocMaxLayers;

static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

// s(h) = (d sum(d_perp phi)^2 / sum |grad phi|^2 - 1) / (d - 1), per layer.
__global__ void k_layers_to_s(const double* __restrict__ sums, int L, int d, double* __restrict__ s)
{
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= L) return;
    const double a = sums[2 * h], b = sums[2 * h + 1];
    s[h] = b > 0 ? (d * a / b - 1.0) / (d - 1) : 0.0;
}

// Device address of the scratch array on the current device, resolved once
// per device (the first call on a device does it; see the header).  The
// cached address belongs to the device's primary context: after that context
// is reset (cudaDeviceReset) the address is stale, so the entry point is not
// for use across a reset.
int noalloc_scratch(double** out)
{
    static std::mutex mu;
    static double* addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LF_ECUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return LF_ECUDA;
        }
        addr[dev] = (double*)p;
    }
    *out = addr[dev];
    return LF_OK;
}

}  // namespace
}  // namespace lf

extern "C" int lf_diag_sums_noalloc(int d, int64_t nx, int64_t ny, int64_t nz, int walls, int precision,
                                    const void* phi, const void* T, const void* moments, double b, double kappa,
                                    double c, double Tc, double* out, void* stream)
{
    using namespace lf;
    if (d != 2 && d != 3) return LF_EINVAL;
    if (nx < 1 || ny < 1 || nz < 1 || (d == 2 && nz != 1)) return LF_EINVAL;
    // bound each extent before forming the product, which could otherwise wrap
    if (nx > (1 << 24) || ny > (1 << 24) || nz > (1 << 24)) return LF_EINVAL;
    if (precision != LF_FP64 && precision != LF_FP32) return LF_EINVAL;
    if (!phi || !T || !moments || !out) return LF_EINVAL;
    if (!(Tc > 0)) return LF_EINVAL;
    const int64_t L = d == 2 ? ny : nz;
    if (L > kNoAllocMaxLayers) return LF_EINVAL;              // the layer sums would not fit
    if (nx * ny * nz >= ((int64_t)1 << 31)) return LF_EINVAL;
    double* scratch = nullptr;
    int rc = noalloc_scratch(&scratch);
    if (rc != LF_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    Geom g{};
    g.d = d;
    g.nx = (int)nx; g.ny = (int)ny; g.nz = (int)nz;
    g.pitch = (int)nx;                                     // caller fields are unpadded
    g.plane = nx * ny * nz;
    g.walls = walls ? 1 : 0;
    // The sums kernel reads n, ux, uy, uz as planes 4..7 of a context's aux
    // block; the caller's moments block holds exactly those four planes, so
    // it is addressed through a base four planes before it (only planes 4..7
    // are ever read).
    const size_t es = precision == LF_FP64 ? 8 : 4;
    const uintptr_t aux_addr = (uintptr_t)moments - 4 * (uintptr_t)g.plane * es;
    const void* aux = (const void*)aux_addr;
    const int64_t N = nx * ny * nz;
    const unsigned nblk = grid_n(N);
    double* part = scratch;
    double* lay = scratch + kNoAllocPartDoubles;
    if (precision == LF_FP64)
        k_diag_partial<double><<<nblk, kThreads, 0, s>>>(g, (const double*)phi, (const double*)T,
                                                         (const double*)aux, b, kappa, c, Tc, part);
    else
        k_diag_partial<float><<<nblk, kThreads, 0, s>>>(g, (const float*)phi, (const float*)T,
                                                        (const float*)aux, b, kappa, c, Tc, part);
    k_diag_final<<<1, kThreads, 0, s>>>(part, (int)nblk, out);
    if (precision == LF_FP64) k_layers<double><<<(unsigned)L, kThreads, 0, s>>>(g, (const double*)phi, lay);
    else k_layers<float><<<(unsigned)L, kThreads, 0, s>>>(g, (const float*)phi, lay);
    k_layers_to_s<<<(unsigned)((L + 127) / 128), 128, 0, s>>>(lay, (int)L, d, out + DQ_N);
    return cudaGetLastError() == cudaSuccess ? LF_OK : LF_ECUDA;
}
