// lf_step2d_f64.cu -- the D2Q9 step of arXiv:1102.3094, Sec. 2, in FP64 with
// either stencil, one tile of sites per CTA.
//
// This GPU's FP64 pipe issues 1.8 operations per clock and SM (about one warp
// instruction in 60 clocks on each of its four partitions), so an FP64 step
// takes as long as its FP64 operations do, and everything else hides behind
// them.  Two things follow:
//   - operations are counted: derivatives stay unscaled sums (the factors 1/2,
//     1/6, 1/12 go into the coefficients of the expressions that use them),
//     products are shared, the collision is per opposite pair with the weights
//     folded into its coefficients: 160 operations per site and step with the
//     compact stencils;
//   - the tile decides how much of them is repeated in halos and how many
//     partitions have work: small lattices take 8 x 4 tiles, so that 64^2 is
//     on 128 SMs, larger ones up to 32 x 16.  Within a tile every stage is a
//     flat list of items; the collision's are (pair, site), so that its work,
//     the largest, is on all partitions even for 32 sites.
// Regions as in lf_tile2d.cuh: phi on the tile + 4, psi + 3, lam, P and mu + 2,
// velocity and flux + 1.  Halo sites read through the boundary map (x wraps; y
// wraps or is mirrored about the half-way walls), so every derived field there
// is that of the mirrored state; the wall-normal flux is odd.
//
// Against the row march (lf_march2d.cuh, lf_march2d_iso.cuh), whose CTAs
// recompute their halo rows and are few on small lattices, per step:
//   64^2 8.6 us (march 21.6), 128^2 14.4 (38), 256^2 36.6 (64), 512^2 123 (175),
//   768^2 258 (277), 1024^2 451 (450);
//   isotropic 64^2 11.5 (33), 256^2 49 (89), 512^2 183 (238), 768^2 365 (360),
//   1024^2 638 (572).
// Longer segments make the march's halo rows cheap on large lattices, so it
// keeps those: f64_tiles() draws the line.
#include "lf_internal.cuh"
#include "lf_march2d.cuh"

namespace lf {

namespace {

using march::map_row;
using march::wrap_near;

// Sums that are a derivative times a constant: KL lap and KD d_a.
template <bool ISO>
struct Fd {
    static constexpr double KL = ISO ? 6.0 : 1.0, KD = ISO ? 12.0 : 2.0;
    template <int W>
    static __device__ __forceinline__ double lap(const double* a, int c)
    {
        const double nn = (a[c - 1] + a[c + 1]) + (a[c - W] + a[c + W]);
        if constexpr (ISO) {
            const double dd = (a[c - W - 1] + a[c - W + 1]) + (a[c + W - 1] + a[c + W + 1]);
            return fma(-20.0, a[c], fma(4.0, nn, dd));
        } else {
            return fma(-4.0, a[c], nn);
        }
    }
    template <int W>
    static __device__ __forceinline__ double dx(const double* a, int c)
    {
        const double m = a[c + 1] - a[c - 1];
        if constexpr (ISO) return fma(4.0, m, (a[c + W + 1] - a[c + W - 1]) + (a[c - W + 1] - a[c - W - 1]));
        else return m;
    }
    template <int W>
    static __device__ __forceinline__ double dy(const double* a, int c)
    {
        const double m = a[c + W] - a[c - W];
        if constexpr (ISO) return fma(4.0, m, (a[c + W + 1] - a[c - W + 1]) + (a[c + W - 1] - a[c - W - 1]));
        else return m;
    }
};

template <int TX, int TY>
struct TileF64 {
    static constexpr int W4 = TX + 8, H4 = TY + 8, W3 = TX + 6, H3 = TY + 6;
    static constexpr int W2 = TX + 4, H2 = TY + 4, W1 = TX + 2, H1 = TY + 2;
    static constexpr int N = TX * TY;
    static constexpr int RING = 2 * W1 + 2 * TY;             // the sites around the tile
    static constexpr int PHI = 0;
    static constexpr int T = PHI + W4 * H4;
    static constexpr int PSI = T + W2 * H2;
    static constexpr int P = PSI + W3 * H3;                  // xx, yy, xy
    static constexpr int MU = P + 3 * W2 * H2;
    static constexpr int G = MU + W2 * H2;                   // gx, gy (tile + 1)
    static constexpr int C = G + 2 * W1 * H1;                // C0, omega n, vx, vy, Fx, Fy per site
    static constexpr int TOTAL = C + 6 * N;
    static constexpr size_t BYTES = sizeof(double) * TOTAL;
};

template <int TX, int TY, int NT, bool ISO>
__global__ void __launch_bounds__(NT) k_step2d_f64(Geom g, Phys<double> p, StepIO<double> io, int ybeg)
{
    using L = D2Q9;
    using TL = TileF64<TX, TY>;
    using D = Fd<ISO>;
    constexpr int W4 = TL::W4, W3 = TL::W3, W2 = TL::W2, H2 = TL::H2, W1 = TL::W1, H1 = TL::H1, N = TL::N;
    extern __shared__ __align__(16) double sm_f64[];
    double* sphi = sm_f64 + TL::PHI;
    double* sT = sm_f64 + TL::T;
    double* spsi = sm_f64 + TL::PSI;
    double* sPxx = sm_f64 + TL::P;
    double* sPyy = sPxx + W2 * H2;
    double* sPxy = sPyy + W2 * H2;
    double* smu = sm_f64 + TL::MU;
    double* sgx = sm_f64 + TL::G;
    double* sgy = sgx + W1 * H1;
    double* sc = sm_f64 + TL::C;

    const int nx = g.nx, ny = g.ny, pitch = g.pitch, walls = g.walls;
    const int plane = (int)g.plane;                          // 32-bit offsets: Q * padded sites < 2^31
    const int x0 = blockIdx.x * TX, y0 = ybeg + blockIdx.y * TY;
    bool bad = false;

    chain_wait();
    for (int k = threadIdx.x; k < W4 * TL::H4; k += NT) {
        const int ly = k / W4, lx = k - ly * W4;
        sphi[k] = io.phi_in[map_row(y0 - 4 + ly, ny, walls) * pitch + wrap_near(x0 - 4 + lx, nx)];
    }
    for (int k = threadIdx.x; k < W2 * H2; k += NT) {
        const int ly = k / W2, lx = k - ly * W2;
        sT[k] = io.T_in[map_row(y0 - 2 + ly, ny, walls) * pitch + wrap_near(x0 - 2 + lx, nx)];
    }
    __syncthreads();

    for (int k = threadIdx.x; k < W3 * TL::H3; k += NT) {    // KL psi
        const int ly = k / W3, lx = k - ly * W3;
        spsi[k] = D::template lap<W4>(sphi, (ly + 1) * W4 + lx + 1);
    }
    __syncthreads();

    // lam, mu, P.  With s = KL psi, l = KL^2 lam, D = KD grad phi, S = KD KL grad psi:
    //   mu  = phi (a + b phi^2) - kappa psi + c lam
    //   iso = phi^2 (a / 2 + 3/4 b phi^2) - kappa (phi psi + |grad phi|^2 / 2)
    //       + c (phi lam + psi^2 / 2 + grad phi . grad psi)
    //   P_ab = iso delta_ab + kappa d_a d_b - c (d_a s_b + d_b s_a)
    // with a = (T - Tc) / Tc from the difference, which is exact near Tc (a fused
    // T / (2 Tc) - 1/2 has the rounding of 1 / Tc instead: 2e-17 at T = Tc)
    {
        const double b34 = 0.75 * p.b;
        const double kL = -p.kappa / D::KL, cL = p.c / (D::KL * D::KL);
        const double g2 = 0.5 / (D::KD * D::KD), p2 = 0.5 / (D::KL * D::KL), gs = 1.0 / (D::KD * D::KD * D::KL);
        const double kD = p.kappa / (D::KD * D::KD), cD = -p.c * gs;
        for (int k = threadIdx.x; k < W2 * H2; k += NT) {
            const int ly = k / W2, lx = k - ly * W2;
            const int cp = (ly + 2) * W4 + lx + 2, cs = (ly + 1) * W3 + lx + 1;
            const double ph = sphi[cp], ps = spsi[cs];
            const double lam = D::template lap<W3>(spsi, cs);
            const double a = (sT[k] - p.Tc) * p.inv_Tc, ph2 = ph * ph;
            smu[k] = fma(cL, lam, fma(kL, ps, ph * fma(p.b, ph2, a)));
            if (p.hydro) {
                const double dx = D::template dx<W4>(sphi, cp), dy = D::template dy<W4>(sphi, cp);
                const double ex = D::template dx<W3>(spsi, cs), ey = D::template dy<W3>(spsi, cs);
                const double xx = dx * dx, yy = dy * dy, ux = dx * ex, uy = dy * ey;
                double iso = ph2 * fma(b34, ph2, 0.5 * a);
                iso = fma(-p.kappa, fma(g2, xx + yy, ph * ps * (1.0 / D::KL)), iso);
                iso = fma(p.c, fma(gs, ux + uy, fma(p2 * ps, ps, ph * lam * (1.0 / (D::KL * D::KL)))), iso);
                sPxx[k] = fma(kD, xx, fma(2.0 * cD, ux, iso));
                sPyy[k] = fma(kD, yy, fma(2.0 * cD, uy, iso));
                sPxy[k] = fma(kD * dx, dy, cD * fma(dx, ey, dy * ex));
            }
        }
    }
    __syncthreads();

    // velocity and flux on the tile (items 0 .. N - 1, from a warp boundary on
    // the ring around it), and what the collision needs on the tile
    constexpr int N32 = (N + 31) / 32 * 32;
    const double omega = p.inv_tau, keep = 1.0 - p.inv_tau;
    for (int k = threadIdx.x; k < N32 + TL::RING; k += NT) {
        const bool inner = k < N32;
        int lx, ly;                                          // in the tile + 1
        if (inner) {
            if (k >= N) continue;
            ly = k / TX;
            lx = k - ly * TX + 1;
            ly += 1;
        } else {
            const int r = k - N32;
            if (r < 2 * W1) { ly = r < W1 ? 0 : H1 - 1; lx = r < W1 ? r : r - W1; }
            else { ly = 1 + (r - 2 * W1) / 2; lx = (r & 1) ? W1 - 1 : 0; }
            if (!ISO && (lx == 0 || lx == W1 - 1) && (ly == 0 || ly == H1 - 1)) continue;
        }
        const int ux = x0 - 1 + lx, uy = y0 - 1 + ly;        // unwrapped
        const int c1 = ly * W1 + lx;
        if (!p.hydro || (walls && (uy < 0 || uy >= ny))) {   // beyond a wall: the images are taken below
            sgx[c1] = 0.0;
            sgy[c1] = 0.0;
            continue;
        }
        const int site = (walls ? uy : wrap_near(uy, ny)) * pitch + wrap_near(ux, nx);
        const double* f = io.f_in + site;
        const double f0 = f[0], f1 = f[plane], f2 = f[2 * plane], f3 = f[3 * plane], f4 = f[4 * plane];
        const double f5 = f[5 * plane], f6 = f[6 * plane], f7 = f[7 * plane], f8 = f[8 * plane];
        const double dn = (((f0 + f1) + (f2 + f3)) + ((f4 + f5) + (f6 + f7))) + f8;
        const double a = f5 - f7, b = f6 - f8;
        const double jx = (f1 - f3) + (a - b), jy = (f2 - f4) + (a + b);
        const int c2 = (ly + 1) * W2 + lx + 1;
        const double Sx = D::template dx<W2>(sPxx, c2) + D::template dy<W2>(sPxy, c2);   // -KD F
        const double Sy = D::template dx<W2>(sPxy, c2) + D::template dy<W2>(sPyy, c2);
        const double n = p.n0 + dn, inv_n = 1.0 / n;
        const double vx = fma(-0.5 / D::KD, Sx, jx) * inv_n, vy = fma(-0.5 / D::KD, Sy, jy) * inv_n;
        const double ph = sphi[(ly + 3) * W4 + lx + 3];
        sgx[c1] = ph * vx;
        sgy[c1] = ph * vy;
        if (!inner || ux >= nx || uy >= ny) continue;
        bad |= !isfinite(n);
        const double Fx = (-1.0 / D::KD) * Sx, Fy = (-1.0 / D::KD) * Sy;
        const double on = omega * n;
        const double C0 = fma(-3.0 * p.guo, fma(vx, Fx, vy * Fy), fma(-1.5 * on, fma(vx, vx, vy * vy), omega * dn));
        sc[k] = C0;
        sc[N + k] = on;
        sc[2 * N + k] = vx;
        sc[3 * N + k] = vy;
        sc[4 * N + k] = Fx;
        sc[5 * N + k] = Fy;
        io.f_out[site] = fma(keep, f0, L::w(0) * C0);
    }
    __syncthreads();

    // collide and push: item = pair N + site, the pair the same for a whole
    // warp when N is a multiple of 32; then phi and T of the tile
    constexpr int kItems = 4 * N;
    if (p.hydro) {
        for (int k = threadIdx.x; k < kItems; k += NT) {
            const int pr = k / N, s = k - pr * N;
            const int ly = s / TX, lx = s - ly * TX;
            const int gx = x0 + lx, gy = y0 + ly;
            if (gx >= nx || gy >= ny) continue;
            // pairs (1, 3), (2, 4), (5, 7), (6, 8): the first's velocity
            const int ex = pr == 0 ? 1 : pr == 1 ? 0 : pr == 2 ? 1 : -1, ey = pr == 0 ? 0 : 1;
            const int i = pr == 0 ? 1 : pr == 1 ? 2 : pr == 2 ? 5 : 6, j = i + 2;
            const double w = pr < 2 ? L::w(1) : L::w(5);
            const double vx = sc[2 * N + s], vy = sc[3 * N + s], Fx = sc[4 * N + s], Fy = sc[5 * N + s];
            const double sv = pr == 0 ? vx : pr == 1 ? vy : pr == 2 ? vx + vy : vy - vx;
            const double ev = pr == 0 ? Fx : pr == 1 ? Fy : pr == 2 ? Fx + Fy : Fy - Fx;
            const double won = w * sc[N + s], we = 3.0 * p.guo * w * ev;
            const double sym = fma(sv, fma(4.5 * won, sv, 3.0 * we), w * sc[s]);
            const double anti = fma(3.0 * won, sv, we);
            const int site = gy * pitch + gx;
            const double pi = fma(keep, io.f_in[i * plane + site], sym) + anti;
            const double pj = fma(keep, io.f_in[j * plane + site], sym) - anti;
            const int xp = gx + 1 == nx ? 0 : gx + 1, xm = gx == 0 ? nx - 1 : gx - 1;
            const int yp = (gy + 1 == ny ? 0 : gy + 1) * pitch, ym = (gy == 0 ? ny - 1 : gy - 1) * pitch, yc = gy * pitch;
            const int to_i = (ey > 0 ? yp : yc) + (ex > 0 ? xp : ex < 0 ? xm : gx);
            const int to_j = (ey > 0 ? ym : yc) + (ex > 0 ? xm : ex < 0 ? xp : gx);
            // a population leaving through a wall returns reversed
            const bool hi = walls && ey > 0 && gy == ny - 1, lo = walls && ey > 0 && gy == 0;
            io.f_out[hi ? j * plane + site : i * plane + to_i] = pi;
            io.f_out[lo ? i * plane + site : j * plane + to_j] = pj;
        }
    }
    for (int k = threadIdx.x; k < N; k += NT) {
        const int ly = k / TX, lx = k - ly * TX;
        const int gx = x0 + lx, gy = y0 + ly;
        if (gx >= nx || gy >= ny) continue;
        const int site = gy * pitch + gx;
        const int c1 = (ly + 1) * W1 + lx + 1, c2 = (ly + 2) * W2 + lx + 2, cp = (ly + 4) * W4 + lx + 4;
        const bool lo = walls && gy == 0, hi = walls && gy == ny - 1;
        double phn = fma(p.Gamma / D::KL, D::template lap<W2>(smu, c2), sphi[cp]);
        if (p.hydro) {
            // the row beyond a wall is the image of the site's own: g_x even, g_y odd
            const int rd = lo ? c1 : c1 - W1, ru = hi ? c1 : c1 + W1;
            double div;
            if constexpr (ISO) {
                const double sd = lo ? -1.0 : 1.0, su = hi ? -1.0 : 1.0;
                const double dgx = fma(4.0, sgx[c1 + 1] - sgx[c1 - 1], (sgx[ru + 1] - sgx[ru - 1]) + (sgx[rd + 1] - sgx[rd - 1]));
                const double gu = fma(4.0, sgy[ru], sgy[ru + 1] + sgy[ru - 1]), gd = fma(4.0, sgy[rd], sgy[rd + 1] + sgy[rd - 1]);
                div = dgx + fma(su, gu, -sd * gd);
            } else {
                const double gu = hi ? -sgy[c1] : sgy[ru], gd = lo ? -sgy[c1] : sgy[rd];
                div = (sgx[c1 + 1] - sgx[c1 - 1]) + (gu - gd);
            }
            phn = fma(-1.0 / D::KD, div, phn);
        }
        const double t0 = sT[c2];
        double Tn = t0;
        if (p.t_update) {
            if ((lo || hi) && g.t_mode == LF_TWALL_LAYERS) {
                Tn = p.T_w;
            } else {
                const bool gl = lo && g.t_mode == LF_TWALL_HALFWAY, gh = hi && g.t_mode == LF_TWALL_HALFWAY;
                const double tw2 = 2.0 * p.T_w;
                const double* d = sT + c2 - W2;
                const double* u = sT + c2 + W2;
                // halfway ghosts: 2 T_w minus the mirror image that the halo row holds
                const double d0 = gl ? tw2 - d[0] : d[0], u0 = gh ? tw2 - u[0] : u[0];
                double lap = (sT[c2 - 1] + sT[c2 + 1]) + (u0 + d0);
                if constexpr (ISO) {
                    const double dl = gl ? tw2 - d[-1] : d[-1], dr = gl ? tw2 - d[1] : d[1];
                    const double ul = gh ? tw2 - u[-1] : u[-1], ur = gh ? tw2 - u[1] : u[1];
                    lap = fma(-20.0, t0, fma(4.0, lap, (ul + ur) + (dl + dr)));
                } else {
                    lap = fma(-4.0, t0, lap);
                }
                Tn = fma(p.dxi / D::KL, lap, t0);
            }
        }
        bad |= !isfinite(phn) || !isfinite(Tn);
        io.phi_out[site] = phn;
        io.T_out[site] = Tn;
    }
    chain_next();
    if (bad) *reinterpret_cast<volatile int*>(io.flag) = 1;
}

// Time of a step in FP64 warp instructions of the busiest SM's partitions, for
// tiles of TX x TY: the rounds of tiles over the SMs times the items of each
// stage, in whole warps; when an SM has a single tile, in whole rows of one
// warp per partition.
template <int TX, int TY>
int64_t tile_cost(int nx, int ny, int sms, bool iso)
{
    using TL = TileF64<TX, TY>;
    const int64_t tiles = (int64_t)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY);
    const int64_t rounds = (tiles + sms - 1) / sms;
    const int q = rounds == 1 ? 128 : 32;
    auto w = [q](int n) { return (int64_t)(n + q - 1) / q * q; };
    const int64_t one = w(TL::W3 * TL::H3) * (iso ? 8 : 4) + w(TL::W2 * TL::H2) * (iso ? 66 : 42) +
                        w(TL::N + TL::RING) * (iso ? 62 : 46) + w(4 * TL::N) * 15 + w(TL::N) * (iso ? 36 : 15);
    return rounds * one;
}

template <int TX, int TY, int NT>
cudaError_t launch_tile(const Geom& g, const Phys<double>& p, const StepIO<double>& io, cudaStream_t s)
{
    constexpr size_t bytes = TileF64<TX, TY>::BYTES;
    const bool iso = g.stencil == LF_STENCIL_ISOTROPIC;
    auto kern = iso ? k_step2d_f64<TX, TY, NT, true> : k_step2d_f64<TX, TY, NT, false>;
    static unsigned long long attr_done[2] = {};             // per instantiation and device
    cudaError_t e = raise_smem_limit(kern, (int)bytes, &attr_done[iso]);
    // A narrow lattice may have more rows of tiles than the grid's y takes: one launch for every 65,535 then.  (Tiles
    // counted on x alone cost a division per block: 512^2 126 us a step instead of 122; folded into y and z, 64^2
    // 8.62 instead of 8.55.)
    constexpr int kRows = 65535;
    for (int r = 0, rows = (g.ny + TY - 1) / TY; r < rows && e == cudaSuccess; r += kRows) {
        const dim3 grid((g.nx + TX - 1) / TX, rows - r < kRows ? rows - r : kRows);
        e = launch_chained(kern, grid, NT, bytes, s, g, p, io, r * TY);
    }
    return e;
}

}  // namespace

bool f64_tiles(const Geom& g)
{
    return (int64_t)g.nx * g.ny <= (g.stencil == LF_STENCIL_ISOTROPIC ? 1 << 19 : 1 << 20);
}

cudaError_t launch_step2d_f64(const Geom& g, const Phys<double>& p, const StepIO<double>& io, cudaStream_t s)
{
    int sms = 0;
    const cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const bool iso = g.stencil == LF_STENCIL_ISOTROPIC;
    const int64_t cost[4] = {tile_cost<8, 4>(g.nx, g.ny, sms, iso), tile_cost<16, 8>(g.nx, g.ny, sms, iso),
                             tile_cost<16, 16>(g.nx, g.ny, sms, iso), tile_cost<32, 16>(g.nx, g.ny, sms, iso)};
    int best = 0;
    for (int i = 1; i < 4; ++i)
        if (cost[i] < cost[best]) best = i;
    switch (best) {
    case 0: return launch_tile<8, 4, 128>(g, p, io, s);
    case 1: return launch_tile<16, 8, 128>(g, p, io, s);
    case 2: return launch_tile<16, 16, 256>(g, p, io, s);
    default: return launch_tile<32, 16, 256>(g, p, io, s);
    }
}

}  // namespace lf
