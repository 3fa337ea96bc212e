// lf_step3d_phi.cu -- pass C of the three-pass D3Q19 step (lf_step3d_split.cu)
// in FP32, with either stencil: phi(t+1) = phi - div(phi u) + Gamma lap(mu)
// (Eq. massdiff) and the first temperature sub-step, four sites per thread.
//
// The pass moves 32 B per site (mu, u, phi, T in; phi, T out), so memory should
// bound it: 267 us at 384^3.  With one site per thread it was bound by
// instructions instead, most of them addresses and 22 (compact) or 44
// (isotropic, through shared memory) loads per site: 433 and 590 us.  Here a
// thread owns four consecutive sites of a row and marches along z: every load
// and store is 16 bytes, x-neighbours inside the four come free, those across
// by one shuffle each way (a scalar load where a row of lanes ends),
// z-neighbours from registers; the two stencils read 13 and 17 vectors per
// plane.  No shared memory, no barriers.  At the register counts this takes
// (122 and 153) too few loads are in flight to cover DRAM latency, so each
// plane is asked for in L2 one iteration before it is loaded: 308 -> 273 us
// (compact, 98 % of the measured copy bandwidth) and 426 -> 373 us (isotropic,
// 72 %; the rest is its 440 instructions per 128 sites at 12 warps per SM).
#include "lf_step3d_common.cuh"
#include "lf_iso3.cuh"

namespace lf {

namespace {

struct Q4 {
    float v[4];
};

__device__ __forceinline__ Q4 mul4(const Q4& a, const Q4& b)
{
    Q4 r;
#pragma unroll
    for (int i = 0; i < 4; ++i) r.v[i] = __fmul_rn(a.v[i], b.v[i]);   // a flux is rounded once for all its readers
    return r;
}

// Four sites of a row with the neighbour on either side: v[-1 .. 4] as e[0 .. 5].
struct Row {
    float e[6];
};

// Where a thread's four sites lie.  A row of the lattice is taken by
// consecutive lanes, LX of them per row and warp; lanes past the end of the
// row hold its first quad (the right neighbour of the last one) and store
// nothing.
template <int LX>
struct Quad {
    int x, y, nv;                 // first site, row, how many of the four are sites
    int xe;                       // the first / last lane's neighbour site beyond its warp's quads
    bool act, edge, first;        // stores; is a first or last lane; is a first lane
    __device__ Quad(const Geom& g)
    {
        const int lane = threadIdx.x % LX;
        const int nq = (g.nx + 3) / 4;
        const unsigned across = (unsigned)(nq + LX - 1) / LX, by = blockIdx.x / across;   // blocks per row of them
        const int q = (int)(blockIdx.x - by * across) * LX + lane;
        y = (int)(by * (blockDim.x / LX)) + threadIdx.x / LX;
        act = q < nq && y < g.ny;
        if (y >= g.ny) y = g.ny - 1;
        x = q < nq ? 4 * q : 0;
        nv = g.nx - x < 4 ? g.nx - x : 4;
        first = lane == 0;
        edge = first || lane == LX - 1;
        xe = first ? (x == 0 ? g.nx - 1 : x - 1) : (x + 4 >= g.nx ? 0 : x + 4);
    }
    __device__ __forceinline__ Q4 load(const float* row) const
    {
        const float4 w = *reinterpret_cast<const float4*>(row + x);
        return Q4{{w.x, w.y, w.z, w.w}};
    }
    // the value beside the quads of this row of lanes (0 in the lanes between)
    __device__ __forceinline__ float beside(const float* row) const { return edge ? row[xe] : 0.f; }
    __device__ __forceinline__ Row around(const Q4& a, float b) const
    {
        Row r;
        const float l = __shfl_up_sync(0xffffffffu, a.v[3], 1, LX);
        float n = __shfl_down_sync(0xffffffffu, a.v[0], 1, LX);
        if (edge && !first) n = b;
        r.e[0] = first ? b : l;
        r.e[1] = a.v[0];
        r.e[2] = nv > 1 ? a.v[1] : n;            // n where the row ends inside the quad
        r.e[3] = nv > 2 ? a.v[2] : n;
        r.e[4] = nv > 3 ? a.v[3] : n;
        r.e[5] = n;
        return r;
    }
    // ask for the thread's sites of plane z, to be loaded an iteration from now, in L2
    template <bool HYD>
    __device__ __forceinline__ void ahead(const StepIO<float>& io, int z, int nz, int zs, int row) const
    {
        if (z >= nz) return;
        const int o = z * zs + row + x;
        auto ask = [&](const float* f) { asm volatile("prefetch.global.L2 [%0];" ::"l"(f + o)); };
        ask(io.mu);
        ask(io.T_in);
        ask(io.phi_in);
        if constexpr (HYD) {
            ask(io.u[0]);
            ask(io.u[1]);
            ask(io.u[2]);
        }
    }
    __device__ __forceinline__ void store(float* row, const Q4& a) const
    {
        if (nv == 4) {
            *reinterpret_cast<float4*>(row + x) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (i < nv) row[x + i] = a.v[i];
        }
    }
};

// Storage plane of z - 1 / z + 1: the wrap, or the plane itself beyond a wall.
__device__ __forceinline__ int z_below(int z, int nz, int walls) { return z == 0 ? (walls ? 0 : nz - 1) : z - 1; }
__device__ __forceinline__ int z_above(int z, int nz, int walls) { return z + 1 == nz ? (walls ? z : 0) : z + 1; }

// Compact stencils.
template <int LX, bool HYD>
__global__ void __launch_bounds__(128) k_phi3d_q(Geom g, Phys<float> p, StepIO<float> io, int zc)
{
    const Quad<LX> q(g);
    const int za = blockIdx.z * zc, zb = min(za + zc, g.nz);
    const int nz = g.nz, pitch = g.pitch, walls = g.walls;
    const int zs = g.ny * pitch;                 // 32-bit offsets: Q * padded sites < 2^31 (checked at creation)
    const int row = q.y * pitch;
    const int rl = (q.y == 0 ? g.ny - 1 : q.y - 1) * pitch, rr = (q.y + 1 == g.ny ? 0 : q.y + 1) * pitch;
    const float half = 0.5f;
    chain_wait();
    int o = z_below(za, nz, walls) * zs + row;
    Q4 mu_d = q.load(io.mu + o), T_d = q.load(io.T_in + o), gz_d{}, gz_c{}, ph_c;
    if constexpr (HYD) gz_d = mul4(q.load(io.phi_in + o), q.load(io.u[2] + o));
    o = za * zs + row;
    Q4 mu_c = q.load(io.mu + o), T_c = q.load(io.T_in + o);
    ph_c = q.load(io.phi_in + o);
    if constexpr (HYD) gz_c = mul4(ph_c, q.load(io.u[2] + o));
    bool bad = false;
    for (int z = za; z < zb; ++z) {
        const int oz = z * zs, oc = oz + row, ou = z_above(z, nz, walls) * zs + row;
        q.template ahead<HYD>(io, z + 2, nz, zs, row);
        const Q4 mu_u = q.load(io.mu + ou), T_u = q.load(io.T_in + ou), ph_u = q.load(io.phi_in + ou);
        const Q4 myl = q.load(io.mu + oz + rl), myr = q.load(io.mu + oz + rr);
        const Q4 tyl = q.load(io.T_in + oz + rl), tyr = q.load(io.T_in + oz + rr);
        const float mb = q.beside(io.mu + oc), tb = q.beside(io.T_in + oc);
        Q4 uz_u{}, gx{}, gyl{}, gyr{};
        float gb = 0.f;
        if constexpr (HYD) {
            uz_u = q.load(io.u[2] + ou);
            gx = q.load(io.u[0] + oc);
            gb = __fmul_rn(q.beside(io.phi_in + oc), q.beside(io.u[0] + oc));
            gyl = mul4(q.load(io.phi_in + oz + rl), q.load(io.u[1] + oz + rl));
            gyr = mul4(q.load(io.phi_in + oz + rr), q.load(io.u[1] + oz + rr));
        }
        const Row m = q.around(mu_c, mb), t = q.around(T_c, tb);
        Row gr{};
        Q4 gz_u{};
        if constexpr (HYD) {
            gz_u = mul4(ph_u, uz_u);
            gr = q.around(mul4(ph_c, gx), gb);
        }
        const bool lo = walls && z == 0, hi = walls && z == nz - 1;
        const bool held = (lo || hi) && g.t_mode == LF_TWALL_LAYERS, half_t = g.t_mode == LF_TWALL_HALFWAY;
        Q4 phn, Tn;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float lapmu = m.e[i] + m.e[i + 2] + myl.v[i] + myr.v[i] + mu_u.v[i] + mu_d.v[i] - 6.f * mu_c.v[i];
            float div = 0.f;
            if constexpr (HYD) {
                const float up = hi ? -gz_c.v[i] : gz_u.v[i], dn = lo ? -gz_c.v[i] : gz_d.v[i];   // no flux through the walls
                div = half * (gr.e[i + 2] - gr.e[i]) + half * (gyr.v[i] - gyl.v[i]) + half * (up - dn);
            }
            phn.v[i] = ph_c.v[i] - div + p.Gamma * lapmu;
            float v = T_c.v[i];
            if (p.t_update) {
                const float gw = 2.f * p.T_w - v;
                const float td = lo && half_t ? gw : T_d.v[i], tu = hi && half_t ? gw : T_u.v[i];
                const float n = v + p.dxi * (t.e[i] + t.e[i + 2] + tyl.v[i] + tyr.v[i] + tu + td - 6.f * v);
                v = held ? p.T_w : n;
            }
            Tn.v[i] = v;
            bad |= q.act && i < q.nv && (!isfinite(phn.v[i]) || !isfinite(v));
        }
        if (q.act) {
            q.store(io.phi_out + oc, phn);
            q.store(io.T_out + oc, Tn);
        }
        mu_d = mu_c; mu_c = mu_u;
        T_d = T_c; T_c = T_u;
        gz_d = gz_c; gz_c = gz_u;
        ph_c = ph_u;
    }
    chain_next();
    if (bad) *reinterpret_cast<volatile int*>(io.flag) = 1;
}

// Isotropic stencils: the parts of each plane (Plane19, Slide19 in
// lf_iso3.cuh) from the rows y - 1, y, y + 1 as they are loaded, the open sums
// of the thread's sites in registers.  Iteration k adds plane k and completes
// plane k - 1; a plane beyond a wall holds the wall plane, its parts enter
// transformed (g_z odd: s -> -s; T with its halfway ghost: s -> 12 T_w - s).
__device__ __forceinline__ Plane19<float> part19(const Row& s, const Row& c, const Row& n, int i)
{
    const float e = c.e[i + 2], w = c.e[i], no = n.e[i + 1], so = s.e[i + 1];
    const float ne = n.e[i + 2], nw = n.e[i], se = s.e[i + 2], sw = s.e[i];
    const float cross = (e + w) + (no + so);
    Plane19<float> r;
    r.s = 2.f * c.e[i + 1] + cross;
    r.l = 2.f * cross + ((ne + nw) + (se + sw)) - 24.f * c.e[i + 1];
    r.ax = e - w;
    r.ay = no - so;
    r.gx = 2.f * r.ax + (ne - nw) + (se - sw);
    r.gy = 2.f * r.ay + (ne - se) + (nw - sw);
    return r;
}

template <int LX, bool HYD>
__global__ void __launch_bounds__(128, 3) k_phi3d_iso_q(Geom g, Phys<float> p, StepIO<float> io, int zc)
{
    const Quad<LX> q(g);
    const int za = blockIdx.z * zc, zb = min(za + zc, g.nz);
    const int nz = g.nz, pitch = g.pitch, walls = g.walls;
    const int zs = g.ny * pitch;
    const int row = q.y * pitch;
    const int rl = (q.y == 0 ? g.ny - 1 : q.y - 1) * pitch, rr = (q.y + 1 == g.ny ? 0 : q.y + 1) * pitch;
    const bool halfway = walls && g.t_mode == LF_TWALL_HALFWAY;
    chain_wait();
    // sums of the open centre and the last plane's parts, per site
    float ml[4], ms[4], tl[4], ts[4];            // lap mu, lap T
    float gxo[4], gxa[4], gyo[4], gya[4];        // d_x g_x, d_y g_y
    float gs0[4], gs1[4];                        // s of g_z, last two planes
#pragma unroll
    for (int i = 0; i < 4; ++i)
        ml[i] = ms[i] = tl[i] = ts[i] = gxo[i] = gxa[i] = gyo[i] = gya[i] = gs0[i] = gs1[i] = 0.f;
    Q4 T1{}, ph1{};                              // own T and phi of plane k - 1
    bool bad = false;
    for (int k = za - 1; k <= zb; ++k) {
        const bool ghost = walls && (k < 0 || k >= nz);
        const int kz = k < 0 ? (walls ? 0 : nz - 1) : k >= nz ? (walls ? nz - 1 : 0) : k;
        const int oz = kz * zs, oc = oz + row, ol = oz + rl, orr = oz + rr;
        q.template ahead<HYD>(io, k + 1, nz, zs, row);
        const Q4 mc = q.load(io.mu + oc), mn = q.load(io.mu + orr), mso = q.load(io.mu + ol);
        const Q4 tc = q.load(io.T_in + oc), tn = q.load(io.T_in + orr), tso = q.load(io.T_in + ol);
        const Q4 pc = q.load(io.phi_in + oc);
        const float mbc = q.beside(io.mu + oc), mbn = q.beside(io.mu + orr), mbs = q.beside(io.mu + ol);
        const float tbc = q.beside(io.T_in + oc), tbn = q.beside(io.T_in + orr), tbs = q.beside(io.T_in + ol);
        float pbc = 0.f, pbn = 0.f, pbs = 0.f, xbc = 0.f, xbn = 0.f, xbs = 0.f, ybn = 0.f, ybs = 0.f, zbc = 0.f;
        Q4 pn{}, pso{}, xc{}, xn{}, xso{}, yn{}, yso{}, zcn{}, zn{}, zso{};
        if constexpr (HYD) {
            pn = q.load(io.phi_in + orr); pso = q.load(io.phi_in + ol);
            xc = q.load(io.u[0] + oc); xn = q.load(io.u[0] + orr); xso = q.load(io.u[0] + ol);
            yn = q.load(io.u[1] + orr); yso = q.load(io.u[1] + ol);
            zcn = q.load(io.u[2] + oc); zn = q.load(io.u[2] + orr); zso = q.load(io.u[2] + ol);
            pbc = q.beside(io.phi_in + oc); pbn = q.beside(io.phi_in + orr); pbs = q.beside(io.phi_in + ol);
            xbc = q.beside(io.u[0] + oc); xbn = q.beside(io.u[0] + orr); xbs = q.beside(io.u[0] + ol);
            ybn = q.beside(io.u[1] + orr); ybs = q.beside(io.u[1] + ol);
            zbc = q.beside(io.u[2] + oc);
        }
        float lapmu[4], lapT[4], div[4];
        {
            const Row a = q.around(mso, mbs), b = q.around(mc, mbc), c = q.around(mn, mbn);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const Plane19<float> w = part19(a, b, c, i);
                lapmu[i] = (ml[i] + w.s) * (1.f / 6.f);
                ml[i] = w.l + ms[i];
                ms[i] = w.s;
            }
        }
        {
            const Row a = q.around(tso, tbs), b = q.around(tc, tbc), c = q.around(tn, tbn);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                Plane19<float> w = part19(a, b, c, i);
                if (ghost && halfway) w.s = 12.f * p.T_w - w.s;
                lapT[i] = (tl[i] + w.s) * (1.f / 6.f);
                tl[i] = w.l + ts[i];
                ts[i] = w.s;
            }
        }
        if constexpr (HYD) {
            const Row xa = q.around(mul4(pso, xso), __fmul_rn(pbs, xbs));
            const Row xb = q.around(mul4(pc, xc), __fmul_rn(pbc, xbc));
            const Row xd = q.around(mul4(pn, xn), __fmul_rn(pbn, xbn));
            const Row ya = q.around(mul4(pso, yso), __fmul_rn(pbs, ybs));
            const Row yd = q.around(mul4(pn, yn), __fmul_rn(pbn, ybn));
            const Row zb_ = q.around(mul4(pc, zcn), __fmul_rn(pbc, zbc));
            const Q4 za_ = mul4(pso, zso), zd_ = mul4(pn, zn);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float ax = xb.e[i + 2] - xb.e[i];
                const float gx = 2.f * ax + (xd.e[i + 2] - xd.e[i]) + (xa.e[i + 2] - xa.e[i]);
                const float ay = yd.e[i + 1] - ya.e[i + 1];
                const float gy = 2.f * ay + (yd.e[i + 2] - ya.e[i + 2]) + (yd.e[i] - ya.e[i]);
                float s = 2.f * zb_.e[i + 1] + ((zb_.e[i + 2] + zb_.e[i]) + (zd_.v[i] + za_.v[i]));
                if (ghost) s = -s;
                const float w = 1.f / 12.f;
                div[i] = fmaf(s - gs0[i], w, fmaf(gxo[i] + ax, w, __fmul_rn(gyo[i] + ay, w)));
                gxo[i] = gx + gxa[i];
                gyo[i] = gy + gya[i];
                gxa[i] = ax;
                gya[i] = ay;
                gs0[i] = gs1[i];
                gs1[i] = s;
            }
        }
        if (k > za) {                            // plane k - 1 is complete
            const int z = k - 1;
            const bool held = walls && g.t_mode == LF_TWALL_LAYERS && (z == 0 || z == nz - 1);
            Q4 phn, Tn;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                phn.v[i] = (HYD ? ph1.v[i] - div[i] : ph1.v[i]) + p.Gamma * lapmu[i];
                float v = T1.v[i];
                if (p.t_update) v = held ? p.T_w : v + p.dxi * lapT[i];
                Tn.v[i] = v;
                bad |= q.act && i < q.nv && (!isfinite(phn.v[i]) || !isfinite(v));
            }
            if (q.act) {
                q.store(io.phi_out + z * zs + row, phn);
                q.store(io.T_out + z * zs + row, Tn);
            }
        }
        T1 = tc;
        ph1 = pc;
    }
    chain_next();
    if (bad) *reinterpret_cast<volatile int*>(io.flag) = 1;
}

// One plane of T around a thread's four sites: the sites, the sums of their
// four in-plane neighbours and (isotropic) of their four diagonal ones, in the
// order of k_tsub3d / k_tsub3d_iso.
struct TPlane {
    Q4 c, cross, diag;
};

// A temperature sub-step (k_tsub3d, k_tsub3d_iso) with four sites per thread
// marching along z, so that each plane's in-plane sums are formed once for the
// three planes that use them and loads are 16 bytes.  Bound by memory on large
// lattices (384^3: 453 MB, 67 us) and by the launch on small ones.  One site per
// thread took 19 (7) loads of 4 bytes per site: isotropic 384^3 335 -> 95 us,
// 250 x 243 x 190 72.7 -> 23.7, 32 x 32 x 256 3.25 -> 2.4; compact 384^3 229 -> 77.
// Every site goes through the scalar kernels' operations in their order (the
// same bits); a plane beyond a wall is 2 T_w minus the wall plane.
template <int LX, bool ISO>
__global__ void __launch_bounds__(128) k_tsub3d_q(Geom g, Phys<float> p, const float* Tin, float* Tout, int zc)
{
    const Quad<LX> q(g);
    const int za = blockIdx.z * zc, zb = min(za + zc, g.nz);
    const int nz = g.nz, pitch = g.pitch, walls = g.walls;
    const int zs = g.ny * pitch;                 // 32-bit offsets: Q * padded sites < 2^31 (checked at creation)
    const int row = q.y * pitch;
    const int rl = (q.y == 0 ? g.ny - 1 : q.y - 1) * pitch, rr = (q.y + 1 == g.ny ? 0 : q.y + 1) * pitch;
    const float tw2 = 2.f * p.T_w;
    chain_wait();
    // plane z; with `image`, also what the plane beyond a wall at z is to it
    auto plane = [&](int z, TPlane* image) {
        const float* f = Tin + z * zs;
        TPlane t;
        t.c = q.load(f + row);
        const Q4 l4 = q.load(f + rl), r4 = q.load(f + rr);
        const Row c = q.around(t.c, q.beside(f + row));
        Row l{}, r{};
        if constexpr (ISO) {
            l = q.around(l4, q.beside(f + rl));
            r = q.around(r4, q.beside(f + rr));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            t.cross.v[i] = c.e[i] + c.e[i + 2] + l4.v[i] + r4.v[i];
            t.diag.v[i] = ISO ? l.e[i] + l.e[i + 2] + r.e[i] + r.e[i + 2] : 0.f;
        }
        if (image) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                image->c.v[i] = tw2 - t.c.v[i];
                image->cross.v[i] = ISO ? (tw2 - c.e[i]) + (tw2 - c.e[i + 2]) + (tw2 - l4.v[i]) + (tw2 - r4.v[i]) : 0.f;
                image->diag.v[i] = 0.f;          // never used beyond a wall
            }
        }
        return t;
    };
    TPlane dn{}, mid, up{}, beyond{};
    const bool lo = walls && za == 0;
    if (!lo) dn = plane(za == 0 ? nz - 1 : za - 1, nullptr);
    mid = plane(za, lo ? &dn : nullptr);
    if (walls && za == nz - 1) plane(za, &beyond);   // the segment starts at the last plane
    for (int z = za; z < zb; ++z) {
        const bool hi = walls && z == nz - 1;
        if (hi) {
            up = beyond;
        } else {
            const int zu = z + 1 == nz ? 0 : z + 1;
            if (z + 2 < nz) asm volatile("prefetch.global.L2 [%0];" ::"l"(Tin + (z + 2) * zs + row + q.x));
            up = plane(zu, walls && zu == nz - 1 ? &beyond : nullptr);
        }
        const bool held = walls && g.t_mode == LF_TWALL_LAYERS && (z == 0 || z == nz - 1);
        Q4 o;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float t0 = mid.c.v[i];
            float lap;
            if constexpr (ISO) {
                const float nn = mid.cross.v[i] + dn.c.v[i] + up.c.v[i];
                const float ed = mid.diag.v[i] + dn.cross.v[i] + up.cross.v[i];
                lap = fmaf(-24.f, t0, fmaf(2.f, nn, ed)) * (1.f / 6.f);
            } else {
                lap = fmaf(-6.f, t0, mid.cross.v[i] + up.c.v[i] + dn.c.v[i]);
            }
            o.v[i] = held ? p.T_w : fmaf(p.dxi, lap, t0);
        }
        if (q.act) q.store(Tout + z * zs + row, o);
        dn = mid;
        mid = up;
    }
    chain_next();
}

// Lanes per row for a row of nq quads: the widest of 32, 16, 8 that leaves the
// fewest lanes past the end of a row.
int quad_lanes(int nq)
{
    int lx = 32;
    for (int c = 16; c >= 8; c /= 2)
        if ((nq + c - 1) / c * c < (nq + lx - 1) / lx * lx) lx = c;
    return lx;
}

// `nt` threads take nt / LX rows over `zc` planes.  The blocks of all rows are on
// x: y takes 65,535, which a long lattice exceeds.
template <int LX>
dim3 quad_grid(const Geom& g, int nt, int zc)
{
    const int ry = nt / LX;
    return dim3((unsigned)(((g.nx + 3) / 4 + LX - 1) / LX) * ((g.ny + ry - 1) / ry), 1, (g.nz + zc - 1) / zc);
}

template <int LX>
cudaError_t launch_tsub_q(const Geom& g, const Phys<float>& p, const float* Tin, float* Tout, int zc, cudaStream_t s)
{
    constexpr int NT = 128;
    const dim3 grid = quad_grid<LX>(g, NT, zc);
    return launch_chained(g.stencil == LF_STENCIL_ISOTROPIC ? k_tsub3d_q<LX, true> : k_tsub3d_q<LX, false>, grid, NT, 0, s, g,
                          p, Tin, Tout, zc);
}

template <int LX>
cudaError_t launch_q(const Geom& g, const Phys<float>& p, const StepIO<float>& io, int zc, cudaStream_t s)
{
    constexpr int NT = 128;
    const dim3 grid = quad_grid<LX>(g, NT, zc);
    if (g.stencil == LF_STENCIL_ISOTROPIC)
        return launch_chained(p.hydro ? k_phi3d_iso_q<LX, true> : k_phi3d_iso_q<LX, false>, grid, NT, 0, s, g, p, io, zc);
    return launch_chained(p.hydro ? k_phi3d_q<LX, true> : k_phi3d_q<LX, false>, grid, NT, 0, s, g, p, io, zc);
}

}  // namespace

cudaError_t launch_phi3d_quads(const Geom& g, const Phys<float>& p, const StepIO<float>& io, int zc, cudaStream_t s)
{
    const int nq = (g.nx + 3) / 4, lx = quad_lanes(nq);
    if (zc <= 0) {
        // Planes per segment: the more the fewer planes are read twice, as long
        // as every SM has its fill of blocks (six compact, three isotropic, of
        // which two suffice).  Between 8 and 64 planes large lattices differ by
        // 3 %; 32 x 32 x 256 takes 8.2 us with 2 planes and 16.4 with 16.
        int sms = 0;
        const cudaError_t e = device_sms(&sms);
        if (e != cudaSuccess) return e;
        const bool iso = g.stencil == LF_STENCIL_ISOTROPIC;
        const int ry = 128 / lx;
        const int64_t cols = (int64_t)((nq + lx - 1) / lx) * ((g.ny + ry - 1) / ry);
        for (int c : {iso ? 28 : 24, 20, 16, 12, 8, 6, 4, 3, 2}) {
            zc = c;
            if (cols * ((g.nz + c - 1) / c) >= (iso ? 2 : 6) * (int64_t)sms) break;
        }
    }
    return lx == 32 ? launch_q<32>(g, p, io, zc, s) : lx == 16 ? launch_q<16>(g, p, io, zc, s) : launch_q<8>(g, p, io, zc, s);
}

cudaError_t launch_tsub3d_quads(const Geom& g, const Phys<float>& p, const float* Tin, float* Tout, cudaStream_t s)
{
    int sms = 0;
    const cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const int nq = (g.nx + 3) / 4, lx = quad_lanes(nq), ry = 128 / lx;
    const int64_t cols = (int64_t)((nq + lx - 1) / lx) * ((g.ny + ry - 1) / ry);
    // Planes per segment: with 8 to 32 large lattices differ by 5 %; small ones
    // take the shortest segments (32 x 32 x 256: 2.4 us with 2 planes, 4.1 with
    // 8), and four blocks per SM hide the loads' latency (128^3 isotropic: 6.0 us
    // with 6 planes, 7.2 with 2, 7.4 with 12).
    int zc = 2;
    for (int c : {12, 8, 6, 4, 3, 2}) {
        zc = c;
        if (cols * ((g.nz + c - 1) / c) >= 4 * (int64_t)sms) break;
    }
    return lx == 32   ? launch_tsub_q<32>(g, p, Tin, Tout, zc, s)
           : lx == 16 ? launch_tsub_q<16>(g, p, Tin, Tout, zc, s)
                      : launch_tsub_q<8>(g, p, Tin, Tout, zc, s);
}

}  // namespace lf
