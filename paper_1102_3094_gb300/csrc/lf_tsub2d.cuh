// lf_tsub2d.cuh -- several explicit temperature sub-steps of a 2D FP32 lattice
// in one pass over it (Sec. 2: d_t T = xi lap T in n_sub steps of xi / n_sub,
// the first of which is part of the step kernel).
//
// A sub-step moves 8 B and costs about ten operations per site, so one launch
// each is all launch and memory time: 23 us at 2999 x 1777, where the 43 MB
// take 6.3 us.  Here a warp owns a strip of 30 quads (120 columns; two more
// quads as halo) and marches up a segment of rows with S sub-steps in flight:
// when row k arrives, stage s forms row k - s from the rows k - s - 1 .. k - s +
// 1 of stage s - 1.  Rows stay in registers, x-neighbours come by shuffle;
// no shared memory, no barriers.  A quad's halo of 4 columns allows S <= 4.
// Each site goes through the operations of tsub2d_site / tsub2d_site_iso in
// their order, so the bits do not depend on how the sub-steps are grouped.
#pragma once

#include "lf_march2d.cuh"

namespace lf {
namespace tsub {

constexpr int kMaxFused = 4;
constexpr int kQuads = 30;       // quads a warp writes per row

// Four neighbouring sites of a row with the one on either side.
struct Row6 {
    float e[6];
};

template <int S, bool ISO>
__device__ __forceinline__ void tsub2d_rows(const Geom& g, const Phys<float>& p, const float* Tin, float* Tout, int strip,
                                            int y0, int y1)
{
    const int lane = threadIdx.x & 31;
    const int nx = g.nx, ny = g.ny, pitch = g.pitch, walls = g.walls;
    const int c0 = 4 * (strip * kQuads - 1 + lane);              // unwrapped first column
    const bool out = lane >= 1 && lane <= kQuads && c0 < nx;
    const int nv = nx - c0 < 4 ? nx - c0 : 4;                    // of an output lane
    int col[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) col[i] = march::wrap_near(c0 + i, nx);
    const bool vec = (col[0] & 3) == 0 && col[3] == col[0] + 3;
    const bool layers = walls && g.t_mode == LF_TWALL_LAYERS;
    const float two_w = 2.f * p.T_w;

    auto load = [&](int r, float v[4]) {
        if (walls) r = r < 0 ? 0 : (r >= ny ? ny - 1 : r);       // rows beyond a wall are never used
        else r = march::wrap_near(r, ny);
        const float* row = Tin + r * pitch;
        if (vec) {
            const float4 w = *reinterpret_cast<const float4*>(row + col[0]);
            v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = row[col[i]];
        }
    };
    auto sides = [&](const float v[4]) {
        Row6 r;
        r.e[0] = __shfl_up_sync(0xffffffffu, v[3], 1);
        r.e[5] = __shfl_down_sync(0xffffffffu, v[0], 1);
#pragma unroll
        for (int i = 0; i < 4; ++i) r.e[i + 1] = v[i];
        return r;
    };

    Row6 older[S], newer[S];                                     // rows k - s - 2, k - s - 1 of stage s
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int i = 0; i < 6; ++i) older[s].e[i] = newer[s].e[i] = 0.f;
    constexpr int kAhead = 4;                                    // rows in flight; the loop is unrolled by as many,
                                                                 // so that no load is waited for to be moved
    float buf[kAhead][4];
    const int kbeg = y0 - S, kend = y1 - 1 + S;
#pragma unroll
    for (int a = 0; a < kAhead; ++a) load(kbeg + a, buf[a]);
    auto iter = [&](int k, float (&now)[4]) {
        Row6 cur = sides(now);                                   // row k of stage 0
        if (k + kAhead <= kend) load(k + kAhead, now);
#pragma unroll
        for (int s = 1; s <= S; ++s) {
            const int r = k - s;
            const Row6& mid = newer[s - 1];                      // row r
            const Row6& dn = older[s - 1];                       // row r - 1; cur is row r + 1
            const bool lo = walls && r == 0, hi = walls && r == ny - 1;
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float t0 = mid.e[i + 1];
                float lap;
                if constexpr (ISO) {
                    const float d0 = lo ? two_w - t0 : dn.e[i + 1], u0 = hi ? two_w - t0 : cur.e[i + 1];
                    const float dl = lo ? two_w - mid.e[i] : dn.e[i], dr = lo ? two_w - mid.e[i + 2] : dn.e[i + 2];
                    const float ul = hi ? two_w - mid.e[i] : cur.e[i], ur = hi ? two_w - mid.e[i + 2] : cur.e[i + 2];
                    const float nn = mid.e[i] + mid.e[i + 2] + u0 + d0;
                    lap = fmaf(-20.f, t0, fmaf(4.f, nn, ul + ur + dl + dr)) * (1.f / 6.f);
                } else {
                    const float d0 = lo ? two_w - t0 : dn.e[i + 1], u0 = hi ? two_w - t0 : cur.e[i + 1];
                    lap = fmaf(-4.f, t0, mid.e[i] + mid.e[i + 2] + u0 + d0);
                }
                v[i] = (lo || hi) && layers ? p.T_w : fmaf(p.dxi, lap, t0);
            }
            older[s - 1] = newer[s - 1];
            newer[s - 1] = cur;
            if (s < S) {
                cur = sides(v);
            } else if (out && r >= y0 && r < y1) {
                float* row = Tout + r * pitch + c0;
                if (nv == 4) {
                    *reinterpret_cast<float4*>(row) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        if (i < nv) row[i] = v[i];
                }
            }
        }
    };
#pragma unroll 1
    for (int k = kbeg; k <= kend; k += kAhead) {
        // rows past kend only repeat work on old values: nothing of theirs is stored
#pragma unroll
        for (int a = 0; a < kAhead; ++a) iter(k + a, buf[a]);
    }
}

// Sub-steps of the next pass when `left` remain: as even as passes of at most
// kMaxFused allow.
inline int fused(int left)
{
    const int passes = (left + kMaxFused - 1) / kMaxFused;
    return (left + passes - 1) / passes;
}

}  // namespace tsub
}  // namespace lf
