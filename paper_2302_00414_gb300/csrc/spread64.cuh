// Two-dimensional float64 spreading (window modes, Algorithm 2.4 step 1 and its form in Algorithm 3.7).
#pragma once

#include <cstdint>

#include "spread.cuh"

namespace infft {

// ---------------------------------------------------------------------------------------
// One warp per work item, the item's padded tile (P x P, P = T + 2m <= 32) in shared memory.
// GB300's float64 rate binds this kernel: a warp's multiply-add takes 18 cycles of its SM, so what
// counts is how many of its 32 lanes do a tap that is not zero.  Off the grid nodes a point has
// 2m taps along each axis (tap 0 only counts on a node); a lane owns one of their columns and the real
// or the imaginary part, and walks down the rows: 2m x 2 x 2m products on 4m lanes, 32 of 32 lanes for
// m = 8 (16 multiply-adds per point; a lane per padded column took 34), in two or more groups of rows
// for small m.  The cells are read, updated and written in shared memory, which costs 85 wavefronts
// per point against 295 cycles of multiply-adds.  Points are taken one after the other, so every
// cell is summed in the item's point order; no atomics.
// The window is evaluated once per point, from the plan's polynomial, while staging 32 points (one lane
// each); the next chunk's points are loaded meanwhile.
template <int MM>
struct Spread64 {
    static constexpr int W = 2 * MM + 1, NT = 2 * MM;      // taps, taps off the nodes
    static constexpr int LN = 2 * NT;                      // lanes of a group of rows
    static constexpr int G = 32 / LN;                      // groups
    static constexpr int RPL = (NT + G - 1) / G;           // rows per lane
    static constexpr int OFF_Y = 0;                        // [32][W] psi_y
    static constexpr int OFF_X = OFF_Y + 32 * W * 8;       // [32][W] psi_x
    static constexpr int OFF_C = OFF_X + 32 * W * 8;       // [32] c_j
    static constexpr int OFF_M = OFF_C + 32 * 16;          // [32] first cell, and whether tap 0 counts along y, x
    static constexpr int OFF_POLY = OFF_M + 32 * 8;
    static constexpr int OFF_PAD = OFF_POLY + WPOLY64_ROWS * wpoly_stride(MM) * 8;
    static constexpr size_t bytes(int P) { return OFF_PAD + (size_t)P * P * 16; }
};

template <int MM>
__device__ __forceinline__ void spread2d_f64_item(const JobSet<double>& js, const int gitem, unsigned char* base) {
    using C = Spread64<MM>;
    constexpr int W = C::W, NT = C::NT;
    const int lane = threadIdx.x & 31;
    const int jb = find_job(js.pre_items, js.njobs, gitem);
    const Job<double>& J = js.job[jb];
    const int it = gitem - js.pre_items[jb];
    const int4 item = J.items[it];
    const int P = J.P, Ms = J.Ms, T = J.T;
    const int ty = item.x / J.ntile, tx = item.x % J.ntile;
    const int logMs = 31 - __clz(Ms);
    const bool dcf = J.mode == INFFT_MODE_DCF;
    const bool use_poly = J.window == WK_KB;
    double* sy = reinterpret_cast<double*>(base + C::OFF_Y);
    double* sx = reinterpret_cast<double*>(base + C::OFF_X);
    double2* sc = reinterpret_cast<double2*>(base + C::OFF_C);
    int2* sm = reinterpret_cast<int2*>(base + C::OFF_M);
    double* poly = reinterpret_cast<double*>(base + C::OFF_POLY);
    double* pad = reinterpret_cast<double*>(base + C::OFF_PAD);   // (re, im) of cell (row, col) at 2 (row P + col)
    if (use_poly)
        for (int e = lane; e < WPOLY64_ROWS * wpoly_stride(MM); e += 32) poly[e] = J.wpoly[e];
    for (int e = lane; e < P * P; e += 32) reinterpret_cast<double2*>(pad)[e] = make_double2(0.0, 0.0);

    const int grp = lane / C::LN, idx = lane % C::LN;
    const int col = 1 + (idx >> 1), part = idx & 1, row0 = 1 + grp * C::RPL;
    const int nrow = grp < C::G ? min(C::RPL, NT + 1 - row0) : 0;   // rows of this lane (may be <= 0)
    double* mine = pad + 2 * (row0 * P + col) + part;

    int perm = 0;
    uint32_t cl = 0;
    double2 u = make_double2(0.5, 0.5), f = make_double2(0.0, 0.0), w = make_double2(1.0, 0.0);
    auto load_point = [&](int c) {
        if (c + lane < item.z) {
            const size_t i = (size_t)item.y + c + lane;
            perm = __ldg(J.perm + i);
            cl = __ldg(J.cell + i);
            u = __ldg(reinterpret_cast<const double2*>(J.u) + i);
            if (dcf) w = __ldg(reinterpret_cast<const double2*>(J.w) + i);
        }
    };
    auto load_sample = [&](int c) {
        if (c + lane < item.z) f = __ldg(reinterpret_cast<const double2*>(J.in) + perm);
    };
    load_point(0);
    load_sample(0);
    for (int c0 = 0; c0 < item.z; c0 += 32) {
        const int np = min(32, item.z - c0);
        __syncwarp();   // the chunk before is read
        if (lane < np) {
            const int oy = (int)(cl >> logMs) - ty * T, ox = (int)(cl & (uint32_t)(Ms - 1)) - tx * T;
            sm[lane] = make_int2(oy * P + ox, (u.x == 0.0 ? 1 : 0) | (u.y == 0.0 ? 2 : 0));
            sc[lane] = dcf ? make_double2(w.x * f.x - w.y * f.y, w.x * f.y + w.y * f.x) : f;
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                double wt[1][W];
                const double v = a == 0 ? u.x : u.y;
                if (use_poly) poly_taps<MM, 1>(poly, &v, wt);
                else bspline_taps<MM>(v, wt[0]);
                double* dst = (a == 0 ? sy : sx) + lane * W;
#pragma unroll
                for (int s = 0; s < W; ++s) dst[s] = wt[0][s];
            }
        }
        load_point(c0 + 32);
        __syncwarp();
        for (int p = 0; p < np; ++p) {
            const int2 o = sm[p];
            const double c = reinterpret_cast<const double*>(sc + p)[part];
            const double* py = sy + p * W;
            const double* px = sx + p * W;
            if (nrow > 0) {
                const double q = c * px[col];
                double* cell = mine + 2 * o.x;
                double v[C::RPL];
#pragma unroll
                for (int r = 0; r < C::RPL; ++r) v[r] = r < nrow ? cell[2 * r * P] : 0.0;
#pragma unroll
                for (int r = 0; r < C::RPL; ++r)
                    if (r < nrow) cell[2 * r * P] = fma(q, py[row0 + r], v[r]);
            }
            if (o.y) {   // on a node along an axis: the row and the column of tap 0
                __syncwarp();
                if (o.y & 1)
                    for (int e = lane; e < 2 * W; e += 32) {
                        double* cell = pad + 2 * (o.x + (e >> 1)) + (e & 1);
                        *cell = fma(reinterpret_cast<const double*>(sc + p)[e & 1] * px[e >> 1], py[0], *cell);
                    }
                if (o.y & 2)
                    for (int e = lane; e < 2 * NT; e += 32) {
                        double* cell = pad + 2 * (o.x + (1 + (e >> 1)) * P) + (e & 1);
                        *cell = fma(reinterpret_cast<const double*>(sc + p)[e & 1] * px[0], py[1 + (e >> 1)], *cell);
                    }
            }
            if (p == 0) load_sample(c0 + 32);   // its index, loaded before the chunk, has arrived
            __syncwarp();
        }
    }
    __syncwarp();
    double2* dst = reinterpret_cast<double2*>(J.padded) + (size_t)it * P * P;
    for (int e = lane; e < P * P; e += 32) dst[e] = reinterpret_cast<const double2*>(pad)[e];
}

}  // namespace infft
