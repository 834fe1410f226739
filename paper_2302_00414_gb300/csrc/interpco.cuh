// Float32 interpolation for d = 3 (Algorithm 2.1 step 3) with the lanes of a warp on one point's cells.
#pragma once

#include <algorithm>

#include "spread.cuh"

namespace infft {

// ---------------------------------------------------------------------------------------
// A block of four warps shares a work item's padded tile of the grid in shared memory and takes a quarter of
// its points each.  Reading the tile binds this kernel: with a lane per point (k_interp_t) the 32 points' cells
// fall into random banks (a 64-bit load took about 7 wavefronts), and one 40 KB tile per warp left 5 warps per SM.
// Here the lanes take the (y, x) cells of one point, rows of W = 2m + 1 neighbours, and a row is rotated by
// W y mod 16 where it fits 16 cells, so that the rows' banks follow one another: 2 wavefronts a load.  Each lane
// adds its cell of the W planes times psi_z first, then times its psi_y psi_x; the sums over the lanes of four
// points at a time share one exchange (11 shuffles).  Every sum has a fixed order.  (In two dimensions, 3
// cells a lane and point, the shuffles and taps outweigh the conflicts: 43 us against 33 for forward 2-D.)
constexpr int INTERP_CO_WARPS = 4;

template <int MM>
struct InterpCo {
    static constexpr int D = 3, W = 2 * MM + 1;
    static constexpr int NR = (W * W + 31) / 32;                       // (y, x) cells per lane
    static constexpr int TAPS = (D * W + 3) / 4 * 4 + 1;               // staged taps of a point, odd stride
    static constexpr bool ROT = 2 * MM + 8 <= 16;                      // tiles of 8: rows of at most 16
    __host__ __device__ static constexpr int pitch(int P) { return ROT ? 16 : P; }
    // bytes before the tile: per warp taps, first cell and caller's index of 32 points; the window table
    static constexpr int PER_WARP = 32 * TAPS * 4 + 32 * 8;
    static constexpr int OFF_POLY = INTERP_CO_WARPS * PER_WARP;
    static constexpr int OFF_PAD = (OFF_POLY + WPOLY_ROWS * wpoly_stride(MM) * 4 + 15) & ~15;
    static size_t bytes(int P) { return OFF_PAD + (size_t)P * P * pitch(P) * 8; }
};

template <int MM>
__global__ void __launch_bounds__(32 * INTERP_CO_WARPS) k_interp_co(const __grid_constant__ JobSet<float> js) {
    using C = InterpCo<MM>;
    constexpr int D = C::D, W = C::W, NR = C::NR, NW = INTERP_CO_WARPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int jb = find_job(js.pre_items, js.njobs, blockIdx.x);
    const Job<float>& J = js.job[jb];
    const int4 item = J.items[blockIdx.x - js.pre_items[jb]];
    const int P = J.P, m = J.m, Ms = J.Ms, T = J.T, nt = J.ntile, PX = C::pitch(P);
    float* st = reinterpret_cast<float*>(smem_raw + warp * C::PER_WARP);       // [32][TAPS] taps y, x, z
    int2* sm = reinterpret_cast<int2*>(smem_raw + warp * C::PER_WARP + 32 * C::TAPS * 4);
    float* poly = reinterpret_cast<float*>(smem_raw + C::OFF_POLY);
    float2* pad = reinterpret_cast<float2*>(smem_raw + C::OFF_PAD);
    const bool use_poly = J.window == WK_KB;
    if (use_poly)
        for (int e = threadIdx.x; e < WPOLY_ROWS * wpoly_stride(MM); e += 32 * NW) poly[e] = J.wpoly[e];
    const int tz = item.x / (nt * nt), ty = (item.x / nt) % nt, tx = item.x % nt;
    const int mask = Ms - 1;   // Ms is a power of two
    auto cell = [&](int y, int x) { return C::ROT ? y * PX + ((x + W * y) & 15) : y * PX + x; };
    for (int e = threadIdx.x; e < P * P * P; e += 32 * NW) {
        const int r1 = e / P, ox = e - r1 * P;
        const int oz = r1 / P, oy = r1 - oz * P;
        const int gx = (tx * T - m + ox) & mask, gy = (ty * T - m + oy) & mask;
        const size_t g = ((size_t)((tz * T - m + oz) & mask) * Ms + gy) * Ms + gx;
        pad[oz * P * PX + cell(oy, ox)] = reinterpret_cast<const float2*>(J.grid)[g];
    }
    int qy[NR], qx[NR];
    bool act[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int q = lane + 32 * r;
        act[r] = q < W * W;
        qy[r] = act[r] ? q / W : 0;
        qx[r] = act[r] ? q % W : 0;
    }
    __syncthreads();
    const int logMs = 31 - __clz(Ms);
    const int per = (item.z + NW - 1) / NW, first = min(item.z, warp * per), last = min(item.z, first + per);
    for (int c0 = first; c0 < last; c0 += 32) {
        const int np = min(32, last - c0);
        __syncwarp();   // the chunk before is read
        if (lane < np) {
            const int i = item.y + c0 + lane;
            const uint32_t cl = __ldg(J.cell + i);
            const int ox = (int)(cl & (uint32_t)mask) - tx * T;
            const int oy = (int)((cl >> logMs) & (uint32_t)mask) - ty * T;
            const int oz = (int)(cl >> (2 * logMs)) - tz * T;
            sm[lane] = make_int2(oz << 16 | oy << 8 | ox, __ldg(J.perm + i));
            float u[D], wt[D][W];
#pragma unroll
            for (int a = 0; a < D; ++a) u[a] = J.u[(size_t)i * D + (a + D - 2) % D];   // y, x, z
            if (use_poly) poly_taps<MM, D>(poly, u, wt);
            else {
#pragma unroll
                for (int a = 0; a < D; ++a) bspline_taps<MM>(u[a], wt[a]);
            }
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
                for (int s = 0; s < W; ++s) st[lane * C::TAPS + a * W + s] = wt[a][s];
        }
        __syncwarp();
        constexpr int U = 4;
        for (int p0 = 0; p0 < np; p0 += U) {
            float v[2 * U];   // (re, im) of the points' sums
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int p = min(p0 + k, np - 1);
                const int o = sm[p].x;
                const float* tp = st + p * C::TAPS;
                const int oy = (o >> 8) & 255, ox = o & 255, oz = o >> 16;
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const float2* g = pad + oz * P * PX + cell(oy + qy[r], ox + qx[r]);
                    const float w = act[r] ? tp[qy[r]] * tp[W + qx[r]] : 0.f;
                    float2 s = make_float2(0.f, 0.f);
#pragma unroll
                    for (int z = 0; z < W; ++z) {
                        const float wz = tp[2 * W + z];
                        s = __ffma2_rn(g[z * P * PX], make_float2(wz, wz), s);
                    }
                    acc = __ffma2_rn(s, make_float2(w, w), acc);
                }
                v[2 * k] = acc.x;
                v[2 * k + 1] = acc.y;
            }
            // sums over the lanes: halves exchange and keep one value in two until a lane holds one, then over its four lanes
#pragma unroll
            for (int h = U, s = 16; h >= 1; h >>= 1, s >>= 1) {
#pragma unroll
                for (int i = 0; i < h; ++i) {
                    const bool up = (lane & s) != 0;
                    const float send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
                }
            }
            float sum = v[0];
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            const int k = ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1), part = (lane >> 2) & 1;
            if ((lane & 3) == 0 && p0 + k < np) reinterpret_cast<float*>(J.out + sm[p0 + k].y)[part] = sum;
        }
    }
}

template <int MM>
static infft_status launch_interp_co(JobSet<float>& js, cudaStream_t st) {
    int P = 0;
    for (int j = 0; j < js.njobs; ++j) P = std::max(P, js.job[j].P);
    const size_t smem = InterpCo<MM>::bytes(P);
    const int nitems = js.pre_items[js.njobs];
    if (nitems == 0) return INFFT_OK;
    INFFT_TRY(smem_limit<k_interp_co<MM>>(smem));
    INFFT_CUDA(cudaFuncSetAttribute(k_interp_co<MM>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    (int)cudaSharedmemCarveoutMaxShared));
    k_interp_co<MM><<<nitems, 32 * INTERP_CO_WARPS, smem, st>>>(js);
    INFFT_LAUNCHED();
    return INFFT_OK;
}

// when every job has the same m (1..6), window taps, and tiles of at most 8 (larger, tuned tiles take k_interp_t)
static infft_status interp_co_try(JobSet<float>& js, cudaStream_t st, bool* used) {
    *used = false;
    const int m = js.job[0].m;
    if (m < 1 || m > 6) return INFFT_OK;
    for (int j = 0; j < js.njobs; ++j)
        if (js.job[j].m != m || js.job[j].mode == INFFT_MODE_BOPT || js.job[j].T > 8) return INFFT_OK;
    *used = true;
    switch (m) {
        case 1: return launch_interp_co<1>(js, st);
        case 2: return launch_interp_co<2>(js, st);
        case 3: return launch_interp_co<3>(js, st);
        case 4: return launch_interp_co<4>(js, st);
        case 5: return launch_interp_co<5>(js, st);
        default: return launch_interp_co<6>(js, st);
    }
}

}  // namespace infft
