// Two-dimensional spreading kernel (register rows) and its launcher, instantiated for
// float32 and float64 in their own translation units (compiled in parallel).
#pragma once

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "spread.cuh"
#include "spread64.cuh"
#include "spreadmma.cuh"

namespace infft {

// Window modes: float32 takes the tensor-core form of spreadmma.cuh, float64 the form of spread64.cuh.

// ---------------------------------------------------------------------------------------
// Two-dimensional spreading with B_opt, the accumulators in registers.  One warp per work
// item; lane l owns column l of the item's P x P padded tile (P = T + 2m + 1 <= 32).
// The item's points are sorted by base row, so the rows a point can touch,
// [oy, oy + 2m + 1] (padded coordinates), only move down: each lane keeps those rows of its
// column in registers, adds the point's coefficients of its column (conjugated) times the sample,
// and when the next point starts lower it stores the rows that no later point can reach.  Every padded
// cell is stored exactly once, no shared-memory read-modify-write, no atomics.
// One warp spreads work item gitem (global over the JobSet's jobs); `base` is the warp's
// shared memory.
template <class R, int MM>
__device__ __forceinline__ void spread2d_bopt_item(const JobSet<R>& js, const int gitem, unsigned char* base) {
    constexpr int S = 2 * MM + 2;              // slots per axis, and rows held in registers
    constexpr bool F32 = sizeof(R) == 4;
    const int lane = threadIdx.x & 31;
    const int jb = find_job(js.pre_items, js.njobs, gitem);
    const Job<R>& J = js.job[jb];
    const int it = gitem - js.pre_items[jb];
    const int4 item = J.items[it];
    const int P = J.P, Ms = J.Ms, T = J.T;
    cx<R>* cst = reinterpret_cast<cx<R>*>(base);            // [32]     c_j
    int* meta = reinterpret_cast<int*>(cst + 32);           // [32][3]  oy, ox, sorted index
    const int ty = item.x / J.ntile, tx = item.x % J.ntile;
    using V2 = typename std::conditional<F32, float2, double2>::type;
    // (re, im) of the rows r0 .. r0 + S - 1 of this lane's column
    V2 acc[S];
#pragma unroll
    for (int k = 0; k < S; ++k) { acc[k].x = R(0); acc[k].y = R(0); }
    int r0 = 0;  // padded row held in acc[0]
    cx<R>* dst = J.padded + (size_t)it * P * P;
    const bool col_ok = lane < P;
    // store row r0 (no later point reaches it) and move the held rows up by one
    auto flush_row = [&]() {
        if (col_ok) dst[(size_t)r0 * P + lane] = mk<R>(acc[0].x, acc[0].y);
#pragma unroll
        for (int k = 0; k < S - 1; ++k) acc[k] = acc[k + 1];
        acc[S - 1].x = R(0);
        acc[S - 1].y = R(0);
        ++r0;
    };
    const int logMs = 31 - __clz(Ms);
    for (int c0 = 0; c0 < item.z; c0 += 32) {
        const int np = min(32, item.z - c0);
        __syncwarp();
        if (lane < np) {
            const int i = item.y + c0 + lane;
            const uint32_t cl = __ldg(J.cell + i);
            meta[lane * 3 + 0] = (int)(cl >> logMs) - ty * T;
            meta[lane * 3 + 1] = (int)(cl & (uint32_t)(Ms - 1)) - tx * T;
            meta[lane * 3 + 2] = i;
            cst[lane] = J.in[__ldg(J.perm + i)];
        }
        __syncwarp();
        // The points are sorted by base row, so the chunk splits into runs of equal oy
        // (found by one ballot): the rows above a run are stored once per run, and the
        // points of a run only add their taps.
        const int my_oy = lane < np ? meta[lane * 3 + 0] : 0x7fffffff;
        int p = 0;
        while (p < np) {
            const int oy = __shfl_sync(0xffffffffu, my_oy, p);
            // store the rows above oy: no later point reaches them
            while (r0 < oy) flush_row();
            const int q = 32 - __clz(__ballot_sync(0xffffffffu, my_oy == oy));
            // float32: four points per unrolled step let the loads of the next points overlap the
            // current FMAs; float64 keeps its registers for the accumulators
            constexpr int UNR = F32 ? 4 : 1;
#pragma unroll UNR
            for (; p < q; ++p) {
                // every lane loads (a column of the point's S x S block, clamped), and the
                // lanes outside the block add zero: with no branch around the loads the
                // unrolled points' coefficient loads are in flight together
                const int sx = lane - meta[p * 3 + 1];
                const bool act = sx >= 0 && sx < S;
                const int sxc = min(max(sx, 0), S - 1);
                const int i = meta[p * 3 + 2];
                const cx<R> cv = act ? cst[p] : mk<R>(0, 0);
                const cx<R>* cf = J.coef + (size_t)i * S * S + sxc;
#pragma unroll
                for (int k = 0; k < S; ++k) {
                    const V2 b = __ldg(reinterpret_cast<const V2*>(cf + k * S));
                    acc[k].x += b.x * cv.re + b.y * cv.im;   // conj(b) f
                    acc[k].y += b.x * cv.im - b.y * cv.re;
                }
            }
        }
    }
    // remaining rows (including rows no point reached)
    while (r0 < P) flush_row();
}

// warps per block: two of the tensor-core form, one of the float64 window form (its shared memory bounds the
// warps per SM), four with B_opt
template <class R, bool BOPT>
constexpr int spread2d_wpb() { return BOPT ? 4 : sizeof(R) == 4 ? 2 : 1; }
template <class R, int MM, bool BOPT>
constexpr int spread2d_blocks() { return BOPT ? 1 : sizeof(R) == 4 ? (MM <= 4 ? 10 : 6) : 1; }

template <class R, int MM, bool BOPT>
__global__ void __launch_bounds__(32 * spread2d_wpb<R, BOPT>(), spread2d_blocks<R, MM, BOPT>())
    k_spread2d(const __grid_constant__ JobSet<R> js) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5;
    const int gitem = blockIdx.x * js.wpb + warp;
    if (gitem >= js.pre_items[js.njobs]) return;
    unsigned char* base = smem_raw + (size_t)warp * js.smem_per_warp;
    if constexpr (BOPT) spread2d_bopt_item<R, MM>(js, gitem, base);
    else if constexpr (sizeof(R) == 4) spread2d_mma_item<MM>(js, gitem, base);
    else spread2d_f64_item<MM>(js, gitem, base);
}

// Per-launch setup: shared memory per warp (js.smem_per_warp), warps per block (js.wpb), and for
// the tensor-core form the jobs' common window polynomial in the parameter block.
template <class R, int MM, bool BOPT>
static void spread2d_setup(JobSet<R>& js) {
    js.wpb = spread2d_wpb<R, BOPT>();
    js.wtab_ok = 0;
    if constexpr (BOPT) {
        js.smem_per_warp = 32 * (int)sizeof(cx<R>) + 96 * (int)sizeof(int);
    } else if constexpr (sizeof(R) == 4) {
        const size_t n = (size_t)WPOLY_ROWS * wpoly_stride(MM);
        bool same = js.job[0].wpoly_h != nullptr;
        for (int j = 1; j < js.njobs && same; ++j)
            same = js.job[j].wpoly_h && memcmp(js.job[j].wpoly_h, js.job[0].wpoly_h, n * sizeof(float)) == 0;
        if (same) {
            for (size_t k = 0; k < n; ++k) js.wtab[k] = js.job[0].wpoly_h[k] * spread_mma_wscale(js.job[0].wexp);
            js.wtab_ok = 1;
        }
        js.smem_per_warp = (SpreadMma<MM>::BYTES + 15) & ~15;
    } else {
        int P = 0;
        for (int j = 0; j < js.njobs; ++j) P = std::max(P, js.job[j].P);
        js.smem_per_warp = (int)((Spread64<MM>::bytes(P) + 15) & ~(size_t)15);
    }
}

// spreading for d = 2 when every job has the same m (2..8) and P <= 32
template <class R, int MM, bool BOPT>
static infft_status launch_spread2d_m(JobSet<R>& js, cudaStream_t st) {
    spread2d_setup<R, MM, BOPT>(js);
    const size_t spw = (size_t)js.smem_per_warp;
    const int nitems = js.pre_items[js.njobs];
    if (nitems == 0) return INFFT_OK;
    const size_t smem = spw * js.wpb;
    INFFT_CUDA(cudaFuncSetAttribute(k_spread2d<R, MM, BOPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (!BOPT)   // shared memory bounds the warps per SM: ask for all of it
        INFFT_CUDA(cudaFuncSetAttribute(k_spread2d<R, MM, BOPT>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        (int)cudaSharedmemCarveoutMaxShared));
    k_spread2d<R, MM, BOPT><<<(nitems + js.wpb - 1) / js.wpb, 32 * js.wpb, smem, st>>>(js);
    INFFT_LAUNCHED();
    return INFFT_OK;
}

template <class R, bool BOPT>
static infft_status launch_spread2d(JobSet<R>& js, cudaStream_t st, int m) {
    switch (m) {
        case 2: return launch_spread2d_m<R, 2, BOPT>(js, st);
        case 3: return launch_spread2d_m<R, 3, BOPT>(js, st);
        case 4: return launch_spread2d_m<R, 4, BOPT>(js, st);
        case 5: return launch_spread2d_m<R, 5, BOPT>(js, st);
        case 6: return launch_spread2d_m<R, 6, BOPT>(js, st);
        case 7: return launch_spread2d_m<R, 7, BOPT>(js, st);
        default: return launch_spread2d_m<R, 8, BOPT>(js, st);
    }
}

template <class R>
static bool spread2d_eligible(const JobSet<R>& js, int* m_out, bool* bopt_out) {
    if (js.njobs < 1) return false;
    const int m = js.job[0].m;
    const bool bopt = js.job[0].mode == INFFT_MODE_BOPT;
    for (int j = 0; j < js.njobs; ++j) {
        const Job<R>& J = js.job[j];
        if (J.d != 2 || J.m != m || (J.mode == INFFT_MODE_BOPT) != bopt || J.P > 32) return false;
        // the two-source halo merge that follows needs P <= 2T, i.e. 2m <= T (2m + 1 <= T with
        // B_opt's extra slot): a tuned tile of 8 at m >= 5 (m >= 4 with B_opt) puts some cells
        // in three tiles along an axis, which the generic path handles
        if (J.P > 2 * J.T) return false;
        if (sizeof(R) == 4 && !bopt && (J.P & 1)) return false;   // 16-byte stores of column pairs
    }
    if (m < 2 || m > 8) return false;   // m = 8 with window taps only: P = 16 + 16 <= 32
    *m_out = m;
    *bopt_out = bopt;
    return true;
}

template <class R>
infft_status spread2d_try(JobSet<R>& js, cudaStream_t st, bool* used) {
    int m = 0;
    bool bopt = false;
    *used = false;
    if (!spread2d_eligible(js, &m, &bopt)) return INFFT_OK;
    *used = true;
    return bopt ? launch_spread2d<R, true>(js, st, m) : launch_spread2d<R, false>(js, st, m);
}

}  // namespace infft
