// Two-dimensional spreading kernel and its launcher, instantiated for float32 and float64 in their own translation
// units (compiled in parallel).
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
// Two-dimensional spreading with B_opt (Algorithm 4.4).  A point's S x S coefficients (S = 2m + 2)
// are one contiguous run of memory, and reading them is what this kernel has to do.  Four warps share a work
// item, each taking a quarter of its points in order; a warp's lanes take the point's coefficients 16 bytes
// each, whole runs at a time (a lane per padded column read ten strided rows of 80 bytes), four
// points' loads in flight before the first is used, and add conj(b) f to the warp's own padded tile in
// shared memory.  The four tiles are summed in warp order, so that the order of every sum is fixed.
constexpr int SPREAD_BOPT_WARPS = 4;

template <class R, int MM>
__device__ __forceinline__ void spread2d_bopt_item(const JobSet<R>& js, const int gitem, unsigned char* smem) {
    using C = BoptLanes<R, MM>;
    constexpr int VEC = C::VEC, NV = C::NV, NR = C::NR, S = C::S, NW = SPREAD_BOPT_WARPS;
    using V = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int jb = find_job(js.pre_items, js.njobs, gitem);
    const Job<R>& J = js.job[jb];
    const int it = gitem - js.pre_items[jb];
    const int4 item = J.items[it];
    const int P = J.P, Ms = J.Ms, T = J.T, cells = P * P;
    const int ty = item.x / J.ntile, tx = item.x % J.ntile;
    const int logMs = 31 - __clz(Ms);
    cx<R>* pad = reinterpret_cast<cx<R>*>(smem) + warp * cells;
    for (int e = lane; e < cells; e += 32) pad[e] = mk<R>(0, 0);
    int off[NR];
    bool act[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int q = VEC * (lane + 32 * r);
        act[r] = lane + 32 * r < NV;
        off[r] = act[r] ? (q / S) * P + q % S : 0;
    }
    __syncwarp();
    const int per = (item.z + NW - 1) / NW, first = min(item.z, warp * per), last = min(item.z, first + per);
    for (int c0 = first; c0 < last; c0 += 32) {
        const int np = min(32, last - c0);
        int o = 0;
        cx<R> f = mk<R>(0, 0);
        if (lane < np) {
            const int i = item.y + c0 + lane;
            const uint32_t cl = __ldg(J.cell + i);
            o = ((int)(cl >> logMs) - ty * T) * P + (int)(cl & (uint32_t)(Ms - 1)) - tx * T;
            f = J.in[__ldg(J.perm + i)];
        }
        const V* cf = reinterpret_cast<const V*>(J.coef + (size_t)(item.y + c0) * S * S);
        constexpr int U = 4;
        for (int p0 = 0; p0 < np; p0 += U) {
            V b[U][NR];
#pragma unroll
            for (int k = 0; k < U; ++k)
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    if (act[r] && p0 + k < np) b[k][r] = __ldg(cf + (size_t)(p0 + k) * NV + lane + 32 * r);
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (p0 + k >= np) break;   // uniform
                const int op = __shfl_sync(0xffffffffu, o, p0 + k);
                const R fr = __shfl_sync(0xffffffffu, f.re, p0 + k), fi = __shfl_sync(0xffffffffu, f.im, p0 + k);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    if (!act[r]) continue;
                    cx<R>* cell = pad + op + off[r];
                    const R* bb = reinterpret_cast<const R*>(&b[k][r]);
#pragma unroll
                    for (int v = 0; v < VEC; ++v) {   // conj(b) f
                        cell[v].re += bb[2 * v] * fr + bb[2 * v + 1] * fi;
                        cell[v].im += bb[2 * v] * fi - bb[2 * v + 1] * fr;
                    }
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    const cx<R>* all = reinterpret_cast<const cx<R>*>(smem);
    cx<R>* dst = J.padded + (size_t)it * cells;
    for (int e = threadIdx.x; e < cells; e += 32 * NW) {
        cx<R> v = all[e];
#pragma unroll
        for (int k = 1; k < NW; ++k) v = add(v, all[k * cells + e]);
        dst[e] = v;
    }
}

// work items and warps per block: two of the tensor-core form, one of the float64 window form (its shared memory
// bounds the warps per SM), one item on four warps with B_opt
template <class R, bool BOPT>
constexpr int spread2d_wpb() { return !BOPT && sizeof(R) == 4 ? 2 : 1; }
template <class R, bool BOPT>
constexpr int spread2d_warps() { return BOPT ? SPREAD_BOPT_WARPS : spread2d_wpb<R, BOPT>(); }
template <class R, int MM, bool BOPT>
constexpr int spread2d_blocks() { return BOPT ? 1 : sizeof(R) == 4 ? (MM <= 4 ? 10 : 6) : 1; }

template <class R, int MM, bool BOPT>
__global__ void __launch_bounds__(32 * spread2d_warps<R, BOPT>(), spread2d_blocks<R, MM, BOPT>())
    k_spread2d(const __grid_constant__ JobSet<R> js) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (BOPT) {
        spread2d_bopt_item<R, MM>(js, blockIdx.x, smem_raw);
    } else {
        const int warp = threadIdx.x >> 5;
        const int gitem = blockIdx.x * js.wpb + warp;
        if (gitem >= js.pre_items[js.njobs]) return;
        unsigned char* base = smem_raw + (size_t)warp * js.smem_per_warp;
        if constexpr (sizeof(R) == 4) spread2d_mma_item<MM>(js, gitem, base);
        else spread2d_f64_item<MM>(js, gitem, base);
    }
}

// Per-launch setup: shared memory per item (js.smem_per_warp), items per block (js.wpb), and for
// the tensor-core form the jobs' common window polynomial in the parameter block.
template <class R, int MM, bool BOPT>
static void spread2d_setup(JobSet<R>& js) {
    js.wpb = spread2d_wpb<R, BOPT>();
    js.wtab_ok = 0;
    if constexpr (BOPT) {
        int P = 0;
        for (int j = 0; j < js.njobs; ++j) P = std::max(P, js.job[j].P);
        js.smem_per_warp = SPREAD_BOPT_WARPS * P * P * (int)sizeof(cx<R>);
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
    INFFT_TRY(smem_limit<k_spread2d<R, MM, BOPT>>(smem));
    // shared memory bounds the warps per SM: ask for all of it
    INFFT_CUDA(cudaFuncSetAttribute(k_spread2d<R, MM, BOPT>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    (int)cudaSharedmemCarveoutMaxShared));
    k_spread2d<R, MM, BOPT><<<(nitems + js.wpb - 1) / js.wpb, 32 * spread2d_warps<R, BOPT>(), smem, st>>>(js);
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
        if (bopt && ((uintptr_t)J.coef & 15)) return false;                 // 16-byte loads of coefficients
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
