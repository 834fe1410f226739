// Fixed-m interpolation for d = 2 (Algorithm 2.1 step 3), with window taps and with B_opt (Remark 4.6).
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "interp.cuh"

namespace infft {

// ---------------------------------------------------------------------------------------
// Interpolation with B_opt for d = 2 (Remark 4.6, f = B_opt F D h): like the B_opt spread, this has to
// read every point's run of S x S coefficients once.  Eight warps share a work item's padded tile of the grid
// in shared memory and take an eighth of its points each; the lanes of a warp take a point's coefficients
// 16 bytes each (a lane per point read them 800 bytes apart), four points' loads in flight, and the
// four points' sums over the lanes share one exchange (11 shuffles for eight values instead of 40).
constexpr int INTERP_BOPT_WARPS = 8;

template <class R, int MM>
__global__ void __launch_bounds__(32 * INTERP_BOPT_WARPS) k_interp_bopt2d(const __grid_constant__ JobSet<R> js) {
    using C = BoptLanes<R, MM>;
    constexpr int VEC = C::VEC, NV = C::NV, NR = C::NR, S = C::S, NW = INTERP_BOPT_WARPS;
    using V = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<R>* pad = reinterpret_cast<cx<R>*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int jb = find_job(js.pre_items, js.njobs, blockIdx.x);
    const Job<R>& J = js.job[jb];
    const int4 item = J.items[blockIdx.x - js.pre_items[jb]];
    const int P = J.P, m = J.m, Ms = J.Ms, T = J.T;
    const int ty = item.x / J.ntile, tx = item.x % J.ntile;
    const int logMs = 31 - __clz(Ms);
    for (int e = threadIdx.x; e < P * P; e += 32 * NW) {
        const int oy = e / P, ox = e - oy * P;
        pad[e] = J.grid[(size_t)((ty * T - m + oy) & (Ms - 1)) * Ms + ((tx * T - m + ox) & (Ms - 1))];
    }
    int off[NR];
    bool act[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int q = VEC * (lane + 32 * r);
        act[r] = lane + 32 * r < NV;
        off[r] = act[r] ? (q / S) * P + q % S : 0;
    }
    __syncthreads();
    const int per = (item.z + NW - 1) / NW, first = min(item.z, warp * per), last = min(item.z, first + per);
    for (int c0 = first; c0 < last; c0 += 32) {
        const int np = min(32, last - c0);
        int o = 0, perm = 0;
        if (lane < np) {
            const int i = item.y + c0 + lane;
            const uint32_t cl = __ldg(J.cell + i);
            o = ((int)(cl >> logMs) - ty * T) * P + (int)(cl & (uint32_t)(Ms - 1)) - tx * T;
            perm = __ldg(J.perm + i);
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
            R v[2 * U];   // (re, im) of the points' sums
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int op = __shfl_sync(0xffffffffu, o, min(p0 + k, np - 1));
                cx<R> acc = mk<R>(0, 0);
                if (p0 + k < np) {
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        if (!act[r]) continue;
                        const cx<R>* cell = pad + op + off[r];
                        const R* bb = reinterpret_cast<const R*>(&b[k][r]);
#pragma unroll
                        for (int q = 0; q < VEC; ++q) acc = add(acc, mul(mk<R>(bb[2 * q], bb[2 * q + 1]), cell[q]));
                    }
                }
                v[2 * k] = acc.re;
                v[2 * k + 1] = acc.im;
            }
            // sums over the lanes: halves exchange and keep one value in two until a lane holds one, then over its four lanes
#pragma unroll
            for (int h = U, s = 16; h >= 1; h >>= 1, s >>= 1) {
#pragma unroll
                for (int i = 0; i < h; ++i) {
                    const bool up = (lane & s) != 0;
                    const R send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
                }
            }
            R sum = v[0];
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            const int k = ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1), part = (lane >> 2) & 1;
            const int j = __shfl_sync(0xffffffffu, perm, min(p0 + k, np - 1));
            if ((lane & 3) == 0 && p0 + k < np) reinterpret_cast<R*>(J.out + j)[part] = sum;
        }
    }
}

template <class R, int MM>
static infft_status launch_interp_bopt2d(JobSet<R>& js, cudaStream_t st) {
    int P = 0;
    for (int j = 0; j < js.njobs; ++j) P = std::max(P, js.job[j].P);
    const size_t smem = (size_t)P * P * sizeof(cx<R>);
    const int nitems = js.pre_items[js.njobs];
    if (nitems == 0) return INFFT_OK;
    INFFT_TRY(smem_limit<k_interp_bopt2d<R, MM>>(smem));
    k_interp_bopt2d<R, MM><<<nitems, 32 * INTERP_BOPT_WARPS, smem, st>>>(js);
    INFFT_LAUNCHED();
    return INFFT_OK;
}

// the B_opt form when every job has it with the same m (2..7), aligned coefficients and power-of-two grids
template <class R>
static infft_status interp_bopt2d_try(JobSet<R>& js, cudaStream_t st, bool* used) {
    *used = false;
    const int m = js.job[0].m;
    if (m < 2 || m > 7) return INFFT_OK;
    for (int j = 0; j < js.njobs; ++j) {
        const Job<R>& J = js.job[j];
        if (J.m != m || J.mode != INFFT_MODE_BOPT || J.P > 64 || ((uintptr_t)J.coef & 15)) return INFFT_OK;
    }
    *used = true;
    switch (m) {
        case 2: return launch_interp_bopt2d<R, 2>(js, st);
        case 3: return launch_interp_bopt2d<R, 3>(js, st);
        case 4: return launch_interp_bopt2d<R, 4>(js, st);
        case 5: return launch_interp_bopt2d<R, 5>(js, st);
        case 6: return launch_interp_bopt2d<R, 6>(js, st);
        default: return launch_interp_bopt2d<R, 7>(js, st);
    }
}

template <class R>
infft_status interp2d_try(JobSet<R>& js, cudaStream_t st, bool* used) {
    INFFT_TRY(interp_bopt2d_try<R>(js, st, used));
    return *used ? INFFT_OK : interp_try_d<R, 2>(js, st, used);
}

template infft_status interp2d_try<float>(JobSet<float>&, cudaStream_t, bool*);
template infft_status interp2d_try<double>(JobSet<double>&, cudaStream_t, bool*);

}  // namespace infft
