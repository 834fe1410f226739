// Three-dimensional float32 spreading on the tensor cores (window modes, m <= 4, tiles of 8^3).
#pragma once

#include "spreadmma.cuh"

namespace infft {

// ---------------------------------------------------------------------------------------
// The scheme of spreadmma.cuh plane by plane.  A work item's padded tile is P <= 16 cells wide, so a plane
// is two blocks of 8 rows (real and imaginary part in one m16 tile each) by two of 8 columns: 16 registers
// per lane.  The points are sorted by plane; a point touches W = 2m + 1 planes from its own on, and all of these
// are held while the points of that first plane pass; then the lowest plane is complete, is stored, and its owner's
// other planes move down (a register move per point layer, at most 8 times an item).  Two warps share an item,
// one holding the even and one the odd planes (at most 5 each, 80 registers), so that 12 warps share an SM.
// Nothing of the tile is in shared memory, where the form before kept all of it (34 KB a warp, six warps
// per SM, a load and a store of 81 cells whenever the base cell changed).
// A chunk is up to 64 points, staged by both warps, half each; it ends where the points leave a plane.  The factors of
// plane s are c psi_y (split once) and psi_x psi_z(s), formed and split into two float16 parts in registers.
template <int MM>
struct SpreadMma3 {
    static constexpr int W = 2 * MM + 1, T = 8, RB = 2;
    static constexpr int SA = 20, SB = 24;              // slots of staged taps, as in spreadmma.cuh
    static constexpr int OFF_A = 7 * 8;
    static constexpr int OFF_B = OFF_A + (32 * SA + 8) * 8 + 7 * 4;
    static constexpr int OFF_Z = (OFF_B + (32 * SB + 8) * 4 + 15) & ~15;
    static constexpr int OFF_PZ = OFF_Z + RB * 64;      // [32][W] psi_z
    static constexpr int OFF_META = (OFF_PZ + 32 * W * 4 + 15) & ~15;
    static constexpr int OFF_US = OFF_META + 32 * 8;    // the half's scale
    static constexpr int HALF = OFF_US + 16;            // bytes of a half chunk
    static constexpr int OFF_POLY = 2 * HALF;
    static constexpr int BYTES = OFF_POLY + WPOLY_ROWS * wpoly_stride(MM) * 4;
    static constexpr int NP = (W + 1) / 2;              // planes of a warp
    static_assert(MM <= 4 && W + 7 <= SA && W + 7 <= SB && 8 * RB <= SA && 8 * RB <= SB, "a window's taps and zeros");
};

template <int MM>
__global__ void __launch_bounds__(64, 6) k_spread3d_mma(const __grid_constant__ JobSet<float> js) {
    using C = SpreadMma3<MM>;
    constexpr int W = C::W, T = C::T, RB = C::RB, NP = C::NP;
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int jb = find_job(js.pre_items, js.njobs, blockIdx.x);
    const Job<float>& J = js.job[jb];
    const int it = blockIdx.x - js.pre_items[jb];
    const int4 item = J.items[it];
    const int P = J.P, Ms = J.Ms, nt = J.ntile;
    const int tz = item.x / (nt * nt), ty = (item.x / nt) % nt, tx = item.x % nt;
    const int logMs = 31 - __clz(Ms);
    const bool dcf = J.mode == INFFT_MODE_DCF;
    unsigned char* own = smem + warp * C::HALF;       // the half chunk this warp stages
    float* poly = reinterpret_cast<float*>(smem + C::OFF_POLY);
    const float wscale = spread_mma_wscale(J.wexp);   // window to at most 2^13
    const float wscale0 = J.window == WK_BSPLINE ? 0.f : wscale;   // tap 0's: on a node
    for (int e = threadIdx.x; e < WPOLY_ROWS * wpoly_stride(MM); e += 64) poly[e] = J.wpoly[e] * wscale;
    for (int e = lane; e < C::OFF_META / 16; e += 32) reinterpret_cast<uint4*>(own)[e] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    // acc[i][k][b]: plane zf + 2 i, where zf is the first plane >= z0 of the warp's parity; block k of 8 rows, b of 8 columns
    float4 acc[NP][RB][2];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int k = 0; k < RB; ++k)
#pragma unroll
            for (int b = 0; b < 2; ++b) acc[i][k][b] = make_float4(0.f, 0.f, 0.f, 0.f);
    int z0 = 0;   // first padded plane held
    cx<float>* dst = J.padded + (size_t)it * P * P * P;
    auto flush_plane = [&]() {   // plane z0 is complete
        if ((z0 & 1) == warp) {
#pragma unroll
            for (int k = 0; k < RB; ++k)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float4 v = acc[0][k][b];
                    const int row = 8 * k + g, col = 8 * b + 2 * t;
                    if (row < P && col < P)   // P is even: a column pair is 16-byte aligned
                        *reinterpret_cast<float4*>(dst + ((size_t)z0 * P + row) * P + col) = make_float4(v.x, v.z, v.y, v.w);
#pragma unroll
                    for (int i = 0; i + 1 < NP; ++i) acc[i][k][b] = acc[i + 1][k][b];
                    acc[NP - 1][k][b] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
        }
        ++z0;
    };

    int perm = 0;
    uint32_t cl0 = 0, cl1 = 0;   // cells of points lane and 32 + lane of the chunk
    float uz = 0.f, uy = 0.f, ux = 0.f;
    float2 f = make_float2(0.f, 0.f), w = make_float2(1.f, 0.f);
    auto load_point = [&](int c) {
        if (c + lane < item.z) cl0 = __ldg(J.cell + item.y + c + lane);
        if (c + 32 + lane < item.z) cl1 = __ldg(J.cell + item.y + c + 32 + lane);
        if (c + 32 * warp + lane < item.z) {
            const size_t i = (size_t)item.y + c + 32 * warp + lane;
            perm = __ldg(J.perm + i);
            uz = __ldg(J.u + 3 * i);
            uy = __ldg(J.u + 3 * i + 1);
            ux = __ldg(J.u + 3 * i + 2);
            if (dcf) w = __ldg(reinterpret_cast<const float2*>(J.w) + i);
        }
    };
    auto load_sample = [&](int c) {
        if (c + 32 * warp + lane < item.z) f = __ldg(reinterpret_cast<const float2*>(J.in) + perm);
    };
    load_point(0);
    load_sample(0);
    for (int c0 = 0; c0 < item.z;) {
        // the chunk ends where the points leave the plane (the points are sorted by plane)
        const int zc = __shfl_sync(0xffffffffu, (int)(cl0 >> (2 * logMs)), 0);
        const int n0 = __popc(__ballot_sync(0xffffffffu, c0 + lane < item.z && (int)(cl0 >> (2 * logMs)) == zc));
        const int n1 = n0 < 32 ? 0 : __popc(__ballot_sync(0xffffffffu, c0 + 32 + lane < item.z && (int)(cl1 >> (2 * logMs)) == zc));
        const int np = n0 + n1, mine = warp == 0 ? n0 : n1;
        while (z0 < zc - tz * T) flush_plane();
        const uint32_t cl = warp == 0 ? cl0 : cl1;
        const int oy = (int)((cl >> logMs) & (uint32_t)(Ms - 1)) - ty * T, ox = (int)(cl & (uint32_t)(Ms - 1)) - tx * T;
        int2 off = make_int2(C::OFF_Z, C::OFF_Z);
        float2 c = f;
        if (dcf) c = make_float2(w.x * f.x - w.y * f.y, w.x * f.y + w.y * f.x);
        const float vz = uz, vy = uy, vx = ux;
        c0 += np;
        load_point(c0);
        const unsigned top = __reduce_max_sync(0xffffffffu, lane < mine ? __float_as_uint(fmaxf(fabsf(c.x), fabsf(c.y))) : 0u);
        const int e = min(max((int)(top >> 23), spread_mma_elow(3 * J.wexp)), 252);
        const float cscale = __int_as_float((253 - e) << 23);
        if (lane < mine) {
            const int ra = C::OFF_A + (lane * C::SA + (lane >> 2)) * 8, rb = C::OFF_B + (lane * C::SB + (lane >> 2)) * 4;
            float* pz = reinterpret_cast<float*>(own + C::OFF_PZ) + lane * W;
            off = make_int2(ra - oy * 8, rb - ox * 4);
            c = make_float2(c.x * cscale, c.y * cscale);
            const float uu[3] = {vy, vx, vz};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                float wt[1][W];
                poly_taps<MM, 1>(poly, uu + a, wt);
                wt[0][0] *= wscale0;
#pragma unroll
                for (int s = 0; s < W; ++s) {
                    if (a == 0) {
                        uint32_t H, L;
                        split_f16<true>(c.x, wt[0][s], c.y, wt[0][s], H, L);
                        *reinterpret_cast<uint2*>(own + ra + 8 * s) =
                            make_uint2(__byte_perm(H, L, 0x5410), __byte_perm(H, L, 0x7632));
                    } else if (a == 1) {
                        *reinterpret_cast<float*>(own + rb + 4 * s) = wt[0][s];
                    } else {
                        pz[s] = wt[0][s] * (1.f / 8192.f);
                    }
                }
            }
        }
        reinterpret_cast<int2*>(own + C::OFF_META)[lane] = off;
        // the samples' scale, 2^13 / 2^wexp of two axes and 1 / 2^wexp of the third
        if (lane == 0)
            *reinterpret_cast<float*>(own + C::OFF_US) =
                __int_as_float((e + 1) << 23) * __int_as_float((127 + 3 * J.wexp - 26) << 23);
        __syncthreads();

        const int ng = (np + 7) >> 3;   // groups 0..3 in the first half, 4..7 in the second
        const int s0 = (z0 ^ warp) & 1;   // tap of the warp's first plane
#pragma unroll 1
        for (int grp = 0; grp < ng; ++grp) {
            const unsigned char* half = smem + (grp >> 2) * C::HALF;
            const int p0 = 8 * (grp & 3) + t, p1 = p0 + 4;
            const int2 o0 = reinterpret_cast<const int2*>(half + C::OFF_META)[p0];
            const int2 o1 = reinterpret_cast<const int2*>(half + C::OFF_META)[p1];
            uint2 a0[RB], a1[RB];
            float x0[2], x1[2];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                a0[r] = *reinterpret_cast<const uint2*>(half + o0.x + 64 * r + 8 * g);
                a1[r] = *reinterpret_cast<const uint2*>(half + o1.x + 64 * r + 8 * g);
            }
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                x0[b] = *reinterpret_cast<const float*>(half + o0.y + 32 * b + 4 * g);
                x1[b] = *reinterpret_cast<const float*>(half + o1.y + 32 * b + 4 * g);
            }
            if (grp == 0) load_sample(c0);
            const float us = *reinterpret_cast<const float*>(half + C::OFF_US);
            const float2 uu = make_float2(us, us);
            const float* pz0 = reinterpret_cast<const float*>(half + C::OFF_PZ) + p0 * W + s0;
            const float* pz1 = pz0 + 4 * W;
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                if (i == NP - 1 && s0 == 1) continue;   // one plane fewer
                const float w0 = pz0[2 * i], w1 = pz1[2 * i];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    uint32_t H, L;
                    split_f16<false>(x0[b], w0, x1[b], w1, H, L);
                    const uint32_t h0 = __byte_perm(H, 0, 0x1010), h1 = __byte_perm(H, 0, 0x3232);
                    const uint32_t l0 = __byte_perm(L, 0, 0x1010), l1 = __byte_perm(L, 0, 0x3232);
                    float4 d[RB];
#pragma unroll
                    for (int k = 0; k < RB; ++k) mma_f16_zero(d[k], a0[k].x, a0[k].y, a1[k].x, a1[k].y, l0, l1);
#pragma unroll
                    for (int k = 0; k < RB; ++k) mma_f16(d[k], a0[k].x, a0[k].y, a1[k].x, a1[k].y, h0, h1);
#pragma unroll
                    for (int k = 0; k < RB; ++k) {
                        float2* q = reinterpret_cast<float2*>(&acc[i][k][b]);
                        q[0] = __ffma2_rn(make_float2(d[k].x, d[k].y), uu, q[0]);
                        q[1] = __ffma2_rn(make_float2(d[k].z, d[k].w), uu, q[1]);
                    }
                }
            }
        }
        __syncthreads();   // the taps are read before the next chunk's are stored
    }
    while (z0 < P) flush_plane();
}

template <int MM>
static infft_status launch_spread3d_mma(JobSet<float>& js, cudaStream_t st) {
    const int nitems = js.pre_items[js.njobs];
    if (nitems == 0) return INFFT_OK;
    const int smem = SpreadMma3<MM>::BYTES;
    INFFT_TRY(smem_limit<k_spread3d_mma<MM>>(smem));
    INFFT_CUDA(cudaFuncSetAttribute(k_spread3d_mma<MM>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    (int)cudaSharedmemCarveoutMaxShared));
    k_spread3d_mma<MM><<<nitems, 64, smem, st>>>(js);
    INFFT_LAUNCHED();
    return INFFT_OK;
}

}  // namespace infft
