// Two-dimensional float32 spreading on the tensor cores (window modes, Algorithm 2.4 step 1 and
// its form in Algorithm 3.7): the body of the float32 k_spread2d and of the spread units of the
// persistent d = 2 kernel.
#pragma once

#include <cuda_fp16.h>

#include <cmath>
#include <cstdint>

#include "spread.cuh"

namespace infft {

// ---------------------------------------------------------------------------------------
// A work item's padded tile is the matrix product  G = (c psi_y)^T psi_x  over its points: rows
// of the padded tile against columns, the contraction index being the point.  A point touches
// 2m + 1 of the rows and columns, so the product is formed on windows of rows and columns only:
//  * the points are sorted by row; those whose first row lies in one band of 8 padded rows touch
//    at most RB = ceil((8 + 2m) / 8) row blocks of 8, held in registers (real and imaginary
//    part).  At the end of a band the top 8 rows are complete: they are stored, and the blocks
//    below move up one block, which in the accumulator layout is a register renaming.
//  * a chunk of up to 32 points (one lane each while staging) is split by one ballot into the
//    points that start in columns 0..7 and in 8..15 of the tile; groups of 8 points then meet RB
//    column blocks of 8 (one more in the one group per chunk that holds both kinds).
// One m16n8k16 instruction takes 8 points: float32 factors are split into two float16 parts h + l
// (h rounded to nearest, so 22 to 23 bits), and the two k slots of a point carry the partial products
//   (h, l) (l', l')  +  (h, l) (h', h'),
// two instructions per 8 points, 16 rows and 8 columns, no product dropped.  Float16's range is met by
// powers of two: the window is scaled to at most 2^13 (its smallest taps then keep their bits to 2^-37
// of its maximum), the chunk's samples to at most 1, and the sum's scale is undone as it is added.  Each
// group's sum starts from zero, the small part first, and is added to the accumulators by a float32
// multiply-add: the tensor cores truncate their sums, which then costs at most one rounding of the
// group's sum and not one of the running total.  Truncation to 24 bits takes 2^-24 E[1 / mantissa], about 3.7e-8, off a
// group's sum on average; the row factors are split with that much added (MMA_TRUNC), each point's alike, so that the mean
// is kept whatever the number of points or groups.  (A factor of 1 + 2^-23 on every other group of a chunk kept it for full
// chunks only, left sparse sets 3.5e-8 low and added its own 6e-8 of scatter to cells of one group.)
//
// A sample that is not finite makes NaN of its group's rows and columns of the tile (the form before:
// of its 2m + 1 rows); after the transforms every coefficient is NaN either way.
//
// Why this form: the register-row form before it (lane = column, every lane adding every point's
// 2m + 1 rows) spent its time in the shared-memory pipe and in issuing multiply-adds of which a
// quarter were not zeros.  Per point (m = 4) that was 9 packed multiply-adds and 9.5 wavefronts;
// here it is 1.7 instructions of the tensor pipe (2.1 cycles each per SM) and 5 wavefronts.
// Accumulation order: groups in point order, so results do not depend on the schedule.
template <int MM>
struct SpreadMma {
    static constexpr int W = 2 * MM + 1;
    static constexpr int RB = (8 + 2 * MM + 7) / 8;     // 8-row (8-column) blocks of a window
    static constexpr int NB = RB + 1;                   // column blocks of a tile of 16 columns
    // Staged taps of a point: W slots, then zeros up to the slot stride, so that a lane reads slot
    // (row - first row) for every row of the window without a test: 7 zeros before (15 of the columns: the
    // zeros of the point before) and the rest of the window after.  Slots of 8 bytes for the rows (the words (h, l)
    // of real and imaginary part), 4 bytes for the columns (h', l').  The strides are 4 mod 16 and +-8
    // mod 32 with one slot more every 4 points: both the stores (one lane per point) and the fragment
    // loads (4 points x consecutive slots) meet distinct banks.
    static constexpr int SA = MM <= 4 ? 20 : 28;
    static constexpr int SB = MM <= 4 ? 24 : 40;
    static constexpr int OFF_A = 7 * 8;
    static constexpr int OFF_B = OFF_A + (32 * SA + 8) * 8 + 15 * 4;
    static constexpr int OFF_Z = (OFF_B + (32 * SB + 8) * 4 + 15) & ~15;   // zeros: taps of no point
    static_assert(RB * 64 >= NB * 32, "the zero block covers the column blocks");
    static constexpr int OFF_META = OFF_Z + RB * 64;   // int2 per point: offsets of row and column taps
    static constexpr int OFF_POLY = OFF_META + 32 * 8;
    static constexpr int BYTES = OFF_POLY + WPOLY_ROWS * wpoly_stride(MM) * 4;
    static_assert(W + 7 <= SA && W + 15 <= SB && 8 * RB <= SA && 8 * NB <= SB, "a window's taps and zeros");
};

// x c and y d as h + l in float16 (the product's own rounding goes into l): H and L hold (x's part, y's part).  With
// TRUNC both are larger by MMA_TRUNC, below the rounding of l and kept by it on average.
constexpr float MMA_TRUNC = 3.7e-8f;
template <bool TRUNC>
__device__ __forceinline__ void split_f16(float x, float c, float y, float d, uint32_t& H, uint32_t& L) {
    const __half2 h = __floats2half2_rn(x * c, y * d);
    H = *reinterpret_cast<const uint32_t*>(&h);
    const float2 b = __half22float2(h);
    float2 r = make_float2(fmaf(x, c, -b.x), fmaf(y, d, -b.y));
    if (TRUNC) r = __ffma2_rn(b, make_float2(MMA_TRUNC, MMA_TRUNC), r);
    const __half2 l = __floats2half2_rn(r.x, r.y);
    L = *reinterpret_cast<const uint32_t*>(&l);
}

// d = a b (mma_f16_zero) or d += a b (mma_f16)
__device__ __forceinline__ void mma_f16_zero(float4& d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                             uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d.x), "=f"(d.y), "=f"(d.z), "=f"(d.w)
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_f16(float4& d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d.x), "+f"(d.y), "+f"(d.z), "+f"(d.w)
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// the power of two that brings a window below 2^wexp to at most 2^13
__host__ __device__ __forceinline__ float spread_mma_wscale(int wexp) {
#ifdef __CUDA_ARCH__
    return __int_as_float((127 + 13 - wexp) << 23);
#else
    return (float)ldexp(1.0, 13 - wexp);
#endif
}

// The least exponent field e of a chunk's largest sample that is scaled up in full: the sum is scaled back by
// 2^(e - 152 + w), w the window's exponent over all axes, which has to stay a power of two that float32 holds (2^-149; a
// subnormal factor is exact).  Kaiser-Bessel windows (w >= 14) reach every normal sample, B-splines (w = 0) all but
// the last two binades, where the products lie below float32's range in the first place.
__device__ __forceinline__ int spread_mma_elow(int w) { return max(1, 3 - w); }

// one warp spreads work item gitem (global over the JobSet's jobs); `base` is the warp's shared memory
template <int MM>
__device__ __forceinline__ void spread2d_mma_item(const JobSet<float>& js, const int gitem, unsigned char* base) {
    using C = SpreadMma<MM>;
    constexpr int W = C::W, RB = C::RB, NB = C::NB;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int jb = find_job(js.pre_items, js.njobs, gitem);
    const Job<float>& J = js.job[jb];
    const int it = gitem - js.pre_items[jb];
    const int4 item = J.items[it];
    const int P = J.P, Ms = J.Ms, T = J.T;
    const int ty = item.x / J.ntile, tx = item.x % J.ntile;
    const int logMs = 31 - __clz(Ms);
    const bool dcf = J.mode == INFFT_MODE_DCF;
    float* poly = reinterpret_cast<float*>(base + C::OFF_POLY);
    const float wscale = spread_mma_wscale(J.wexp), wscale0 = J.window == WK_BSPLINE ? 0.f : wscale;   // tap 0's: on a node
    if (!js.wtab_ok)
        for (int e = lane; e < WPOLY_ROWS * wpoly_stride(MM); e += 32) poly[e] = J.wpoly[e] * wscale;
    for (int e = lane; e < C::OFF_META / 16; e += 32) reinterpret_cast<uint4*>(base)[e] = make_uint4(0, 0, 0, 0);
    __syncwarp();   // before lanes read others' rows of the table and store taps over slots others cleared

    // acc[k][b]: row g of the k-th block of 8 rows held, columns 8b + 2t and 8b + 2t + 1; (x, y) real, (z, w)
    // imaginary parts (the two 8-row halves of an m16 tile)
    float4 acc[RB][NB];
#pragma unroll
    for (int k = 0; k < RB; ++k)
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[k][b] = make_float4(0.f, 0.f, 0.f, 0.f);
    int r0 = 0;   // first padded row held
    cx<float>* dst = J.padded + (size_t)it * P * P;
    auto flush_rows = [&]() {   // rows r0 .. r0 + 7 are complete
        const int row = r0 + g;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const float4 v = acc[0][b];
            // P and the item's base are even: a column pair is 16-byte aligned
            if (row < P && 8 * b + 2 * t < P)
                *reinterpret_cast<float4*>(dst + (size_t)row * P + 8 * b + 2 * t) = make_float4(v.x, v.z, v.y, v.w);
#pragma unroll
            for (int k = 0; k + 1 < RB; ++k) acc[k][b] = acc[k + 1][b];
            acc[RB - 1][b] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        r0 += 8;
    };

    // the lane's point of the next chunk is loaded while this one is staged, its sample (whose index has
    // arrived by then) while this one is multiplied
    int perm = 0;
    uint32_t cl = 0;
    float2 u = make_float2(0.f, 0.f), f = u, w = make_float2(1.f, 0.f);
    auto load_point = [&](int c) {
        if (c + lane < item.z) {
            const size_t i = (size_t)item.y + c + lane;
            perm = __ldg(J.perm + i);
            cl = __ldg(J.cell + i);
            u = __ldg(reinterpret_cast<const float2*>(J.u) + i);
            if (dcf) w = __ldg(reinterpret_cast<const float2*>(J.w) + i);
        }
    };
    auto load_sample = [&](int c) {
        if (c + lane < item.z) f = __ldg(reinterpret_cast<const float2*>(J.in) + perm);
    };
    auto taps = [&](float2 v, float (*wt)[W]) {   // of both coordinates, scaled to at most 2^13
        const float vv[2] = {v.x, v.y};
        if (js.wtab_ok) {
            poly_taps<MM, 1>(js.wtab, vv, wt);
            poly_taps<MM, 1>(js.wtab, vv + 1, wt + 1);
        } else {
            poly_taps<MM, 2>(poly, vv, wt);
        }
        wt[0][0] *= wscale0;
        wt[1][0] *= wscale0;
    };
    load_point(0);
    load_sample(0);

    for (int c0 = 0; c0 < item.z;) {
        const int oy = (int)(cl >> logMs) - ty * T, ox = (int)(cl & (uint32_t)(Ms - 1)) - tx * T;
        // the chunk ends where the points leave its band of rows (the points are sorted by row)
        const int band = __shfl_sync(0xffffffffu, oy >> 3, 0);
        const unsigned in = __ballot_sync(0xffffffffu, c0 + lane < item.z && (oy >> 3) == band);
        const int np = __popc(in);
        while (r0 < 8 * band) flush_rows();
        // the points that start in the first 8 columns come first
        const unsigned right = __ballot_sync(0xffffffffu, ox >= 8) & in;
        const int n0 = np - __popc(right);
        const unsigned below = (1u << lane) - 1u;
        const int pos = lane >= np ? lane : ox >= 8 ? n0 + __popc(right & below) : __popc(~right & in & below);
        int2 off = make_int2(C::OFF_Z, C::OFF_Z);
        const float2 uc = u;
        float2 c = f;
        if (dcf) c = make_float2(w.x * f.x - w.y * f.y, w.x * f.y + w.y * f.x);
        c0 += np;
        load_point(c0);
        // 2^(126 - e) brings the chunk's samples to at most 1 (4 for the last exponents of float32)
        const unsigned top = __reduce_max_sync(0xffffffffu, lane < np ? __float_as_uint(fmaxf(fabsf(c.x), fabsf(c.y))) : 0u);
        const int e = min(max((int)(top >> 23), spread_mma_elow(2 * J.wexp)), 252);
        const float cscale = __int_as_float((253 - e) << 23);
        const float us1 = __int_as_float((e + 1) << 23) * __int_as_float((127 + 2 * (J.wexp - 13)) << 23);
        const float2 us = make_float2(us1, us1);
        if (lane < np) {
            const int ra = C::OFF_A + (pos * C::SA + (pos >> 2)) * 8, rb = C::OFF_B + (pos * C::SB + (pos >> 2)) * 4;
            off = make_int2(ra - (oy & 7) * 8, rb - ox * 4);
            c = make_float2(c.x * cscale, c.y * cscale);
            float wt[2][W];
            taps(uc, wt);
#pragma unroll
            for (int s = 0; s < W; ++s) {
                uint32_t H, L;
                split_f16<true>(c.x, wt[0][s], c.y, wt[0][s], H, L);
                *reinterpret_cast<uint2*>(base + ra + 8 * s) =
                    make_uint2(__byte_perm(H, L, 0x5410), __byte_perm(H, L, 0x7632));
            }
#pragma unroll
            for (int s = 0; s < W; s += 2) {
                uint32_t H, L;
                split_f16<false>(wt[1][s], 1.f, s + 1 < W ? wt[1][s + 1] : 0.f, 1.f, H, L);
                *reinterpret_cast<uint32_t*>(base + rb + 4 * s) = __byte_perm(H, L, 0x5410);
                if (s + 1 < W) *reinterpret_cast<uint32_t*>(base + rb + 4 * s + 4) = __byte_perm(H, L, 0x7632);
            }
        }
        reinterpret_cast<int2*>(base + C::OFF_META)[pos] = off;
        __syncwarp();

        const int ng = (np + 7) >> 3;
#pragma unroll 2
        for (int grp = 0; grp < ng; ++grp) {
            const int p0 = 8 * grp + t, p1 = p0 + 4;
            const int2 o0 = reinterpret_cast<const int2*>(base + C::OFF_META)[p0];
            const int2 o1 = reinterpret_cast<const int2*>(base + C::OFF_META)[p1];
            uint2 a0[RB], a1[RB];   // the (h, l) words of real and imaginary part, points p0 and p1
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                a0[r] = *reinterpret_cast<const uint2*>(base + o0.x + 64 * r + 8 * g);
                a1[r] = *reinterpret_cast<const uint2*>(base + o1.x + 64 * r + 8 * g);
            }
            if (grp == 0) load_sample(c0);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                // no tap of the points from column 8 on lies in the first column block, none of the others' in the last
                if (b == 0 && 8 * grp >= n0) continue;
                if (b == NB - 1 && 8 * grp + 7 < n0) continue;
                const uint32_t v0 = *reinterpret_cast<const uint32_t*>(base + o0.y + 32 * b + 4 * g);
                const uint32_t v1 = *reinterpret_cast<const uint32_t*>(base + o1.y + 32 * b + 4 * g);
                const uint32_t h0 = __byte_perm(v0, 0, 0x1010), l0 = __byte_perm(v0, 0, 0x3232);
                const uint32_t h1 = __byte_perm(v1, 0, 0x1010), l1 = __byte_perm(v1, 0, 0x3232);
                float4 d[RB];
#pragma unroll
                for (int k = 0; k < RB; ++k)
                    mma_f16_zero(d[k], a0[k].x, a0[k].y, a1[k].x, a1[k].y, l0, l1);
#pragma unroll
                for (int k = 0; k < RB; ++k)
                    mma_f16(d[k], a0[k].x, a0[k].y, a1[k].x, a1[k].y, h0, h1);
#pragma unroll
                for (int k = 0; k < RB; ++k) {
                    float2* q = reinterpret_cast<float2*>(&acc[k][b]);
                    q[0] = __ffma2_rn(make_float2(d[k].x, d[k].y), us, q[0]);
                    q[1] = __ffma2_rn(make_float2(d[k].z, d[k].w), us, q[1]);
                }
            }
        }
        __syncwarp();   // the taps are read before the next chunk's are stored
    }
    while (r0 < P) flush_rows();
}

}  // namespace infft
