// Shared device/host definitions of the iNFFT library (sm_103a).
//
// Notation follows Sections 2-4 of Kircheis & Potts: d dimensions, degree M,
// oversampled grid M_sigma ("Ms"), truncation m, points x_j (j = 1..N).
// Grid cells are stored at l mod Ms along every axis, C order (first axis
// slowest); coefficients k in I_M at k + M/2, C order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <string>

#include "../../include/infft.h"

namespace infft {

// ----------------------------------------------------------------------------------------
// complex numbers of float or double
template <class R>
struct alignas(2 * sizeof(R)) cx {
    R re, im;
};

template <class R>
__host__ __device__ __forceinline__ cx<R> mk(R a, R b) { cx<R> z; z.re = a; z.im = b; return z; }
template <class R>
__host__ __device__ __forceinline__ cx<R> add(cx<R> a, cx<R> b) { return mk<R>(a.re + b.re, a.im + b.im); }
template <class R>
__host__ __device__ __forceinline__ cx<R> sub(cx<R> a, cx<R> b) { return mk<R>(a.re - b.re, a.im - b.im); }
template <class R>
__host__ __device__ __forceinline__ cx<R> mul(cx<R> a, cx<R> b) {
    return mk<R>(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <class R>
__host__ __device__ __forceinline__ cx<R> mulconj(cx<R> a, cx<R> b) {  // conj(a) * b
    return mk<R>(a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re);
}
template <class R>
__host__ __device__ __forceinline__ cx<R> scale(cx<R> a, R s) { return mk<R>(a.re * s, a.im * s); }
template <class R>
__host__ __device__ __forceinline__ cx<R> conjg(cx<R> a) { return mk<R>(a.re, -a.im); }

// ----------------------------------------------------------------------------------------
// Kaiser-Bessel window in grid units (Section 2.1 with the I0 form of the window):
//   phi(delta) = I0(beta sqrt(1 - (delta/m)^2)) for |delta| <= m, 0 otherwise,
// delta = M_sigma x - l, beta = pi m (2 - M/M_sigma).  The closed support is used:
// |delta| = m is inside.
__device__ __forceinline__ float bessel_i0(float z) { return cyl_bessel_i0f(z); }
__device__ __forceinline__ double bessel_i0(double z) { return cyl_bessel_i0(z); }

template <class R>
__device__ __forceinline__ R kb_phi(R delta, R inv_m, R beta) {
    R t = delta * inv_m;
    R s = R(1) - t * t;
    return (s >= R(0)) ? bessel_i0(beta * sqrt(s)) : R(0);
}

enum WindowKind { WK_KB = 0, WK_BSPLINE = 1, WK_DIRICHLET = 2 };

// Window value of tap s = 0..2m of a point with fractional offset u = M_sigma x - b in
// [0, 1] (b = floor(M_sigma x)); the tap sits at l = b - m + s, delta = u + m - s.
// Membership in the index set (eq. indexset_x) is decided exactly: taps 1..2m always
// satisfy |delta| <= m, tap 0 only when u = 0 (the point on a grid node).
template <class R>
__device__ __forceinline__ R kb_tap(R u, int s, int m, R inv_m, R beta) {
    if (s == 0 && u != R(0)) return R(0);
    return kb_phi<R>(u + R(m - s), inv_m, beta);
}

// The taps of the centred cardinal B-spline of order n = 2m (eq. window_bspline; 2m <= 16) by the Cox-de Boor
// recursion on the uniform knots -m..m, once for all taps: with w_j the value at u + j above the first knot,
//   order k + 1:  w_j <- (u + j) w_j + (k + 1 - j - u) w_{j-1}
// without the 1 / k of each order, which is 1 / (n - 1)! at the end.  All terms are positive: no digits are lost.
// Tap s is w_{2m-s}; tap 0, on a node, is zero.  (A recursion for each tap by itself takes 2m times the work: where a
// kernel stages few points at a time, sparse d = 3 sets in float32, it was three quarters of the call.)
template <int MM, class R>
__device__ __forceinline__ void bspline_taps(R u, R* out) {
    constexpr int n = 2 * MM;
    R w[n];
    w[0] = R(1);
    double fact = 1;
#pragma unroll
    for (int k = 1; k < n; ++k) {
        fact *= k;
        w[k] = (R(1) - u) * w[k - 1];
#pragma unroll
        for (int j = n - 1; j >= 1; --j)
            if (j < k) w[j] = fma(u + R(j), w[j], (R(k + 1 - j) - u) * w[j - 1]);
        w[0] *= u;
    }
    // 1 / (n - 1)! to twice the precision: rounded, it would scale every value alike
    const double inv = 1.0 / fact;
    const R hi = R(inv), lo = R(sizeof(R) == 4 ? inv - (double)hi : fma(-inv, fact, 1.0) * inv);
    out[0] = R(0);
#pragma unroll
    for (int s = 1; s <= n; ++s) out[s] = fma(w[n - s], hi, w[n - s] * lo);
}
// for m known at run time only; out[0..2m] holds the triangle
template <class R>
__device__ __forceinline__ void bspline_taps_any(int m, R u, R* out) {
    const int n = 2 * m;
    R fact = R(1);
    out[n] = R(1);
    for (int k = 1; k < n; ++k) {
        fact *= R(k);
        R* w = out + n;   // w_j at w[-j]
        w[-k] = (R(1) - u) * w[1 - k];
        for (int j = k - 1; j >= 1; --j) w[-j] = fma(u + R(j), w[-j], (R(k + 1 - j) - u) * w[1 - j]);
        w[0] *= u;
    }
    out[0] = R(0);
    for (int s = 1; s <= n; ++s) out[s] /= fact;
}

// Float32 plans evaluate the Kaiser-Bessel taps s = 1..2m from per-plan polynomials:
// phi(u + m - s) = sum_k c[k][s] v^k, v = 2u - 1, u in [0, 1], degree WPOLY_DEG, obtained
// by Chebyshev interpolation in float64 at plan creation (piecewise-polynomial kernel
// evaluation in the manner of Barnett, Magland and af Klinteberg, SIAM J. Sci. Comput.
// 2019).  Degree 10 reaches the float32 rounding level of the window.  The window is even, so
// tap 2m + 1 - s has the polynomial of tap s in -v: the table holds s = 1..m, and the even and
// odd parts of one polynomial give both taps (11 multiply-adds for two taps instead of 20).  Tap 0
// keeps the exact membership rule: I0(0) = 1 on a grid node, 0 otherwise.
constexpr int WPOLY_DEG = 10;
// rows of the table: c[0..WPOLY_DEG], then what rounding took from c[0] (every point of a grid node has v = -1
// along that axis, so the coefficients' errors there do not average out)
constexpr int WPOLY_ROWS = WPOLY_DEG + 2;

// row stride of the coefficient table (tap s at s - 1), padded to a multiple of 4 (16-byte rows)
__host__ __device__ constexpr int wpoly_stride(int m) { return (m + 3) & ~3; }

// the 2m + 1 taps of NC coordinates at once, two taps s, s + 1 per packed multiply-add; the table's
// rows are read with 16-byte loads (c 16-byte aligned, best in shared memory: a constant operand would
// have to be moved to registers for every use)
template <int MM, int NC>
__device__ __forceinline__ void poly_taps(const float* __restrict__ c, const float* u, float (*out)[2 * MM + 1]) {
    constexpr int WP = wpoly_stride(MM);
    constexpr int NP = WP / 2;   // pairs of taps, padded
    float2 ev[NC][NP], od[NC][NP];
    float v[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) v[a] = 2.f * u[a] - 1.f;
#pragma unroll
    for (int k = WPOLY_DEG; k >= 0; --k) {
#pragma unroll
        for (int q = 0; q < NP; q += 2) {
            const int row = k == 0 ? WPOLY_DEG + 1 : k;   // c[0] is added last, its low part first
            const float4 t = *reinterpret_cast<const float4*>(c + row * WP + 2 * q);
            const float2 t0 = make_float2(t.x, t.y), t1 = make_float2(t.z, t.w);
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                float2* p = (k & 1) ? od[a] : ev[a];
                const float2 ww = make_float2(v[a] * v[a], v[a] * v[a]);
                p[q] = k >= WPOLY_DEG - 1 ? t0 : __ffma2_rn(p[q], ww, t0);
                if (2 * q + 2 < MM) p[q + 1] = k >= WPOLY_DEG - 1 ? t1 : __ffma2_rn(p[q + 1], ww, t1);
            }
        }
    }
#pragma unroll
    for (int q = 0; 2 * q < MM; ++q) {
        const float2 t0 = *reinterpret_cast<const float2*>(c + 2 * q);
#pragma unroll
        for (int a = 0; a < NC; ++a) ev[a][q] = __fadd2_rn(ev[a][q], t0);
    }
#pragma unroll
    for (int a = 0; a < NC; ++a) {
#pragma unroll
        for (int q = 0; 2 * q < MM; ++q) {
            const float2 x = __ffma2_rn(od[a][q], make_float2(v[a], v[a]), ev[a][q]);
            const float2 y = __ffma2_rn(od[a][q], make_float2(-v[a], -v[a]), ev[a][q]);
            out[a][2 * q + 1] = x.x;
            out[a][2 * MM - 2 * q] = y.x;
            if (2 * q + 2 <= MM) {
                out[a][2 * q + 2] = x.y;
                out[a][2 * MM - 2 * q - 1] = y.y;
            }
        }
        out[a][0] = (u[a] == 0.f) ? 1.f : 0.f;
    }
}

// Float64 plans: the same polynomials of degree 21 (from values to twice the precision, made on the host at
// plan creation: polytable.h).  Interpolation is off by at most 1e-23 of the window's largest value for every m and
// oversampling, and by less than 1e-17 of a tap's own largest value but for the outermost taps of m > 10 with
// M < M_sigma / 2 (5e-14 for m = 15, M = M_sigma / 10, where that tap is 2e-25 of the window).  A tap costs 11
// multiply-adds; the double Bessel function cost several times that, at 1/32 of the float32 rate.
constexpr int WPOLY64_DEG = 21;
constexpr int WPOLY64_ROWS = WPOLY64_DEG + 1;

template <class R>
__host__ __device__ constexpr int wpoly_rows() { return sizeof(R) == 4 ? WPOLY_ROWS : WPOLY64_ROWS; }

template <int MM, int NC>
__device__ __forceinline__ void poly_taps(const double* __restrict__ c, const double* u, double (*out)[2 * MM + 1]) {
    constexpr int WP = wpoly_stride(MM);
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        const double v = 2.0 * u[a] - 1.0, v2 = v * v;
        double ev[MM], od[MM];
#pragma unroll
        for (int k = WPOLY64_DEG; k >= 0; --k) {
#pragma unroll
            for (int s = 0; s < MM; ++s) {
                double* p = (k & 1) ? od : ev;
                p[s] = k >= WPOLY64_DEG - 1 ? c[k * WP + s] : fma(p[s], v2, c[k * WP + s]);
            }
        }
#pragma unroll
        for (int s = 0; s < MM; ++s) {
            out[a][s + 1] = fma(od[s], v, ev[s]);
            out[a][2 * MM - s] = fma(od[s], -v, ev[s]);
        }
        out[a][0] = (u[a] == 0.0) ? 1.0 : 0.0;
    }
}

// the 2m + 1 taps for m known at run time only
template <class R>
__device__ __forceinline__ void poly_taps_any(const R* __restrict__ c, int m, R u, R* out) {
    const int WP = wpoly_stride(m);
    constexpr int DEG = sizeof(R) == 4 ? WPOLY_DEG : WPOLY64_DEG;
    const R v = R(2) * u - R(1), v2 = v * v;
#pragma unroll 4
    for (int s = 0; s < m; ++s) {
        R ev = R(0), od = R(0);
#pragma unroll
        for (int k = DEG; k >= 0; --k) {
            R& p = (k & 1) ? od : ev;
            const bool low = sizeof(R) == 4 && k == 0;   // float32: c[0]'s low part first
            p = fma(p, v2, __ldg(c + (low ? DEG + 1 : k) * WP + s));
            if (low) p += __ldg(c + s);
        }
        out[s + 1] = fma(od, v, ev);
        out[2 * m - s] = fma(od, -v, ev);
    }
    out[0] = (u == R(0)) ? R(1) : R(0);
}

// the 2m + 1 taps of a job's window for m known at run time only
template <class R>
__device__ __forceinline__ void taps_any(int window, const R* __restrict__ wpoly, int m, R inv_m, R beta, R u, R* out) {
    if (window == WK_BSPLINE) bspline_taps_any<R>(m, u, out);
    else if (wpoly) poly_taps_any<R>(wpoly, m, u, out);
    else for (int s = 0; s <= 2 * m; ++s) out[s] = kb_tap<R>(u, s, m, inv_m, beta);
}

// ----------------------------------------------------------------------------------------
// Work descriptors.  One Job describes one transform (one plan, one in/out pair);
// kernels receive an array of Jobs with the same d and precision and map their
// blocks onto the jobs through prefix sums.
template <class R>
struct Job {
    int d, M, Ms, m;
    int N, T, ntile, P;        // T tile edge, ntile tiles per axis, P = T + 2m + 1 padded edge
    int nitems, window;        // work items (tile, start, count); window kind
    int mode;                  // INFFT_MODE_*
    int S;                     // B_opt slots per axis (2m+2)
    int wexp;                  // the window is below 2^wexp
    int prefetch, fused_fft;   // the plan's tuning of these choices (0 = library default)
    R beta, inv_m;
    const int* perm;           // sorted position -> caller's index
    const uint32_t* cell;      // row-major wrapped base cell of each sorted point
    const R* u;                // N*d fractional offsets M_sigma x - floor(M_sigma x)
    const cx<R>* w;            // weights in sorted order (DCF)
    const cx<R>* coef;         // B_opt coefficients, sorted order, N*S^d (BOPT)
    const int4* items;         // (tile, start, count, 0)
    const int* tile_items;     // ntile^d + 1 prefix of items per tile
    const int* cell_start;     // sorted position of each cell's first point, cells tile-major
    const R* dinv;             // M entries 1/(Ms w^(k)) (per axis); float32: then their low parts
    const R* wpoly;            // wpoly_rows x wpoly_stride(m) window polynomial (Kaiser-Bessel; float32 B-spline) or null
    const float* wpoly_h;      // host copy of the same table (read by the launchers only) or null
    const cx<R>* tw;           // Ms/2 twiddles exp(-2 pi i k / Ms); float32: then their low parts
    cx<R>* padded;             // nitems * P^d
    cx<R>* grid;               // Ms^d
    cx<R>* tmp1;               // FFT intermediates
    cx<R>* tmp2;
    const cx<R>* in;           // adjoint: f (N), forward: fhat (M^d)
    cx<R>* out;                // adjoint: fhat (M^d), forward: f (N)
};

// ----------------------------------------------------------------------------------------
// small helpers
__host__ __device__ __forceinline__ int ipow(int b, int e) {
    int r = 1;
    for (int i = 0; i < e; ++i) r *= b;
    return r;
}

__device__ __forceinline__ int find_job(const int* prefix, int njobs, int idx) {
    // largest j with prefix[j] <= idx (prefix has njobs+1 entries, prefix[0] = 0)
    int lo = 0, hi = njobs;  // invariant prefix[lo] <= idx < prefix[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (prefix[mid] <= idx) lo = mid; else hi = mid;
    }
    return lo;
}

__host__ __device__ __forceinline__ int mod_pos(int a, int n) {
    int r = a % n;
    return r < 0 ? r + n : r;
}

__device__ __forceinline__ int bitrev(int i, int logn) {
    return (int)(__brev((unsigned)i) >> (32 - logn));
}

}  // namespace infft
