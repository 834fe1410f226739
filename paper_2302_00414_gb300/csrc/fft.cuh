// FFT passes over lines held in shared memory (Algorithm 2.4 steps 2-3, Algorithm 2.1 steps
// 1-2): the block body shared by the FFT kernels of nfft.cu and the persistent d = 2 adjoint.
#pragma once

#include <algorithm>

#include "jobset.cuh"
#include "spread.cuh"

namespace infft {

// FFT pass along one axis for a batch of lines: Stockham radix-8 (and radix-4) butterflies in
// registers, exchanged through shared memory.  Adjoint direction (FWD = false): forward DFT
// (sign -) of length Ms, keep the M outputs k in I_M, multiply by 1/(Ms w^(k)) of this axis.
// Forward direction (FWD = true): the M inputs of I_M times 1/(Ms w^(k)) are placed at
// k mod Ms, the rest is zero, inverse DFT (sign +).
// A pass sees a tensor (A, n_in, B): lines run along the middle index with stride B.
//
// A line of 512 takes three stages (8, 8, 8): the first reads global memory (or the merged row), the
// last writes it, and shared memory is crossed twice with two barriers, where the radix-2 pairs before
// it crossed it six times.  The two line buffers alternate, so a stage needs one barrier and no registers
// across it.  Fewer twiddle products (two of three stages) also round less: float32 results of the
// 512 x 512 grids are nearer the exact sums.  The passes are bound by load latency and barriers, not by
// bandwidth (event-timed stages, batched d = 2, 64 sets: pass along y 0.034 -> 0.026 ms, merging pass along x
// 0.082 -> 0.080).
// Shared-memory position of element i of a line: one padding slot every 16 elements, so that the
// first stage's stores (stride 8) and the twiddles' strides spread over banks.
__device__ __forceinline__ int skew(int i) { return i + (i >> 4); }

// lines of length n per FFT block: a 16 KB budget of complex elements, at most 32 lines (more,
// smaller blocks hide the passes' load latency better: batched d = 2, n = 512: 64 / 32 / 16 / 8 KB
// of lines per block gave FFT passes of 0.140 / 0.109 / 0.100 / 0.104 ms).  Per job, so that the
// blocks of small grids are as full as those of large ones.
__host__ __device__ inline int fft_lines(int n, int elem) {
    int L = 1;
    while (L < 32 && 2 * L * n * elem <= 16 * 1024) L *= 2;
    return L;
}

// line stride in shared memory: 16 / L (odd for L >= 16) modulo 16 elements, so that the lanes of the
// passes along y and z, which take consecutive lines of the same few elements, meet distinct banks
__host__ __device__ inline int fft_stride(int n, int L) {
    const int want = L < 16 ? 16 / L : 1;
    return n + (n >> 4) + ((want - n - (n >> 4)) & 15);
}

// elements of the line buffers (two: a stage reads one and writes the other) and of the twiddles
__host__ __device__ inline int fft_buf_elems(int n, int L) { return 2 * L * fft_stride(n, L); }
template <class R>
__host__ __device__ inline int fft_tw_elems(int n) { return (sizeof(R) == 4 ? 2 : 1) * ((n >> 1) + (n >> 5) + 1); }

// bytes of a deconvolution factor in shared memory (float32 with its low part)
template <class R>
constexpr size_t fft_dv_bytes() { return 8; }

// threads of an FFT block: one radix-8 butterfly each for the line budget
template <class R>
constexpr int fft_threads() { return sizeof(R) == 4 ? 256 : 128; }

// rows of tiles whose item ranges a merge-on-load block of L lines (grid rows) consults: its
// own one or L / T, and one above and below
__host__ __device__ inline int mrg_tile_rows(int L, int T) { return (L <= T ? 1 : L / T) + 2; }

// a w: float64 with two roundings per part; float32 with w = w + wl to twice the precision and the
// products' errors carried along, so that one rounding is left (the passes wait for loads and barriers,
// the extra multiply-adds are free, and the twiddles were a third of the passes' float32 error)
template <class R>
__device__ __forceinline__ cx<R> mul_w(cx<R> a, cx<R> w, cx<R> wl) {
    if constexpr (sizeof(R) == 8) {
        return mk<R>(fma(a.re, w.re, -(a.im * w.im)), fma(a.re, w.im, a.im * w.re));
    } else {
        const R p = __fmul_rn(a.im, w.im), q = __fmul_rn(a.im, w.re);
        const R ep = fmaf(a.im, w.im, -p), eq = fmaf(a.im, w.re, -q);
        const R lr = fmaf(a.re, wl.re, fmaf(-a.im, wl.im, -ep)), li = fmaf(a.re, wl.im, fmaf(a.im, wl.re, eq));
        const R r = fmaf(a.re, w.re, -p), i = fmaf(a.re, w.im, q);
        return mk<R>(__fadd_rn(r, lr), __fadd_rn(i, li));
    }
}
// v d, in float32 with d's low part
template <class R>
__device__ __forceinline__ cx<R> mul_d(cx<R> v, R d, R dl) {
    if constexpr (sizeof(R) == 8) return scale(v, d);
    else return mk<R>(fmaf(v.re, d, __fmul_rn(v.re, dl)), fmaf(v.im, d, __fmul_rn(v.im, dl)));
}
// a times -i (adjoint direction) or i (forward direction)
template <class R, bool FWD>
__device__ __forceinline__ cx<R> rot(cx<R> a) { return FWD ? mk<R>(-a.im, a.re) : mk<R>(a.im, -a.re); }

// DFT of RX = 4 or 8 values in place, natural order, sign - (FWD = false) or + (FWD = true)
template <class R, bool FWD, int RX>
__device__ __forceinline__ void dft(cx<R>* v) {
    if constexpr (RX == 4) {
        const cx<R> a = add(v[0], v[2]), b = sub(v[0], v[2]), c = add(v[1], v[3]), d = rot<R, FWD>(sub(v[1], v[3]));
        v[0] = add(a, c); v[2] = sub(a, c);
        v[1] = add(b, d); v[3] = sub(b, d);
    } else {
        cx<R> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft<R, FWD, 4>(e);
        dft<R, FWD, 4>(o);
        const R c = R(0.70710678118654752440);
        // o[1] W_8, o[2] W_8^2, o[3] W_8^3 with W_8 = (1 -+ i) c: the factor c goes into the last additions
        const cx<R> r1 = rot<R, FWD>(o[1]), r3 = rot<R, FWD>(o[3]);
        const cx<R> p = add(o[1], r1), q = sub(r3, o[3]), h = rot<R, FWD>(o[2]);
        v[0] = add(e[0], o[0]); v[4] = sub(e[0], o[0]);
        v[2] = add(e[2], h);    v[6] = sub(e[2], h);
        v[1] = mk<R>(fma(p.re, c, e[1].re), fma(p.im, c, e[1].im));
        v[5] = mk<R>(fma(p.re, -c, e[1].re), fma(p.im, -c, e[1].im));
        v[3] = mk<R>(fma(q.re, c, e[3].re), fma(q.im, c, e[3].im));
        v[7] = mk<R>(fma(q.re, -c, e[3].re), fma(q.im, -c, e[3].im));
    }
}

// One Stockham stage of radix RX on L lines of n elements, Ns the product of the radices before it:
// butterfly j of a line takes elements j + r n / RX (through ld), multiplies them by
// exp(-+2 pi i r k / (RX Ns)), k = j mod Ns, and writes its results at (j - k) RX + k + r Ns
// (through st).  L_FAST: consecutive threads take consecutive lines.
template <class R, bool FWD, int RX, int NTH, class Ld, class St>
__device__ __forceinline__ void fft_stage(int L, int logL, int logn, int logNs, bool l_fast, const cx<R>* tws,
                                          const Ld& ld, const St& st) {
    constexpr int LOGR = RX == 8 ? 3 : 2;
    const int n = 1 << logn, logq = logn - LOGR, q = 1 << logq;
    const int twl = skew(n >> 1) + 1;   // the twiddles' low parts (float32)
    for (int e = threadIdx.x; e < (L << logq); e += NTH) {
        const int l = l_fast ? (e & (L - 1)) : (e >> logq), j = l_fast ? (e >> logL) : (e & (q - 1));
        cx<R> v[RX];
        ld(l, j, q, v);
        const int k = j & ((1 << logNs) - 1);
        if (logNs > 0) {
            const int step = k << (logq - logNs);   // of n-th roots of unity
#pragma unroll
            for (int r = 1; r < RX; ++r) {
                const int i = r * step, h = i & ((n >> 1) - 1);
                cx<R> w = tws[skew(h)], wl = sizeof(R) == 4 ? tws[twl + skew(h)] : mk<R>(0, 0);
                if (FWD) { w.im = -w.im; wl.im = -wl.im; }
                const cx<R> x = mul_w(v[r], w, wl);
                v[r] = (i & (n >> 1)) ? mk<R>(-x.re, -x.im) : x;
            }
        }
        dft<R, FWD, RX>(v);
        const int o = ((j - k) << LOGR) + k;
#pragma unroll
        for (int r = 0; r < RX; ++r) st(l, o + (r << logNs), v[r]);
    }
}

// Sum of every padded-tile cell that maps onto grid cell `cidx` (row-major over Ms^D).
template <class R, int D>
__device__ __forceinline__ cx<R> merged_cell(const Job<R>& J, long long cidx) {
    const int Ms = J.Ms, T = J.T, m = J.m, P = J.P, nt = J.ntile;
    int c[D];
    {
        long long rem = cidx;
        for (int t = D - 1; t >= 0; --t) { c[t] = (int)(rem % Ms); rem /= Ms; }
    }
    int cnt[D], tl[D][8], of[D][8];
    for (int t = 0; t < D; ++t) {
        cnt[t] = 0;
        const int own = c[t] / T;
        const int ncand = nt >= 3 ? 3 : nt;
        for (int k = 0; k < ncand; ++k) {
            const int tile = (nt >= 3) ? mod_pos(own - 1 + k, nt) : k;
            int o = mod_pos(c[t] - tile * T + m, Ms);
            for (; o < P && cnt[t] < 8; o += Ms) {
                tl[t][cnt[t]] = tile;
                of[t][cnt[t]] = o;
                ++cnt[t];
            }
        }
    }
    const int cells = ipow(P, D);
    cx<R> acc = mk<R>(0, 0);
    int idx[D];
    for (int t = 0; t < D; ++t) idx[t] = 0;
    bool any = true;
    for (int t = 0; t < D; ++t) any = any && cnt[t] > 0;
    while (any) {
        int tile_lin = 0, pidx = 0;
        for (int t = 0; t < D; ++t) {
            tile_lin = tile_lin * nt + tl[t][idx[t]];
            pidx = pidx * P + of[t][idx[t]];
        }
        int i0 = __ldg(J.tile_items + tile_lin), i1 = __ldg(J.tile_items + tile_lin + 1);
        if (D == 1 && i1 - i0 > 1) {
            // the points that touch padded cell o start at offsets o - S + 1 .. o of the tile: of its items, all of
            // them as long as the first but the last, only those that hold such points (the others' cells are zeros).
            // Float32, M_sigma = 128, 4,000 points: 35.4 us with all of them read (by a kernel of its own), 22.3 here.
            const int S = J.mode == INFFT_MODE_BOPT ? J.S : 2 * m + 1;
            const int a = __ldg(J.cell_start + tile_lin * T + max(0, pidx - S + 1));
            const int b = __ldg(J.cell_start + tile_lin * T + min(T - 1, pidx) + 1);
            const int4 first = __ldg(J.items + i0);
            i1 = b > a ? i0 + (b - 1 - first.y) / first.z + 1 : i0;
            i0 += (a - first.y) / first.z;
        }
#pragma unroll 4
        for (int itm = i0; itm < i1; ++itm) acc = add(acc, J.padded[(size_t)itm * cells + pidx]);
        int t = D - 1;
        while (t >= 0) {
            if (++idx[t] < cnt[t]) break;
            idx[t] = 0;
            --t;
        }
        if (t < 0) break;
    }
    return acc;
}

// the sum of a cell over the items of its (at most four) sources, in order: item k of source q at s_q + k cells.
// All sources' items are one sequence, U loads of it in flight: a polar centre's cell has dozens, and with four
// at a time source by source its block's threads waited for one round of loads after the other (float32, 131,072 polar
// points, m = 6, first FFT pass: 43 us so, 36 with eight of the sequence, 53 with sixteen; float64,
// linogram of 524,288 points: 129 so, 142 with eight, 132 with sixteen; polar 112 with eight, 108 with sixteen).
template <class R>
__device__ __noinline__ cx<R> merge_items(const cx<R>* padded, unsigned cells, size_t s0, size_t s1, size_t s2, size_t s3,
                                          int n0, int n1, int n2, int n3) {
    constexpr int U = sizeof(R) == 4 ? 8 : 16;
    cx<R> acc = mk<R>(0, 0);
    const int p1 = n0, p2 = p1 + n1, p3 = p2 + n2, total = p3 + n3;
    const cx<R>*b0 = padded + s0, *b1 = padded + s1, *b2 = padded + s2, *b3 = padded + s3;
#pragma unroll 1
    for (int k = 0; k < total; k += U) {
        cx<R> v[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int e = k + i;
            const cx<R>* b = e < p1 ? b0 : e < p2 ? b1 : e < p3 ? b2 : b3;
            const unsigned f = (unsigned)(e - (e < p1 ? 0 : e < p2 ? p1 : e < p3 ? p2 : p3));
            v[i] = e < total ? b[(size_t)f * cells] : mk<R>(0, 0);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) acc = add(acc, v[i]);
    }
    return acc;
}

// With MRG (d = 1 and 2 adjoint, pass 0 only) the block's lines are grid rows whose cells are summed
// from the padded tiles as they are loaded: the halo merge of k_merge2d in the same order per
// cell, with no grid written or read in between.  The item ranges of the tiles the block's
// rows draw on are staged in shared memory after the twiddles first.
//
// One block's lines of FFT pass `pass` (block gblk of the pass, global over the JobSet's jobs),
// with the block's dynamic shared memory at smem_raw: the body of k_fft, and the FFT units of the
// persistent d = 2 kernel.  Generic in the block size (a power of two, >= 32).
template <class R, int D, bool FWD, bool MRG, int NTH>
__device__ __forceinline__ void fft_block(const JobSet<R>& js, const int pass, const int gblk,
                                          unsigned char* smem_raw) {
    const int jb = find_job(js.pre_fft[pass], js.njobs, gblk);
    const Job<R>& J = js.job[jb];
    const int lb = gblk - js.pre_fft[pass][jb];
    const int Ms = J.Ms, M = J.M, L = fft_lines(J.Ms, (int)sizeof(cx<R>));
    const int t = FWD ? pass : D - 1 - pass;
    const bool expl = !FWD && js.axA > 0;   // one explicit pass over an (A, Ms, B) tensor
    const long long A = expl ? js.axA : ipow(Ms, t);
    const long long B = expl ? js.axB : ipow(M, D - 1 - t);
    const int MB = expl ? M / js.axblk : M;   // output block along the middle index
    const int n = Ms, logn = 31 - __clz(n);
    const int ns = fft_stride(n, L);
    const long long nlines = A * B;
    const long long q0 = (long long)lb * L;
    const bool lanes_b = (B >= L);  // consecutive lines are consecutive b: coalesce along b

    cx<R>* buf0 = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* buf1 = buf0 + L * ns;
    cx<R>* tws = buf1 + L * ns;     // the n/2 twiddles, skewed, after the lines
    for (int k = threadIdx.x; k < (n >> 1); k += NTH) {
        tws[skew(k)] = J.tw[k];
        if (sizeof(R) == 4) tws[skew(n >> 1) + 1 + skew(k)] = J.tw[(n >> 1) + k];
    }
    // then (merging pass only) the table of tile item ranges, then the M deconvolution factors
    const int nrng = (MRG && D == 2 && pass == 0) ? mrg_tile_rows(L, J.T) * J.ntile : 0;
    int2* rng = reinterpret_cast<int2*>(tws + fft_tw_elems<R>(n));
    R* dvs = reinterpret_cast<R*>(rng + nrng);
    for (int k = threadIdx.x; k < (sizeof(R) == 4 ? 2 : 1) * M; k += NTH) dvs[k] = J.dinv[k];

    const cx<R>* src;
    cx<R>* dst;
    if (expl) {
        src = J.grid;
        dst = J.out;
    } else if (!FWD) {
        src = (pass == 0) ? J.grid : (pass == 1 ? J.tmp1 : J.tmp2);
        dst = (pass == D - 1) ? J.out : (pass == 0 ? J.tmp1 : J.tmp2);
    } else {
        src = (pass == 0) ? J.in : (pass == 1 ? J.tmp1 : J.tmp2);
        dst = (pass == D - 1) ? J.grid : (pass == 0 ? J.tmp1 : J.tmp2);
    }
    const int tid = threadIdx.x;
    const int logL = 31 - __clz(L);   // L is a power of two

    // offsets of each line's first element in the source and destination tensors (line l of
    // the block is (a, b) = divmod(q0 + l, B); element i sits i * B further), or -1 past the end
    __shared__ long long s_in[32], s_out[32];
    if (tid < L) {
        const long long q = q0 + tid;
        long long bi = -1, bo = -1;
        if (q < nlines) {
            // a 32-bit division where the counts allow (a 64-bit one is a long software routine
            // that the whole block would wait for)
            long long a;
            if (nlines <= 0x7fffffffLL && B <= 0x7fffffffLL) a = (long long)((unsigned)q / (unsigned)B);
            else a = q / B;
            const long long b = q - a * B;
            bi = (a * (FWD ? M : n)) * B + b;
            bo = (a * (FWD ? n : MB)) * B + b;
        }
        s_in[tid] = bi;
        s_out[tid] = bo;
    }
    int ty0 = 0, logT = 0, lognt = 0;
    if (MRG && D == 2 && pass == 0) {
        const int T = J.T, nt = J.ntile;
        logT = 31 - __clz(T);
        lognt = 31 - __clz(nt);
        ty0 = (int)(q0 >> logT);
        for (int k = tid; k < nrng; k += NTH) {
            const int tyw = (ty0 - 1 + (k >> lognt)) & (nt - 1), tx = k & (nt - 1);
            const int a = __ldg(J.tile_items + tyw * nt + tx), b = __ldg(J.tile_items + tyw * nt + tx + 1);
            rng[k] = make_int2(a, b - a);   // [tile row][tile] first item, count
        }
    }
    __syncthreads();

    // the merge: every element of the block's rows into buf0, in order.  Thread columns: i = tid + NTH kc
    // for n >= NTH (every line), else i = tid mod n on lines l = tid / n + (NTH / n) k.  The x-sources
    // of a column and the y-sources of a line are found once each; an element then looks up its (at most
    // four) tiles' item ranges.
    if constexpr (MRG && D == 1) {   // one line, every cell from its own and the neighbouring tiles
        for (int i = tid; i < L * n; i += NTH)
            buf0[(i >> logn) * ns + skew(i & (n - 1))] = i < n ? merged_cell<R, 1>(J, i) : mk<R>(0, 0);
        __syncthreads();
    } else if (MRG && pass == 0) {
        const int T = J.T, m = J.m, P = J.P, nt = J.ntile;
        const unsigned cells = (unsigned)(P * P);
        const int ncol = n >= NTH ? n / NTH : 1, dl = n >= NTH ? 1 : NTH / n;
        const int i0 = n >= NTH ? tid : (tid & (n - 1)), l0 = n >= NTH ? 0 : (tid >> logn);
        for (int kc = 0; kc < ncol; ++kc) {
            const int i = i0 + kc * NTH;
            const int c = i & (T - 1), tx = i >> logT;
            int xcol[2], xoff[2], nx = 1;
            xcol[0] = tx; xoff[0] = c + m;
            xcol[1] = 0; xoff[1] = 0;
            if (c + T + m < P) { xcol[1] = (tx - 1) & (nt - 1); xoff[1] = c + T + m; nx = 2; }
            else if (c - T + m >= 0) { xcol[1] = (tx + 1) & (nt - 1); xoff[1] = c - T + m; nx = 2; }
#pragma unroll 2
            for (int l = l0; l < L; l += dl) {
                const long long y = q0 + l;
                cx<R> acc = mk<R>(0, 0);
                if (y < nlines) {
                    const int r = (int)y & (T - 1), trow = (int)(y >> logT) - ty0 + 1;
                    int yrow[2], yoff[2], ny = 1;
                    yrow[0] = trow << lognt; yoff[0] = (r + m) * P;
                    yrow[1] = 0; yoff[1] = 0;
                    if (r + T + m < P) { yrow[1] = (trow - 1) << lognt; yoff[1] = (r + T + m) * P; ny = 2; }
                    else if (r - T + m >= 0) { yrow[1] = (trow + 1) << lognt; yoff[1] = (r - T + m) * P; ny = 2; }
                    // the first item of every source, loaded together; then the sum in
                    // k_merge2d's order (y-source major, x-source minor, items in order)
                    size_t src0[4];
                    int cnt[4];
                    cx<R> v[4];
#pragma unroll
                    for (int a = 0; a < 2; ++a)
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            const int q = 2 * a + b;
                            const bool has = a < ny && b < nx;
                            const int2 g = has ? rng[yrow[a] + xcol[b]] : make_int2(0, 0);
                            cnt[q] = g.y;
                            src0[q] = (size_t)(unsigned)g.x * cells + (unsigned)(yoff[a] + xoff[b]);
                        }
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = cnt[q] > 0 ? J.padded[src0[q]] : mk<R>(0, 0);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (cnt[q] > 0) acc = add(acc, v[q]);
                    // tiles with more points than one item holds (rare; kept out of this loop's registers)
                    if (max(max(cnt[0], cnt[1]), max(cnt[2], cnt[3])) > 1)
                        acc = merge_items<R>(J.padded, cells, src0[0], src0[1], src0[2], src0[3], cnt[0], cnt[1], cnt[2], cnt[3]);
                }
                buf0[l * ns + skew(i)] = acc;
            }
        }
        __syncthreads();
    }
    cx<R>*from = MRG && pass == 0 ? buf0 : buf1, *to = MRG && pass == 0 ? buf1 : buf0;
    // the first stage's inputs: elements j + r q of line l, all loads issued before any is used
    auto ld_in = [&](int l, int j, int q, auto& v) {
        constexpr int RX = sizeof(v) / sizeof(v[0]);
        if (MRG && pass == 0) {
#pragma unroll
            for (int r = 0; r < RX; ++r) v[r] = from[l * ns + skew(j + r * q)];
        } else {
            const long long g0 = s_in[l];
#pragma unroll
            for (int r = 0; r < RX; ++r) {
                int i = j + r * q;
                if (FWD) i = (i + M / 2) & (n - 1);   // coefficient of this bin, if below M
                v[r] = (g0 >= 0 && (!FWD || i < M)) ? src[g0 + (long long)i * B] : mk<R>(0, 0);
            }
            if (FWD) {
#pragma unroll
                for (int r = 0; r < RX; ++r) {
                    const int i = (j + r * q + M / 2) & (n - 1);
                    if (i < M) v[r] = mul_d(v[r], dvs[i], sizeof(R) == 4 ? dvs[M + i] : R(0));
                }
            }
        }
    };
    // a result: bin i of line l
    auto st_out = [&](int l, int i, cx<R> v) {
        const long long g0 = s_out[l];
        if (g0 < 0) return;
        if (FWD) {
            dst[g0 + (long long)i * B] = v;
            return;
        }
        const int k = (i + M / 2) & (n - 1);
        if (k >= M) return;
        // explicit passes: block k / MB of the middle index holds the (A, MB, B) tensor of its indices
        const long long o = expl ? (long long)(k / MB) * A * MB * B + (long long)(k % MB) * B : (long long)k * B;
        dst[g0 + o] = mul_d(v, dvs[k], sizeof(R) == 4 ? dvs[M + k] : R(0));
    };
    auto ld_buf = [&](int l, int j, int q, auto& v) {
        constexpr int RX = sizeof(v) / sizeof(v[0]);
#pragma unroll
        for (int r = 0; r < RX; ++r) v[r] = from[l * ns + skew(j + r * q)];
    };
    auto st_to = [&](int l, int i, cx<R> v) { to[l * ns + skew(i)] = v; };

    // radices: eights, then one or two fours (n = 4^2 or 4: fours only)
    const int nfour = logn % 3 == 0 ? 0 : logn % 3 == 2 ? 1 : 2, neight = (logn - 2 * nfour) / 3;
    auto swap_bufs = [&]() {
        __syncthreads();
        cx<R>* const s = from;
        from = to;
        to = s;
    };
    if (neight > 0) fft_stage<R, FWD, 8, NTH>(L, logL, logn, 0, lanes_b && !(MRG && pass == 0), tws, ld_in, st_to);
    else fft_stage<R, FWD, 4, NTH>(L, logL, logn, 0, lanes_b && !(MRG && pass == 0), tws, ld_in, st_to);
    swap_bufs();
    int logNs = neight > 0 ? 3 : 2;
    while (logNs < logn) {
        const bool eight = logNs < 3 * neight;
        const int next = logNs + (eight ? 3 : 2);
        if (next == logn) {
            if (eight) fft_stage<R, FWD, 8, NTH>(L, logL, logn, logNs, lanes_b, tws, ld_buf, st_out);
            else fft_stage<R, FWD, 4, NTH>(L, logL, logn, logNs, lanes_b, tws, ld_buf, st_out);
            return;
        }
        if (eight) fft_stage<R, FWD, 8, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_to);
        else fft_stage<R, FWD, 4, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_to);
        swap_bufs();
        logNs = next;
    }
    // n = 4 or 8: a single stage
    for (int e = tid; e < L * n; e += NTH) st_out(e >> logn, e & (n - 1), from[(e >> logn) * ns + skew(e & (n - 1))]);
}


// Lines of a circular convolution along the last axis (run_fft_conv): each of the A = Ms^(D-1) lines of M
// values (k in I_M) is zero-padded, transformed with sign +, multiplied by its line of the spectrum,
// transformed back with sign - and cropped, without leaving shared memory (as two passes and a product it crossed
// global memory four times at the full length).  The destination may be the source: a block reads its lines
// before it writes them.
template <class R, int D, int NTH>
__device__ __forceinline__ void fft_conv_block(const JobSet<R>& js, const int lb, unsigned char* smem_raw) {
    const Job<R>& J = js.job[0];
    const int n = J.Ms, M = J.M, L = fft_lines(n, (int)sizeof(cx<R>)), ns = fft_stride(n, L);
    const int logn = 31 - __clz(n), logL = 31 - __clz(L);
    const int nlines = ipow(n, D - 1), q0 = lb * L;
    cx<R>* from = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* to = from + L * ns;
    cx<R>* tws = to + L * ns;
    for (int k = threadIdx.x; k < (n >> 1); k += NTH) {
        tws[skew(k)] = J.tw[k];
        if (sizeof(R) == 4) tws[skew(n >> 1) + 1 + skew(k)] = J.tw[(n >> 1) + k];
    }
    __syncthreads();
    const cx<R>* src = (D == 1 ? J.in : D == 2 ? J.tmp1 : J.tmp2) + (size_t)q0 * M;
    cx<R>* dst = (D == 1 ? J.out : J.tmp1) + (size_t)q0 * M;
    const cx<R>* spec = J.coef + (size_t)q0 * n;
    auto ld_in = [&](int l, int j, int q, auto& v) {
        constexpr int RX = sizeof(v) / sizeof(v[0]);
#pragma unroll
        for (int r = 0; r < RX; ++r) {
            const int i = (j + r * q + M / 2) & (n - 1);
            v[r] = (i < M && q0 + l < nlines) ? src[(size_t)l * M + i] : mk<R>(0, 0);
        }
    };
    auto ld_buf = [&](int l, int j, int q, auto& v) {
        constexpr int RX = sizeof(v) / sizeof(v[0]);
#pragma unroll
        for (int r = 0; r < RX; ++r) v[r] = from[l * ns + skew(j + r * q)];
    };
    auto st_to = [&](int l, int i, cx<R> v) { to[l * ns + skew(i)] = v; };
    auto st_spec = [&](int l, int i, cx<R> v) {
        if (q0 + l < nlines) v = mul(v, spec[(size_t)l * n + i]);
        to[l * ns + skew(i)] = v;
    };
    auto st_out = [&](int l, int i, cx<R> v) {
        const int k = (i + M / 2) & (n - 1);
        if (k < M && q0 + l < nlines) dst[(size_t)l * M + k] = v;
    };
    auto swap_bufs = [&]() {
        __syncthreads();
        cx<R>* const s = from;
        from = to;
        to = s;
    };
    const int nfour = logn % 3 == 0 ? 0 : logn % 3 == 2 ? 1 : 2, neight = (logn - 2 * nfour) / 3;
    // forward; the last stage multiplies by the spectrum as it stores
    int logNs = 0;
    while (logNs < logn) {
        const bool eight = logNs < 3 * neight, first = logNs == 0;
        const int next = logNs + (eight ? 3 : 2);
        const bool end = next == logn;
        if (eight) {
            if (first && end) fft_stage<R, true, 8, NTH>(L, logL, logn, logNs, false, tws, ld_in, st_spec);
            else if (first) fft_stage<R, true, 8, NTH>(L, logL, logn, logNs, false, tws, ld_in, st_to);
            else if (end) fft_stage<R, true, 8, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_spec);
            else fft_stage<R, true, 8, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_to);
        } else {
            if (first && end) fft_stage<R, true, 4, NTH>(L, logL, logn, logNs, false, tws, ld_in, st_spec);
            else if (first) fft_stage<R, true, 4, NTH>(L, logL, logn, logNs, false, tws, ld_in, st_to);
            else if (end) fft_stage<R, true, 4, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_spec);
            else fft_stage<R, true, 4, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_to);
        }
        swap_bufs();
        logNs = next;
    }
    // and back
    logNs = 0;
    while (logNs < logn) {
        const bool eight = logNs < 3 * neight;
        const int next = logNs + (eight ? 3 : 2);
        if (next == logn) {
            if (eight) fft_stage<R, false, 8, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_out);
            else fft_stage<R, false, 4, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_out);
            return;
        }
        if (eight) fft_stage<R, false, 8, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_to);
        else fft_stage<R, false, 4, NTH>(L, logL, logn, logNs, false, tws, ld_buf, st_to);
        swap_bufs();
        logNs = next;
    }
}

// The halo merge of d = 2 folded into the first FFT pass (fft_block with
// MRG), unless INFFT_FFT_MERGE=0 or a job's table of tile item ranges would pass 16 KB: the
// grid is then neither written nor read between the two.  Both forms give bitwise the same
// result.
template <class R>
inline bool merge_on_load_ok(const JobSet<R>& js) {
    if (env_form("INFFT_FFT_MERGE") == 0 || js.axA > 0) return false;
    for (int j = 0; j < js.njobs; ++j) {
        const Job<R>& J = js.job[j];
        const int L = fft_lines(J.Ms, (int)sizeof(cx<R>));
        if ((size_t)mrg_tile_rows(L, J.T) * J.ntile * sizeof(int2) > 16 * 1024) return false;
    }
    return true;
}

// dynamic shared memory of a merging first pass (MRG) over the jobs of js
template <class R>
inline size_t fft_smem_mrg(const JobSet<R>& js) {
    size_t mx = 0;
    for (int j = 0; j < js.njobs; ++j) {
        const Job<R>& J = js.job[j];
        const int n = J.Ms, L = fft_lines(n, (int)sizeof(cx<R>));
        mx = std::max(mx, ((size_t)fft_buf_elems(n, L) + fft_tw_elems<R>(n)) * sizeof(cx<R>) +
                              (size_t)mrg_tile_rows(L, J.T) * J.ntile * sizeof(int2) + (size_t)J.M * fft_dv_bytes<R>());
    }
    return mx;
}

// dynamic shared memory of an FFT pass over the jobs of js: the largest of the jobs' line
// buffers plus twiddles and deconvolution factors
template <class R>
inline size_t fft_smem(const JobSet<R>& js) {
    size_t mx = 0;
    for (int j = 0; j < js.njobs; ++j) {
        const int n = js.job[j].Ms, L = fft_lines(n, (int)sizeof(cx<R>));
        mx = std::max(mx, ((size_t)fft_buf_elems(n, L) + fft_tw_elems<R>(n)) * sizeof(cx<R>) + (size_t)js.job[j].M * fft_dv_bytes<R>());
    }
    return mx;
}

}  // namespace infft
