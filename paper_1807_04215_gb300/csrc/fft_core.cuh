// Register-resident Stockham FFT used by every transform pass of the library.
//
// A batch of independent length-L transforms ("columns") is processed by one
// thread block. Thread p (0 <= p < P = L / E) of a column holds the E elements
// n = p + P * i (i = 0..E-1) in registers. Each radix-R stage does E / R
// butterflies per thread entirely in registers; between stages the outputs go
// through a shared-memory exchange buffer (Stockham autosort ordering), and
// after the last stage the thread again holds n = p + P * i in natural order,
// so a forward transform can feed an inverse transform without touching
// shared memory (used by the fused spectral-derivative pass).
//
// Sign convention: DIR = +1 computes y[n] = sum_t x[t] e^{+2 pi i n t / L}
// (the backward/synthesis sum of the paper's transform pair, Sec. II.C),
// DIR = -1 the analysis sum with e^{-...}; neither is normalised.
//
// Twiddle factors are read from a table of the N-th roots of unity
// e^{+2 pi i j / N} (FP64 on the host, rounded to FP32) held in shared memory;
// a length-L transform (L divides N) uses every (N / L)-th entry.
#pragma once
#include <cuda_runtime.h>

namespace gridspt {

// ----------------------------------------------------------- complex helpers
// The real and imaginary parts are combined with the packed two-lane FP32
// instructions of sm_100 and later (add/sub/mul/fma .rn .f32x2): each lane is
// rounded exactly as the scalar instruction would round it, so the results are
// those of the scalar forms below, with half the arithmetic instructions.
#ifndef GRIDSPT_PACKED_F32X2
#define GRIDSPT_PACKED_F32X2 1
#endif
#if GRIDSPT_PACKED_F32X2
__device__ __forceinline__ unsigned long long f2u(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 u2f(unsigned long long r) {
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2u(a)), "l"(f2u(b)));
    return u2f(r);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2u(a)), "l"(f2u(b)));
    return u2f(r);
}
__device__ __forceinline__ float2 cscale(float2 a, float s) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2u(a)), "l"(f2u(make_float2(s, s))));
    return u2f(r);
}
// (a.x b.x - a.y b.y, a.x b.y + a.y b.x): t = (a.y b.y, a.y b.x) rounded, then
// fma((a.x, a.x), (b.x, b.y), (-t.x, t.y)), as the scalar form
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    unsigned long long t, r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(f2u(make_float2(a.y, a.y))), "l"(f2u(make_float2(b.y, b.x))));
    const float2 tf = u2f(t);
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r)
        : "l"(f2u(make_float2(a.x, a.x))), "l"(f2u(b)), "l"(f2u(make_float2(-tf.x, tf.y))));
    return u2f(r);
}
#else
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
#endif
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }

// Lane-wise forms used by the pair products of real fields stored as float2
// pairs of cells: (a.x b.x, a.y b.y) and (fma(s, v.x, c.x), fma(s, v.y, c.y)),
// rounded as the scalar instructions.
#if GRIDSPT_PACKED_F32X2
__device__ __forceinline__ float2 lmul(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2u(a)), "l"(f2u(b)));
    return u2f(r);
}
__device__ __forceinline__ float2 lfma(float s, float2 v, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2u(make_float2(s, s))), "l"(f2u(v)), "l"(f2u(c)));
    return u2f(r);
}
#else
__device__ __forceinline__ float2 lmul(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ float2 lfma(float s, float2 v, float2 c) {
    return make_float2(fmaf(s, v.x, c.x), fmaf(s, v.y, c.y));
}
#endif
// multiply by DIR * i
template <int DIR>
__device__ __forceinline__ float2 cmul_i(float2 a) {
    return DIR > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// ------------------------------------------------------- radix schedule (L)
// Power-of-two lengths use E = 8 elements per thread: radix-8 stages and one
// final radix-2 or radix-4 stage. Lengths 3 * 2^a use E = 12 (E = 6 for L = 6):
// one radix-3 stage, then radix-4 stages and possibly one radix-2 stage.
__host__ __device__ constexpr bool fft_has3(int L) { return L % 3 == 0; }
__host__ __device__ constexpr int fft_pow2_part(int L) { return fft_has3(L) ? L / 3 : L; }
__host__ __device__ constexpr int fft_base(int L) { return fft_has3(L) ? 4 : 8; }
__host__ __device__ constexpr int fft_fullb(int m, int b) { return m >= b ? 1 + fft_fullb(m / b, b) : 0; }
__host__ __device__ constexpr int fft_remb(int m, int b) { return m >= b ? fft_remb(m / b, b) : m; }
__host__ __device__ constexpr int fft_nstages(int L) {
    return (fft_has3(L) ? 1 : 0) + fft_fullb(fft_pow2_part(L), fft_base(L)) +
           (fft_remb(fft_pow2_part(L), fft_base(L)) > 1 ? 1 : 0);
}
__host__ __device__ constexpr int fft_radix_p2(int m, int s, int b) {
    return s < fft_fullb(m, b) ? b : fft_remb(m, b);
}
__host__ __device__ constexpr int fft_radix(int L, int s) {
    return fft_has3(L) ? (s == 0 ? 3 : fft_radix_p2(fft_pow2_part(L), s - 1, 4))
                       : fft_radix_p2(L, s, 8);
}
__host__ __device__ constexpr int fft_ls(int L, int s) {  // product of radices before stage s
    return s == 0 ? 1 : fft_ls(L, s - 1) * fft_radix(L, s - 1);
}
__host__ __device__ constexpr int fft_elems(int L) {
    return fft_has3(L) ? (L >= 12 ? 12 : L) : (L >= 8 ? 8 : L);
}

// ------------------------------------------------------------ small DFTs
template <int R, int DIR>
__device__ __forceinline__ void dft_small(float2* v) {
    if constexpr (R == 2) {
        float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (R == 3) {
        const float h = 0.86602540378443864676f;  // sqrt(3) / 2
        float2 s = cadd(v[1], v[2]);
        float2 d = csub(v[1], v[2]);
        float2 m = make_float2(fmaf(-0.5f, s.x, v[0].x), fmaf(-0.5f, s.y, v[0].y));
        float2 r = cscale(cmul_i<DIR>(d), h);
        v[0] = cadd(v[0], s);
        v[1] = cadd(m, r);
        v[2] = csub(m, r);
    } else if constexpr (R == 4) {
        float2 a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
        float2 b0 = cadd(v[1], v[3]), b1 = cmul_i<DIR>(csub(v[1], v[3]));
        v[0] = cadd(a0, b0);
        v[2] = csub(a0, b0);
        v[1] = cadd(a1, b1);
        v[3] = csub(a1, b1);
    } else if constexpr (R == 8) {
        const float r2 = 0.70710678118654752440f;  // 1 / sqrt(2)
        float2 e[4] = {v[0], v[2], v[4], v[6]};
        float2 o[4] = {v[1], v[3], v[5], v[7]};
        dft_small<4, DIR>(e);
        dft_small<4, DIR>(o);
        // o[t] *= w8^t, w8 = (1 + DIR i) / sqrt(2)
        o[1] = cscale(cadd(o[1], cmul_i<DIR>(o[1])), r2);
        o[2] = cmul_i<DIR>(o[2]);
        o[3] = cscale(csub(cmul_i<DIR>(o[3]), o[3]), r2);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            v[t] = cadd(e[t], o[t]);
            v[t + 4] = csub(e[t], o[t]);
        }
    }
}

// ------------------------------------------------------------- one stage
// Shared-memory exchange buffer of one column: element n at col[n * SN].
template <int L, int S, int DIR, int N>
__device__ __forceinline__ void fft_stage(float2 (&x)[fft_elems(L)], int p, float2* col, int SN,
                                          const float2* __restrict__ tw) {
    constexpr int E = fft_elems(L);
    constexpr int P = L / E;
    constexpr int R = fft_radix(L, S);
    constexpr int Ls = fft_ls(L, S);
    constexpr int Q = E / R;              // butterflies per thread
    constexpr int NS = fft_nstages(L);
    constexpr bool last = (S == NS - 1);
    constexpr int TWS = N / (Ls * R);     // table stride for angle t * k / (Ls * R)
    float2 y[E];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float2 v[R];
        const int b = p + q * P;          // butterfly index
        const int k = (Ls == 1) ? 0 : (b % Ls);
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = x[q + t * Q];
        if constexpr (Ls > 1) {
#pragma unroll
            for (int t = 1; t < R; ++t) {
                float2 w = tw[t * k * TWS];  // t * k < Ls * R, so the index is < N
                if (DIR < 0) w.y = -w.y;
                v[t] = cmul(v[t], w);
            }
        }
        dft_small<R, DIR>(v);
        if constexpr (last) {
#pragma unroll
            for (int t = 0; t < R; ++t) y[q + t * Q] = v[t];
        } else {
            const int base = (b / Ls) * Ls * R + k;
#pragma unroll
            for (int t = 0; t < R; ++t) col[(base + t * Ls) * SN] = v[t];
        }
    }
    if constexpr (last) {
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = y[i];
    } else {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = col[(p + P * i) * SN];
        __syncthreads();
    }
}

template <int L, int S, int DIR, int N>
__device__ __forceinline__ void fft_stages(float2 (&x)[fft_elems(L)], int p, float2* col, int SN,
                                           const float2* __restrict__ tw) {
    if constexpr (S < fft_nstages(L)) {
        fft_stage<L, S, DIR, N>(x, p, col, SN, tw);
        fft_stages<L, S + 1, DIR, N>(x, p, col, SN, tw);
    }
}

// Full length-L transform of the column whose exchange buffer is `col`
// (stride SN float2). Every thread of the block must call it the same number
// of times (it contains __syncthreads). tw: shared table of N-th roots.
template <int L, int DIR, int N>
__device__ __forceinline__ void fft_column(float2 (&x)[fft_elems(L)], int p, float2* col, int SN,
                                           const float2* __restrict__ tw) {
    fft_stages<L, 0, DIR, N>(x, p, col, SN, tw);
}


// ------------------------------------------------------- warp-row variant
// The same transform with the P threads of one length-L row on P consecutive
// lanes of one warp (P <= 32 and 32 % P == 0, so a warp holds 32 / P rows), or
// of two warps for P = 64 (L = 512): the stage exchanges go through a buffer of
// those warps, ordered by __syncwarp or a 64-thread named barrier (row_sync),
// so rows never wait on a block-wide barrier. Stage arithmetic and twiddle
// values are those of fft_stage, so results are bitwise equal.
//
// Exchange buffer: element n of a row at xpad(n) = n + n / 16 (one float2 of
// padding per 16). With it every stage's scatter writes and gather reads of a
// warp take the minimum two shared-memory wavefronts for power-of-two L.
//
// Stage twiddles are read from a lane-major table twl[j][p] (conflict-free,
// identical for every row): j enumerates (stage S >= 1, butterfly q, t >= 1).
__device__ __forceinline__ int xpad(int n) { return n + (n >> 4); }

// Barrier of the threads that share a row: the warp, or for P > 32 the P
// threads of named barrier `bar` (1 .. 15, one per team of the block).
template <int P>
__device__ __forceinline__ void row_sync(int bar) {
    if constexpr (P <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;\n" ::"r"(bar), "n"(P) : "memory");
}

template <int L>
__host__ __device__ constexpr int fft_row_tw_count(int S) {   // stage twiddles of stages < S
    return S <= 0 ? 0
                  : fft_row_tw_count<L>(S - 1) +
                        (fft_ls(L, S - 1) > 1 ? (fft_elems(L) / fft_radix(L, S - 1)) * (fft_radix(L, S - 1) - 1) : 0);
}
template <int L>
__host__ __device__ constexpr int fft_row_tw_total() { return fft_row_tw_count<L>(fft_nstages(L)); }

// Fill twl[j * P + p] for p < P from the shared table of N-th roots tw.
template <int L, int N, int S = 0>
__device__ __forceinline__ void fft_row_twiddles(float2* twl, const float2* tw, int p) {
    if constexpr (S < fft_nstages(L)) {
        constexpr int E = fft_elems(L), P = L / E, R = fft_radix(L, S), Ls = fft_ls(L, S), Q = E / R;
        constexpr int TWS = N / (Ls * R);
        if constexpr (Ls > 1) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int k = (p + q * P) % Ls;
#pragma unroll
                for (int t = 1; t < R; ++t)
                    twl[(fft_row_tw_count<L>(S) + q * (R - 1) + (t - 1)) * P + p] = tw[t * k * TWS];
            }
        }
        fft_row_twiddles<L, N, S + 1>(twl, tw, p);
    }
}

template <int L, int S, int DIR>
__device__ __forceinline__ void fft_row_stage(float2 (&x)[fft_elems(L)], int p, float2* row,
                                              const float2* __restrict__ twl, int bar) {
    constexpr int E = fft_elems(L);
    constexpr int P = L / E;
    constexpr int R = fft_radix(L, S);
    constexpr int Ls = fft_ls(L, S);
    constexpr int Q = E / R;
    constexpr bool last = (S == fft_nstages(L) - 1);
    constexpr int J0 = fft_row_tw_count<L>(S);
    float2 y[E];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float2 v[R];
        const int b = p + q * P;
        const int k = (Ls == 1) ? 0 : (b % Ls);
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = x[q + t * Q];
        if constexpr (Ls > 1) {
#pragma unroll
            for (int t = 1; t < R; ++t) {
                float2 w = twl[(J0 + q * (R - 1) + (t - 1)) * P + p];
                if (DIR < 0) w.y = -w.y;
                v[t] = cmul(v[t], w);
            }
        }
        dft_small<R, DIR>(v);
        if constexpr (last) {
#pragma unroll
            for (int t = 0; t < R; ++t) y[q + t * Q] = v[t];
        } else {
            const int base = (b / Ls) * Ls * R + k;
#pragma unroll
            for (int t = 0; t < R; ++t) row[xpad(base + t * Ls)] = v[t];
        }
    }
    if constexpr (last) {
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = y[i];
    } else {
        row_sync<P>(bar);
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = row[xpad(p + P * i)];
        row_sync<P>(bar);
    }
}

template <int L, int S, int DIR>
__device__ __forceinline__ void fft_row_stages(float2 (&x)[fft_elems(L)], int p, float2* row,
                                               const float2* __restrict__ twl, int bar) {
    if constexpr (S < fft_nstages(L)) {
        fft_row_stage<L, S, DIR>(x, p, row, twl, bar);
        fft_row_stages<L, S + 1, DIR>(x, p, row, twl, bar);
    }
}

// Full length-L transform of one row held by P lanes (exchange buffer `row`,
// padded layout). Every lane of the warp (for P > 32: of the team with named
// barrier `bar`) must call it the same number of times.
template <int L, int DIR>
__device__ __forceinline__ void fft_row(float2 (&x)[fft_elems(L)], int p, float2* row,
                                        const float2* __restrict__ twl, int bar = 0) {
    fft_row_stages<L, 0, DIR>(x, p, row, twl, bar);
}


// ------------------------------------------------ column-pass variant (fft_col)
// The column transform of the column passes (colpass, x and y expansion), with
//  * NB = 2 exchange buffers used in turn (stage S writes buffer S % 2): a
//    buffer is rewritten only after a later block barrier that every reader of
//    its previous contents has passed, so each exchange takes one barrier
//    instead of two. A transform with an odd number of exchanges ends with a
//    barrier, so back-to-back transforms keep the alternation safe. NB = 1:
//    one buffer and two barriers per exchange, as fft_column.
//  * a padded exchange layout: element n of a column at col_row(n) * SN, one
//    padding row per 8 rows. The scatter of a radix-8 stage by a warp that
//    spans several butterflies of a narrow tile then hits distinct banks.
//  * the lane-major stage-twiddle table of fft_row, twl[j * P + p] (filled by
//    col_twiddles): the P-indexed twiddle loads of a warp read consecutive
//    entries instead of entries t * k * TWS apart.
// Butterfly arithmetic and twiddle values are those of fft_stage, so results
// are bitwise equal to fft_column.
__host__ __device__ constexpr int col_rows(int L) { return L + L / 8; }
__device__ __forceinline__ int col_row(int n) { return n + (n >> 3); }

// Fill the lane-major stage-twiddle table of a length-L column transform from
// the table of N-th roots (global or shared); threads p < P of the block each
// fill their own entries. The caller orders the table before its first use by
// a block barrier (the first exchange of fft_col has one before any stage
// that reads twiddles).
template <int L, int N>
__device__ __forceinline__ void col_twiddles(float2* twl, const float2* tw) {
    constexpr int P = L / fft_elems(L);
    if (threadIdx.x < P) fft_row_twiddles<L, N>(twl, tw, threadIdx.x);
}

template <int L, int S, int DIR, int NB>
__device__ __forceinline__ void fft_col_stage(float2 (&x)[fft_elems(L)], int p, float2* colA, float2* colB, int SN,
                                              const float2* __restrict__ twl) {
    constexpr int E = fft_elems(L);
    constexpr int P = L / E;
    constexpr int R = fft_radix(L, S);
    constexpr int Ls = fft_ls(L, S);
    constexpr int Q = E / R;
    constexpr bool last = (S == fft_nstages(L) - 1);
    constexpr int J0 = fft_row_tw_count<L>(S);
    float2* col = (NB == 2 && (S & 1)) ? colB : colA;
    float2 y[E];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float2 v[R];
        const int b = p + q * P;
        const int k = (Ls == 1) ? 0 : (b % Ls);
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = x[q + t * Q];
        if constexpr (Ls > 1) {
#pragma unroll
            for (int t = 1; t < R; ++t) {
                float2 w = twl[(J0 + q * (R - 1) + (t - 1)) * P + p];
                if (DIR < 0) w.y = -w.y;
                v[t] = cmul(v[t], w);
            }
        }
        dft_small<R, DIR>(v);
        if constexpr (last) {
#pragma unroll
            for (int t = 0; t < R; ++t) y[q + t * Q] = v[t];
        } else {
            const int base = (b / Ls) * Ls * R + k;
#pragma unroll
            for (int t = 0; t < R; ++t) col[col_row(base + t * Ls) * SN] = v[t];
        }
    }
    if constexpr (last) {
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = y[i];
    } else {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = col[col_row(p + P * i) * SN];
        if constexpr (NB == 1) __syncthreads();
    }
}

template <int L, int S, int DIR, int NB>
__device__ __forceinline__ void fft_col_stages(float2 (&x)[fft_elems(L)], int p, float2* colA, float2* colB, int SN,
                                               const float2* __restrict__ twl) {
    if constexpr (S < fft_nstages(L)) {
        fft_col_stage<L, S, DIR, NB>(x, p, colA, colB, SN, twl);
        fft_col_stages<L, S + 1, DIR, NB>(x, p, colA, colB, SN, twl);
    }
}

// Every thread of the block must call it the same number of times.
template <int L, int DIR, int NB>
__device__ __forceinline__ void fft_col(float2 (&x)[fft_elems(L)], int p, float2* colA, float2* colB, int SN,
                                        const float2* __restrict__ twl) {
    fft_col_stages<L, 0, DIR, NB>(x, p, colA, colB, SN, twl);
    if constexpr (NB == 2 && (fft_nstages(L) - 1) % 2 == 1) __syncthreads();
}

// --------------------------------------------- one-exchange column transform (col2)
// The column transform of the power-of-two lengths L = 128 .. 1024 with its stages
// grouped so that an element crosses shared memory once:
//   L = 128, 256: radix 8, exchange, then 8 x 2 or 8 x 4 inside a thread (P = 8
//     threads a column, E = 16 or 32 elements each);
//   L = 512, 1024: 8 x 8 inside a pair of threads of a warp, exchange, then radix 8
//     or 8 x 2 inside a thread (P = 16 or 32, E = 32). Half of a pair's values
//     change threads by shuffles between its two stages.
// Stages, butterflies and twiddle values are those of fft_column: the results are
// bitwise equal (signs that the pair form moves around are exact).
// The column passes are bound by shared-memory wavefronts, barriers and the warps
// that 64 registers leave (512^3, one exchange per stage: 0.5 wavefronts and 50
// instructions a point); here a thread carries 16 or 32 elements as independent
// chains, most twiddles serve several butterflies, and a transform has two
// barriers. 64 elements a thread (8, exchange, 8 x 8) spills and is slower.
template <int L>
struct Col2 {
    static constexpr bool ok = L >= 128 && L <= 1024 && (L & (L - 1)) == 0;
    static constexpr bool pair = L >= 512;
    static constexpr int P = pair ? L / 32 : 8, E = L / P;
    static constexpr int G = P / 2;                         // pairs of a column
    static constexpr int R2 = pair ? (L == 512 ? 1 : 2) : L / 64;   // radix of the last stage (1: none)
    // shared twiddles. P = 8: per thread p [8] stage 1, [8][R2] stage 2. Pair form: [2][4][8]
    // of the second stage common to all pairs, then per thread 512: [4][8] stage 2;
    // 1024: [2][8] stage 2, [2][8] stage 3. The pitch (two entries more) puts the
    // threads of a warp on other banks.
    static constexpr int PER = pair ? 32 : 8 + 8 * R2, PITCH = PER + 2;
    static constexpr int TW = P * PITCH + (pair ? 64 : 0);        // float2, even
    static constexpr int ROWS = L + L / 64;                       // exchange rows (row of n: n + n / 64)
    static constexpr size_t bytes(int tz) { return sizeof(float2) * (TW + (size_t)ROWS * tz); }
    // element held by thread p in x[i]: in_base(p) + in_step(i) before the transform, p + P i after
    __host__ __device__ static constexpr int in_base(int p) { return pair ? (p >> 1) + 4 * G * (p & 1) : p; }
    __host__ __device__ static constexpr int in_step(int i) { return pair ? G * ((i & 3) + 8 * (i >> 2)) : P * i; }
};
__device__ __forceinline__ int col2_row(int n) { return n + (n >> 6); }
// sign that the pair form leaves on element m of the exchange: -1 where the index
// inside the group of 64, r + 8 t, has r >= 4 and t odd
__device__ __forceinline__ float col2_sign(int m) { return (m & 4) && (m & 8) ? -1.f : 1.f; }

// Fill the table (whole block) from the L-th roots of unity in global memory; the
// pair form ends with a block barrier (the others read it after an exchange's).
template <int L>
__device__ __forceinline__ void col2_table(float2* twl, const float2* __restrict__ twg) {
    using C = Col2<L>;
    if constexpr (!C::pair) {
        for (int j = threadIdx.x; j < C::P * C::PER; j += blockDim.x) {
            const int p = j / C::PER, r = j - p * C::PER, m = r - 8;
            twl[p * C::PITCH + r] = r < 8 ? twg[r * p * (L / 64)] : twg[(m % C::R2) * (p + 8 * (m / C::R2))];
        }
    } else {
        for (int j = threadIdx.x; j < 64; j += blockDim.x) {      // [h][s][own 4, received 4]: w64^(q r)
            const int h = j / 32, r = (j / 8) % 4 + 4 * h, q = (j % 8) ^ (4 * h);
            twl[j] = twg[q * r * (L / 64)];
        }
        for (int j = threadIdx.x; j < C::P * 32; j += blockDim.x) {
            const int p = j / 32, r = j % 32, t = r % 8;
            float2 w;
            float g = 1.f;
            if (L == 512) {                                       // butterfly p + 16 (r / 8)
                const int k = p + 16 * (r / 8);
                w = twg[t * k];
                g = col2_sign(k);
            } else if (r < 16) {                                  // k = p + 32 (r / 8), w512^(t k)
                const int k = p + 32 * (r / 8);
                w = twg[t * k * 2];
                g = col2_sign(k);
            } else {
                w = twg[p + 32 * (r / 8 - 2) + 64 * t];           // w1024^(k + 64 t)
            }
            twl[64 + p * C::PITCH + r] = make_float2(g * w.x, g * w.y);
        }
        __syncthreads();                       // read before the first exchange's barrier
    }
}

template <int DIR>
__device__ __forceinline__ float2 col2_tw(float2 a, float wx, float wy) {   // a w (DIR > 0) or a conj w
    const float y = DIR < 0 ? -wy : wy;
    return make_float2(fmaf(a.x, wx, -a.y * y), fmaf(a.x, y, a.y * wx));
}
// v[t] *= w[t], T0 <= t < R, from consecutive table entries, two per 16-byte load;
// with sign, v[0] is scaled by the real w[0] = +-1
template <int R, int DIR, int T0 = 1, bool SIGN = false>
__device__ __forceinline__ void col2_twiddle(float2* v, const float2* __restrict__ w) {
#pragma unroll
    for (int t = 0; t < R; t += 2) {
        const float4 u = *reinterpret_cast<const float4*>(w + t);
        if (t >= T0) v[t] = col2_tw<DIR>(v[t], u.x, u.y);
        else if (SIGN) v[t] = cscale(v[t], u.x);
        v[t + 1] = col2_tw<DIR>(v[t + 1], u.z, u.w);
    }
}
// dft_small<8> with outputs s and s + 4 exchanged for g = -1. The products with
// 1 / sqrt(2) and the sums after them are single roundings, as the compiler makes
// them in dft_small.
template <int DIR>
__device__ __forceinline__ void dft8_half(float2* v, float g) {
    const float r2 = g * 0.70710678118654752440f;
    float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft_small<4, DIR>(e);
    dft_small<4, DIR>(o);
    o[1] = cadd(o[1], cmul_i<DIR>(o[1]));
    o[2] = cmul_i<DIR>(o[2]);
    o[3] = csub(cmul_i<DIR>(o[3]), o[3]);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float w = t & 1 ? r2 : g;
        v[t] = lfma(w, o[t], e[t]);
        v[t + 4] = lfma(-w, o[t], e[t]);
    }
}

// Thread p of a column holds elements in_base(p) + in_step(i) in x[i] before and
// p + P i after. Every thread of the block calls it the same number of times; the
// TZ columns of a thread index p are consecutive lanes (TZ = 8, 16 or 32). col: exchange
// buffer of the column (element n at col[col2_row(n) * TZ]); the barrier before the
// writes lets the readers of the previous transform finish.
template <int L, int DIR, int TZ>
__device__ __forceinline__ void fft_col2(float2 (&x)[Col2<L>::E], int p, float2* col,
                                         const float2* __restrict__ twl) {
    using C = Col2<L>;
    constexpr int E = C::E, R2 = C::R2;
    if constexpr (!C::pair) {
        // stage 0: butterflies b = p + 8 q, outputs 8 b + t
#pragma unroll
        for (int q = 0; q < E / 8; ++q) {
            float2 v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = x[q + t * (E / 8)];
            dft_small<8, DIR>(v);
#pragma unroll
            for (int t = 0; t < 8; ++t) x[q + t * (E / 8)] = v[t];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < E / 8; ++q)
#pragma unroll
            for (int t = 0; t < 8; ++t) col[col2_row(8 * (p + 8 * q) + t) * TZ] = x[q + t * (E / 8)];
        __syncthreads();
        // stage 1: butterflies b = p + 8 s (k = p), inputs b + u L / 8; outputs of index
        // u feed input s of the last stage's butterfly p + 8 u
        const float2* tw = twl + p * C::PITCH;
        float2 w1[8];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            const float4 w = *reinterpret_cast<const float4*>(tw + u);
            w1[u] = make_float2(w.x, w.y);
            w1[u + 1] = make_float2(w.z, w.w);
        }
#pragma unroll
        for (int s = 0; s < R2; ++s) {
            float2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = col[col2_row(p + 8 * s + u * (L / 8)) * TZ];
#pragma unroll
            for (int u = 1; u < 8; ++u) v[u] = col2_tw<DIR>(v[u], w1[u].x, w1[u].y);
            dft_small<8, DIR>(v);
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u + 8 * s] = v[u];
        }
        // last stage: butterflies p + 8 u, outputs p + 8 (u + 8 t)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            float2 v[R2];
#pragma unroll
            for (int s = 0; s < R2; ++s) v[s] = x[u + 8 * s];
            col2_twiddle<R2, DIR>(v, tw + 8 + u * R2);
            dft_small<R2, DIR>(v);
#pragma unroll
            for (int t = 0; t < R2; ++t) x[u + 8 * t] = v[t];
        }
    } else {
        // stage 0: butterflies g + G q of the pair, this thread q = 4 h + j; output r
        // goes to slot r ^ 4 h, so slots 0 .. 3 are the ones this thread keeps
        const int h = p & 1, g = p >> 1;
        const float sg = h ? -1.f : 1.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = x[j + 4 * t];
            dft8_half<DIR>(v, sg);
#pragma unroll
            for (int t = 0; t < 8; ++t) x[j + 4 * t] = v[t];
        }
#pragma unroll
        for (int i = 16; i < 32; ++i) {                           // slots 4 .. 7 change threads
            x[i].x = __shfl_xor_sync(0xffffffffu, x[i].x, TZ);
            x[i].y = __shfl_xor_sync(0xffffffffu, x[i].y, TZ);
        }
        // stage 1: for r = s + 4 h, inputs q: own 4 h + j, received 4 (1 - h) + j. For h = 1
        // the two halves are exchanged, which leaves (-1)^t on output t (col2_sign)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            float2 v[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v[j] = x[j + 4 * s];
                v[j + 4] = x[j + 4 * (s + 4)];
            }
            col2_twiddle<8, DIR, 0>(v, twl + 32 * h + 8 * s);
            dft_small<8, DIR>(v);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[j + 4 * s] = v[j];
                x[j + 4 * (s + 4)] = v[j + 4];
            }
        }
        __syncthreads();
        float2* wr = col + col2_row(64 * g + 4 * h) * TZ;         // (all rows of a group share the padding)
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int t = 0; t < 8; ++t) wr[(s + 8 * t) * TZ] = t < 4 ? x[t + 4 * s] : x[t - 4 + 4 * (s + 4)];
        __syncthreads();
        const float2* tw = twl + 64 + p * C::PITCH;
        if constexpr (L == 512) {
            // stage 2: butterflies k = p + 16 m, outputs k + 64 t
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                float2 v[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) v[t] = col[(col2_row(64 * t) + p + 16 * m) * TZ];
                col2_twiddle<8, DIR, 1, true>(v, tw + 8 * m);
                dft_small<8, DIR>(v);
#pragma unroll
                for (int t = 0; t < 8; ++t) x[m + 4 * t] = v[t];
            }
        } else {
            // stages 2 and 3 for k = p + 32 j: butterflies k and k + 64, then the pairs
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float2 v[2][8];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
#pragma unroll
                    for (int t = 0; t < 8; ++t) v[hh][t] = col[(col2_row(64 * hh + 128 * t) + p + 32 * j) * TZ];
                    col2_twiddle<8, DIR, 1, true>(v[hh], tw + 8 * j);
                    dft_small<8, DIR>(v[hh]);
                }
#pragma unroll
                for (int t = 0; t < 8; t += 2) {
                    const float4 w = *reinterpret_cast<const float4*>(tw + 16 + 8 * j + t);
                    const float2 a = col2_tw<DIR>(v[1][t], w.x, w.y), b = col2_tw<DIR>(v[1][t + 1], w.z, w.w);
                    x[j + 2 * t] = cadd(v[0][t], a);
                    x[j + 2 * t + 16] = csub(v[0][t], a);
                    x[j + 2 * t + 2] = cadd(v[0][t + 1], b);
                    x[j + 2 * t + 18] = csub(v[0][t + 1], b);
                }
            }
        }
    }
}

}  // namespace gridspt
