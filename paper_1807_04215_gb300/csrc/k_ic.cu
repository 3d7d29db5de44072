// Gaussian initial field delta_1(k) (Sec. II.C step (1); Eq. recursion_n=1).
//
// One warp per row (kx, ky) of the half spectrum float2[N][N][M]. Only modes
// with 0 < |s|^2 <= s2_cut and no Nyquist component draw random numbers; the
// rest are written as zero. The draw is keyed by the canonical member c of the
// pair {s, -s} (c_z > 0, or c_z = 0 and c_y > 0, or c_z = c_y = 0 and c_x > 0),
// so the two members of a pair on the kz = 0 plane get conjugate values.
//
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11), written
// from its published definition: 10 rounds of two 32x32->64-bit multiplies
// with constants 0xD2511F53 and 0xCD9E8D57 and a key bumped by the Weyl
// constants 0x9E3779B9, 0xBB67AE85. Key = seed; counter = (packed c low word,
// packed c high word, 0, 0) with c packed as three 21-bit two's-complement
// fields (x bits 0-20, y 21-41, z 42-62).
//
// Spectrum: P(k) = A k^{n_s} T(k / Gamma)^2 with the BBKS transfer function
// T(q) = ln(1 + 2.34 q)/(2.34 q) [1 + 3.89 q + (16.1 q)^2 + (5.46 q)^3 + (6.71 q)^4]^{-1/4}.
// delta(c) = sqrt(P / L^3) (g1 + i g2) / sqrt(2), g1 + i g2 = sqrt(-2 ln u1) e^{2 pi i u2},
// stored as FP32.
//
// What bounds it: FP64 arithmetic is some 60 times slower than FP32 here (a log
// and a sincospi per mode inside the cut held the FP64 pipe for most of a launch
// whose writes take 80 us), so the two normal deviates are formed in pairs of
// FP32 numbers (value and rounding error; T. J. Dekker, Numer. Math. 18, 1971),
// by table and short polynomial (P. T. P. Tang's table-driven scheme, ACM TOMS 16,
// 1990: ln u = k ln 2 - ln r + log1p(h r - 1), h r - 1 exact in integers; the
// angle-addition theorem; one Newton step for the square root). Their relative
// error is below 1e-12 of the modulus (4e-13: the tail of log1p in FP32), the FP32
// result's rounding 6e-8. Rows are visited plane by plane in a scattered order of kx,
// so planes with modes inside the cut run beside planes that are only written. 512^3: 345 us a realisation with FP64 log,
// sincospi and a 64-bit division per element, 250 with FP64 tables, 93 now.
// The amplitude A is the Simpson sum of gridspt_linear_amplitude, formed on the
// device in FP64 (65537 integrands: 4.6 ms per call on the host, 32 us here).
#include <cstdint>

#include "gridspt_internal.h"

namespace gridspt {

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k.x += W0;
            k.y += W1;
        }
        const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// T_BBKS(q)^2 = (ln(1 + 2.34 q) / (2.34 q))^2 / sqrt(poly)
__device__ __forceinline__ double bbks_t2(double q) {
    if (q <= 0.0) return 1.0;
    const double a = 16.1 * q, b = 5.46 * q, c = 6.71 * q;
    const double poly = 1.0 + 3.89 * q + a * a + b * b * b + (c * c) * (c * c);
    const double l = log1p(2.34 * q) / (2.34 * q);
    return l * l / sqrt(poly);
}

// Pairs (x: value, y: error of it): exact sum and product of two FP32 numbers,
// and the product of two pairs.
__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ float2 two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return make_float2(p, __fmaf_rn(a, b, -p));
}
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
    float2 p = two_prod(a.x, b.x);
    p.y = __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, p.y));
    return p;
}
__device__ __forceinline__ float2 renorm(float h, float l) {          // |l| small against |h|
    const float s = __fadd_rn(h, l);
    return make_float2(s, __fsub_rn(l, __fsub_rn(s, h)));
}

// A pair rounded to FP32. An infinite value's error is infinite or not a number: it is
// clamped (a finite one is below 2^-24 of FP32's largest number), so the value stays.
__device__ __forceinline__ float pair_value(float2 p) { return __fadd_rn(p.x, fminf(fmaxf(p.y, -3e31f), 3e31f)); }

// (g1, g2) = sqrt(-2 ln u1) (cos 2 pi u2, sin 2 pi u2), u = (r + 1/2) 2^-32, as pairs.
// logt[i - 128] = -ln(r_i / 512) with r_i = 131072 / i rounded to an integer;
// cst[j] = (cos, sin)(2 pi j / 512), values then errors.
__device__ __forceinline__ void box_muller(uint32_t r1, uint32_t r2, const float2* __restrict__ logt,
                                           const float4* __restrict__ cst, float2& g1, float2& g2) {
    // u1 = h 2^k, h = w / 2^33 in [1/2, 1)
    const unsigned long long v1 = 2ull * r1 + 1ull;                 // u1 2^33
    const int lz = __clzll((long long)v1);
    const unsigned long long w = v1 << (lz - 31);
    const int i = (int)((w + (1ull << 24)) >> 25);                  // 256 h rounded, 128 .. 256
    const int r = (131072 + i / 2) / i;
    const long long P = (long long)(w * (unsigned)r) - (1ll << 42);   // f = h r / 512 - 1 = P 2^-42, |f| < 2^-7
    const float ph = (float)P, pl = (float)(P - (long long)ph);
    const float fh = ph * 0x1p-42f, fl = pl * 0x1p-42f;
    const float2 L = logt[i - 128];
    const float k = (float)(31 - lz);
    float2 e = two_prod(k, 0.693147182464599609375f);               // k ln 2
    e.y = __fmaf_rn(k, -1.904654323148236e-9f, e.y);
    float2 q = two_prod(fh, fh);                                    // f^2
    q.y = __fmaf_rn(2.f * fh, fl, q.y);
    const float tail = fh * q.x * (0.33333333f + fh * (-0.25f + fh * (0.2f + fh * (-0.16666667f + fh * 0.14285714f))));
    const float2 s1 = two_sum(e.x, L.x), s2 = two_sum(s1.x, fh), s3 = two_sum(s2.x, -0.5f * q.x);
    const float2 ln = renorm(s3.x, ((s1.y + s2.y) + (s3.y + e.y)) + ((L.y + fl) + __fmaf_rn(-0.5f, q.y, tail)));
    const float xh = -2.f * ln.x, xl = -2.f * ln.y;                 // -2 ln u1 > 0
    const float y = rsqrtf(xh), s = __fmul_rn(xh, y);
    const float2 rad = renorm(s, __fmul_rn(__fadd_rn(__fmaf_rn(-s, s, xh), xl), 0.5f * y));
    // u2: nearest of 512 angles, remainder |d| <= 2 pi / 1024
    const unsigned long long v2 = 2ull * r2 + 1ull;                 // u2 2^33
    const int j = (int)((v2 + (1ull << 23)) >> 24);
    const float rem = (float)(int)((long long)v2 - ((long long)j << 24));   // exact, |rem| <= 2^23
    const float4 c4 = cst[j & 511];
    float2 d = two_prod(rem, kIcAngleUnitHi);                       // 2 pi 2^-33 rem
    d.y = __fmaf_rn(rem, kIcAngleUnitLo, d.y);
    float2 d2 = two_prod(d.x, d.x);
    d2.y = __fmaf_rn(2.f * d.x, d.y, d2.y);
    const float2 sd = make_float2(d.x, __fmaf_rn(d.x * d2.x, -0.16666667f + d2.x * 8.3333333e-3f, d.y));
    const float2 c1 = make_float2(-0.5f * d2.x, __fmaf_rn(d2.x * d2.x, 0.041666667f - d2.x * 1.3888889e-3f, -0.5f * d2.y));
    const float2 C = make_float2(c4.x, c4.z), S = make_float2(c4.y, c4.w);
    auto turn = [&](float2 a, float2 b) {                           // a + a c1 + b sd
        const float2 p = pair_mul(b, sd), t = pair_mul(a, c1), u = two_sum(a.x, p.x), v = two_sum(u.x, t.x);
        return renorm(v.x, (u.y + v.y) + (a.y + (p.y + t.y)));
    };
    g1 = pair_mul(rad, turn(C, make_float2(-S.x, -S.y)));
    g2 = pair_mul(rad, turn(S, C));
}

constexpr int kIcWarps = 8;
__global__ void __launch_bounds__(kIcWarps * 32)
k_ic(IcArgs a, int N, int M, int step) {
    __shared__ float4 cst[kIcAngles];
    __shared__ float2 logt[kIcLogs];
    for (int i = threadIdx.x; i < kIcAngles; i += kIcWarps * 32) cst[i] = a.angles[i];
    for (int i = threadIdx.x; i < kIcLogs; i += kIcWarps * 32) logt[i] = a.logs[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, half = N / 2, s2cut = (int)a.s2_cut;
    const int rows = N * N;
    for (int row = blockIdx.x * kIcWarps + (threadIdx.x >> 5); row < rows; row += gridDim.x * kIcWarps) {
        const int plane = row / N, ky = row - plane * N;
        const int kx = (int)((long long)plane * step % N);          // step coprime to N: every kx once
        const int sx = kx < half ? kx : kx - N, sy = ky < half ? ky : ky - N;
        float2* out = a.out + ((long long)kx * N + ky) * M;
        const int left = sx != -half && sy != -half ? s2cut - sx * sx - sy * sy : -1;
        int z0 = 0;                                                 // first kz of the zeros
        if (left >= 0) {
            for (; z0 < M; z0 += 32) {
                const int kz = z0 + lane;
                if (z0 * z0 > left) break;
                if (kz >= M) continue;
                const int s2 = sx * sx + sy * sy + kz * kz;
                float2 v = make_float2(0.f, 0.f);
                if (s2 > 0 && s2 <= s2cut) {
                    const bool canon = kz > 0 || sy > 0 || (sy == 0 && sx > 0);
                    const long long cx = canon ? sx : -sx, cy = canon ? sy : -sy, cz = kz;
                    const unsigned long long packed = ((unsigned long long)cx & 0x1FFFFFull) |
                                                      (((unsigned long long)cy & 0x1FFFFFull) << 21) |
                                                      (((unsigned long long)cz & 0x1FFFFFull) << 42);
                    const uint4 r = philox4x32_10(make_uint4((uint32_t)packed, (uint32_t)(packed >> 32), 0u, 0u),
                                                  make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32)));
                    float2 g1, g2;
                    box_muller(r.x, r.y, logt, cst, g1, g2);
                    const float2 sd = a.table[s2], re = pair_mul(sd, g1), im = pair_mul(sd, g2);
                    const float a1 = pair_value(re), a2 = pair_value(im);
                    v = make_float2(a1, canon ? a2 : -a2);
                }
                out[kz] = v;
            }
        }
        // zeros from z0 (a multiple of 32) to the row's end (M is even for every supported N)
        for (int q = z0 / 2 + lane; q < M / 2; q += 32)
            reinterpret_cast<float4*>(out)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Unnormalised integrand of sigma_8^2 in ln k: k^(3 + n_s) T^2 W(8 k)^2 (W the
// top-hat window), at the same 65537 Simpson points as gridspt_linear_amplitude;
// block b sums its points in a fixed order into part[b].
constexpr int kAmpThreads = 128;
__global__ void __launch_bounds__(kAmpThreads) k_ic_amp(IcArgs a) {
    constexpr int n = 1 << 16;
    const double lo = log(1e-5), hi = log(1e3), step = (hi - lo) / n;
    double s = 0.0;
    for (int i = blockIdx.x * kAmpThreads + threadIdx.x; i <= n; i += kIcParts * kAmpThreads) {
        const double lk = lo + step * i, k = exp(lk), x = 8.0 * k;
        double w;
        if (x < 1e-3) {
            w = 1.0 - x * x / 10.0 + x * x * x * x / 280.0;
        } else {
            double sn, cs;
            sincos(x, &sn, &cs);
            w = 3.0 * (sn - x * cs) / (x * x * x);
        }
        s += exp((3.0 + a.n_s) * lk) * bbks_t2(k * (1.0 / a.gamma)) * w * w * (i == 0 || i == n ? 1.0 : (i & 1 ? 4.0 : 2.0));
    }
    __shared__ double r[kAmpThreads / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kAmpThreads / 32; ++w) t += r[w];
        a.parts[blockIdx.x] = step / 3.0 * t / (2.0 * M_PI * M_PI);
    }
}

// sqrt(P(k) / L^3) / sqrt(2) with P(k) = A k^n_s T_BBKS(k / Gamma)^2 at
// k = k_F sqrt(s2), one thread per integer s2 (FP64, stored as a pair); A = sigma_8^2 over the sum
// of the parts. Small blocks: the FP64 pipes of every SM take part.
__global__ void __launch_bounds__(64) k_ic_table(IcArgs a) {
    double p = 0.0;
    for (int q = threadIdx.x & 31; q < kIcParts; q += 32) p += a.parts[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) p += __shfl_xor_sync(0xffffffffu, p, off);
    const double amp = a.sigma8 * a.sigma8 / p;
    const long long s2 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s2 > a.s2_cut) return;
    double sd = 0.0;
    if (s2 > 0) {
        const double k = a.kF * sqrt((double)s2);
        const double pk = amp * exp(a.n_s * log(k)) * bbks_t2(k / a.gamma);
        sd = sqrt(pk * a.inv_vol) * 0.70710678118654752440;
    }
    const float h = (float)sd;
    a.table[s2] = make_float2(h, (float)(sd - (double)h));   // value and error
}

cudaError_t launch_ic_table(const IcArgs& a, cudaStream_t s) {
    k_ic_amp<<<kIcParts, kAmpThreads, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_ic_table<<<(unsigned)((a.s2_cut + 1 + 63) / 64), 64, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_ic(const Geo& g, const IcArgs& a, cudaStream_t s) {
    const int rows = g.N * g.N, need = (rows + kIcWarps - 1) / kIcWarps;
    // planes in steps of about 0.38 N, coprime to N = 2^a 3^b
    int step = (int)(0.381966 * g.N) | 1;
    while (step % 3 == 0) step += 2;
    k_ic<<<(unsigned)(need < 152 * 8 ? need : 152 * 8), kIcWarps * 32, 0, s>>>(a, g.N, g.M, step);
    return cudaGetLastError();
}

// Self-test: the two deviates of given Philox words, value and error added in FP64.
__global__ void k_normals_selftest(const uint2* __restrict__ words, int n, const float2* __restrict__ logs,
                                   const float4* __restrict__ angles, double2* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float2 g1, g2;
    box_muller(words[i].x, words[i].y, logs, angles, g1, g2);
    out[i] = make_double2((double)g1.x + (double)g1.y, (double)g2.x + (double)g2.y);
}
cudaError_t launch_normals_selftest(const uint2* words, int n, const float2* logs, const float4* angles, double2* out,
                                    cudaStream_t s) {
    k_normals_selftest<<<(n + 255) / 256, 256, 0, s>>>(words, n, logs, angles, out);
    return cudaGetLastError();
}

}  // namespace gridspt
