// Multilayer-perceptron emulator kernels (not part of the GridSPT paper: the
// emulator maps linear-spectrum parameters to binned P-terms).
//
// Network: I -> H -> H -> O, SiLU(z) = z / (1 + e^{-z}) after the two hidden
// layers, linear output. Parameter vector (row-major [in][out] weights):
// W1[I][H], b1[H], W2[H][H], b2[H], W3[H][O], b3[O]. Storage type T of the
// weights and of the saved activations is float or bfloat16; every product is
// accumulated in FP32. Activations saved for the backward pass, per row:
// z1[H], a1[H], z2[H], a2[H] as FP32 (a1, a2 hold T-rounded values).
//
// What bounds these kernels is latency, not arithmetic: a forward pass of 256
// rows is 19 MFLOP over 74 KB of weights. So the rows are spread over the SMs
// (as few as two per block), every weight chunk is copied to shared memory by
// cp.async ahead of its use, and one thread carries a few independent
// accumulators. Each output keeps one FMA chain in the order of k, whatever the
// tile, so results do not depend on the tile chosen.
// Measured (kernel times, bf16, 3 -> 128 -> 128 -> 160, against 8/16-block
// kernels that read the weights from global memory in the chains):
//   forward 256 rows 61 -> 9.5 us, 4096 rows 57 -> 21; backward 256 rows
//   267 -> 19; mse 41 k elements 26 -> 7. One after the other in a graph: forward of 256
//   rows 42.6 -> 7.6 us, 4096 rows 43 -> 18.2, backward 257 -> 12.6 and 501 -> 80. Where
//   the row kernels of before are the faster ones (narrow networks): fwd_rows, mlp_backward.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

#include "fft_core.cuh"
#include "gridspt_internal.h"
#include "pdl.cuh"

namespace gridspt {

namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <typename T> __device__ __forceinline__ float round_t(float v) { return to_f<T>(from_f<T>(v)); }

__device__ __forceinline__ float silu(float z) { return z / (1.f + expf(-z)); }
__device__ __forceinline__ float silu_grad(float z) {
    const float s = 1.f / (1.f + expf(-z));
    return s * (1.f + z * (1.f - s));
}

constexpr int kGradRows = 16;          // rows of one FMA chain of the parameter gradients
constexpr int kWBytes = 49152;         // one of the two weight buffers at most (32-bit 128 x 128 takes two chunks)

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async16b(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(LEFT) : "memory"); }
__device__ __forceinline__ bool aligned_to(const void* p, int bytes) {
    return (reinterpret_cast<unsigned long long>(p) & (bytes - 1)) == 0;
}

// Copy rows x C elements (contiguous in global memory) to shared rows of `pitch`
// elements: 16-byte or 4-byte asynchronous copies where addresses and lengths
// allow, plain loads otherwise (an odd C of bfloat16), eight in flight a thread
// (one at a time: 97 columns to 161, 25 of the 31 us of any batch up to 4096 rows).
template <typename T>
__device__ __noinline__ void stage_plain(T* dst, int pitch, const T* src, int rows, int C, long long src_pitch) {
    const int nt = blockDim.x, dr = nt / C, dj = nt - dr * C;
    int r = threadIdx.x / C, j = threadIdx.x - r * C;
    while (r < rows) {
        T v[8];
        int to[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            to[u] = r < rows ? r * pitch + j : -1;
            if (to[u] >= 0) v[u] = src[r * src_pitch + j];
            r += dr;
            j += dj;
            if (j >= C) {
                j -= C;
                ++r;
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (to[u] >= 0) dst[to[u]] = v[u];
    }
}
template <typename T>
__device__ void stage_rows(T* dst, int pitch, const T* src, int rows, int C, long long src_pitch) {
    constexpr int S = sizeof(T), V = 16 / S, W = 4 / S;
    const bool vec = C % V == 0 && pitch % V == 0 && src_pitch % V == 0 && aligned_to(src, 16);
    if constexpr (W > 1) {
        if (!vec && !(C % W == 0 && pitch % W == 0 && src_pitch % W == 0 && aligned_to(src, 4))) {
            stage_plain(dst, pitch, src, rows, C, src_pitch);
            return;
        }
    }
    const int e = vec ? V : W, nt = blockDim.x, q = C / e, dr = nt / q, dj = nt - dr * q;   // stepping (r, j): no division per copy
    int r = threadIdx.x / q, j = threadIdx.x - r * q;
    while (r < rows) {
        T* d = dst + r * pitch + j * e;
        const T* g = src + r * src_pitch + j * e;
        if (vec) cp_async16b(d, g);
        else cp_async4(d, g);
        r += dr;
        j += dj;
        if (j >= q) {
            j -= q;
            ++r;
        }
    }
}

// One FMA step of RT rows (pairs): acc[r] += in[r] * w, each lane rounded as fmaf.
template <int RT>
__device__ __forceinline__ void fma_rows(float2 (&acc)[RT / 2], const float* in, float w) {
    if constexpr (RT % 4 == 0) {
#pragma unroll
        for (int j = 0; j < RT / 4; ++j) {
            const float4 v = *reinterpret_cast<const float4*>(in + 4 * j);
            acc[2 * j] = lfma(w, make_float2(v.x, v.y), acc[2 * j]);
            acc[2 * j + 1] = lfma(w, make_float2(v.z, v.w), acc[2 * j + 1]);
        }
    } else {
        acc[0] = lfma(w, *reinterpret_cast<const float2*>(in), acc[0]);
    }
}

// Forward tiles: R rows per block, RT rows x CT columns per thread. A block has one
// thread per such piece of the widest layer (at most 1024).
template <int R> struct FwdTile;
template <> struct FwdTile<2> { static constexpr int RT = 2, CT = 1; };
template <> struct FwdTile<8> { static constexpr int RT = 4, CT = 1; };
template <> struct FwdTile<32> { static constexpr int RT = 4, CT = 2; };
// row pitch of a transposed activation [k][R]: 16-byte rows, and tasks that write
// neighbouring columns spread over the banks
template <int R> __host__ __device__ constexpr int row_pitch() { return R == 2 ? 2 : R + 4; }
__host__ __device__ constexpr int even(int n) { return (n + 1) & ~1; }
// Weight chunks of the forward pass: k rows of K at once, elements of a row in shared memory.
template <typename T>
__host__ __device__ constexpr int fwd_chunk(int K, int C) {
    const int fit = kWBytes / (even(C) * (int)sizeof(T));
    return K < fit ? K : fit;
}
template <typename T>
__host__ __device__ constexpr int fwd_pitch(int C) { return C % (16 / (int)sizeof(T)) == 0 ? C : even(C); }

}  // namespace

// y = net(x), activations saved. Activations are held transposed ([k][row]) in
// shared memory, so one 8- or 16-byte load feeds several rows; the weights pass
// through two buffers in chunks of whole k rows, the next chunk (or the next
// layer's first) in flight while one is used.
template <typename T, int R>
__global__ void __launch_bounds__(256 / FwdTile<R>::CT * (R / FwdTile<R>::RT))
k_mlp_forward(const float* __restrict__ x, int B, int I, int H, int O, const T* __restrict__ theta,
              float* __restrict__ y, float* __restrict__ act, int wbytes) {
    pdl_wait();
    pdl_fresh(x);
    pdl_fresh(theta);
    constexpr int RT = FwdTile<R>::RT, CT = FwdTile<R>::CT, RP = row_pitch<R>(), G = R / RT;
    extern __shared__ __align__(16) char smraw[];
    T* wb[2] = {reinterpret_cast<T*>(smraw), reinterpret_cast<T*>(smraw + wbytes)};
    float* hin = reinterpret_cast<float*>(smraw + 2 * wbytes);     // [max(I, H)][RP], input of the layer
    float* hout = hin + (H > I ? H : I) * RP;                      // [H][RP]
    float* bs = hout + H * RP;                                     // b1[H], b2[H], b3[O]
    const T* W1 = theta;
    const T* W2 = W1 + (long long)I * H + H;
    const T* W3 = W2 + (long long)H * H + H;
    const int r0 = blockIdx.x * R;
    // chunk s of the weights in order of use: layer, first k, number of k rows
    auto layer_w = [&](int l) { return l == 0 ? W1 : l == 1 ? W2 : W3; };
    auto layer_c = [&](int l) { return l == 2 ? O : H; };
    auto layer_k = [&](int l) { return l == 0 ? I : H; };
    auto chunk_k = [&](int l) { return fwd_chunk<T>(layer_k(l), layer_c(l)); };
    const bool pairs = O % 2 == 0 && aligned_to(y, 8);
    int nl = 0, nk = 0, nbuf = 0;                                  // next chunk to issue
    auto issue = [&]() {
        if (nl < 3) {
            const int C = layer_c(nl), kc = chunk_k(nl), left = layer_k(nl) - nk, n = left < kc ? left : kc;
            stage_rows(wb[nbuf], fwd_pitch<T>(C), layer_w(nl) + (long long)nk * C, n, C, C);
            nk += n;
            if (nk == layer_k(nl)) { nk = 0; ++nl; }
            nbuf ^= 1;
        }
        cp_commit();                                               // (an empty group past the end)
    };
    issue();
    issue();
    for (int i = threadIdx.x; i < R * I; i += blockDim.x) {
        const int r = i / I, k = i - r * I;
        hin[k * RP + r] = r0 + r < B ? x[(long long)(r0 + r) * I + k] : 1.f;   // (0 / n: the division's slow path)
    }
    for (int i = threadIdx.x; i < 2 * H + O; i += blockDim.x)
        bs[i] = to_f<T>(i < H ? W1[(long long)I * H + i] : i < 2 * H ? W2[(long long)H * H + i - H]
                                                                     : W3[(long long)H * O + i - 2 * H]);
    __syncthreads();
    int buf = 0;
    for (int l = 0; l < 3; ++l) {
        const int K = layer_k(l), C = layer_c(l), kc = chunk_k(l);
        const int CP = fwd_pitch<T>(C);
        const int nc = (C + CT - 1) / CT, ntask = nc * G;         // a warp's tasks: neighbouring columns, one row group
        const float* bias = bs + l * H;
        float2 acc[CT][RT / 2];
        const int t = threadIdx.x, ct = (t % nc) * CT, rt = (t / nc) * RT;
#pragma unroll
        for (int q = 0; q < CT; ++q) {
            const float b = t < ntask && ct + q < C ? bias[ct + q] : 0.f;
#pragma unroll
            for (int j = 0; j < RT / 2; ++j) acc[q][j] = make_float2(b, b);
        }
        for (int k0 = 0; k0 < K; k0 += kc) {
            const int n = K - k0 < kc ? K - k0 : kc;
            cp_wait<1>();
            __syncthreads();                                       // this chunk and the layer's input are in place
            if (t < ntask) {
                const T* w = wb[buf] + ct;
                const float* in = hin + k0 * RP + rt;
#pragma unroll 8
                for (int k = 0; k < n; ++k, w += CP, in += RP) {
                    if constexpr (CT == 1) {
                        fma_rows<RT>(acc[0], in, to_f<T>(*w));
                    } else if constexpr (sizeof(T) == 2) {         // CP is even: two neighbouring columns
                        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(w);
                        fma_rows<RT>(acc[0], in, __low2float(v));
                        fma_rows<RT>(acc[CT - 1], in, __high2float(v));
                    } else {
                        const float2 v = *reinterpret_cast<const float2*>(w);
                        fma_rows<RT>(acc[0], in, v.x);
                        fma_rows<RT>(acc[CT - 1], in, v.y);
                    }
                }
            }
            __syncthreads();                                       // the buffer (and, at the end, hin) is free
            issue();
            buf ^= 1;
        }
        if (t < ntask && CT == 2 && l == 2 && pairs) {             // both columns of a row in one store
#pragma unroll
            for (int j = 0; j < RT; ++j)
                if (r0 + rt + j < B)
                    *reinterpret_cast<float2*>(y + (long long)(r0 + rt + j) * O + ct) =
                        (j & 1) ? make_float2(acc[0][j / 2].y, acc[CT - 1][j / 2].y)
                                : make_float2(acc[0][j / 2].x, acc[CT - 1][j / 2].x);
        } else if (t < ntask) {
#pragma unroll
            for (int q = 0; q < CT; ++q) {
                const int c = ct + q;
                if (c >= C) continue;
                float a[RT];
#pragma unroll
                for (int j = 0; j < RT; ++j) {
                    const int row = r0 + rt + j;
                    const float z = (j & 1) ? acc[q][j / 2].y : acc[q][j / 2].x;
                    if (l == 2) {
                        if (row < B) y[(long long)row * O + c] = z;
                    } else {
                        a[j] = round_t<T>(silu(z));
                        if (act && row < B) {
                            act[(long long)row * 4 * H + 2 * l * H + c] = z;
                            act[(long long)row * 4 * H + (2 * l + 1) * H + c] = a[j];
                        }
                    }
                }
                if (l < 2) {
                    if constexpr (RT % 4 == 0) {
#pragma unroll
                        for (int j = 0; j < RT; j += 4)
                            *reinterpret_cast<float4*>(hout + c * RP + rt + j) = make_float4(a[j], a[j + 1], a[j + 2], a[j + 3]);
                    } else {
                        *reinterpret_cast<float2*>(hout + c * RP + rt) = make_float2(a[0], a[1]);
                    }
                }
            }
        }
        float* sw = hin;
        hin = hout;
        hout = sw;
    }
}

// The network for 32 rows per block, the weights read from global memory in the
// chains (same chains): a block of 256 threads and a few kilobytes, so many share an SM.
constexpr int kDenseRows = 32;
template <typename T>
__device__ void dense(const float* __restrict__ in, int K, const T* __restrict__ W, const T* __restrict__ b, int C,
                      float* __restrict__ out) {
    constexpr int RG = kDenseRows / 16;
    for (int w = threadIdx.x; w < C * RG; w += blockDim.x) {       // one column of 16 rows
        const int c = w % C, g = w / C;
        float acc[16];
        const float bc = to_f<T>(b[c]);
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[j] = bc;
        for (int k = 0; k < K; ++k) {
            const float wk = to_f<T>(W[(long long)k * C + c]);
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[j] = fmaf(in[(g * 16 + j) * K + k], wk, acc[j]);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) out[(g * 16 + j) * C + c] = acc[j];
    }
}
template <typename T>
__global__ void __launch_bounds__(256)
k_mlp_forward_rows(const float* __restrict__ x, int B, int I, int H, int O, const T* __restrict__ theta,
                   float* __restrict__ y, float* __restrict__ act) {
    constexpr int R = kDenseRows;
    extern __shared__ float smf[];
    float* in = smf;                                               // R x max(I, H)
    float* out = in + R * (I > H ? I : H);                         // R x max(H, O)
    const int r0 = blockIdx.x * R;
    for (int i = threadIdx.x; i < R * I; i += blockDim.x)
        in[i] = r0 + i / I < B ? x[(long long)r0 * I + i] : 0.f;
    __syncthreads();
    const T* W = theta;
    for (int l = 0; l < 3; ++l) {
        const int K = l ? H : I, C = l == 2 ? O : H;
        dense<T>(in, K, W, W + (long long)K * C, C, out);
        W += (long long)K * C + C;
        __syncthreads();
        for (int i = threadIdx.x; i < R * C; i += blockDim.x) {
            const int r = i / C, c = i - r * C;
            const bool on = r0 + r < B;
            if (l == 2) {
                if (on) y[(long long)r0 * O + i] = out[i];
            } else {
                const float z = out[i], a = round_t<T>(silu(z));
                if (act && on) {
                    act[(long long)(r0 + r) * 4 * H + 2 * l * H + c] = z;
                    act[(long long)(r0 + r) * 4 * H + (2 * l + 1) * H + c] = a;
                }
                in[i] = a;
            }
        }
        __syncthreads();
    }
}

// Deltas of the hidden layers for R rows per block, d2 = (dy W3^T) silu'(z2) and
// d1 = (d2 W2^T) silu'(z1), to [row][H] scratch. The weights' rows are staged
// with an odd pitch in 4-byte words, so the threads of a warp (one hidden unit
// each) read distinct banks; the chain of an output runs over the columns in
// order, in chunks where a row block does not fit a buffer.
// Columns per chunk: an even number, pitch = columns + one or two words (odd in words).
template <typename T>
__host__ __device__ constexpr int delta_cols(int all, int H) {
    constexpr int W = 4 / (int)sizeof(T);
    const int n = (kWBytes / (H * (int)sizeof(T)) - 2 * W - 2) & ~(2 * W - 1);
    return all < n ? all : n;
}
template <typename T>
__host__ __device__ constexpr int delta_pitch(int n) {             // elements; odd in 4-byte words
    constexpr int W = 4 / (int)sizeof(T);
    return (((n + W - 1) / W) | 1) * W;
}
template <typename T, int R>
__global__ void __launch_bounds__(R == 2 ? 256 : 512)
k_mlp_delta(int B, int I, int H, int O, const T* __restrict__ theta, const float* __restrict__ act,
            const float* __restrict__ dy, float* __restrict__ d2, float* __restrict__ d1, int wbytes, int early) {
    pdl_wait();
    if (early) pdl_release();
    pdl_fresh(theta);
    pdl_fresh(act);
    pdl_fresh(dy);
    constexpr int RT = R == 2 ? 2 : 4, G = R / RT, RP = row_pitch<R>();
    extern __shared__ __align__(16) char smraw[];
    T* wb[2] = {reinterpret_cast<T*>(smraw), reinterpret_cast<T*>(smraw + wbytes)};
    float* din = reinterpret_cast<float*>(smraw + 2 * wbytes);     // [max(O, H)][RP]
    float* dmid = din + (O > H ? O : H) * RP;                      // [H][RP]
    const T* W2 = theta + (long long)I * H + H;
    const T* W3 = W2 + (long long)H * H + H;
    const int r0 = blockIdx.x * R;
    auto cols = [&](int l) { return delta_cols<T>(l ? H : O, H); };
    int nl = 0, nk = 0, nbuf = 0;
    auto issue = [&]() {
        if (nl < 2) {
            const int all = nl ? H : O, kc = cols(nl), n = all - nk < kc ? all - nk : kc;
            stage_rows(wb[nbuf], delta_pitch<T>(kc), (nl ? W2 : W3) + nk, H, n, (long long)all);
            nk += n;
            if (nk == all) { nk = 0; ++nl; }
            nbuf ^= 1;
        }
        cp_commit();
    };
    issue();
    issue();
    for (int i = threadIdx.x; i < R * O; i += blockDim.x) {
        const int r = i / O, o = i - r * O;
        din[o * RP + r] = r0 + r < B ? dy[(long long)(r0 + r) * O + o] : 0.f;
    }
    int buf = 0;
    for (int l = 0; l < 2; ++l) {
        const int K = l ? H : O, kc = cols(l), WP = delta_pitch<T>(kc);
        const int h = threadIdx.x % H, rt = (threadIdx.x / H) * RT;
        const bool on = threadIdx.x < H * G;
        float2 acc[RT / 2];
        float z[RT];                                               // read before the chain hides their latency
#pragma unroll
        for (int j = 0; j < RT; ++j) {
            const int row = r0 + rt + j;
            z[j] = on && row < B ? act[(long long)row * 4 * H + (l ? 0 : 2) * H + h] : 0.f;
            if (j % 2 == 0) acc[j / 2] = make_float2(0.f, 0.f);
        }
        for (int k0 = 0; k0 < K; k0 += kc) {
            const int n = K - k0 < kc ? K - k0 : kc;
            cp_wait<1>();
            __syncthreads();
            if (on) {
                const float* in = (l ? dmid : din) + k0 * RP + rt;
                const T* w = wb[buf] + h * WP;
                int k = 0;
                if constexpr (sizeof(T) == 2) {
#pragma unroll 4
                    for (; k + 1 < n; k += 2) {
                        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(w + k);
                        fma_rows<RT>(acc, in + k * RP, __low2float(v));
                        fma_rows<RT>(acc, in + (k + 1) * RP, __high2float(v));
                    }
                }
#pragma unroll 8
                for (; k < n; ++k) fma_rows<RT>(acc, in + k * RP, to_f<T>(w[k]));
            }
            __syncthreads();
            issue();
            buf ^= 1;
        }
        if (on) {
#pragma unroll
            for (int j = 0; j < RT; ++j) {
                const int row = r0 + rt + j;
                const float s = (j & 1) ? acc[j / 2].y : acc[j / 2].x;
                float d = 0.f;
                if (row < B) {
                    d = s * silu_grad(z[j]);
                    (l ? d1 : d2)[(long long)row * H + h] = d;
                }
                if (l == 0) dmid[h * RP + rt + j] = d;
            }
        }
    }
}

// Parameter gradients as 16 x 16 tiles of the three products (rows contracted):
// W3: a2^T dy, W2: a1^T d2, W1: x^T d1; one element a thread, the next 64 rows
// loaded into registers while the current ones are summed. Rows are summed in
// chains of 16, the chains added in row order; tiles of the first k rows add the bias
// sums. blockIdx.y: a part of `per` rows, to grad + blockIdx.y * np.
constexpr int kGT = 16, kGChunk = 64;
__global__ void __launch_bounds__(kGT * kGT)
k_mlp_grad(const float* __restrict__ x, int B, int per, int I, int H, int O, const float* __restrict__ act,
           const float* __restrict__ dy, const float* __restrict__ d2, const float* __restrict__ d1,
           float* __restrict__ grad, long long np) {
    pdl_wait();
    pdl_fresh(x);
    pdl_fresh(act);
    pdl_fresh(dy);
    pdl_fresh(d2);
    pdl_fresh(d1);
    const int row0 = blockIdx.y * per, rows = B - row0 < per ? B - row0 : per;
    grad += blockIdx.y * np;
    constexpr int PER = kGChunk / kGT;
    __shared__ float ls[2][kGChunk][kGT], rs[2][kGChunk][kGT];
    const int th = (H + kGT - 1) / kGT, to = (O + kGT - 1) / kGT;
    int b = blockIdx.x, layer, kt, nt;
    if (b < th * to) { layer = 2; kt = b / to; nt = b % to; }
    else if ((b -= th * to) < th * th) { layer = 1; kt = b / th; nt = b % th; }
    else { layer = 0; kt = 0; nt = b - th * th; }
    const int K = layer == 0 ? I : H, C = layer == 2 ? O : H;
    float* gw = grad + (layer == 0 ? 0 : layer == 1 ? (long long)I * H + H : (long long)I * H + 2 * H + (long long)H * H);
    float* gb = gw + (long long)K * C;
    const int tk = threadIdx.x / kGT, tn = threadIdx.x % kGT, k = kt * kGT + tk, n = nt * kGT + tn;
    // this thread loads rows tk + 16 q of the chunk: left column lk, right column n
    const int lk = kt * kGT + tn;
    const bool lok = lk < K, rok = n < C, live = k < K && rok, bias = kt == 0 && tk == 0 && rok;
    const int lp = layer == 0 ? I : 4 * H, rp = C;
    const float* left = (layer == 0 ? x : act + (layer == 1 ? H : 3 * H)) + (long long)(row0 + tk) * lp + lk;
    const float* right = (layer == 2 ? dy : layer == 1 ? d2 : d1) + (long long)(row0 + tk) * rp + n;
    float lv[PER], rv[PER];
    auto load = [&](int c0) {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int r = c0 + q * kGT;
            lv[q] = lok && r + tk < rows ? left[(long long)r * lp] : 0.f;
            rv[q] = rok && r + tk < rows ? right[(long long)r * rp] : 0.f;
        }
    };
    float tot = 0.f, tb = 0.f;
    load(0);
    int buf = 0;
    for (int c0 = 0; c0 < rows; c0 += kGChunk) {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            ls[buf][q * kGT + tk][tn] = lv[q];
            rs[buf][q * kGT + tk][tn] = rv[q];
        }
        __syncthreads();                       // (the other buffer's readers passed the previous barrier's chunk)
        if (c0 + kGChunk < rows) load(c0 + kGChunk);
        auto chain = [&](int g) {
            float s = 0.f, sb = 0.f;
#pragma unroll
            for (int r = 0; r < kGradRows; ++r) {
                const float d = rs[buf][g + r][tn];
                s = fmaf(ls[buf][g + r][tk], d, s);
                sb += d;
            }
            tot += s;
            tb += sb;
        };
        if (c0 + kGChunk <= rows) {            // four chains side by side
#pragma unroll
            for (int g = 0; g < kGChunk; g += kGradRows) chain(g);
        } else {
#pragma unroll 1
            for (int g = 0; c0 + g < rows; g += kGradRows) chain(g);
        }
        buf ^= 1;
    }
    if (live) gw[(long long)k * C + n] = tot;
    if (bias) gb[n] = tb;
}

// Backward of sum(dy * y) for kGradRows rows in one block, the deltas in shared memory:
// the block's gradient (one chain, parameter layout) to part + blockIdx.x * np. For
// networks whose workspace does not hold the deltas of the batch (I + H + O below about 30),
// and for H, O <= 16 between 64 and 1024 rows (3 -> 16 -> 16 -> 16, 256 rows: 6.2 against 7.4 us).
template <typename T>
__global__ void __launch_bounds__(256)
k_mlp_backward_rows(const float* __restrict__ x, int B, int I, int H, int O, const T* __restrict__ theta,
               const float* __restrict__ act, const float* __restrict__ dy, float* __restrict__ part) {
    constexpr int R = kGradRows;
    extern __shared__ float sm[];
    float* xs = sm;              // R x I
    float* z1 = xs + R * I;      // R x H
    float* a1 = z1 + R * H;
    float* z2 = a1 + R * H;
    float* a2 = z2 + R * H;
    float* d3 = a2 + R * H;      // R x O
    float* d2 = d3 + R * O;      // R x H
    float* d1 = d2 + R * H;      // R x H
    const T* W2 = theta + I * H + H;
    const T* W3 = W2 + H * H + H;
    const long long np = (long long)I * H + H + (long long)H * H + H + (long long)H * O + O;
    float* g = part + blockIdx.x * np;
    float* gW1 = g;
    float* gb1 = gW1 + I * H;
    float* gW2 = gb1 + H;
    float* gb2 = gW2 + H * H;
    float* gW3 = gb2 + H;
    float* gb3 = gW3 + H * O;
    const int r0 = blockIdx.x * R;
    for (int i = threadIdx.x; i < R * I; i += blockDim.x) {
        const int r = i / I;
        xs[i] = r0 + r < B ? x[(long long)(r0 + r) * I + (i % I)] : 0.f;
    }
    for (int i = threadIdx.x; i < R * H; i += blockDim.x) {
        const int r = i / H, c = i % H;
        const bool ok = r0 + r < B;
        const float* ar = act + (long long)(r0 + r) * 4 * H;
        z1[i] = ok ? ar[c] : 0.f;
        a1[i] = ok ? ar[H + c] : 0.f;
        z2[i] = ok ? ar[2 * H + c] : 0.f;
        a2[i] = ok ? ar[3 * H + c] : 0.f;
    }
    for (int i = threadIdx.x; i < R * O; i += blockDim.x) {
        const int r = i / O;
        d3[i] = r0 + r < B ? dy[(long long)(r0 + r) * O + (i % O)] : 0.f;
    }
    __syncthreads();
    // output layer
    for (int w = threadIdx.x; w < H * O; w += blockDim.x) {
        const int h = w / O, o = w % O;
        float s = 0.f;
        for (int r = 0; r < R; ++r) s = fmaf(a2[r * H + h], d3[r * O + o], s);
        gW3[w] = s;
    }
    for (int o = threadIdx.x; o < O; o += blockDim.x) {
        float s = 0.f;
        for (int r = 0; r < R; ++r) s += d3[r * O + o];
        gb3[o] = s;
    }
    for (int w = threadIdx.x; w < R * H; w += blockDim.x) {
        const int r = w / H, h = w % H;
        float s = 0.f;
        for (int o = 0; o < O; ++o) s = fmaf(d3[r * O + o], to_f<T>(W3[(long long)h * O + o]), s);
        d2[w] = s * silu_grad(z2[w]);
    }
    __syncthreads();
    // second hidden layer
    for (int w = threadIdx.x; w < H * H; w += blockDim.x) {
        const int k = w / H, h = w % H;
        float s = 0.f;
        for (int r = 0; r < R; ++r) s = fmaf(a1[r * H + k], d2[r * H + h], s);
        gW2[w] = s;
    }
    for (int h = threadIdx.x; h < H; h += blockDim.x) {
        float s = 0.f;
        for (int r = 0; r < R; ++r) s += d2[r * H + h];
        gb2[h] = s;
    }
    for (int w = threadIdx.x; w < R * H; w += blockDim.x) {
        const int r = w / H, k = w % H;
        float s = 0.f;
        for (int h = 0; h < H; ++h) s = fmaf(d2[r * H + h], to_f<T>(W2[(long long)k * H + h]), s);
        d1[w] = s * silu_grad(z1[w]);
    }
    __syncthreads();
    // first layer
    for (int w = threadIdx.x; w < I * H; w += blockDim.x) {
        const int i = w / H, h = w % H;
        float s = 0.f;
        for (int r = 0; r < R; ++r) s = fmaf(xs[r * I + i], d1[r * H + h], s);
        gW1[w] = s;
    }
    for (int h = threadIdx.x; h < H; h += blockDim.x) {
        float s = 0.f;
        for (int r = 0; r < R; ++r) s += d1[r * H + h];
        gb1[h] = s;
    }
}

// grad[i] = sum (in order) of part[b][i]
__global__ void k_mlp_reduce(const float* __restrict__ part, int nblocks, long long np, float* __restrict__ grad) {
    pdl_wait();
    pdl_fresh(part);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (long long)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int b = 0; b < nblocks; ++b) s += part[b * np + i];
        grad[i] = s;
    }
}

// Masked mean-squared error: dy = 2 mask (y - t) / sum(mask); loss = sum(mask (y - t)^2) / sum(mask).
__device__ __forceinline__ void mse_term(float y, float t, float mask, float& s, float& c) {
    const float d = (y - t) * mask;
    s = fmaf(d, d, s);
    c += mask;
}
__device__ __forceinline__ float2 warp_sum2(float s, float c) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, off);
        c += __shfl_down_sync(0xffffffffu, c, off);
    }
    return make_float2(s, c);
}
// Sum over 1024 threads by a fixed tree, in thread 0 (rs: 32 entries).
__device__ __forceinline__ float2 block_sum2(float s, float c, float2* rs) {
    float2 v = warp_sum2(s, c);
    if ((threadIdx.x & 31) == 0) rs[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) v = warp_sum2(rs[threadIdx.x].x, rs[threadIdx.x].y);
    return v;
}
// The sums are needed by every element of dy, and one block alone is bound by its own
// load latency, so the blocks are one cluster: the elements form kOptParts parts
// (1024 consecutive ones in turn), whose sums are exchanged through distributed
// shared memory and added in order. A cluster of fewer blocks (most_cluster) takes
// several parts a block; the sums are the same bits.
constexpr int kOptParts = 16;
__global__ void __launch_bounds__(1024)
k_mlp_mse(const float* __restrict__ y, const float* __restrict__ t, const float* __restrict__ mask, long long n,
          float* __restrict__ dy, float* __restrict__ loss) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ float2 rs[32];
    __shared__ float2 tot[kOptParts];
    const int blocks = gridDim.x;                                 // one cluster: 16, 8 or 1
    const long long step = 1024LL * kOptParts;
    for (int part = blockIdx.x; part < kOptParts; part += blocks) {
        float s = 0.f, c = 0.f;
#pragma unroll 4
        for (long long i = part * 1024LL + threadIdx.x; i < n; i += step) mse_term(y[i], t[i], mask[i], s, c);
        const float2 v = block_sum2(s, c, rs);
        if (threadIdx.x == 0) tot[part] = v;
        if (part + blocks < kOptParts) __syncthreads();           // rs is free for the next part
    }
    cl.sync();
    if (threadIdx.x < 32) {                                       // the parts, added in order
        const float2 v = threadIdx.x < kOptParts ? *cl.map_shared_rank(&tot[threadIdx.x], threadIdx.x % blocks)
                                                 : make_float2(0.f, 0.f);
        float s = 0.f, c = 0.f;
#pragma unroll
        for (int q = 0; q < kOptParts; ++q) {
            s += __shfl_sync(0xffffffffu, v.x, q);
            c += __shfl_sync(0xffffffffu, v.y, q);
        }
        if (threadIdx.x == 0) rs[0] = make_float2(s, c);
    }
    cl.sync();                                                    // rs[0] in place; no block leaves while its sums are read
    const float s = rs[0].x, c = rs[0].y, cnt = c > 0.f ? c : 1.f;
    for (int part = blockIdx.x; part < kOptParts; part += blocks)
#pragma unroll 4
        for (long long i = part * 1024LL + threadIdx.x; i < n; i += step) dy[i] = 2.f * (y[i] - t[i]) * mask[i] / cnt;
    if (blockIdx.x == 0 && threadIdx.x == 0 && loss) *loss = s / cnt;
}
// n <= 1024: the one part that has elements, in one block without the cluster's barriers; same bits
// (in a graph 1.9 .. 2.3 us, a cluster 3.3 .. 3.8).
__global__ void __launch_bounds__(1024)
k_mlp_mse_one(const float* __restrict__ y, const float* __restrict__ t, const float* __restrict__ mask, int n,
              float* __restrict__ dy, float* __restrict__ loss) {
    __shared__ float2 rs[32], tot;
    const int i = threadIdx.x;
    const bool on = i < n;
    const float yi = on ? y[i] : 0.f, ti = on ? t[i] : 0.f, mi = on ? mask[i] : 0.f;
    float s = 0.f, c = 0.f;
    if (on) mse_term(yi, ti, mi, s, c);
    const float2 v = block_sum2(s, c, rs);
    if (i == 0) tot = v;
    __syncthreads();
    const float cnt = tot.y > 0.f ? tot.y : 1.f;
    if (on) dy[i] = 2.f * (yi - ti) * mi / cnt;
    if (i == 0 && loss) *loss = tot.x / cnt;
}

// Adam (Kingma & Ba 2015) on the FP32 master parameters; the step count lives
// in device memory (incremented by a launch before) so that a captured training
// step can be replayed. Blocks over the whole GPU: one cluster of 16 blocks that
// increments the count itself, without the first launch, took 5.7 us at 38 k
// parameters, 11.8 at 133 k and 66 at 1 M in a graph against 3.2, 4.4 and 15, and a
// whole step of 256 rows (38 k) takes 36 us either way.
__global__ void k_step_inc(int* step) {
    pdl_enter();
    pdl_fresh(step);
    *step += 1;
}
template <typename T>
__global__ void __launch_bounds__(256)
k_mlp_adam(float* master, T* __restrict__ lowp, const float* grad, float* m, float* v, const int* step, long long n,
           float lr, float b1, float b2, float eps) {
    pdl_wait();
    const int t = *step;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float g = grad[i];
        const float mi = b1 * m[i] + (1.f - b1) * g;
        const float vi = b2 * v[i] + (1.f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        const float p = master[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        master[i] = p;
        if (lowp) lowp[i] = from_f<T>(p);
    }
}

template <typename T>
__global__ void k_convert(const float* __restrict__ src, T* __restrict__ dst, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = from_f<T>(src[i]);
}

// ---------------------------------------------------------------- launchers
long long mlp_params(int I, int H, int O) { return (long long)I * H + H + (long long)H * H + H + (long long)H * O + O; }
int mlp_bwd_blocks(int B) { return (B + kGradRows - 1) / kGradRows; }

// All of a block's shared memory as the limit, set once per kernel and device: two threads
// with networks of different widths must not lower it under one another's launch (and the
// call takes a fifth of a microsecond of the host's three a launch).
template <auto K>
static cudaError_t smem_attr() {
    static std::atomic<unsigned long long> set{0};                 // bit d: set on device d
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (set.load() & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
    if (e == cudaSuccess) set.fetch_or(bit);
    return e;
}

// Rows per block: two while that gives at most two blocks per SM (304), eight
// up to eight rows an SM block pair, then 32 (the weights are read once per block).
// 0: k_mlp_forward_rows, where a block's fixed cost counts for more than its loads do:
// a few hidden units (3 -> 1 -> 1 -> 1, 4096 rows: 3.4 us against 4.8), and large batches
// with a layer that is wide against the hidden ones (block of 640 threads for little work; 3 -> 16 ->
// 16 -> 160, 65536 rows: 44 against 92; 64 hidden units: 136 / 144) or with odd rows,
// which are copied by single elements (97 -> 161, 65536 rows: bf16 241 / 275, FP32 244 / 265).
static int fwd_rows(int B, int H, int O, bool bf16) {
    if (H <= 2 || (H <= 4 && B > 608) || (B >= 8192 && O >= 5 * H) ||
        (B >= (bf16 ? 16384 : 32768) && H < 128 && (O & 1)))
        return 0;
    return B <= 608 ? 2 : B <= 2432 ? 8 : 32;
}

// The weight buffers hold the largest chunk, no more: blocks of a narrow network are
// short chains, and several of them have to share an SM (3 -> 64 -> 64 -> 64, 65536 rows:
// 102 us with two 48 KB buffers, 63 now; 3 -> 16 -> 16 -> 16 38 and 16).
template <typename T, int R>
static cudaError_t mlp_forward_r(const float* x, int B, int I, int H, int O, const void* theta, float* y, float* act,
                                 cudaStream_t s) {
    const int K[3] = {I, H, H}, C[3] = {H, H, O};
    int wbytes = 0;
    for (int l = 0; l < 3; ++l)
        wbytes = std::max(wbytes, fwd_chunk<T>(K[l], C[l]) * fwd_pitch<T>(C[l]) * (int)sizeof(T));
    wbytes = (wbytes + 15) & ~15;
    const size_t sm = 2 * (size_t)wbytes +
                      sizeof(float) * ((size_t)row_pitch<R>() * ((H > I ? H : I) + H) + 2 * H + O);
    cudaError_t e = smem_attr<k_mlp_forward<T, R>>();
    if (e != cudaSuccess) return e;
    const int wide = H > O ? H : O, ct = FwdTile<R>::CT;
    int nt = (((wide + ct - 1) / ct) * (R / FwdTile<R>::RT) + 31) / 32 * 32;
    const int copies = std::min(256, std::max(128, (wbytes / 16 + 31) / 32 * 32));   // the copies want threads too
    if (nt < copies) nt = copies;
    pdl(k_mlp_forward<T, R>, (unsigned)((B + R - 1) / R), nt, sm, s)(x, B, I, H, O, static_cast<const T*>(theta),
                                                                         y, act, wbytes);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t mlp_forward_rows(const float* x, int B, int I, int H, int O, const void* theta, float* y, float* act,
                                    cudaStream_t s) {
    const size_t sm = sizeof(float) * kDenseRows * (size_t)((I > H ? I : H) + (H > O ? H : O));
    cudaError_t e = smem_attr<k_mlp_forward_rows<T>>();
    if (e != cudaSuccess) return e;
    k_mlp_forward_rows<T><<<(unsigned)((B + kDenseRows - 1) / kDenseRows), 256, sm, s>>>(
        x, B, I, H, O, static_cast<const T*>(theta), y, act);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t mlp_forward(const float* x, int B, int I, int H, int O, const void* theta, float* y, float* act,
                               cudaStream_t s) {
    switch (fwd_rows(B, H, O, sizeof(T) == 2)) {
        case 2: return mlp_forward_r<T, 2>(x, B, I, H, O, theta, y, act, s);
        case 8: return mlp_forward_r<T, 8>(x, B, I, H, O, theta, y, act, s);
        case 32: return mlp_forward_r<T, 32>(x, B, I, H, O, theta, y, act, s);
        default: return mlp_forward_rows<T>(x, B, I, H, O, theta, y, act, s);
    }
}
cudaError_t launch_mlp_forward(const float* x, int B, int I, int H, int O, const void* theta, int bf16, float* y,
                               float* act, cudaStream_t s) {
    return bf16 ? mlp_forward<__nv_bfloat16>(x, B, I, H, O, theta, y, act, s)
                : mlp_forward<float>(x, B, I, H, O, theta, y, act, s);
}

template <typename T, int R>
static cudaError_t mlp_delta_r(int B, int I, int H, int O, const void* theta, const float* act, const float* dy,
                               float* d2, float* d1, int next, cudaStream_t s) {
    int wbytes = 0;
    for (int all : {O, H})
        wbytes = std::max(wbytes, H * delta_pitch<T>(delta_cols<T>(all, H)) * (int)sizeof(T));
    wbytes = (wbytes + 15) & ~15;
    const size_t sm = 2 * (size_t)wbytes + sizeof(float) * (size_t)row_pitch<R>() * ((O > H ? O : H) + H);
    cudaError_t e = smem_attr<k_mlp_delta<T, R>>();
    if (e != cudaSuccess) return e;
    const int need = (H * (R == 2 ? 1 : 2) + 31) / 32 * 32, nt = need < 256 ? 256 : need, blocks = (B + R - 1) / R;
    pdl(k_mlp_delta<T, R>, (unsigned)blocks, nt, sm, s)(B, I, H, O, static_cast<const T*>(theta), act, dy, d2, d1, wbytes,
                                                        blocks + next <= 152);
    return cudaGetLastError();
}
// Parts of the rows that the gradient tiles are split into: one tile an SM, 128 rows a
// part at least. Backward of 16384 rows (bf16), unsplit / split: 3 -> 16 -> 16 -> 16
// (3 tiles) 223 / 31 us, 3 -> 16 -> 16 -> 160 (12) 244 / 59, 3 -> 64 -> 64 -> 160 (60) 261 / 160.
// The parts' sums are added in order; against 64 bits the gradients are off by 0.4 to 1.0 of
// the unsplit ones' error (16 .. 97 hidden units, 300 .. 16384 rows).
static int grad_parts(int B, int tiles) { return std::max(1, std::min(152 / tiles, B / 128)); }

// The deltas of all rows, then the gradient tiles over the rows: in parts of rows
// where the tiles are fewer than the SMs, added in order.
template <typename T>
static cudaError_t mlp_backward(const float* x, int B, int I, int H, int O, const void* theta, const float* act,
                                const float* dy, float* ws, float* grad, cudaStream_t s) {
    const long long np = mlp_params(I, H, O), room = (long long)mlp_bwd_blocks(B) * np;
    const int th = (H + kGT - 1) / kGT, to = (O + kGT - 1) / kGT, tiles = th * (to + th + 1);
    int parts = grad_parts(B, tiles);
    const int per = ((B + parts - 1) / parts + kGChunk - 1) / kGChunk * kGChunk;
    parts = (B + per - 1) / per;
    cudaError_t e;
    if (2LL * H * B + (parts > 1 ? parts * np : 0) > room || (tiles <= 3 && B > 64 && B < 1024)) {
        e = smem_attr<k_mlp_backward_rows<T>>();
        if (e != cudaSuccess) return e;
        k_mlp_backward_rows<T><<<mlp_bwd_blocks(B), 256, sizeof(float) * (size_t)kGradRows * (I + 6 * H + O), s>>>(
            x, B, I, H, O, static_cast<const T*>(theta), act, dy, ws);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        pdl(k_mlp_reduce, (unsigned)((np + 255) / 256), 256, 0, s)(ws, mlp_bwd_blocks(B), np, grad);
        return cudaGetLastError();
    }
    float* d2 = ws;
    float* d1 = d2 + (long long)B * H;
    float* part = d1 + (long long)B * H;
    e = B <= 608 ? mlp_delta_r<T, 2>(B, I, H, O, theta, act, dy, d2, d1, tiles * parts, s)
                 : mlp_delta_r<T, 8>(B, I, H, O, theta, act, dy, d2, d1, tiles * parts, s);
    if (e != cudaSuccess) return e;
    pdl(k_mlp_grad, dim3(tiles, parts), kGT * kGT, 0, s)(x, B, per, I, H, O, act, dy, d2, d1, parts > 1 ? part : grad, np);
    if ((e = cudaGetLastError()) != cudaSuccess || parts == 1) return e;
    pdl(k_mlp_reduce, (unsigned)((np + 255) / 256), 256, 0, s)(part, parts, np, grad);
    return cudaGetLastError();
}
cudaError_t launch_mlp_backward(const float* x, int B, int I, int H, int O, const void* theta, int bf16,
                                const float* act, const float* dy, float* part, float* grad, cudaStream_t s) {
    return bf16 ? mlp_backward<__nv_bfloat16>(x, B, I, H, O, theta, act, dy, part, grad, s)
                : mlp_backward<float>(x, B, I, H, O, theta, act, dy, part, grad, s);
}

// One cluster of `blocks` blocks of 1024 threads (one block: an ordinary launch).
static void cluster_config(cudaLaunchConfig_t& c, cudaLaunchAttribute& at, int blocks, cudaStream_t s) {
    c.gridDim = dim3(blocks);
    c.blockDim = dim3(1024);
    c.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    c.attrs = &at;
    c.numAttrs = blocks > 1 ? 1 : 0;
}
template <typename... P, typename... A>
static cudaError_t launch_cluster(void (*k)(P...), int blocks, cudaStream_t s, A... a) {
    if (blocks > 1 && fault_inject("cluster")) return cudaErrorInvalidClusterSize;
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at{};
    cluster_config(c, at, blocks, s);
    return cudaLaunchKernelEx(&c, k, static_cast<P>(a)...);
}

// Largest cluster of 1024-thread blocks, of 16 (beyond the portable 8), 8 and 1, that
// the device can hold (an SM limit or a partition may leave less room): asked once per
// device.
template <typename... P>
static cudaError_t most_cluster(void (*k)(P...), int* blocks) {
    static std::atomic<int> known[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::atomic<int>& most = known[dev & 63];
    *blocks = 1;
    if (fault_inject("cluster")) return cudaSuccess;
    if (!most.load()) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        int got = 1;
        for (int want : {8, 16}) {
            cudaLaunchConfig_t c{};
            cudaLaunchAttribute at{};
            cluster_config(c, at, want, nullptr);
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, k, &c) == cudaSuccess && fit > 0) got = want;
            else cudaGetLastError();                              // (a size the device refuses)
        }
        most.store(got);
    }
    *blocks = most.load();
    return cudaSuccess;
}

cudaError_t launch_mlp_mse(const float* y, const float* t, const float* mask, long long n, float* dy, float* loss,
                           cudaStream_t s) {
    if (n <= 1024) {
        k_mlp_mse_one<<<1, 1024, 0, s>>>(y, t, mask, (int)n, dy, loss);
        return cudaGetLastError();
    }
    int blocks = 1;
    const cudaError_t e = most_cluster(k_mlp_mse, &blocks);
    return e != cudaSuccess ? e : launch_cluster(k_mlp_mse, blocks, s, y, t, mask, n, dy, loss);
}

template <typename T>
static cudaError_t mlp_adam(float* master, void* lowp, const float* grad, float* m, float* v, int* step, long long n,
                            float lr, float b1, float b2, float eps, cudaStream_t s) {
    pdl(k_step_inc, 1, 1, 0, s)(step);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long g = (n + 255) / 256;
    pdl(k_mlp_adam<T>, (unsigned)(g < (1 << 30) ? g : 1 << 30), 256, 0, s)(master, static_cast<T*>(lowp), grad, m, v,
                                                                          step, n, lr, b1, b2, eps);
    return cudaGetLastError();
}
cudaError_t launch_mlp_adam(float* master, void* lowp, int bf16, const float* grad, float* m, float* v, int* step,
                            long long n, float lr, float b1, float b2, float eps, cudaStream_t s) {
    return bf16 ? mlp_adam<__nv_bfloat16>(master, lowp, grad, m, v, step, n, lr, b1, b2, eps, s)
                : mlp_adam<float>(master, lowp, grad, m, v, step, n, lr, b1, b2, eps, s);
}

cudaError_t launch_mlp_convert(const float* src, void* dst, int bf16, long long n, cudaStream_t s) {
    const unsigned g = (unsigned)((n + 255) / 256);
    if (bf16)
        k_convert<__nv_bfloat16><<<g, 256, 0, s>>>(src, (__nv_bfloat16*)dst, n);
    else
        k_convert<float><<<g, 256, 0, s>>>(src, (float*)dst, n);
    return cudaGetLastError();
}

}  // namespace gridspt
