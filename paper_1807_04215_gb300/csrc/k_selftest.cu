// Self-tests: a bounded device-side wait, the column transforms.
//
// The wait and its status path: one block waits
// on an mbarrier whose phase never completes (no arrival is ever
// made). The wait gives up after its iteration limit, the kernel records the
// timeout in the status word and returns. Used only by the failure-detection
// test; no GPU fault, trap or unbounded spin is involved.
#include "fft_core.cuh"
#include "gridspt_internal.h"

namespace gridspt {

__global__ void k_wait_selftest(int* status) {
    __shared__ uint64_t bar;
    const unsigned a = (unsigned)__cvta_generic_to_shared(&bar);
    if (threadIdx.x == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(a) : "memory");
    __syncthreads();
    bool done = false;
    for (unsigned it = 0; it < (1u << 14) && !done; ++it) {
        unsigned d;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(d) : "r"(a) : "memory");
        done = d != 0;
        __nanosleep(64);
    }
    if (!done && threadIdx.x == 0) atomicOr(status, kStatusWaitSelftest);
}

cudaError_t launch_wait_selftest(int* status, cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>(status);
    return cudaGetLastError();
}

// Two sets of TZ columns ([set][element][column]) through the one-exchange transform
// (ONE) or the transform with one exchange per stage, whose results it has to equal.
// A block takes W columns: all, or as many as 1024 threads hold.
template <int L, int TZ, bool ONE>
struct ColumnsTest {
    static constexpr int E = ONE ? Col2<L>::E : fft_elems(L), P = L / E, W = P * TZ <= 1024 ? TZ : 1024 / P;
    static constexpr size_t smem = ONE ? Col2<L>::bytes(W) : sizeof(float2) * (size_t)(L + L * W);
    static_assert(TZ % W == 0 && smem <= 232448, "self-test columns");
};
template <int L, int DIR, int TZ, bool ONE>
__global__ void __launch_bounds__(ColumnsTest<L, TZ, ONE>::P * ColumnsTest<L, TZ, ONE>::W)
k_columns_selftest(const float2* __restrict__ in, float2* __restrict__ out, const float2* __restrict__ twg) {
    extern __shared__ __align__(16) float2 sm[];
    using C = ColumnsTest<L, TZ, ONE>;
    constexpr int E = C::E, P = C::P, W = C::W;
    const int c = threadIdx.x % W, p = threadIdx.x / W;
    in += blockIdx.x * W;
    out += blockIdx.x * W;
    if constexpr (ONE) {
        col2_table<L>(sm, twg);
    } else {
        for (int i = threadIdx.x; i < L; i += blockDim.x) sm[i] = twg[i];
        __syncthreads();
    }
    for (int set = 0; set < 2; ++set, in += L * TZ, out += L * TZ) {
        float2 x[E];
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = in[(ONE ? Col2<L>::in_base(p) + Col2<L>::in_step(i) : p + P * i) * TZ + c];
        if constexpr (ONE) fft_col2<L, DIR, W>(x, p, sm + Col2<L>::TW + c, sm);
        else fft_column<L, DIR, L>(x, p, sm + L + c, W, sm);
#pragma unroll
        for (int i = 0; i < E; ++i) out[(p + P * i) * TZ + c] = x[i];
    }
}

template <int L, int DIR, int TZ, bool ONE>
static cudaError_t columns_selftest(const float2* in, float2* out, const float2* tw, cudaStream_t s) {
    using C = ColumnsTest<L, TZ, ONE>;
    const cudaError_t e = cudaFuncSetAttribute(k_columns_selftest<L, DIR, TZ, ONE>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem);
    if (e != cudaSuccess) return e;
    k_columns_selftest<L, DIR, TZ, ONE><<<TZ / C::W, C::P * C::W, C::smem, s>>>(in, out, tw);
    return cudaGetLastError();
}
template <int L, int TZ>
static cudaError_t columns_selftest(int dir, int one, const float2* in, float2* out, const float2* tw, cudaStream_t s) {
    return dir > 0 ? (one ? columns_selftest<L, +1, TZ, true>(in, out, tw, s) : columns_selftest<L, +1, TZ, false>(in, out, tw, s))
                   : (one ? columns_selftest<L, -1, TZ, true>(in, out, tw, s) : columns_selftest<L, -1, TZ, false>(in, out, tw, s));
}
cudaError_t launch_columns_selftest(int N, int width, int dir, int one, const float2* in, float2* out, const float2* tw,
                                    cudaStream_t s) {
    if (width == 32 && N == 128) return columns_selftest<128, 32>(dir, one, in, out, tw, s);
    if (width == 32 && N == 256) return columns_selftest<256, 32>(dir, one, in, out, tw, s);
    if (width != 16) return cudaErrorInvalidValue;
    switch (N) {
        case 128: return columns_selftest<128, 16>(dir, one, in, out, tw, s);
        case 256: return columns_selftest<256, 16>(dir, one, in, out, tw, s);
        case 512: return columns_selftest<512, 16>(dir, one, in, out, tw, s);
        case 1024: return columns_selftest<1024, 16>(dir, one, in, out, tw, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gridspt
