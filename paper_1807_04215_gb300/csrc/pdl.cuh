#pragma once
#include <cuda_runtime.h>

namespace gridspt {

// Programmatic dependent launch. Every block of these kernels first waits for the
// whole previous kernel of the stream (its writes are then visible), so results and
// order are as without it; only the launch itself and the block start overlap
// the previous kernel's end. The next kernel is let in when all blocks have started (no
// block of this one then waits for an SM that the next one holds); the persistent z
// passes let it in only when they end, except where each team has one row group:
// blocks that only wait would keep SMs from the kernels of other streams.
// A pointer that an earlier kernel writes through is not __restrict__ here, or passes
// pdl_fresh(): the compiler may move loads through a restrict parameter over the wait.
// Recursion 64^3 85.5 -> 77.1 us, 16 bispectrum shells of 256^3 274 -> 225 us, 192^3
// 2.29 -> 2.25 ms, from 256^3 on no difference; six 512^3 spectra 230 -> 207 us,
// emulator: 4096 rows predicted 20.5 -> 18.6 us, training step 41 -> 39.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
    pdl_wait();
    pdl_release();
}
#define pdl_fresh(p) asm volatile("" : "+l"(p)::"memory")

// A launch that may be placed on the SMs while the stream's previous kernel ends
// (a programmatic edge, also under capture); the kernel's pdl_wait() orders it.
template <typename... P>
struct PdlCall {
    void (*k)(P...);
    cudaLaunchConfig_t c;
    template <typename... A>
    void operator()(A&&... a) {
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        c.attrs = &at;
        c.numAttrs = 1;
        cudaLaunchKernelEx(&c, k, static_cast<P>(a)...);   // the caller reads cudaGetLastError()
    }
};
template <typename... P>
static PdlCall<P...> pdl(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    PdlCall<P...> r{k, {}};
    r.c.gridDim = grid;
    r.c.blockDim = block;
    r.c.dynamicSmemBytes = smem;
    r.c.stream = s;
    return r;
}

}  // namespace gridspt
