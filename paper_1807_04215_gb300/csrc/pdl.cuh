#pragma once
#include <cuda_runtime.h>

namespace gridspt {

// Programmatic dependent launch. Every block of these kernels first waits for the
// whole previous kernel of the stream (its writes are then visible), so results and
// order are as without it; only the launch itself overlaps the previous kernel's end.
// The transform and shell passes (pdl_wait) let the next kernel in when their last block ends.
// Letting it in as soon as all blocks have started places the next kernel's blocks
// wherever there is room while this one runs: several on one SM, none on others, and
// they stay there. Fifth order, early / at the end / no programmatic launch, replayed
// from a graph and launched on a stream: 96^3 481 / 365 / 360 and 491 / 374 / 406 us,
// 64^3 201 / 147 / 150 and 212 / 156 / 197, 128^3 533 / 492 / 492; r2c at 96^3 18.4 /
// 14.6 / 15.6. So do the emulator's layers (2400 rows of 3 -> 64 -> 64 -> 160, one call after the
// other: 11.9 / 9.0 us; backward of 1024 rows of 3 -> 128 -> 128 -> 160: 44 / 25), except a delta
// kernel that leaves an SM to each block of its successor. The power and shell-sum kernels
// let it in early (pdl_enter): their successors are small (the final sums of a power call:
// 0.6 us of 7 later otherwise), so do the passes of grids up to 24^3, which leave most SMs
// empty (divergence form, eighth order: 8^3 98 / 112 us, 24^3 223 / 235; at 48^3 272 / 250),
// and warp-row z passes up to 48^3 (c2r 12.4 / 12.9; fifth order at 96^3 375 / 369).
// A pointer that an earlier kernel writes through is not __restrict__ here, or passes
// pdl_fresh(): the compiler may move loads through a restrict parameter over the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
    pdl_wait();
    pdl_release();
}
template <int N>
__device__ __forceinline__ void pdl_pass() {
    pdl_wait();
    if constexpr (N <= 24) pdl_release();
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
