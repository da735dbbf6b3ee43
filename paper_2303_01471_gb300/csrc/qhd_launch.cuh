// qhd_launch.cuh -- launches that overlap with the end of the kernel before them.
//
// A small grid's pass is a few microseconds long, and between two passes of a
// stream the GPU drains, launches and refills for one to two of them.  With
// programmatic stream serialization the next grid's blocks are placed as soon
// as every block of the previous grid has started (grid_release) and SM
// resources come free; they do what depends on no earlier kernel (index
// arithmetic, the static tables) and then wait for the previous grid's
// completion (grid_wait).
//
// Rules: every kernel launched through launch_overlapped calls grid_wait in all
// its threads before it touches anything an earlier kernel writes, or writes
// anything an earlier kernel reads.  grid_wait returns when the previous grid is
// complete and its writes are visible; that grid waited for the one before it,
// so the order is transitive.  Nothing that a kernel of the same stream wrote may be
// read before it unless the host has waited for that kernel since: what is left is
// what set_potential, set_schedule and init_grid write (they synchronise the
// stream).  A kernel without grid_release counts as well: the wait, not the end of
// its blocks, is what makes its writes visible.  And nothing that an overlapped
// kernel writes is read with __ldg or through a restrict pointer, wait or not: those
// loads are for memory that nobody writes while the kernel is resident, and the
// compiler may move them across the wait.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace qhd {

__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Passes over fewer points than this overlap.  Measured per step, with and
// without: 64x16x128 x 5 19.4 / 23.4 us, 512^2 x 16 48.8 / 53.6, 128^3 x 4 114.8 /
// 118.8, 512^2 x 32 95.9 / 101.1; at 2^24 points the gap no longer counts and
// 256^3, whose plane and axis passes want different shared-memory splits of the
// SM, loses: 257.8 / 244.5.
constexpr int64_t OVERLAP_POINTS = int64_t(1) << 24;

template <typename... P, typename... A>
cudaError_t launch_overlapped(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace qhd
