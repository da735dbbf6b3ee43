// qhd_launch.cuh -- launches that overlap with the end of the kernel before them.
//
// A small grid's pass is a few microseconds long, and between two passes of a
// stream the GPU drains, launches and refills for one to two of them.  With
// programmatic stream serialization the next grid's blocks are placed as soon
// as every block of the previous grid has released it (grid_release) or ended;
// they do what depends on no earlier kernel (index arithmetic, the static tables)
// and then wait for the previous grid's completion (grid_wait).
//
// Where a kernel releases decides where the next one's blocks land.  Released at the
// start, they take the room that the running blocks leave, several to an SM while
// others stay empty: kernels of about one block per SM then take up to twice as
// long, and k_plane_whole, placed behind k_prep, keeps that for a whole chunk (per
// step, released at the start / at the end / without overlap: 256^2 x 8 19.8 / 13.0 /
// 13.1 us, 128x256 x 30 19.3 / 12.5 / 12.7, 64^3 17.1 / 9.8 / 14.7, 64x16x128 x 5
// 17.5 / 15.1 / 22.8).  So the passes, and k_prep where a whole-run kernel follows,
// release at their end, with these exceptions.  A grid of up to 16 blocks is in
// nobody's way and releases at its start (16x1024 x 1 6.4 us, 7.2 at the end); one of up to a block per SM before its last
// transform (256x16 x 1 6.1 and 6.6, 128x16 x 4 5.4 and 6.1; with more threads than
// that the early blocks get in the way again: 512x256 x 4 13.2 and 11.3); more than 24
// one-warp blocks per SM at their start (4x1024 x 300 15.6 and 17.7; not with 13 per
// SM, 8x128x256 x 4 25.9 and 17.3).  Kernels that k_prep or the observables follow
// release at their start, so that those compute beside them: the observables,
// k_uniform, the whole-run kernels (k_solo_whole, which clusters may follow, at its
// end) and an evolution's last pass (1024^2 x 2, 8 evolutions of 3 steps: 832 us, 859
// released at the end).
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

// No order with memory accesses is needed: the next kernel waits for this grid's end.
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;"); }
// Released by grids of at most `threads` threads.
__device__ __forceinline__ void grid_release_upto(unsigned threads) {
    if (gridDim.x * blockDim.x <= threads) grid_release();
}
constexpr unsigned TINY_GRID = 16 * 128, SMALL_GRID = 152 * 128;
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Passes over fewer points than this overlap.  Measured per step, with (released at
// the start) and without: 64x16x128 x 5 19.4 / 23.4 us, 512^2 x 16 48.8 / 53.6, 128^3 x 4 114.8 /
// 118.8, 512^2 x 32 95.9 / 101.1; at 2^24 points the gap no longer counts and
// 256^3, whose plane and axis passes want different shared-memory splits of the
// SM, loses: 257.8 / 244.5.
constexpr int64_t OVERLAP_POINTS = int64_t(1) << 24;

// Kernels that run a whole chunk overlap k_prep for chunks of up to this many steps:
// the overlap saves 2.4 us per launch (64^2, chunks of 10 steps: 403 us per 100 steps,
// 427 without), but clusters placed while k_prep's last blocks run can be slower for
// all of their steps (128x256 7.11 us per step, 6.75 without; 256x32 4.54 and 4.17).
// 1-D, 64 points, 100 steps in chunks of 10: 228 us, 246 without; in one chunk 140 and
// 131.  One instance alone is the exception: in plain order its cluster always lands on
// the same SMs, good ones or bad ones by GPU (128^2 x 200 steps, 888 to 950 us on eight
// GPUs); k_prep releases it at the start and it takes what is free (886 to 898).
constexpr int OVERLAP_STEPS = 32;

// A launch's error is its caller's to report: it does not stay behind as the thread's
// last error, where the next plain launch, of any context, would find it.
inline cudaError_t launched(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

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
    return launched(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
}

}  // namespace qhd
