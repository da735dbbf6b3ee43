// qhd_plane.cu -- kernels built on the plane engines.
//
// k_solo_pass, k_plane_pass: one fused pass over the last two axes of a 3-D grid
//   (for every (instance, i0) plane): inverse transform of the previous step along
//   axes 2 and 1, potential phase, forward transform along axes 1 and 2.  With
//   the axis-0 pass (forward, kinetic phase, inverse) a 3-D Strang step then
//   reads and writes psi twice instead of four times.  Planes of up to 16384
//   points take one CTA each, larger ones a cluster.
// k_solo_whole, k_plane_whole: a whole 2-D instance resident in one CTA or one
//   cluster for every step of a chunk: per step the potential phase between the
//   column transforms and the kinetic phase between the row transforms.  psi
//   touches global memory only at the chunk's start and end.
#include <cmath>

#include "qhd_kernels.h"
#include "qhd_launch.cuh"
#include "qhd_plane.cuh"
#include "qhd_plane2.cuh"

namespace qhd {

// Resident CTAs per SM a kernel on pairs of rows is compiled for: 512 threads of
// 128 registers where one holds 16 pairs of points, 768 of 80 where it holds 8
// (64^3 x 32 84.4 us per step, 90.3 with 512 threads, 86.6 with 1024), or what the
// tiles' shared memory allows.
template <typename P> constexpr int plane2_min_blocks(int threads) {
    constexpr int by_smem = (int)((227 * 1024) / (P::SMEM + 1024));
    const int by_regs = threads / P::THREADS < 1 ? 1 : threads / P::THREADS;
    return by_smem < by_regs ? by_smem : by_regs;
}
template <typename P> constexpr int solo_min_blocks() {
    return plane2_min_blocks<P>(P::E2 == 16 || P::RP == 64 ? 512 : 768);
}

template <int N1, int N2>
__global__ void __launch_bounds__(Solo<N1, N2>::THREADS, solo_min_blocks<Solo<N1, N2>>()) k_solo_pass(PlaneArgs a) {
    using P = Solo<N1, N2>;
    extern __shared__ __align__(16) float4 smem4[];
    float4 *ptab = smem4;
    ulonglong2 *tile = reinterpret_cast<ulonglong2 *>(smem4 + PHASE_TAB);
    const int tid = (int)threadIdx.x;
    const int64_t plane = blockIdx.x;
    float2 *g = a.psi + plane * (int64_t)N1 * N2;
    const uint32_t *fq = a.fq + plane * (int64_t)N1 * N2;
    const float4 *tw_row = a.tw_row + P::V * TW2_TABLE * N2;
    const bool inv = a.mode & MODE_INV, fwd = a.mode & MODE_FWD;
    if (!fwd) grid_release();
    load_phase_tab(ptab, a.ptab);
    grid_wait();
    const uint64_t coef = a.pot[plane >> a.log_planes];
    if (inv) plane2_rows_global<P, true>(tile, g, tw_row, tid);
    else plane2_copy<P, true>(tile, g, tid);
    __syncthreads();
    solo_columns<P>(tile, inv, true, fwd, a.twx, fq, coef, a.dither, ptab, tid);
    __syncthreads();
    if (fwd) plane2_rows_global<P, false>(tile, g, tw_row, tid);
    else plane2_copy<P, false>(tile, g, tid);
    grid_release();
}

template <int N1, int N2, int C>
__global__ void __launch_bounds__(Plane2<N1, N2, C, 1>::THREADS, plane2_min_blocks<Plane2<N1, N2, C, 1>>(512))
    k_plane_pass(PlaneArgs a) {
    using P = Plane2<N1, N2, C, 1>;
    extern __shared__ __align__(16) float4 smem4[];
    float4 *ptab = smem4;
    ulonglong2 *tile = reinterpret_cast<ulonglong2 *>(smem4 + PHASE_TAB);
    const int rank = (int)(blockIdx.x % C), tid = (int)threadIdx.x;
    const int64_t plane = blockIdx.x / C;
    uint32_t tiles[C];
#pragma unroll
    for (int q = 0; q < C; ++q) tiles[q] = cluster_addr(tile, (uint32_t)q);
    float2 *g = a.psi + plane * (int64_t)N1 * N2 + (int64_t)rank * P::R * N2;
    const float4 *tw_row = a.tw_row + P::V * TW2_TABLE * N2;
    const bool inv = a.mode & MODE_INV, fwd = a.mode & MODE_FWD;
    const uint32_t *fq = a.fq + plane * (int64_t)N1 * N2;
    // the potential rows this CTA's exchange positions read (R / C rows in each of the C
    // row blocks) go to L2 now, during the tile load and the inverse transform (20 steps of
    // 256^3: 4871 us without, 4822 with)
    static_assert(P::R % C == 0, "whole rows per CTA");
    if (!fwd) grid_release();
    if (tid < C) {
        const uint32_t *rows = fq + (int64_t)(P::R * tid + rank * (P::R / C)) * N2;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(rows), "r"(P::R / C * N2 * 4) : "memory");
    }
    load_phase_tab(ptab, a.ptab);
    grid_wait();
    const uint64_t coef = a.pot[plane >> a.log_planes];
    if (inv) {
        plane2_rows_global<P, true>(tile, g, tw_row, tid);
        __syncthreads();
        plane2_columns<P, true>(tile, tid);
    } else {
        plane2_copy<P, true>(tile, g, tid);
    }
    cluster_sync();
    plane2_exchange<P>(tiles, rank, inv, true, fwd, a.twx, fq, coef, a.dither, ptab, tid);
    cluster_sync();
    if (fwd) {
        plane2_columns<P, false>(tile, tid);
        __syncthreads();
        plane2_rows_global<P, false>(tile, g, tw_row, tid);
    } else {
        plane2_copy<P, false>(tile, g, tid);
    }
    grid_release();
}

// A block's instance.  HIDDEN: the compiler cannot tell that the index is a small
// unsigned number and keeps fewer of a step's addresses in registers, which spill in
// some shapes.
template <bool HIDDEN> __device__ __forceinline__ int64_t instance_of(unsigned i) {
    int64_t zero = 0;
    if (HIDDEN) asm volatile("" : "+l"(zero));
    return zero + i;
}

// Hidden index: per step, without / with, 32x256 x 608 41.3 / 39.7 us, 64x32 x 304 6.86 /
// 6.74; against 128^2 x 608 72.3 / 74.9, 64^2 x 304 10.3 / 10.4.
template <int N1, int N2>
__global__ void __launch_bounds__(Solo<N1, N2>::THREADS, solo_min_blocks<Solo<N1, N2>>()) k_solo_whole(PlaneArgs a) {
    using P = Solo<N1, N2>;
    extern __shared__ __align__(16) float4 smem4[];
    float4 *ptab = smem4;
    ulonglong2 *tile = reinterpret_cast<ulonglong2 *>(smem4 + PHASE_TAB);
    load_phase_tab(ptab, a.ptab);
    grid_wait();
    solo_whole_run<P>(a, instance_of<N2 == 256 || N2 == 32>(blockIdx.x), ptab, tile, (int)threadIdx.x);
    grid_release();
}

// MINB: CTAs per SM the kernel is compiled for (2 for batches; 1 for the wide
// split, which runs only when every CTA has an SM of its own).
// Args: PlaneArgsLong for shapes that spill with the arguments in registers.  Per
// step, in registers / in constant memory: 64x128 x 60 9.81 / 8.47 us, 256x64 x 60 13.1 /
// 12.8, 256x128 x 456 146.6 / 143.8, 128^2 on 8 CTAs 4.64 / 4.59; against 32x128 x 30 5.91 /
// 6.07, 64^2 x 30 3.04 / 3.12, 128x64 x 1 2.86 / 2.91, 128x256 x 1 6.66 / 6.82, 256x32 x 38
// 8.53 / 8.70.  Hidden index, without / with: 32x256 x 30 9.70 / 7.08, 256x128 x 456 143.8 /
// 139.9 and x 1 8.57 / 8.02, 256^2 x 8 13.1 / 12.9; against 256x32 x 38 8.57 / 8.78, 128^2 x 30
// 8.13 / 8.34.
template <int N1, int N2, int C>
using WholeArgs =
    std::conditional_t<(N1 == 64 && N2 == 128 && C == 2) || (N1 == 128 && N2 == 128 && C == 8) ||
                           (N1 == 256 && (N2 == 64 || N2 == 128)),
                       PlaneArgsLong, PlaneArgs>;
template <int N1, int N2> constexpr bool WHOLE_HIDDEN = (N1 == 32 && N2 == 256) || (N1 == 256 && N2 >= 128);

template <int N1, int N2, int C, int MINB>
__global__ void __launch_bounds__(PLANE_THREADS, MINB) k_plane_whole(WholeArgs<N1, N2, C> a) {
    extern __shared__ __align__(16) float4 smem4[];
    float4 *ptab = smem4;
    float2 *tile = reinterpret_cast<float2 *>(smem4 + PHASE_TAB);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    uint32_t tiles[C];
#pragma unroll
    for (int q = 0; q < C; ++q) tiles[q] = cluster_addr(tile, (uint32_t)q);
    grid_release();
    plane_whole_run<N1, N2, C, 1>(a, instance_of<WHOLE_HIDDEN<N1, N2>>(blockIdx.x / C), rank, tiles, ptab, tile, true,
                                  cluster);
}

// ---------------------------------------------------------------- launchers
template <typename Args>
static cudaError_t launch_cluster(void (*kernel)(Args), bool overlap, int64_t clusters, int c, int threads, size_t smem,
                                  const PlaneArgs &a, cudaStream_t s, bool &attr_done) {
    if (!attr_done) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_done = true;
    }
    if (clusters == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * c), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int k = 0;
    if (overlap) {  // the kernels follow qhd_launch.cuh's rules
        attr[k].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[k++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (c > 1) {
        attr[k].id = cudaLaunchAttributeClusterDimension;
        attr[k].val.clusterDim.x = (unsigned)c;
        attr[k].val.clusterDim.y = 1;
        attr[k++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)k;
    Args args{};
    static_cast<PlaneArgs &>(args) = a;
    return launched(cudaLaunchKernelEx(&cfg, kernel, args));
}

// Cluster size per distributed-axis length: R = 32 rows per CTA (16 for 32).
__host__ __device__ constexpr int plane_c(int n1) { return n1 >= 256 ? 8 : n1 >= 128 ? 4 : n1 >= 64 ? 2 : n1 >= 32 ? 2 : 0; }

// The shared-memory attribute is a per-device property of the kernel; it is set
// on the first launch of each instantiation (one device per process here).
template <int N1, int N2>
static cudaError_t plane_pass_impl(const PlaneArgs &a, cudaStream_t s) {
    static bool attr_done = false;
    const bool overlap = a.count * N1 * N2 < OVERLAP_POINTS;
    if constexpr (plane_solo(N1, N2)) {
        using P = Solo<N1, N2>;
        return launch_cluster(k_solo_pass<N1, N2>, overlap, a.count, 1, P::THREADS, P::SMEM, a, s, attr_done);
    } else {
        using P = Plane2<N1, N2, plane_c(N1), 1>;
        return launch_cluster(k_plane_pass<N1, N2, plane_c(N1)>, overlap, a.count, plane_c(N1), P::THREADS, P::SMEM, a, s,
                              attr_done);
    }
}

template <int N1, int N2>
static cudaError_t solo_whole_impl(const PlaneArgs &a, cudaStream_t s) {
    if constexpr (plane_solo(N1, N2)) {
        using P = Solo<N1, N2>;
        static bool attr_done = false;
        return launch_cluster(k_solo_whole<N1, N2>, a.cnt <= OVERLAP_STEPS, a.count, 1, P::THREADS, P::SMEM, a, s,
                              attr_done);
    } else {
        return cudaErrorInvalidValue;
    }
}

template <int N1, int N2, int C = plane_c(N1), int MINB = 2>
static cudaError_t plane_whole_impl(const PlaneArgs &a, cudaStream_t s) {
    static bool attr_done = false;
    return launch_cluster(k_plane_whole<N1, N2, C, MINB>, a.cnt <= OVERLAP_STEPS || a.batch == 1, a.count, C, PLANE_THREADS,
                          PlaneCfg<N1, N2, C>::SMEM, a, s, attr_done);
}

bool plane_supported(int n1, int n2) {
    return (n1 == 32 || n1 == 64 || n1 == 128 || n1 == 256) && (n2 == 32 || n2 == 64 || n2 == 128 || n2 == 256);
}

int plane_cluster(int n1) { return plane_c(n1); }
bool plane_fits_solo(int n1, int n2) { return plane_supported(n1, n2) && plane_solo(n1, n2); }

template <int N1, int N2> static int solo_per_sm_of() {
    if constexpr (plane_solo(N1, N2)) return solo_min_blocks<Solo<N1, N2>>();
    else return 0;
}

#define QHD_PLANE_DISPATCH(fn)                                                        \
    switch (n1 * 1000 + n2) {                                                         \
    case 32032: return fn<32, 32>(a, s);    \
    case 32064: return fn<32, 64>(a, s);    \
    case 32128: return fn<32, 128>(a, s);    \
    case 32256: return fn<32, 256>(a, s);    \
    case 64032: return fn<64, 32>(a, s);    \
    case 64064: return fn<64, 64>(a, s);    \
    case 64128: return fn<64, 128>(a, s);    \
    case 64256: return fn<64, 256>(a, s);    \
    case 128032: return fn<128, 32>(a, s);    \
    case 128064: return fn<128, 64>(a, s);    \
    case 128128: return fn<128, 128>(a, s);    \
    case 128256: return fn<128, 256>(a, s);    \
    case 256032: return fn<256, 32>(a, s);    \
    case 256064: return fn<256, 64>(a, s);    \
    case 256128: return fn<256, 128>(a, s);    \
    case 256256: return fn<256, 256>(a, s);    \
    default: return cudaErrorInvalidValue;                                            \
    }

// Instances an SM runs at once in the one-CTA form.
static int solo_per_sm(int n1, int n2) {
    switch (n1 * 1000 + n2) {
    case 32032: return solo_per_sm_of<32, 32>();
    case 32064: return solo_per_sm_of<32, 64>();
    case 32128: return solo_per_sm_of<32, 128>();
    case 32256: return solo_per_sm_of<32, 256>();
    case 64032: return solo_per_sm_of<64, 32>();
    case 64064: return solo_per_sm_of<64, 64>();
    case 64128: return solo_per_sm_of<64, 128>();
    case 64256: return solo_per_sm_of<64, 256>();
    case 128032: return solo_per_sm_of<128, 32>();
    case 128064: return solo_per_sm_of<128, 64>();
    case 128128: return solo_per_sm_of<128, 128>();
    default: return 0;
    }
}

// Microseconds per step of a batch of n1 x n2 instances in the two forms (152 SMs,
// 200 steps): tail, the first of few instances behind full waves of clusters; c1 and
// c2, clusters on up to one and two CTAs per SM; solo[k - 1], one CTA each with k
// instances per SM.
struct FormTimes {
    int n1, n2;
    float tail, c1, c2, solo[6];
};
constexpr FormTimes FORM_TIMES[] = {
    {32, 32, 2.16f, 2.96f, 3.60f, {5.84f, 7.16f, 8.65f, 10.47f, 12.95f, 15.18f}},
    {32, 64, 3.12f, 3.44f, 4.41f, {6.23f, 8.45f, 11.02f}},
    {32, 128, 5.67f, 6.25f, 7.45f, {6.20f}},
    {32, 256, 5.70f, 7.50f, 10.67f, {10.06f}},
    {64, 32, 3.18f, 3.87f, 4.78f, {5.14f, 6.74f, 9.43f, 12.14f, 15.19f, 18.07f}},
    {64, 64, 3.76f, 5.48f, 6.76f, {6.12f, 10.32f, 14.79f}},
    {64, 128, 6.13f, 8.52f, 10.97f, {10.41f}},
    {64, 256, 9.75f, 12.72f, 18.75f, {18.87f}},
    {128, 32, 2.90f, 3.36f, 4.28f, {8.36f, 10.78f, 15.94f, 25.40f}},
    {128, 64, 4.28f, 5.08f, 6.48f, {9.84f, 17.38f}},
    {128, 128, 5.93f, 7.70f, 10.95f, {18.48f}},
};

// How many of a batch's instances (the first ones) run in one CTA each: all, none,
// or the whole waves of that form with the rest on clusters, whichever the times
// above make shortest.  A split has to win by 8%: it costs a second launch, and its two
// parts round differently.  Measured with every choice forced: 128^2 x 100 17.7 us on
// clusters, 18.2 in one CTA each; x 120 21.4 / 18.3; x 512 74.5 / 72.6, split 65.4; 64^2 x
// 78 6.05 / 5.60; 32^2 x 200 6.26 / 6.50, x 400 10.2 / 8.3; 128x32 x 78 7.67 / 7.32, x 152
// 11.7 / 8.4; 64x256 x 304 36.8 / 37.3.  Batches of 8 instances per SM and more stay in
// one CTA each where that is up to 4% behind (64x256 x 1216 143.8 / 148.9).
int64_t solo_instances(int n1, int n2, int64_t batch, int sms) {
    if (!plane_fits_solo(n1, n2)) return 0;
    const FormTimes *f = FORM_TIMES;
    while (f->n1 != n1 || f->n2 != n2) ++f;
    const int c = plane_c(n1), per_sm = solo_per_sm(n1, n2);
    // pairs of CTAs find room on every SM, clusters of four not quite (74 of 76)
    const int64_t wave_c = 2 * (int64_t)sms / c - (c > 2 ? 2 : 0);
    const double spread = c > 2 ? 0.8 : 1.0;  // share of the SMs up to which CTAs are alone on theirs
    auto clusters = [&](int64_t b) {
        const int64_t full = b / wave_c, rem = b % wave_c;
        if (rem == 0) return (double)full * f->c2;
        const double load = (double)(rem * c) / sms;
        if (load > spread) return (double)(full + 1) * f->c2;
        return full * f->c2 + (full ? f->tail + (f->c1 - f->tail) * load / spread : (double)f->c1);
    };
    const int64_t wave_s = (int64_t)sms * per_sm, full = batch / wave_s, rem = batch % wave_s;
    const double whole = (double)full * f->solo[per_sm - 1];
    const double solo = whole + (rem ? f->solo[(rem + sms - 1) / sms - 1] : 0.f);
    const double split = full && rem ? whole + clusters(rem) : INFINITY;
    const double limit = clusters(batch) * (batch >= 8 * (int64_t)sms ? 1.04 : 1.0);
    if (split * 1.08 <= solo || solo > limit) return split <= limit ? full * wave_s : 0;
    return batch;
}

cudaError_t launch_plane_pass(int n1, int n2, const PlaneArgs &a, cudaStream_t s) {
    QHD_PLANE_DISPATCH(plane_pass_impl)
}

cudaError_t launch_plane_whole(int n1, int n2, const PlaneArgs &a, cudaStream_t s) {
    QHD_PLANE_DISPATCH(plane_whole_impl)
}

cudaError_t launch_solo_whole(int n1, int n2, const PlaneArgs &a, cudaStream_t s) {
    QHD_PLANE_DISPATCH(solo_whole_impl)
}

// The whole-run kernel with twice the CTAs per instance (half the rows each) for
// distributed axes of 64 and 128: a batch too small to fill the GPU then runs on
// twice the SMs.
__host__ __device__ constexpr int plane_c_wide(int n1) { return n1 == 128 ? 8 : n1 == 64 ? 4 : 0; }

int plane_cluster_wide(int n1) { return plane_c_wide(n1); }

cudaError_t launch_plane_whole_wide(int n1, int n2, const PlaneArgs &a, cudaStream_t s) {
    switch (n1 * 1000 + n2) {
    case 64032: return plane_whole_impl<64, 32, plane_c_wide(64), 1>(a, s);
    case 64064: return plane_whole_impl<64, 64, plane_c_wide(64), 1>(a, s);
    case 64128: return plane_whole_impl<64, 128, plane_c_wide(64), 1>(a, s);
    case 64256: return plane_whole_impl<64, 256, plane_c_wide(64), 1>(a, s);
    case 128032: return plane_whole_impl<128, 32, plane_c_wide(128), 1>(a, s);
    case 128064: return plane_whole_impl<128, 64, plane_c_wide(128), 1>(a, s);
    case 128128: return plane_whole_impl<128, 128, plane_c_wide(128), 1>(a, s);
    case 128256: return plane_whole_impl<128, 256, plane_c_wide(128), 1>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

// exp(-2 pi i m / n) as (re, im) values and their FP32 residuals
static void unit_root(int64_t m, int64_t n, float *hr, float *hi, float *lr, float *li) {
    const double ang = 2.0 * 3.141592653589793238462643383279502884 * (double)(m % n) / (double)n;
    const double cr = cos(ang), ci = -sin(ang);
    *hr = (float)cr;
    *hi = (float)ci;
    *lr = (float)(cr - (double)*hr);
    *li = (float)(ci - (double)*hi);
}

void exchange_twiddles(float4 *out, int n1, int c) {
    const int r = n1 / c;
    for (int q = 0; q < c; ++q)
        for (int j = 0; j < r; ++j) {
            float4 &o = out[q * r + j];
            unit_root((int64_t)j * q, n1, &o.x, &o.y, &o.z, &o.w);
        }
}

void exchange_twiddles2(float4 *out, int n1, int c) {
    const int rp = n1 / c / 2;
    for (int q = 0; q < c; ++q)
        for (int p = 0; p < rp; ++p) {
            float4 &h = out[q * rp + p], &l = out[n1 / 2 + q * rp + p];
            unit_root((int64_t)(2 * p) * q, n1, &h.x, &h.z, &l.x, &l.z);
            unit_root((int64_t)(2 * p + 1) * q, n1, &h.y, &h.w, &l.y, &l.w);
        }
}

template <int RP> static void solo_fill(float4 *out) {
    using L = Line2<RP, 2>;
    constexpr int R1 = L::P::R[0], R2 = L::P::R[1];
    static_assert(L::STAGES == 2 && R1 * R2 == RP, "two stages");
    for (int k = 0; k < RP; ++k) unit_root(k, 2 * RP, &out[k].x, &out[k].y, &out[k].z, &out[k].w);
    for (int i = 0; i < RP; ++i) {
        float4 &o = out[RP + i];
        unit_root((int64_t)(i % R1) * (i / R1), RP, &o.x, &o.y, &o.z, &o.w);
    }
}

void solo_twiddles(float4 *out, int n1) {
    switch (n1) {
    case 32: return solo_fill<16>(out);
    case 64: return solo_fill<32>(out);
    case 128: return solo_fill<64>(out);
    }
}

}  // namespace qhd
