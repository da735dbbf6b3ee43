// qhd_kernels.cu -- the hot path of the split-operator QHD step on sm_103a.
//
// One Strang step (Eq. (prod_qhd_fft) in its symmetric form) is
//   psi <- P(dt b/2) F^-1 K(dt a) F P(dt b/2) psi
// with P the potential phase exp(-i theta f(x)) (diagonal in position) and K
// the kinetic phase exp(-i dt a |k|^2/2) (diagonal in Fourier space,
// k = 2 pi m / L).  The half potential phases of consecutive steps commute and
// are merged: theta_j = dt (b_{j-1} + b_j)/2.  The multi-dimensional DFT is
// split by axis, and the per-axis transforms are fused with the phases so that
// each launch reads and writes psi once:
//   2-D:  row pass    F_1 . P . F_1^-1           (contiguous rows)
//         column pass F_0^-1 . K . F_0           (strided columns)
//   3-D:  x pass F_2 . P . F_2^-1,  y pass F_1,  z pass F_0^-1 K F_0,  y pass F_1^-1
//   1-D:  one launch runs every step of a chunk with the line in registers.
// Between passes psi is stored with the fastest axis in Fourier space
// (natural frequency order), the others in position space.
//
// Phase arithmetic is exact in fixed point: the potential uses f quantised to
// 32 bits with a per-instance power-of-two scale, and a 64-bit fraction of a
// turn per unit of f; the kinetic phase uses integer m^2 and a 64-bit fraction
// of a turn per unit of m^2.  The product modulo one turn is exact to 2^-32,
// so the FP32 sine/cosine only ever sees a reduced argument.
#include <cmath>
#include <type_traits>

#include "qhd_device.cuh"
#include "qhd_kernels.h"
#include "qhd_launch.cuh"
#include "qhd_packed.cuh"
#include "qhd_sched.cuh"
#include "qhd_prep.cuh"

namespace qhd {

struct WarpSync {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};
struct BlockSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

constexpr int ROW_THREADS = 128;

// The row and axis passes work on pairs of lines in packed FP32
// (qhd_packed.cuh): rows 2i and 2i + 1, columns 2i and 2i + 1.  Every axis
// length is even, so the pairs never straddle an instance or a plane.

// --------------------------------------------------------------- row pass
template <int N, int V>
__global__ void __launch_bounds__(ROW_THREADS, 4) k_row(RowArgs a) {
    using C = Line2<N, V>;
    using B = RowBuf<N, V>;
    const RowAddr<C::LOG_R1> at;
    constexpr int E = C::E, T = C::T;
    using Sync = std::conditional_t<(T > 32), BlockSync, WarpSync>;
    extern __shared__ __align__(16) float4 smem4[];
    float4 *ptab = smem4;
    if (!(a.mode & MODE_FWD)) grid_release();
    else grid_release_upto(TINY_GRID);
    load_phase_tab(ptab, a.ptab);
    __syncthreads();
    const int line = threadIdx.x / T, t = threadIdx.x % T;
    const int64_t row = 2 * ((int64_t)blockIdx.x * (blockDim.x / T) + line);
    const bool valid = row < a.rows;
    const int64_t r = valid ? row : 0;
    float2 *g = a.psi + r * N;
    const uint32_t *fq = a.fq + r * N;
    grid_wait();
    c2 x[E];
    // a thread that holds whole rows moves two of their points at a time: its lanes lie
    // 16 N bytes apart, and an access per point touched every sector twice as often
    // (8x1024x8 x 256, the pass over 8-point rows: 161 us, 88 so)
    if constexpr (T == 1) {
        const float4 *g4 = reinterpret_cast<const float4 *>(g);
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            const float4 u = g4[e], v = g4[N / 2 + e];
            x[2 * e] = c2_make(make_float2(u.x, u.y), make_float2(v.x, v.y));
            x[2 * e + 1] = c2_make(make_float2(u.z, u.w), make_float2(v.z, v.w));
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = c2_make(g[t + T * e], g[N + t + T * e]);
    }
    ulonglong2 *sm = reinterpret_cast<ulonglong2 *>(smem4 + PHASE_TAB) + line * B::S;
    const float4 *tw = a.tw2;
    if (a.mode & MODE_INV) line_fft2<N, V, true>(x, sm, t, tw, Sync{}, at);
    const uint64_t c = a.pot[r >> a.log_rows];
    if constexpr (T == 1) {
        const uint2 *f2 = reinterpret_cast<const uint2 *>(fq);
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            const uint2 p = __ldg(&f2[e]), q = __ldg(&f2[N / 2 + e]);
            x[2 * e] = apply_phase_tab2(x[2 * e], turns_mul(c, p.x) + a.dither, turns_mul(c, q.x) + a.dither, ptab);
            x[2 * e + 1] = apply_phase_tab2(x[2 * e + 1], turns_mul(c, p.y) + a.dither, turns_mul(c, q.y) + a.dither, ptab);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = t + T * e;
            x[e] = apply_phase_tab2(x[e], turns_mul(c, __ldg(&fq[i])) + a.dither,
                                    turns_mul(c, __ldg(&fq[N + i])) + a.dither, ptab);
        }
    }
    // not at 1024 points, where the check alone costs the passes 1%
    if constexpr (N < 1024) grid_release_upto(SMALL_GRID);
    if (a.mode & MODE_FWD) line_fft2<N, V, false>(x, sm, t, tw, Sync{}, at);
    if (valid) {
        if constexpr (T == 1) {
            float4 *g4 = reinterpret_cast<float4 *>(g);
#pragma unroll
            for (int e = 0; e < E / 2; ++e) {
                const float2 a0 = c2_first(x[2 * e]), b0 = c2_second(x[2 * e]);
                const float2 a1 = c2_first(x[2 * e + 1]), b1 = c2_second(x[2 * e + 1]);
                g4[e] = make_float4(a0.x, a0.y, a1.x, a1.y);
                g4[N / 2 + e] = make_float4(b0.x, b0.y, b1.x, b1.y);
            }
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                g[t + T * e] = c2_first(x[e]);
                g[N + t + T * e] = c2_second(x[e]);
            }
        }
    }
    grid_release();
}

// ------------------------------------------------------ strided axis pass
// Lines of length N at stride `inner`; a block owns CP adjacent pairs of columns
// of one plane, lanes run along the pairs, so each 16-byte access moves both
// columns of a pair and each row of a tile is 16 CP contiguous bytes.
// FLAT: a plane has fewer than CP pairs, and a block takes several planes' (the
// last block what is left); with one plane per block such passes ran on blocks of
// inner / 2 * T threads (1024x8x8 x 256, whose axis 1 had blocks of 4 threads: 816 us
// per step, 366 with full ones).
// Resident blocks: 4 of 128 threads with 8 points per thread; 3 with 16 (at 4,
// the 128 registers a thread may then use spill: 256^3 axis-0 pass 69 us, 66 at 3).
template <int N, int V, int CP> constexpr int axis_min_blocks() {
    constexpr int threads = CP * Line2<N, V>::T;
    return threads < 128 ? 1 : (Line2<N, V>::E == 16 ? 3 : 4) * 128 / threads;
}

template <int N, int V, int CP, bool FLAT>
__global__ void __launch_bounds__(CP * Line2<N, V>::T, axis_min_blocks<N, V, CP>()) k_axis(AxisArgs a) {
    using C = Line2<N, V>;
    using B = ColBuf<N, V, CP>;
    const ColBufAddr<N, V, CP> at;
    constexpr int E = C::E, T = C::T;
    extern __shared__ __align__(16) float4 smem4[];
    const int c = threadIdx.x % CP, t = threadIdx.x / CP;
    constexpr int LOG_W = CP == 32 ? 6 : CP == 16 ? 5 : CP == 8 ? 4 : CP == 4 ? 3 : CP == 2 ? 2 : 1;  // log2(2 CP)
    static_assert(1 << LOG_W == 2 * CP, "tile width");
    int64_t o, tile, ci;
    if (FLAT) {
        const int64_t pair = (int64_t)blockIdx.x * CP + c;
        o = pair >> (a.log_inner - 1);
        tile = 0;
        ci = 2 * (pair - (o << (a.log_inner - 1)));
    } else {
        o = blockIdx.x >> (a.log_inner - LOG_W);
        tile = blockIdx.x - (o << (a.log_inner - LOG_W));
        ci = tile * (2 * CP) + 2 * c;
    }
    const bool valid = !FLAT || o < a.planes;
    if (!valid) o = 0;
    float4 *g = reinterpret_cast<float4 *>(a.psi + o * (int64_t)N * a.inner + ci);
    const int64_t stride = a.inner / 2;
    // so many one-warp blocks leave even room everywhere
    if (T == 1 && gridDim.x > 152 * 24) grid_release();
    grid_release_upto(TINY_GRID);
    grid_wait();
    c2 x[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const float4 v = valid ? g[(int64_t)(t + T * e) * stride] : make_float4(0.f, 0.f, 0.f, 0.f);
        x[e] = c2_make(make_float2(v.x, v.y), make_float2(v.z, v.w));
    }
    ulonglong2 *sm = reinterpret_cast<ulonglong2 *>(smem4) + c * B::S;
    const float4 *tw = a.tw2;
    // zero-mode split (qhd_device.cuh) in the forward-kinetic-inverse pass, for
    // the tile holding column 0 (frequency 0 of the other axes) of each
    // instance: the T threads of a column span several warps, so their partial
    // sums meet in the exchange buffer's space and every thread adds them in the
    // same order.  The sum, later its part of the result, waits in a slot behind
    // the buffer, so that no other tile's pass holds registers for it.
    constexpr int ALL3 = MODE_FWD | MODE_KIN | MODE_INV;
    const bool split0 = (a.mode & ALL3) == ALL3 && tile == 0;  // FLAT: every block has a column 0
    ulonglong2 *slot = reinterpret_cast<ulonglong2 *>(smem4) + (C::STAGES > 1 ? CP * B::S : 0) + c;
    if (split0) {
        ulonglong2 *red = reinterpret_cast<ulonglong2 *>(smem4);
        c2 s = x[0];
#pragma unroll
        for (int e = 1; e < E; ++e) s = s + x[e];
        if (T > 1) {
            st_c2(&red[t * CP + c], s);
            __syncthreads();
            s = ld_c2(&red[c]);
#pragma unroll 1
            for (int q = 1; q < T; ++q) s = s + ld_c2(&red[q * CP + c]);
            __syncthreads();
        }
        const c2 mu{s.x * pf_dup(1.0f / N), s.y * pf_dup(1.0f / N)};
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = x[e] - mu;
        if (t == 0) st_c2(slot, s);
    }
    if (a.mode & MODE_FWD) line_fft2<N, V, false>(x, sm, t, tw, BlockSync{}, at);
    if (a.mode & MODE_KIN) {
        // axis 0 pass: plane index o is the instance.  The per-axis factors are
        // FP32 hi/lo pairs applied with compensated products: a table entry is
        // shared by every point with the same frequency index, so a plain FP32
        // rounding of it would perturb the norm coherently.  The factors of axes 1
        // and 2 are the same for the whole column: their product (hi/lo again) is
        // formed once.  Plain loads: k_prep may still write the tables when this
        // block starts, which the read-only path does not allow.
        const float4 *kb = a.kt + (a.kt_batch == 1 ? 0 : o) * a.ksum;
        w2 kc;
        if (a.ndim == 2) {
            kc = w2_make(kb[a.koff1 + ci], kb[a.koff1 + ci + 1]);
        } else {
            int64_t i1 = ci >> a.log_n2;
            const int i2 = (int)(ci & ((1 << a.log_n2) - 1));
            if (a.perm1_c) i1 = (i1 >> a.perm1_log_r) + a.perm1_c * (i1 & ((1 << a.perm1_log_r) - 1));
            const float4 k1 = kb[a.koff1 + i1];
            kc = w2_mul(w2_make(k1, k1), w2_make(kb[a.koff2 + i2], kb[a.koff2 + i2 + 1]));
        }
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = c2_mul<false>(c2_mul_shared<false>(x[e], kb[t + T * e]), kc);
        // the mean's part: N mu = sum through the factor of frequency 0
        if (split0 && t == 0) st_c2(slot, c2_mul<false>(c2_mul_shared<false>(ld_c2(slot), kb[0]), kc));
    }
    if constexpr (N < 1024) grid_release_upto(SMALL_GRID);
    if (a.mode & MODE_INV) line_fft2<N, V, true>(x, sm, t, tw, BlockSync{}, at);
    if (split0) {
        // written by the column's thread 0 before the inverse transform's barriers
        const c2 mean_part = ld_c2(slot);
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = x[e] + mean_part;
    }
    if (valid) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float2 p = c2_first(x[e]), q = c2_second(x[e]);
            g[(int64_t)(t + T * e) * stride] = make_float4(p.x, p.y, q.x, q.y);
        }
    }
    grid_release();
}

// --------------------------------------------- 1-D: a whole chunk per launch
// OVERLAP: launched to overlap k_prep, so the kinetic tables are read with plain
// loads, as in k_axis; those wait for the exchanges before them, where __ldg may be
// issued ahead (100 steps of 256 points: 259 us with plain loads, 248 with __ldg), so
// chunks that do not overlap keep it.
template <int N, bool OVERLAP>
__global__ void __launch_bounds__(ROW_THREADS) k_oned(OneDArgs a) {
    using C = LineCfg<N>;
    constexpr int E = C::E, T = C::T;
    constexpr int S = line_stride<N>();
    extern __shared__ __align__(16) float4 smem4[];
    float4 *ptab = smem4;
    float2 *smem = reinterpret_cast<float2 *>(smem4 + PHASE_TAB);
    grid_release();
    load_phase_tab(ptab, a.ptab);
    __syncthreads();
    grid_wait();
    const int lpb = blockDim.x / T;
    const int line = threadIdx.x / T, t = threadIdx.x % T;
    const int64_t row = (int64_t)blockIdx.x * lpb + line;
    const bool valid = row < a.batch;
    const int64_t b = valid ? row : 0;
    float2 *g = a.psi + b * N;
    const uint32_t *fq = a.fq + b * N;
    float2 x[E];
    uint32_t fv[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        x[e] = g[t + T * e];
        fv[e] = fq[t + T * e];
    }
    float2 *sm = smem + (C::TWO_STAGE ? line * S : 0);
    for (int j = 0; j < a.cnt; ++j) {
        const uint64_t c = a.pot[(int64_t)j * a.batch + b];
        const uint32_t dz = step_dither(a.dither_base + (uint64_t)j);
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = apply_phase_tab(x[e], turns_mul(c, fv[e]) + dz, ptab);
        // zero-mode split (qhd_device.cuh): the line is the whole instance, so
        // its zero mode is the global one
        const float2 sum = line_sum_lanes<E, T>(x);
        sub_line_mean<N, E>(x, sum);
        line_fft<N, false>(x, sm, t, a.tw2, WarpSync{});
        const float4 *kb = a.kt + ((int64_t)j * a.kt_batch + (a.kt_batch == 1 ? 0 : b)) * N;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float4 k0 = OVERLAP ? kb[t + T * e] : __ldg(&kb[t + T * e]);
            x[e] = cmul_comp(x[e], make_float2(k0.x, k0.y), make_float2(k0.z, k0.w));
        }
        const float4 z0 = OVERLAP ? kb[0] : __ldg(&kb[0]);
        const float2 mean_part = cmul_comp(sum, make_float2(z0.x, z0.y), make_float2(z0.z, z0.w));
        line_fft<N, true>(x, sm, t, a.tw2, WarpSync{});
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = cadd(x[e], mean_part);
    }
    if (a.final_phase) {
        const uint64_t c = a.pot[(int64_t)a.cnt * a.batch + b];
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = apply_phase_tab(x[e], turns_mul(c, fv[e]), ptab);
    }
    if (valid) {
#pragma unroll
        for (int e = 0; e < E; ++e) g[t + T * e] = x[e];
    }
}

// ------------------------------------------------------------- prep kernel
// Schedule evaluation at the step midpoints, the merged potential coefficients
// and the per-axis kinetic phase tables of one chunk of steps (qhd_prep.cuh).

// EARLY: releases the next kernel at the start (qhd_launch.cuh).
template <bool EARLY>
__global__ void k_prep(PrepArgs a) {
    const int64_t jl = blockIdx.x;  // local step 0..cnt (cnt is the extra potential entry)
    const int64_t b = blockIdx.y;
    __shared__ uint64_t s_k[3];
    __shared__ double s_fd[3];
    if (EARLY) grid_release();
    uint64_t pot = 0;
    if (threadIdx.x == 0) pot = prep_coefficients(a, jl, b, s_k, s_fd);
    __syncthreads();
    // the schedules and the potential's scale were loaded under a synchronisation,
    // the tables are read by the passes before: compute first, wait, then write
    const bool row = jl < a.cnt && b < a.kt_batch;
    const int i0 = (int)(blockIdx.z * blockDim.x + threadIdx.x), stride = (int)(gridDim.z * blockDim.x);
    const bool one = row && i0 < a.ksum;
    const float4 first = one ? prep_kinetic_entry(a, i0, s_k, s_fd) : make_float4(0.f, 0.f, 0.f, 0.f);
    grid_wait();
    if (threadIdx.x == 0 && blockIdx.z == 0) a.pot[jl * a.batch + b] = pot;
    if (one) {
        float4 *out = a.kt + (jl * a.kt_batch + b) * a.ksum;
        out[i0] = first;
        for (int i = i0 + stride; i < a.ksum; i += stride) out[i] = prep_kinetic_entry(a, i, s_k, s_fd);
    }
    if (!EARLY) grid_release();
}

// ------------------------------------------------------------ small kernels
__global__ void k_uniform(float2 *psi, int64_t count, float v) {
    grid_release();
    grid_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        psi[i] = make_float2(v, 0.0f);
}

// Lowest value (lowest index on ties), highest value and non-finite count of the
// block's 256 threads, in thread 0.
__device__ __forceinline__ MinMaxPart minmax_block(MinMaxPart v) {
    __shared__ MinMaxPart sh[256];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w /= 2) {
        if ((int)threadIdx.x < w) {
            const MinMaxPart o = sh[threadIdx.x + w];
            MinMaxPart &m = sh[threadIdx.x];
            if (o.fmin < m.fmin || (o.fmin == m.fmin && o.argmin < m.argmin)) {
                m.fmin = o.fmin;
                m.argmin = o.argmin;
            }
            m.fmax = fmax(m.fmax, o.fmax);
            m.nonfinite += o.nonfinite;
        }
        __syncthreads();
    }
    return sh[0];
}

__global__ void __launch_bounds__(256) k_minmax(const double *f, int64_t g, MinMaxPart *part) {
    const int64_t b = blockIdx.y;
    const double *fb = f + b * g;
    MinMaxPart m{INFINITY, -INFINITY, INT64_MAX, 0};
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < g;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double v = fb[i];
        if (!isfinite(v)) {
            ++m.nonfinite;
            continue;
        }
        if (v < m.fmin || (v == m.fmin && i < m.argmin)) {
            m.fmin = v;
            m.argmin = i;
        }
        m.fmax = fmax(m.fmax, v);
    }
    m = minmax_block(m);
    if (threadIdx.x == 0) part[b * gridDim.x + blockIdx.x] = m;
}

// out[b] of the nblk partials of instance b.
__global__ void __launch_bounds__(256) k_minmax_final(const MinMaxPart *part, int nblk, MinMaxPart *out) {
    const int64_t b = blockIdx.x;
    MinMaxPart m{INFINITY, -INFINITY, INT64_MAX, 0};
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
        const MinMaxPart p = part[b * nblk + i];
        if (p.fmin < m.fmin || (p.fmin == m.fmin && p.argmin < m.argmin)) {
            m.fmin = p.fmin;
            m.argmin = p.argmin;
        }
        m.fmax = fmax(m.fmax, p.fmax);
        m.nonfinite += p.nonfinite;
    }
    m = minmax_block(m);
    if (threadIdx.x == 0) out[b] = m;
}

__global__ void k_quantize(const double *f, uint32_t *fq, const InstDev *inst, int64_t g, int64_t total) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const InstDev &p = inst[i / g];
        double q = rint(ldexp(f[i] - p.fmin, p.shift));
        q = fmin(fmax(q, 0.0), 4294967295.0);
        fq[i] = (uint32_t)q;
    }
}

// Observables: FP64 partial sums per block, then a fixed-order final sum.
__device__ __forceinline__ double block_sum(double v, double *sh) {
    for (int o = 16; o > 0; o /= 2) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x / 32, l = threadIdx.x % 32;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x / 32); ++i) s += sh[i];
    return s;
}

// FP64 bounds it (5.3e11 FMA/s on the whole GPU, 1/74 of the FP32 rate), so each
// point costs only its own products: the squared coordinate distances to x* are one
// table per block, and the distance is compared squared, with the largest square
// whose root is below the radius.  256^3 with |psi|^2, the call: 932 us with a square
// root and the coordinates' arithmetic per point, 449 so.
__global__ void __launch_bounds__(256) k_obs_partial(ObsArgs a) {
    extern __shared__ double d2[];  // (x - x*)^2 per axis, at a.coff[d]
    const int64_t b = blockIdx.y;
    const float2 *psi = a.psi + b * a.g;
    const double *f = a.f64 + b * a.g;
    const InstDev &ip = a.inst[b];
    grid_release();
    if (a.await_tables) grid_wait();
    for (int d = 0; d < a.ndim; ++d)
        for (int i = threadIdx.x; i < a.n[d]; i += blockDim.x) {
            const double dx = __dsub_rn(a.coord[a.coff[d] + i], ip.xs[d]);
            d2[a.coff[d] + i] = __dmul_rn(dx, dx);
        }
    __syncthreads();
    grid_wait();
    double sn = 0.0, sf = 0.0, sp = 0.0;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.g;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float2 z = psi[i];
        const double p = __dadd_rn(__dmul_rn((double)z.x, (double)z.x), __dmul_rn((double)z.y, (double)z.y));
        if (a.prob) a.prob[b * a.g + i] = (float)p;
        sn += p;
        sf += p * f[i];
        // squared Euclidean distance to x*, summed in the same order as a plain
        // loop over the axes from the last to the first
        const uint32_t idx = (uint32_t)i;  // G <= 2^30
        double r2 = d2[a.coff[a.ndim - 1] + (idx & (a.n[a.ndim - 1] - 1))];
        if (a.ndim > 1) {
            uint32_t rem = idx >> a.log_n[a.ndim - 1];
            r2 = __dadd_rn(r2, d2[a.coff[a.ndim - 2] + (rem & (a.n[a.ndim - 2] - 1))]);
            if (a.ndim > 2) r2 = __dadd_rn(r2, d2[rem >> a.log_n[1]]);
        }
        if (r2 <= a.r2_max) sp += p;
    }
    __shared__ double sh[32];
    const double tn = block_sum(sn, sh);
    const double tf = block_sum(sf, sh);
    const double tp = block_sum(sp, sh);
    if (threadIdx.x == 0) {
        double *o = a.partial + (b * a.nblk + blockIdx.x) * 3;
        o[0] = tn;
        o[1] = tf;
        o[2] = tp;
    }
}

__global__ void k_obs_final(ObsArgs a) {
    const int64_t b = blockIdx.x;
    __shared__ double sh[3][256];
    grid_release();
    grid_wait();
    for (int k = 0; k < 3; ++k) {
        double s = 0.0;
        for (int i = threadIdx.x; i < a.nblk; i += blockDim.x) s += a.partial[(b * a.nblk + i) * 3 + k];
        sh[k][threadIdx.x] = s;
    }
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w /= 2) {
        if (threadIdx.x < w)
            for (int k = 0; k < 3; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 3; ++k) a.result[b * 3 + k] = sh[k][0];
}

// ---------------------------------------------------------------- launchers
template <int N, int V>
static cudaError_t row_v_impl(const RowArgs &a, cudaStream_t s) {
    using C = Line2<N, V>;
    constexpr int PAIRS = ROW_THREADS / C::T;
    const int64_t blocks = (a.rows / 2 + PAIRS - 1) / PAIRS;
    constexpr size_t sm =
        PHASE_TAB * sizeof(float4) + (C::STAGES > 1 ? (size_t)PAIRS * RowBuf<N, V>::S * sizeof(ulonglong2) : 0);
    static_assert(sm <= 48 * 1024, "default shared-memory limit");
    RowArgs r = a;
    r.tw2 += V * TW2_TABLE * N;
    return launch_overlapped(a.rows * N < OVERLAP_POINTS, k_row<N, V>, dim3((unsigned)blocks), dim3(ROW_THREADS), sm, s, r);
}

template <int N>
static cudaError_t row_impl(const RowArgs &a, cudaStream_t s) {
    if constexpr (two_plans(N))
        if (a.rows * N > BIG_PLAN_POINTS) return row_v_impl<N, 1>(a, s);
    return row_v_impl<N, 0>(a, s);
}

// Pairs of columns per tile of a strided pass: 128 threads per block, at most
// 32 pairs (512-byte row segments); 256 threads at 512 points, where 2 pairs are
// only 32 bytes of each row (512^2 x 64 188 us per step, 183 with 4 pairs).
__host__ __device__ constexpr int axis_cp(int n, int t) {
    return n == 512 ? 4 : t >= 64 ? 2 : 128 / t > 32 ? 32 : 128 / t;
}

template <int N, int V, int CP, bool FLAT>
static cudaError_t axis_tile_impl(const AxisArgs &a, cudaStream_t s) {
    using C = Line2<N, V>;
    const int64_t blocks = FLAT ? (a.planes * (a.inner / 2) + CP - 1) / CP : a.planes * (a.inner / (2 * CP));
    // exchange buffer (the zero-mode split's CP T partial sums use it too), then
    // that split's slot per pair
    constexpr size_t xch = ((C::STAGES > 1 ? (size_t)CP * ColBuf<N, V, CP>::S : 0) + CP) * sizeof(ulonglong2);
    static_assert(xch <= 48 * 1024, "default shared-memory limit");
    AxisArgs r = a;
    r.tw2 += V * TW2_TABLE * N;
    return launch_overlapped(a.planes * a.inner * N < OVERLAP_POINTS, k_axis<N, V, CP, FLAT>, dim3((unsigned)blocks),
                             dim3(CP * C::T), xch, s, r);
}

// Planes narrower than a tile: full blocks where they reach every SM, else blocks of
// about a warp (512x2 x 16: 6.7 us per step, 8.3 with 4 blocks of 256 threads).
template <int N, int V>
static cudaError_t axis_v_impl(const AxisArgs &a, cudaStream_t s) {
    constexpr int T = Line2<N, V>::T, CP = axis_cp(N, T), NARROW = T >= 32 ? 1 : 32 / T;
    if (a.inner >= 2 * CP) return axis_tile_impl<N, V, CP, false>(a, s);
    if (a.planes * (a.inner / 2) >= 152 * CP) return axis_tile_impl<N, V, CP, true>(a, s);
    if (a.inner >= 2 * NARROW) return axis_tile_impl<N, V, NARROW, false>(a, s);
    return axis_tile_impl<N, V, NARROW, true>(a, s);
}

template <int N>
static cudaError_t axis_impl(const AxisArgs &a, cudaStream_t s) {
    if constexpr (two_plans(N))
        if (a.planes * a.inner * N > BIG_PLAN_POINTS) return axis_v_impl<N, 1>(a, s);
    return axis_v_impl<N, 0>(a, s);
}

template <int N>
static cudaError_t oned_impl(const OneDArgs &a, cudaStream_t s) {
    using C = LineCfg<N>;
    constexpr int S = line_stride<N>();
    const int lpb = ROW_THREADS / C::T;
    const int64_t blocks = (a.batch + lpb - 1) / lpb;
    const size_t sm = PHASE_TAB * sizeof(float4) + (C::TWO_STAGE ? (size_t)lpb * S * sizeof(float2) : 0);
    const dim3 grid((unsigned)blocks), block(ROW_THREADS);
    return a.cnt <= OVERLAP_STEPS ? launch_overlapped(true, k_oned<N, true>, grid, block, sm, s, a)
                                  : launch_overlapped(false, k_oned<N, false>, grid, block, sm, s, a);
}

#define QHD_DISPATCH_N(n, fn, ...)                        \
    switch (n) {                                          \
    case 2: return fn<2>(__VA_ARGS__);                    \
    case 4: return fn<4>(__VA_ARGS__);                    \
    case 8: return fn<8>(__VA_ARGS__);                    \
    case 16: return fn<16>(__VA_ARGS__);                  \
    case 32: return fn<32>(__VA_ARGS__);                  \
    case 64: return fn<64>(__VA_ARGS__);                  \
    case 128: return fn<128>(__VA_ARGS__);                \
    case 256: return fn<256>(__VA_ARGS__);                \
    case 512: return fn<512>(__VA_ARGS__);                \
    case 1024: return fn<1024>(__VA_ARGS__);              \
    default: return cudaErrorInvalidValue;                \
    }

cudaError_t launch_row(int n, const RowArgs &a, cudaStream_t s) { QHD_DISPATCH_N(n, row_impl, a, s) }
cudaError_t launch_axis(int n, const AxisArgs &a, cudaStream_t s) { QHD_DISPATCH_N(n, axis_impl, a, s) }
cudaError_t launch_oned(int n, const OneDArgs &a, cudaStream_t s) { QHD_DISPATCH_N(n, oned_impl, a, s) }

cudaError_t launch_prep(const PrepArgs &a, bool early, cudaStream_t s) {
    // FP64 bounds a row's entries (1.7 FMA per clock and SM): short chunks of few
    // instances share each row among blocks (1024^2 x 2, 8 evolutions of 3 steps: 985 us
    // with a block per row, 832 so)
    const int64_t split = (a.ksum + 255) / 256;
    dim3 grid((unsigned)(a.cnt + 1), (unsigned)a.batch, (a.cnt + 1) * a.batch * split <= 152 * 8 ? (unsigned)split : 1u);
    return launch_overlapped(true, early ? k_prep<true> : k_prep<false>, grid, dim3(256), 0, s, a);
}

cudaError_t load_prep() {
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, k_prep<true>);
    return e == cudaSuccess ? cudaFuncGetAttributes(&fa, k_prep<false>) : e;
}

cudaError_t launch_uniform(float2 *psi, int64_t count, float value, cudaStream_t s) {
    int64_t blocks = (count + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    return launch_overlapped(true, k_uniform, dim3((unsigned)blocks), dim3(256), 0, s, psi, count, value);
}

cudaError_t launch_minmax(const double *f, int64_t g, int64_t batch, MinMaxPart *part, int nblk,
                          cudaStream_t s) {
    k_minmax<<<dim3((unsigned)nblk, (unsigned)batch), 256, 0, s>>>(f, g, part);
    return cudaGetLastError();
}

cudaError_t launch_quantize(const double *f, uint32_t *fq, const InstDev *inst, int64_t g,
                            int64_t batch, cudaStream_t s) {
    const int64_t total = g * batch;
    int64_t blocks = (total + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    k_quantize<<<(unsigned)blocks, 256, 0, s>>>(f, fq, inst, g, total);
    return cudaGetLastError();
}

cudaError_t launch_observables(const ObsArgs &a, int64_t batch, cudaStream_t s) {
    int ksum = 0;
    for (int d = 0; d < a.ndim; ++d) ksum += a.n[d];
    ObsArgs o = a;
    // squares up to this are the ones whose (correctly rounded) root is below the radius
    o.r2_max = a.radius * a.radius;
    while (std::sqrt(o.r2_max) < a.radius) o.r2_max = std::nextafter(o.r2_max, INFINITY);
    while (!(std::sqrt(o.r2_max) < a.radius)) o.r2_max = std::nextafter(o.r2_max, 0.0);
    // as many blocks as fill the GPU: the tables and the block sums cost as much as
    // hundreds of points
    const int64_t want = (152 * 8 + batch - 1) / batch;
    if (want < o.nblk) o.nblk = (int)want;
    cudaError_t e = launch_overlapped(true, k_obs_partial, dim3((unsigned)o.nblk, (unsigned)batch), dim3(256),
                                      ksum * sizeof(double), s, o);
    if (e != cudaSuccess) return e;
    return launch_overlapped(true, k_obs_final, dim3((unsigned)batch), dim3(256), 0, s, o);
}

template <int N> static void plan2_radix(int v, int *radix, int *stages) {
    for (int k = 0; k < 4; ++k) radix[k] = v ? Plan2<N, 1>::R[k] : Plan2<N, 0>::R[k];
    *stages = v ? Line2<N, 1>::STAGES : Line2<N, 0>::STAGES;
}
void plan2_of(int n, int v, int *radix, int *stages) {
    switch (n) {
#define QHD_PLAN2_CASE(N) \
    case N: return plan2_radix<N>(v, radix, stages);
        QHD_PLAN2_CASE(2) QHD_PLAN2_CASE(4) QHD_PLAN2_CASE(8) QHD_PLAN2_CASE(16) QHD_PLAN2_CASE(32)
        QHD_PLAN2_CASE(64) QHD_PLAN2_CASE(128) QHD_PLAN2_CASE(256) QHD_PLAN2_CASE(512) QHD_PLAN2_CASE(1024)
#undef QHD_PLAN2_CASE
    default: *stages = 0;
    }
}

cudaError_t launch_minmax_final(const MinMaxPart *part, int nblk, int64_t batch, MinMaxPart *out, cudaStream_t s) {
    k_minmax_final<<<(unsigned)batch, 256, 0, s>>>(part, nblk, out);
    return cudaGetLastError();
}

void plan_of(int n, int *r1, int *r2) {
    switch (n) {
#define QHD_PLAN_CASE(N)      \
    case N:                   \
        *r1 = Plan<N>::R1;    \
        *r2 = Plan<N>::R2;    \
        return;
        QHD_PLAN_CASE(2) QHD_PLAN_CASE(4) QHD_PLAN_CASE(8) QHD_PLAN_CASE(16) QHD_PLAN_CASE(32)
        QHD_PLAN_CASE(64) QHD_PLAN_CASE(128) QHD_PLAN_CASE(256) QHD_PLAN_CASE(512) QHD_PLAN_CASE(1024)
#undef QHD_PLAN_CASE
    default:
        *r1 = 0;
        *r2 = 0;
    }
}

bool supported_n(int64_t n) { return n >= 2 && n <= 1024 && (n & (n - 1)) == 0; }

}  // namespace qhd
