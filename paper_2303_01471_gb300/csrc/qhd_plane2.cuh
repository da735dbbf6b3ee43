// qhd_plane2.cuh -- plane engine on pairs of rows in packed FP32.
//
// A plane of N1 x N2 points (a whole 2-D instance, or the last two axes of a 3-D
// grid for one index of axis 0) is held in shared memory as pairs of rows: a tile
// element is 16 bytes, one column of two rows, and all arithmetic is on packed
// pairs (qhd_packed.cuh).  Two forms:
//
// * Solo (planes of up to 16384 points, 151 KB): one CTA holds the plane.  Row
//   transforms as in the line engine, T2 threads per pair of rows; column
//   transforms by T1 = 4 threads per column, 8 columns and 4 threads in a warp, so
//   that both exchange inside a warp and a step has two block barriers, no cluster
//   barrier and no distributed shared memory.  On 128^2 the scalar cluster engine
//   spent 3.1 of 6.8 cycles between issues on barriers, fences and remote loads;
//   152 instances take 18.6 us per step, 26.6 on clusters.
// * Cluster (larger planes of 3-D passes): C CTAs of R = N1 / C rows each and a
//   four-step transform along axis N1 through distributed shared memory, as in
//   qhd_plane.cuh.
//
// Pairs: in position space pair p of a CTA's rows holds rows 2p and 2p + 1, in
// Fourier space rows p and p + RP (RP = half the rows).  The transform along the
// column turns the one into the other without moving lanes: an RP-point packed
// DFT transforms the even rows in one lane and the odd rows in the other, and the
// last radix-2 step combines the two lanes of each register pair (the inverse
// runs the same steps backwards).
#pragma once
#include <cooperative_groups.h>
#include <type_traits>

#include "qhd_kernels.h"
#include "qhd_launch.cuh"
#include "qhd_packed.cuh"
#include "qhd_plane.cuh"

namespace qhd {

namespace cg = cooperative_groups;

// Largest plane of the solo form, in points (and columns of at most 128: four
// threads hold 16 pairs of points each).
constexpr int SOLO_POINTS = 16384;
__host__ __device__ constexpr bool plane_solo(int n1, int n2) { return n1 <= 128 && n1 * n2 <= SOLO_POINTS; }

// C = 1: solo.  V: plan of the rows.
template <int N1_, int N2_, int C_, int V_> struct Plane2 {
    static constexpr int N1 = N1_, N2 = N2_, C = C_, V = V_;
    static constexpr int R = N1 / C;                       // rows per CTA
    static constexpr int RP = R / 2;                       // row pairs
    static constexpr int T1 = 4;                           // solo: threads per column
    static constexpr int THREADS = C > 1 ? N2 : T1 * N2 > 512 ? 512 : T1 * N2;
    using RowC = Line2<N2, V>;
    static constexpr int S = RowBuf<N2, V>::S;             // row-pair stride in 16-byte elements
    static constexpr int T2 = RowC::T, E2 = RowC::E;
    static constexpr int PAIRS_PER_ITER = THREADS / T2;
    static constexpr int OWNED = RP * N2 / C;              // exchange positions (pairs of rows) per CTA
    // rows, then the slot of the zero-mode split
    static constexpr size_t TILE = ((size_t)RP * S + 1) * sizeof(ulonglong2);
    static constexpr size_t SMEM = PHASE_TAB * sizeof(float4) + TILE;
    static_assert(RowC::STAGES > 1, "rows of at least 32 points");
    static_assert(N1 % C == 0 && R % 2 == 0 && RP * N2 % C == 0, "even rows per CTA, equal exchange shares");
    static_assert(C == 1 || RP <= 16, "cluster form: local column transform held in registers");
    static_assert(T2 <= 32 && 32 % T2 == 0, "a pair of rows lives in one warp");
};

// Solo form: 16 points of a row pair per thread (plan 1) where that leaves no
// thread idle in the row phase (64x128 x 512: 39.9 us per step with 8 points, 52.8
// with 16 and half of the threads idle); rows of 256 points with 8 (64x256 x 1216 148.9,
// 151.9 with 16).
template <int N1, int N2> constexpr int solo_row_plan() {
    using P = Plane2<N1, N2, 1, 1>;
    return N2 < 256 && P::RP * P::T2 >= P::THREADS ? 1 : 0;
}
template <int N1, int N2> using Solo = Plane2<N1, N2, 1, solo_row_plan<N1, N2>()>;

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Global <-> shared copy of this CTA's rows (contiguous in global memory) in position
// space: pair p = rows 2p, 2p + 1.  16-byte global accesses, two columns
// of one row each.
template <typename P, bool TO_SHARED>
__device__ __forceinline__ void plane2_copy(ulonglong2 *tile, float2 *g, int tid) {
    constexpr int N2 = P::N2;
    constexpr int Q = P::RP * N2 / 2;  // column pairs of a row pair
#pragma unroll 4
    for (int i = tid; i < Q; i += P::THREADS) {
        const int p = (2 * i) / N2, col = (2 * i) % N2;
        float4 *r0 = reinterpret_cast<float4 *>(g + (int64_t)(2 * p) * N2 + col);
        float4 *r1 = reinterpret_cast<float4 *>(g + (int64_t)(2 * p + 1) * N2 + col);
        ulonglong2 *s = tile + p * P::S + col;
        if (TO_SHARED) {
            const float4 a = *r0, b = *r1;
            st_c2(&s[0], c2_make(make_float2(a.x, a.y), make_float2(b.x, b.y)));
            st_c2(&s[1], c2_make(make_float2(a.z, a.w), make_float2(b.z, b.w)));
        } else {
            const c2 u = ld_c2(&s[0]), v = ld_c2(&s[1]);
            const float2 a = c2_first(u), b = c2_first(v), c = c2_second(u), d = c2_second(v);
            *r0 = make_float4(a.x, a.y, b.x, b.y);
            *r1 = make_float4(c.x, c.y, d.x, d.y);
        }
    }
}

// Last radix-2 step of the local column transform on one register pair: lane 0
// holds E[k], lane 1 O[k]; out (E + w O, E - w O), w = W_R^k.  Inverse: lanes
// (X[k], X[k + RP]) to (X[k] + X[k + RP], (X[k] - X[k + RP]) conj(w)).
template <int R, bool INV> __device__ __forceinline__ c2 lane_butterfly(c2 v, int k) {
    float2 a = c2_first(v), b = c2_second(v);
    if (!INV) {
        b = twiddle_const<R, false>(b, k);
        return c2_make(cadd(a, b), csub(a, b));
    }
    return c2_make(cadd(a, b), twiddle_const<R, true>(csub(a, b), k));
}

// Cluster form: local transform along the distributed axis, one thread per column.
template <typename P, bool INV>
__device__ __forceinline__ void plane2_columns(ulonglong2 *tile, int tid) {
    {
        c2 v[P::RP];
#pragma unroll
        for (int p = 0; p < P::RP; ++p) v[p] = ld_c2(&tile[p * P::S + tid]);
        if (INV) {
#pragma unroll
            for (int p = 0; p < P::RP; ++p) v[p] = lane_butterfly<P::R, true>(v[p], p);
        }
        dft2<P::RP, INV>(v);
        if (!INV) {
#pragma unroll
            for (int p = 0; p < P::RP; ++p) v[p] = lane_butterfly<P::R, false>(v[p], p);
        }
#pragma unroll
        for (int p = 0; p < P::RP; ++p) st_c2(&tile[p * P::S + tid], v[p]);
    }
}

// lane_butterfly with the twiddle from memory (hi, lo).
template <bool INV> __device__ __forceinline__ c2 lane_butterfly_tab(c2 v, float4 w) {
    const float2 a = c2_first(v), b = c2_second(v);
    const float2 hi = make_float2(w.x, w.y), lo = make_float2(w.z, w.w);
    if (!INV) {
        const float2 wb = cmul_comp(b, hi, lo);
        return c2_make(cadd(a, wb), csub(a, wb));
    }
    return c2_make(cadd(a, b), cmulc_comp(csub(a, b), hi, lo));
}

struct Warp2Sync {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};

// Solo form: the columns, in one pass over the tile: inverse transform of the
// previous step, potential phase, forward transform.  T1 threads per column; lane
// = 8 t + column, so that a quarter warp moves 8 neighbouring columns.  twc:
// exp(-2 pi i k / N1), k < RP, then the stage twiddles of an RP-point line
// (solo_twiddles).
template <typename P>
__device__ __forceinline__ void solo_columns(ulonglong2 *tile, bool inv, bool phase, bool fwd,
                                             const float4 *__restrict__ twc, const uint32_t *__restrict__ fq,
                                             uint64_t coef, uint32_t dither, const float4 *ptab, int tid) {
    using L = Line2<P::RP, 2>;
    constexpr int E = L::E, T = L::T, N2 = P::N2;
    static_assert(T == P::T1, "four threads per column");
    const int t = (tid % 32) / 8;
#pragma unroll 1
    for (int c = tid / 32 * 8 + tid % 8; c < N2; c += P::THREADS / T) {
        ulonglong2 *col = tile + c;
        const ColAddr<P::S> at;
        c2 x[E];
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = ld_c2(&col[(t + T * e) * P::S]);
        __syncwarp();
        if (inv) {
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = lane_butterfly_tab<true>(x[e], __ldg(&twc[t + T * e]));
            line_fft2<P::RP, 2, true>(x, col, t, twc + P::RP, Warp2Sync{}, at);
        }
        if (phase) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t *f = &fq[(int64_t)(2 * (t + T * e)) * N2 + c];
                x[e] = apply_phase_tab2(x[e], turns_mul(coef, __ldg(f)) + dither, turns_mul(coef, __ldg(f + N2)) + dither,
                                        ptab);
            }
        }
        if (fwd) {
            line_fft2<P::RP, 2, false>(x, col, t, twc + P::RP, Warp2Sync{}, at);
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = lane_butterfly_tab<false>(x[e], __ldg(&twc[t + T * e]));
        }
#pragma unroll
        for (int e = 0; e < E; ++e) st_c2(&col[(t + T * e) * P::S], x[e]);
        __syncwarp();
    }
}

// Zero-mode split (qhd_device.cuh): the row transform is the last forward
// transform before the kinetic factor, and local row 0 of CTA 0 (frequency 0
// along the column axis), lane 0 of pair 0, holds the global zero mode.  Its T2
// threads (lanes 0..T2-1 of warp 0, the ones that transform it) take the mean out
// of the shared-memory row before the row transforms and add the mean's part back
// after them, so those are the same for every row.  Out of line, with the part
// waiting behind the tile, so that the row transforms hold no registers for it.
template <typename P>
__device__ __noinline__ void plane2_zero_row_out(ulonglong2 *tile, const float4 *kt0, const float4 *kt1, int t) {
    constexpr int T2 = P::T2, E2 = P::E2;
    float2 v[E2];
#pragma unroll
    for (int e = 0; e < E2; ++e) v[e] = c2_first(ld_c2(&tile[t + T2 * e]));
    const float2 sum = line_sum_lanes<E2, T2>(v, T2 >= 32 ? 0xffffffffu : (1u << (T2 % 32)) - 1u);
    sub_line_mean<P::N2, E2>(v, sum);
#pragma unroll
    for (int e = 0; e < E2; ++e) st_c2(&tile[t + T2 * e], c2_make(v[e], c2_second(ld_c2(&tile[t + T2 * e]))));
    const float4 k0 = kt0[0], k1 = kt1[0];
    const float2 y = cmul_comp(sum, make_float2(k0.x, k0.y), make_float2(k0.z, k0.w));
    const float2 part = cmul_comp(y, make_float2(k1.x, k1.y), make_float2(k1.z, k1.w));
    if (t == 0) st_c2(&tile[P::RP * P::S], c2_make(part, make_float2(0.f, 0.f)));
}
template <typename P> __device__ __noinline__ void plane2_zero_row_back(ulonglong2 *tile, int t) {
    // each thread adds to the elements it stored itself; the part was stored before
    // the row transforms' warp barriers
    const c2 part = ld_c2(&tile[P::RP * P::S]);
#pragma unroll
    for (int e = 0; e < P::E2; ++e) st_c2(&tile[t + P::T2 * e], ld_c2(&tile[t + P::T2 * e]) + part);
}

// Rows along N2 with the kinetic phase in between (forward, factor, inverse), for
// the pairs in Fourier space.  The pair's own storage is the exchange buffer of
// the line engine (its content is in registers at that point).
template <typename P>
__device__ __forceinline__ void plane2_rows_kinetic(ulonglong2 *tile, const float4 *__restrict__ tw_row,
                                                    const float4 *kt0, const float4 *kt1, int tid) {
    static_assert(P::C == 1, "solo form");
    constexpr int T2 = P::T2, E2 = P::E2, N2 = P::N2, V = P::V;
    const RowAddr<Line2<N2, V>::LOG_R1> at;
    const int t = tid % T2;
    if (tid < T2) plane2_zero_row_out<P>(tile, kt0, kt1, t);
#pragma unroll 1
    for (int base = 0; base < P::RP; base += P::PAIRS_PER_ITER) {
        const int p = base + tid / T2;
        if (P::RP % P::PAIRS_PER_ITER == 0 || p < P::RP) {
            ulonglong2 *rp = tile + p * P::S;
            c2 x[E2];
#pragma unroll
            for (int e = 0; e < E2; ++e) x[e] = ld_c2(&rp[t + T2 * e]);
            __syncwarp();
            line_fft2<N2, V, false>(x, rp, t, tw_row, Warp2Sync{}, at);
            // rows p and p + RP hold these frequencies along the column axis; plain
            // loads: the step tables may still be written when the block starts
            const w2 k0 = w2_make(kt0[p], kt0[p + P::RP]);
#pragma unroll
            for (int e = 0; e < E2; ++e) x[e] = c2_mul_shared<false>(c2_mul<false>(x[e], k0), kt1[t + T2 * e]);
            line_fft2<N2, V, true>(x, rp, t, tw_row, Warp2Sync{}, at);
#pragma unroll
            for (int e = 0; e < E2; ++e) st_c2(&rp[t + T2 * e], x[e]);
        }
    }
    if (tid < T2) plane2_zero_row_back<P>(tile, t);
}

// Rows along N2, one direction, between global memory and the tile: inverse reads
// the CTA's rows (Fourier space, natural row order) from global memory,
// forward writes them there.
template <typename P, bool INV>
__device__ __forceinline__ void plane2_rows_global(ulonglong2 *tile, float2 *g, const float4 *__restrict__ tw_row,
                                                  int tid) {
    constexpr int T2 = P::T2, E2 = P::E2, N2 = P::N2, C = P::C, V = P::V;
    const RowAddr<Line2<N2, V>::LOG_R1> at;
    const int t = tid % T2;
#pragma unroll 1
    for (int base = 0; base < P::RP; base += P::PAIRS_PER_ITER) {
        const int p = base + tid / T2;
        if (P::RP % P::PAIRS_PER_ITER == 0 || p < P::RP) {
            ulonglong2 *rp = tile + p * P::S;
            float2 *g0 = g + (int64_t)p * N2, *g1 = g0 + (int64_t)P::RP * N2;
            c2 x[E2];
#pragma unroll
            for (int e = 0; e < E2; ++e)
                x[e] = INV ? c2_make(g0[t + T2 * e], g1[t + T2 * e]) : ld_c2(&rp[t + T2 * e]);
            __syncwarp();
            line_fft2<N2, V, INV>(x, rp, t, tw_row, Warp2Sync{}, at);
#pragma unroll
            for (int e = 0; e < E2; ++e) {
                if (INV) {
                    st_c2(&rp[t + T2 * e], x[e]);
                } else {
                    g0[t + T2 * e] = c2_first(x[e]);
                    g1[t + T2 * e] = c2_second(x[e]);
                }
            }
        }
    }
}

__device__ __forceinline__ c2 ld_cluster2(uint32_t addr) {
    c2 v;
    asm volatile("ld.shared::cluster.v2.u64 {%0, %1}, [%2];" : "=l"(v.x.v), "=l"(v.y.v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster2(uint32_t addr, c2 v) {
    asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(addr), "l"(v.x.v), "l"(v.y.v) : "memory");
}

// Exchange twiddles exp(-2 pi i n2 q / N1) of the rows n2 = 2p, 2p + 1 of a pair:
// entry [q * RP + p] of the value array, then of the residual array (N1 / 2 each).
template <int N1, int RP> __device__ __forceinline__ w2 exchange_twiddle(const float4 *__restrict__ twx, int q, int p) {
    const ulonglong2 *t = reinterpret_cast<const ulonglong2 *>(twx) + q * RP + p;
    const ulonglong2 h = __ldg(t), l = __ldg(t + N1 / 2);
    return {{h.x}, {h.y}, {l.x}, {l.y}};
}

// The cross-cluster step over the positions this CTA owns: pair p = row pair
// of position space, one column.  base[q] = cluster address of CTA q's tile;
// fq: this plane's fixed-point potential.
template <typename P>
__device__ __forceinline__ void plane2_exchange(const uint32_t *base, int rank, bool inv, bool phase, bool fwd,
                                               const float4 *__restrict__ twx, const uint32_t *__restrict__ fq,
                                               uint64_t coef, uint32_t dither, const float4 *ptab, int tid) {
    constexpr int R = P::R, N1 = P::N1, N2 = P::N2, C = P::C;
#pragma unroll 1
    for (int i = tid; i < P::OWNED; i += P::THREADS) {
        const int pos = rank * P::OWNED + i;
        const int p = pos / N2, c = pos % N2;
        const uint32_t off = (uint32_t)((p * P::S + c) * sizeof(ulonglong2));
        c2 v[C];
        uint32_t f0[C], f1[C];
#pragma unroll
        for (int q = 0; q < C; ++q) v[q] = ld_cluster2(base[q] + off);
        if (phase) {
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const uint32_t *f = &fq[(R * q + 2 * p) * N2 + c];
                f0[q] = __ldg(f);
                f1[q] = __ldg(f + N2);
            }
        }
        if (inv) {
#pragma unroll
            for (int q = 1; q < C; ++q) v[q] = c2_mul<true>(v[q], exchange_twiddle<N1, P::RP>(twx, q, p));
            dft2<C, true>(v);
        }
        if (phase) {
#pragma unroll
            for (int q = 0; q < C; ++q)
                v[q] = apply_phase_tab2(v[q], turns_mul(coef, f0[q]) + dither, turns_mul(coef, f1[q]) + dither, ptab);
        }
        if (fwd) {
            dft2<C, false>(v);
#pragma unroll
            for (int q = 1; q < C; ++q) v[q] = c2_mul<false>(v[q], exchange_twiddle<N1, P::RP>(twx, q, p));
        }
#pragma unroll
        for (int q = 0; q < C; ++q) st_cluster2(base[q] + off, v[q]);
    }
}

// Every step of a chunk for one 2-D instance b in the solo form; psi touches
// global memory only at the chunk's start and end.
template <typename P>
__device__ __forceinline__ void solo_whole_run(const PlaneArgs &a, int64_t b, const float4 *ptab, ulonglong2 *tile,
                                               int tid) {
    constexpr int N2 = P::N2;
    float2 *g = a.psi + b * (int64_t)P::N1 * N2;
    const uint32_t *fq = a.fq + b * (int64_t)P::N1 * N2;
    const float4 *tw_row = a.tw_row + P::V * TW2_TABLE * N2;
    plane2_copy<P, true>(tile, g, tid);
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < a.cnt; ++j) {
        solo_columns<P>(tile, j > 0, true, true, a.twx, fq, a.pot[(int64_t)j * a.batch + b],
                        step_dither(a.dither_base + (uint64_t)j), ptab, tid);
        __syncthreads();
        const float4 *kb = a.kt + ((int64_t)j * a.kt_batch + (a.kt_batch == 1 ? 0 : b)) * a.ksum;
        plane2_rows_kinetic<P>(tile, tw_row, kb, kb + P::N1, tid);
        __syncthreads();
    }
    solo_columns<P>(tile, a.cnt > 0, a.final_phase != 0, false, a.twx, fq, a.pot[(int64_t)a.cnt * a.batch + b], 0u, ptab,
                    tid);
    __syncthreads();
    plane2_copy<P, false>(tile, g, tid);
}

}  // namespace qhd
