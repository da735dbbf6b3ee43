// qhd_packed.cuh -- the line FFT on pairs of lines in packed FP32.
//
// Two complex numbers of two neighbouring lines travel together: a c2 holds
// (re0, re1) and (im0, im1) as packed FP32 pairs, and every addition, product
// and FMA of the transform is one add/mul/fma.rn.f32x2.  Each lane rounds as
// the scalar instruction does.  A packed instruction occupies the FP32 pipe for
// as long as two scalar ones but takes one issue slot: the scalar line FFT
// kept the issue slots 55-60% and the FP32 pipe 42-48% busy, with the loads,
// stores and address arithmetic competing for the rest, so halving the issue
// slots of the additions is what brings the pipe closer to its peak.
//
// Shared-memory exchanges move 16-byte elements (one c2), the width at which a
// warp needs the fewest instructions per byte.
#pragma once
#include <type_traits>

#include "qhd_device.cuh"

namespace qhd {

// ------------------------------------------------------- two FP32 lanes
struct pf {
    unsigned long long v;
};
__device__ __forceinline__ pf pf_make(float a, float b) {
    pf r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 pf_lanes(pf a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ pf pf_dup(float a) { return pf_make(a, a); }
__device__ __forceinline__ pf operator+(pf a, pf b) {
    pf r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ pf operator-(pf a, pf b) {
    pf r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ pf operator*(pf a, pf b) {
    pf r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ pf pf_fma(pf a, pf b, pf c) {
    pf r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ pf operator-(pf a) {
    const float2 t = pf_lanes(a);
    return pf_make(-t.x, -t.y);
}

// ------------------------------------------------- two complex numbers
struct c2 {
    pf x, y;  // (re0, re1), (im0, im1)
};
__device__ __forceinline__ c2 operator+(c2 a, c2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ c2 operator-(c2 a, c2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ c2 c2_make(float2 a, float2 b) { return {pf_make(a.x, b.x), pf_make(a.y, b.y)}; }
__device__ __forceinline__ float2 c2_first(c2 a) { return make_float2(pf_lanes(a.x).x, pf_lanes(a.y).x); }
__device__ __forceinline__ float2 c2_second(c2 a) { return make_float2(pf_lanes(a.x).y, pf_lanes(a.y).y); }
// a + w b and a - w b for w = -i (forward) or +i (inverse)
template <bool INV> __device__ __forceinline__ c2 c2_add_mi(c2 a, c2 b) {
    return INV ? c2{a.x - b.y, a.y + b.x} : c2{a.x + b.y, a.y - b.x};
}

// A twiddle with both lanes filled: value and FP32 rounding residual.
struct w2 {
    pf hx, hy, lx, ly;
};
// v * (hi + lo), or its conjugate, in the operation order of cmul_comp: the
// residual products first, then the cross term, then the diagonal term.
template <bool CONJ> __device__ __forceinline__ c2 c2_mul(c2 v, w2 w) {
    if (CONJ) {
        const pf nx = -v.x;
        const pf cre = pf_fma(v.y, w.ly, v.x * w.lx), cim = pf_fma(nx, w.ly, v.y * w.lx);
        return {pf_fma(v.x, w.hx, pf_fma(v.y, w.hy, cre)), pf_fma(v.y, w.hx, pf_fma(nx, w.hy, cim))};
    }
    const pf ny = -v.y;
    const pf cre = pf_fma(ny, w.ly, v.x * w.lx), cim = pf_fma(v.x, w.ly, v.y * w.lx);
    return {pf_fma(v.x, w.hx, pf_fma(ny, w.hy, cre)), pf_fma(v.y, w.hx, pf_fma(v.x, w.hy, cim))};
}

// v * (hi + lo) for one twiddle shared by both lanes, kept as it is in memory
// (hr, hi, lr, li): a packed product would want it with both lanes filled, which
// costs either eight moves or twice the loaded bytes (a warp's 128-bit load takes
// four cycles of the L1 data path even when its lanes share addresses).
template <bool CONJ> __device__ __forceinline__ c2 c2_mul_shared(c2 v, float4 w) {
    const float2 hi = make_float2(w.x, CONJ ? -w.y : w.y), lo = make_float2(w.z, CONJ ? -w.w : w.w);
    return c2_make(cmul_comp(c2_first(v), hi, lo), cmul_comp(c2_second(v), hi, lo));
}

// v * W_R^k (forward) or its conjugate, k a compile-time constant other than the
// multiples of R/4.  Odd multiples of R/8 are (+-1 +-i)/sqrt(2): the sum and the
// difference of the components times one constant, 6 operations instead of 8.
template <int R, bool INV> __device__ __forceinline__ c2 c2_twiddle(c2 v, int k) {
    static_assert(64 % R == 0, "in-register DFT sizes up to 64");
    const double cd = cos64(k * (64 / R));
    const double sd = INV ? sin64(k * (64 / R)) : -sin64(k * (64 / R));
    if (R >= 8 && (k % (R / 4)) * 8 == R) {
        const float h = (float)cd, l = (float)(cd - (double)h);
        const pf hp = pf_dup(h), lp = pf_dup(l);
        const bool same = (cd > 0) == (sd > 0);  // w = cd (1 + i) or cd (1 - i)
        const pf p = same ? v.x - v.y : v.x + v.y;
        const pf q = same ? v.y + v.x : v.y - v.x;
        return {pf_fma(p, hp, p * lp), pf_fma(q, hp, q * lp)};
    }
    const float ch = (float)cd, sh = (float)sd;
    return c2_mul<false>(v, {pf_dup(ch), pf_dup(sh), pf_dup((float)(cd - (double)ch)), pf_dup((float)(sd - (double)sh))});
}

// In-place R-point DFT of v[0..R), natural order in and out, unnormalised: the
// radix-4 recursion of dft() (qhd_device.cuh) on packed pairs.
template <int R, bool INV> __device__ __forceinline__ void dft2(c2 *v) {
    if constexpr (R == 1) {
        return;
    } else if constexpr (R == 2) {
        const c2 a = v[0], b = v[1];
        v[0] = a + b;
        v[1] = a - b;
    } else if constexpr (R == 4) {
        const c2 t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], d = v[1] - v[3];
        v[0] = t0 + t2;
        v[2] = t0 - t2;
        v[1] = c2_add_mi<INV>(t1, d);
        v[3] = c2_add_mi<!INV>(t1, d);
    } else if constexpr (R == 8) {
        c2 e[4], o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            e[i] = v[2 * i];
            o[i] = v[2 * i + 1];
        }
        dft2<4, INV>(e);
        dft2<4, INV>(o);
        v[0] = e[0] + o[0];
        v[4] = e[0] - o[0];
        v[2] = c2_add_mi<INV>(e[2], o[2]);
        v[6] = c2_add_mi<!INV>(e[2], o[2]);
#pragma unroll
        for (int k = 1; k < 4; k += 2) {
            const c2 w = c2_twiddle<8, INV>(o[k], k);
            v[k] = e[k] + w;
            v[k + 4] = e[k] - w;
        }
    } else {
        constexpr int Q = R / 4;
        c2 d[4][Q];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int i = 0; i < Q; ++i) d[r][i] = v[4 * i + r];
#pragma unroll
        for (int r = 0; r < 4; ++r) dft2<Q, INV>(d[r]);
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const c2 a0 = d[0][k];
            const c2 a1 = k ? c2_twiddle<R, INV>(d[1][k], k) : d[1][k];
            const c2 a3 = k ? c2_twiddle<R, INV>(d[3][k], 3 * k) : d[3][k];
            c2 t0, t1;
            if (8 * k == R) {  // W_R^(2k) = -i (forward)
                t0 = c2_add_mi<INV>(a0, d[2][k]);
                t1 = c2_add_mi<!INV>(a0, d[2][k]);
            } else {
                const c2 a2 = k ? c2_twiddle<R, INV>(d[2][k], 2 * k) : d[2][k];
                t0 = a0 + a2;
                t1 = a0 - a2;
            }
            const c2 t2 = a1 + a3, t3 = a1 - a3;
            v[k] = t0 + t2;
            v[k + 2 * Q] = t0 - t2;
            v[k + Q] = c2_add_mi<INV>(t1, t3);
            v[k + 3 * Q] = c2_add_mi<!INV>(t1, t3);
        }
    }
}

// ------------------------------------------------------------ line plans
// N = product of the stage radices; each thread holds E points of both lines
// (4 E registers), T = N / E threads per pair of lines.  V = 0 holds 8 points at
// most: many threads with a short chain each, for launches that do not fill the
// GPU (and for every launch where more points per thread gained nothing).
// V = 1 (128, 256 and 1024 points) holds 16: fewer exchanges per point.
// Measured per step, V = 0 / V = 1: 1024^2 x 1 (2^20 points) 20.3 / 25.4 us, x 2
// 32.3 / 30.8, x 8 114 / 101; 256x16x256 x 2 (2^21) 32.8 / 31.6, x 4 57.6 / 50.8;
// 64x16x128 x 5 17.2 / 22.3.  (16 points in one thread held 168 registers:
// 16x128x16 x 32 41 us, 4 x 4 20.9.)
constexpr int64_t BIG_PLAN_POINTS = int64_t(1) << 20;  // launches over more points than this take V = 1

template <int N, int V> struct Plan2;
template <int V> struct Plan2<2, V>  { static constexpr int E = 2, R[4] = {2, 1, 1, 1}; };
template <int V> struct Plan2<4, V>  { static constexpr int E = 4, R[4] = {4, 1, 1, 1}; };
template <int V> struct Plan2<8, V>  { static constexpr int E = 8, R[4] = {8, 1, 1, 1}; };
template <int V> struct Plan2<16, V> { static constexpr int E = 4, R[4] = {4, 4, 1, 1}; };
template <int V> struct Plan2<32, V> { static constexpr int E = 8, R[4] = {4, 8, 1, 1}; };
template <int V> struct Plan2<64, V> { static constexpr int E = 8, R[4] = {8, 8, 1, 1}; };
template <> struct Plan2<128, 0>     { static constexpr int E = 8, R[4] = {8, 8, 2, 1}; };
template <> struct Plan2<128, 1>     { static constexpr int E = 16, R[4] = {8, 16, 1, 1}; };
template <> struct Plan2<256, 0>     { static constexpr int E = 8, R[4] = {8, 8, 4, 1}; };
template <> struct Plan2<256, 1>     { static constexpr int E = 16, R[4] = {16, 16, 1, 1}; };
template <int V> struct Plan2<512, V> { static constexpr int E = 8, R[4] = {8, 8, 8, 1}; };
template <> struct Plan2<1024, 0>    { static constexpr int E = 8, R[4] = {8, 4, 4, 8}; };
template <> struct Plan2<1024, 1>    { static constexpr int E = 16, R[4] = {16, 8, 8, 1}; };
// V = 2: half-length columns of the solo plane engine, four threads each
template <> struct Plan2<64, 2>      { static constexpr int E = 16, R[4] = {8, 8, 1, 1}; };
__host__ __device__ constexpr bool two_plans(int n) { return n == 128 || n == 256 || n == 1024; }

template <int N, int V> struct Line2 {
    using P = Plan2<N, V>;
    static constexpr int E = P::E, T = N / E;
    static constexpr int STAGES = P::R[1] == 1 ? 1 : P::R[2] == 1 ? 2 : P::R[3] == 1 ? 3 : 4;
    static constexpr int LOG_R1 = P::R[0] == 4 ? 2 : P::R[0] == 8 ? 3 : 4;
    static constexpr int PADDED = N + (N >> LOG_R1);
};

// Line stride and padding of the exchange buffer in 16-byte elements.  A
// quarter warp (8 lanes) moves 128 bytes per cycle; these choices give every
// exchange of every plan eight distinct 16-byte banks (checked for all plans
// by enumeration).  Columns: CP pairs of columns side by side over the lanes;
// rows: the T threads of a line are consecutive lanes.
template <int N, int V, int CP> struct ColBuf {
    static constexpr bool PAD = CP < 8;
    static constexpr int S = CP >= 8 ? N + 1 : Line2<N, V>::PADDED + (CP == 4 ? 2 : CP == 2 ? 4 : 0);
};
template <int N, int V> struct RowBuf {
    static constexpr int S = Line2<N, V>::PADDED + (Line2<N, V>::T == 4 ? 4 : 0);
};

// Where element i of a line lives in its exchange buffer.
struct PlainAddr {
    __device__ __forceinline__ int operator()(int i) const { return i; }
};
template <int LOG_R1> struct RowAddr {
    __device__ __forceinline__ int operator()(int i) const { return i + (i >> LOG_R1); }
};
template <int S> struct ColAddr {  // a column of a row-major tile, in place
    __device__ __forceinline__ int operator()(int i) const { return i * S; }
};
template <int N, int V, int CP>
using ColBufAddr = std::conditional_t<ColBuf<N, V, CP>::PAD, RowAddr<Line2<N, V>::LOG_R1>, PlainAddr>;

__device__ __forceinline__ c2 ld_c2(const ulonglong2 *p) {
    const ulonglong2 q = *p;
    return {{q.x}, {q.y}};
}
__device__ __forceinline__ void st_c2(ulonglong2 *p, c2 v) { *p = make_ulonglong2(v.x.v, v.y.v); }

// Twiddle table of a line, (hr, hi, lr, li) per entry.  Stage 2 has entries
// [m * R1 + j], exp(-2 pi i j m / (R1 R2)); the later stages follow in the same
// form, stage 3 with [m * R1 R2 + j] and so on.
// One stage: L = product of the radices before it, TW0 = its first table entry.
template <int N, int V, bool INV, int S, int L, int TW0, typename Sync, typename At>
__device__ __forceinline__ void line_stage2(c2 *x, ulonglong2 *sm, int t, const float4 *__restrict__ tw, Sync sync, At at) {
    using C = Line2<N, V>;
    constexpr int R = C::P::R[S], E = C::E, T = C::T;
    constexpr bool LAST = S + 1 == C::STAGES;
#pragma unroll
    for (int q = 0; q < E / R; ++q) {
        const int j = t + T * q;
        c2 v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = x[q + m * (E / R)];
        if (S > 0) {
#pragma unroll
            for (int m = 1; m < R; ++m) v[m] = c2_mul_shared<INV>(v[m], __ldg(&tw[TW0 + m * L + (j % L)]));
        }
        dft2<R, INV>(v);
        if (LAST) {
#pragma unroll
            for (int m = 0; m < R; ++m) x[q + m * (E / R)] = v[m];
        } else {
#pragma unroll
            for (int m = 0; m < R; ++m) st_c2(&sm[at((j / L) * (L * R) + (j % L) + m * L)], v[m]);
        }
    }
    if constexpr (!LAST) {
        sync();
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = ld_c2(&sm[at(t + T * e)]);
        sync();
        line_stage2<N, V, INV, S + 1, L * R, (S == 0 ? 0 : TW0 + L * R)>(x, sm, t, tw, sync, at);
    }
}

// x[e] holds element t + T e of both lines on entry and transform element
// t + T e on exit.  sm: the pair's exchange buffer; sync orders the exchange
// among the T threads.
template <int N, int V, bool INV, typename Sync, typename At>
__device__ __forceinline__ void line_fft2(c2 *x, ulonglong2 *sm, int t, const float4 *__restrict__ tw, Sync sync, At at) {
    // a transform and its inverse load the same twiddles; kept in registers from the
    // one to the other (60 of them for 16 points) they would be spilled
    asm volatile("" : "+l"(tw));
    line_stage2<N, V, INV, 0, 1, 0>(x, sm, t, tw, sync, at);
}

// Two hi/lo values (hr, hi, lr, li) side by side.
__device__ __forceinline__ w2 w2_make(float4 a, float4 b) {
    return {pf_make(a.x, b.x), pf_make(a.y, b.y), pf_make(a.z, b.z), pf_make(a.w, b.w)};
}

// Product of two unit factors carried as value and residual, again as value and
// residual: the exact products' errors and the cross terms with the residuals
// are gathered in the new residual (relative error ~2^-46).
__device__ __forceinline__ w2 w2_mul(w2 a, w2 b) {
    const pf p = a.hx * b.hx, q = a.hy * b.hy;
    const pf pe = pf_fma(a.hx, b.hx, -p), qe = pf_fma(a.hy, b.hy, -q);
    const pf r = a.hx * b.hy, s = a.hy * b.hx;
    const pf re = pf_fma(a.hx, b.hy, -r), se = pf_fma(a.hy, b.hx, -s);
    // two-sums p - q and r + s
    const pf x = p - q, xb = x - p, xe = (p - (x - xb)) - (q + xb);
    const pf y = r + s, yb = y - r, ye = (r - (y - yb)) + (s - yb);
    const pf lx = pf_fma(a.hx, b.lx, a.lx * b.hx) - pf_fma(a.hy, b.ly, a.ly * b.hy);
    const pf ly = pf_fma(a.hx, b.ly, a.lx * b.hy) + pf_fma(a.hy, b.lx, a.ly * b.hx);
    const pf tx = xe + ((pe - qe) + lx), ty = ye + ((re + se) + ly);
    // renormalise: the residual is at most half a unit of the value
    const pf ox = x + tx, oy = y + ty;
    return {ox, oy, tx - (ox - x), ty - (oy - y)};
}

// apply_phase_tab (qhd_device.cuh) on a pair of points with their own turns.
__device__ __forceinline__ c2 apply_phase_tab2(c2 z, uint32_t u0, uint32_t u1, const float4 *tab) {
    const float4 t0 = tab[u0 >> 24], t1 = tab[u1 >> 24];
    const pf d = pf_make((float)((int32_t)(u0 & 0xFFFFFFu) - (1 << 23)), (float)((int32_t)(u1 & 0xFFFFFFu) - (1 << 23))) *
                 pf_dup(1.4629180792671596e-09f);  // 2 pi / 2^32
    const pf d2 = d * d;
    const pf cm1 = d2 * pf_fma(d2, pf_dup(1.0f / 24.0f), pf_dup(-0.5f));
    const pf sn = d * pf_fma(d2, pf_dup(-1.0f / 6.0f), pf_dup(1.0f));
    w2 w = w2_make(t0, t1);
    const pf lx = pf_fma(w.hx, cm1, pf_fma(w.hy, sn, w.lx));
    const pf ly = pf_fma(w.hy, cm1, pf_fma(-w.hx, sn, w.ly));
    w.lx = lx;
    w.ly = ly;
    return c2_mul<false>(z, w);
}

}  // namespace qhd
