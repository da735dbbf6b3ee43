// qhd_kernels.h -- launch interface between the host library and the kernels.
// Host-only declarations; the kernels themselves live in qhd_kernels.cu.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace qhd {

// Pass modes.
enum : int { MODE_FWD = 1, MODE_INV = 2, MODE_KIN = 4 };

// Damping schedule as the device evaluates it (one per instance).
struct SchedDev {
    int32_t kind;  // 0 Nesterov, 1 table, 2 power family
    int32_t ns;    // table samples
    double c_phi, eps, c_chi;
    const double *t, *phi, *chi;  // workspace copies of the samples
    double power;  // power family: p
};

// Per-instance potential data written by set_potential.
struct InstDev {
    double fmin;     // offset of the fixed-point potential
    int32_t shift;   // fq = rint((f - fmin) * 2^shift)
    int32_t pad_;
    double xs[3];    // grid minimiser coordinates
};

// Per-block partial of the min/max/argmin reduction over f.
struct MinMaxPart {
    double fmin, fmax;
    int64_t argmin;
    int64_t nonfinite;
};

struct RowArgs {
    float2 *psi;
    const uint32_t *fq;
    const uint64_t *pot;   // potential coefficient of this pass, one per instance
    const float4 *tw2;     // twiddles of the row length (line_fft2), both plans
    int64_t rows;          // batch * rows per instance
    int log_rows;          // log2 of the rows per instance
    int mode;              // MODE_INV: inverse FFT before the phase; MODE_FWD: forward after
    uint32_t dither;       // global phase of this pass in 2^-32 turns (step_dither)
    const float4 *ptab;    // potential phase table (PHASE_TAB hi/lo entries)
};

struct AxisArgs {
    float2 *psi;
    const float4 *tw2;     // twiddles of the line length (line_fft2), both plans
    const float4 *kt;      // kinetic tables of this step: [batch][ksum] (MODE_KIN only)
    int64_t inner;         // product of the axis lengths after this axis (line stride)
    int log_inner;         // its log2
    int64_t planes;        // product of batch and the axis lengths before this axis
    int ksum;              // sum of the axis lengths
    int koff1, koff2;      // table offsets of axes 1 and 2
    int log_n2;            // log2 n[2] (3-D only)
    int ndim;
    int mode;
    int64_t kt_batch;      // 1: every instance shares the kinetic table; else batch
    int perm1_log_r, perm1_c;  // 3-D after a plane pass: stored axis-1 row s holds frequency
                               // s / r + perm1_c * (s % r), r = 2^perm1_log_r; perm1_c = 0: natural
};

// Plane engine (qhd_plane.cu): N1 distributed over a cluster, N2 per row.  Up to 144
// bytes of arguments the compiler loads into registers once, longer ones it reads
// where they are used (PlaneArgsLong, for the shapes where that is faster).
struct PlaneArgs {
    float2 *psi;
    const uint32_t *fq;
    const uint64_t *pot;     // pass: coefficients of this pass [batch]; whole: chunk [cnt+1][batch]
    const float4 *kt;        // whole: chunk kinetic tables [cnt][batch][ksum]
    const float4 *tw_row;    // row twiddles: line_fft's (cluster whole run) or line_fft2's, both plans (others)
    const float4 *twx;       // column twiddles: exchange_twiddles (cluster whole run), exchange_twiddles2
                             // (cluster pass), solo_twiddles (one CTA)
    int64_t count;           // planes (pass) or instances (whole) of this launch
    int64_t batch;
    int mode;                // pass: MODE_INV (previous step's inverse first), MODE_FWD
    uint32_t dither;         // pass: global phase of this step
    int cnt;                 // whole: steps in the chunk
    int final_phase;         // whole: apply pot[cnt] at the end
    int ksum;
    int log_planes;          // pass: log2 of the planes per instance (n0)
    uint64_t dither_base;    // whole: global index of the chunk's first step
    const float4 *ptab;      // potential phase table
    int64_t kt_batch;        // whole: 1 = shared kinetic table, else batch
};
static_assert(sizeof(PlaneArgs) <= 144, "costs the cluster engine registers");
struct PlaneArgsLong : PlaneArgs {
    char unused[48];
};

struct OneDArgs {
    float2 *psi;
    const uint32_t *fq;
    const uint64_t *pot;   // chunk potential coefficients [cnt+1][batch]
    const float4 *kt;      // chunk kinetic tables [cnt][batch][n]
    const float4 *tw2;
    int64_t batch;
    int cnt;
    int final_phase;       // apply pot[cnt] after the last step
    uint64_t dither_base;  // global step index of the chunk's first step
    const float4 *ptab;    // potential phase table
    int64_t kt_batch;      // 1: shared kinetic table; else batch
};

struct PrepArgs {
    const SchedDev *sched;
    const InstDev *inst;
    uint64_t *pot;         // [cnt+1][batch]
    float4 *kt;            // [cnt][kt_batch][ksum], (hi.re, hi.im, lo.re, lo.im)
    int64_t kt_batch;      // 1 when every instance has the same kinetic schedule
    double t_start, dt;
    int64_t j0, cnt, nsteps, batch;
    int ndim;
    int n[3];
    double len[3];
    int koff[3];
    int ksum;
    double inv_g;          // 1/G (exact power of two)
    int split;             // 0 Strang (midpoint, merged halves), 1 first-order Lie-Trotter
    int kinetic;           // 0 spectral |k|^2, 1 central second difference (4/h^2) sin^2(pi m/N)
};

struct ObsArgs {
    const float2 *psi;
    const double *f64;
    const InstDev *inst;
    const double *coord;   // mesh coordinates per axis, concatenated
    float *prob;           // optional
    double *partial;       // [batch][nblk][3]
    double *result;        // [batch][3]
    int64_t g;
    int ndim;
    int n[3];
    int log_n[3];
    int coff[3];
    double radius;
    double r2_max;         // set by launch_observables
    int nblk;              // partials per instance at most
    bool await_tables;     // coord and inst come from a kernel on this stream, not from a synchronised upload
};

// Launchers; each returns the launch error (cudaSuccess on success).
cudaError_t launch_row(int n, const RowArgs &a, cudaStream_t s);
cudaError_t launch_axis(int n, const AxisArgs &a, cudaStream_t s);
cudaError_t launch_oned(int n, const OneDArgs &a, cudaStream_t s);
cudaError_t launch_prep(const PrepArgs &a, bool early, cudaStream_t s);  // early: releases the next kernel at its start
// Loads launch_prep's kernels (a first launch inside a stream capture must not).
cudaError_t load_prep();
cudaError_t launch_uniform(float2 *psi, int64_t count, float value, cudaStream_t s);
cudaError_t launch_minmax(const double *f, int64_t g, int64_t batch, MinMaxPart *part, int nblk,
                          cudaStream_t s);
cudaError_t launch_minmax_final(const MinMaxPart *part, int nblk, int64_t batch, MinMaxPart *out, cudaStream_t s);
cudaError_t launch_quantize(const double *f, uint32_t *fq, const InstDev *inst, int64_t g,
                            int64_t batch, cudaStream_t s);
cudaError_t launch_observables(const ObsArgs &a, int64_t batch, cudaStream_t s);
cudaError_t launch_plane_pass(int n1, int n2, const PlaneArgs &a, cudaStream_t s);
cudaError_t launch_plane_whole(int n1, int n2, const PlaneArgs &a, cudaStream_t s);
cudaError_t launch_solo_whole(int n1, int n2, const PlaneArgs &a, cudaStream_t s);
bool plane_supported(int n1, int n2);
bool plane_fits_solo(int n1, int n2);  // one CTA holds the plane
int64_t solo_instances(int n1, int n2, int64_t batch, int sms);  // 2-D: how many of a batch run in one CTA each
int plane_cluster(int n1);
// Whole-run kernel with twice the CTAs per instance (distributed axis 64 or 128; 0: none).
int plane_cluster_wide(int n1);
cudaError_t launch_plane_whole_wide(int n1, int n2, const PlaneArgs &a, cudaStream_t s);

// Plans shared with the host (twiddle tables are built on the host).
void plan_of(int n, int *r1, int *r2);         // scalar line FFT (line_fft)
void plan2_of(int n, int v, int *radix, int *stages);  // packed line FFT (line_fft2), plan v
constexpr int TW2_TABLE = 2;  // table of plan v starts at v * TW2_TABLE * N; each holds at most TW2_TABLE * N entries
bool supported_n(int64_t n);
// Exchange twiddles of a distributed axis of n1 = c * r points, n1 entries:
// exp(-2 pi i q j / n1) at [q * r + j], (re, im, residuals).
void exchange_twiddles(float4 *out, int n1, int c);
// The same for pairs of rows j = 2p, 2p + 1: values (re, re, im, im) at
// [q * r / 2 + p], their FP32 residuals n1 / 2 entries later.
void exchange_twiddles2(float4 *out, int n1, int c);
// Column twiddles of the solo form, n1 entries: exp(-2 pi i k / n1), k < n1 / 2,
// then the stage twiddles of a line of n1 / 2 points.
void solo_twiddles(float4 *out, int n1);

}  // namespace qhd
