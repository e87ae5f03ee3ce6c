// Internal declarations shared by the translation units of libbz (not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <vector>

#include "../../include/bz.h"

#ifndef EXTRA_STREAMS
#define EXTRA_STREAMS 1
#endif

namespace bz {

// One radial node's part-II theta rule (Sec. 4.1): nodes t_n on [eps, pi] with
// weights W_n = w_n g(t_n), stored as (1 - cos t_n, sin t_n, W_n).
struct ThetaRule {
    std::vector<double> omc, sn, W;
};

struct HostTerms {
    std::vector<double> r, wr, q, wq, c;   // per term p = i*M + j; q is [P][3]
    std::vector<int> radial_index;          // i for each p
};

// Optional per-kernel CUDA-event timing (bz_plan_set_timing).
enum { TK_PLANE_INV = 0, TK_PENCIL = 1, TK_PLANE_FWD = 2, TK_REDUCE = 3, TK_OTHER = 4, TK_FUSED = 5, TK_COUNT = 6 };
struct Timing {
    bool on = false;
    std::vector<cudaEvent_t> ev;    // pairs (start, end)
    std::vector<int> kind;          // per pair
    size_t used = 0;                // pairs recorded since the last collect
    double ms[TK_COUNT] = {0, 0, 0, 0, 0, 0};
    long n[TK_COUNT] = {0, 0, 0, 0, 0, 0};
};

// Streams of the chunked pipeline beside the caller's.
constexpr int kExtraStreams = EXTRA_STREAMS;

struct Plan {
    // parameters
    int N = 0, N_rho = 0, M = 0, P = 0, kernel = 0, precision = 0, device = 0;
    int Nin = 0;                    // BZ_CONV_PADDED: the caller's modes per axis (N = 2 Nin); 0 = circular
    int dim = 3;                    // 3: the 3D operator; 2: the 2D operator on an N x N grid
    double L = 0, R = 0, gamma = 0, s = 0, eps = 0;
    double theta0 = 0;              // angular cutoff (0: none)
    double A[3] = {0, 0, 0};        // part I kernel moments
    double kc = 0;                  // kernel constant (c_s, 1/(4 pi), 5/(192 pi))
    HostTerms terms;
    std::vector<ThetaRule> rules;   // one per radial node
    // device tables
    float2 *alpha = nullptr;        // [P][N^3]  c_p F / N^3
    float2 *tw = nullptr;           // [P][3][N] exp(-i pi r q_d m / L)
    double *rule_buf = nullptr;     // concatenated (omc, sn, W) per radial node
    int *rule_off = nullptr;        // [N_rho + 1] node offsets
    int rule_max = 0;               // largest node count of one radial node
    double *term_dev = nullptr;     // [P][5]: r, q0, q1, q2, c
    // workspace
    int chunk = 0;                  // terms per chunk
    float2 *S = nullptr;            // [chunk][N^3]
    float2 *h = nullptr;            // [N^3]
    float2 *fin = nullptr;          // [N^3] FP32 input
    const float2 *f32 = nullptr;    // the FP32 input of the call being issued: fin, or a complex64 caller's array
    float2 *fcopy = nullptr;        // where the h pass stores it (complex128 callers), or null
    double2 *acc = nullptr;         // [N^3] FP64 accumulator (while a chunked collide runs, the same
                                    // bytes hold k_reduce's compensated FP32 state: s, c per mode pair)
    double2 *rk = nullptr;          // [2][N^3] RK4 state (f0, fsum)
    double *mom = nullptr;          // moments scratch
    // fused cluster pipeline (N <= 32)
    int use_fused = 0;              // 1: bz_collide runs k_fused
    int fused_C = 0;                // CTAs per cluster
    int fused_G = 0;                // resident clusters (persistent grid)
    float fused_ms = 0.f;           // timed collide of the selected cluster size
    int h_fp64 = 1;                 // fused path: bits of the h pass, HFF_*; HFF_FP32 in the term kernel but for k_col32
    double2 *fin64 = nullptr;       // [N^3] FP64 stage input (RK4) for the h pass
    double2 *scr64 = nullptr;       // [N^3] scratch of the h pass (16 bytes per mode)
    const void *src = nullptr;      // FP64-capable source of h for the next fused collide
    int src_dtype = BZ_C128;
    float2 *part = nullptr;         // [fused_G][N^3] per-cluster partial sums
    uint4 *wimg = nullptr;          // BZ_PREC_BF16X3: split DFT matrix (tensor-core B operand)
    // BZ_DATA_REAL: terms 2q and 2q + 1 share one pair of transforms
    int real = 0;
    int col32 = 0;                  // N = 32: one term per SM (k_col32): the default of the fused pipeline
    int cube32 = 0;                 // the same for complex data (k_cube32)
    int few_G = 0;                  // its 8-CTA clusters of k_fused, for collides of few terms (0: not used)
    float2 *acol = nullptr;         // their table [P][18][32][32] (bz_col32.cu), [P][32][32][32] (bz_cube32.cu)
    float2 *fcol = nullptr;         // input [k3 (< 16)][k1][k2] (N^3 allocated)
    float *hcol = nullptr;          // h [j3][j1][j2], packed floats (k_cube32: float2)
    int pair3 = 0;                  // N = 32, on request: the three-CTA-per-SM pair kernel (k_pair3) instead of k_fused
    float2 *apair = nullptr;        // [P / 2][N^3] A = (alpha_2q - i alpha_2q+1) / 2
    float2 *cpair = nullptr;        // [P / 2][3][N][N] C = conj B(-k), B = (alpha_2q + i alpha_2q+1) / 2, on the
                                    // Nyquist planes (families k1 = -N/2, k2 = -N/2, k3 = -N/2), 0 elsewhere
    float2 *part_s = nullptr;       // [fused_G][3][N][N] per-item sums X on the Nyquist planes
    float2 *S_s = nullptr;          // chunked pipeline: [chunk][3][N][N] the chunk's Nyquist sums
    double2 *acc_s = nullptr;       // chunked pipeline: [3][N][N] FP64 sum of X
    // chunked pipeline on several streams: chunk i runs on lane i % (1 + xn), lane 0 the
    // caller's stream over S / acc, lane e > 0 the plan's stream xst[e - 1] over its own
    // scratch and accumulators; the lanes overlap and their sums are added at the end
    int xn = 0;                                      // extra streams in use
    cudaStream_t xst[kExtraStreams] = {};
    cudaEvent_t ev_fork = nullptr, xev_join[kExtraStreams] = {};
    float2 *xS[kExtraStreams] = {};                  // [chunk][N^3]
    float2 *xS_s[kExtraStreams] = {};                // [chunk][3][N][N] (BZ_DATA_REAL)
    double2 *xacc[kExtraStreams] = {};               // [N^3]
    double2 *xacc_s[kExtraStreams] = {};             // [3][N][N] (BZ_DATA_REAL)
    // N = 48, 64 (bz_lines.cu): running sums per lane and split [lanes][splits][N^3], and the term
    // pairs' products [P / 2][3][N][N] on the Nyquist planes (BZ_DATA_REAL)
    float4 *lstate = nullptr;
    float2 *xs = nullptr;
    float2 *fsym = nullptr;         // [N^3] Hermitian part of fhat, Nyquist planes zero (FP32)
    const float *gsc_cur = nullptr; // chunked pipeline inside a batch call: the slot's radial scale
                                    // r_i^(gamma_slot - gamma) per radial node (null: none)
    int *dev_err = nullptr;         // device flags: [0] a bounded wait of a kernel gave up,
                                    // [1] a result written since the last check held NaN or Inf
    size_t ws_bytes = 0;
    int last_launches = 0;
    Timing tm;
};

// Raises the non-finite flag (Plan::dev_err[1]) if the value written is NaN or Inf.
#ifdef __CUDACC__
__device__ __forceinline__ void note_finite(double2 v, int *flag) {
    if (flag && !(isfinite(v.x) && isfinite(v.y))) atomicOr(flag, 1);
}
__device__ __forceinline__ void note_finite(float2 v, int *flag) {
    if (flag && !(isfinite(v.x) && isfinite(v.y))) atomicOr(flag, 1);
}
#endif
inline int *nonfinite_flag(const Plan &pl) { return pl.dev_err ? pl.dev_err + 1 : nullptr; }

// Where a collide's result goes: each kernel that finishes a mode's sum over the terms hands it on.
struct Sink {
    enum { ACC, OUT, RK };
    int mode = ACC;
    double2 *acc = nullptr;          // ACC: the plan's FP64 accumulator
    void *out = nullptr;             // OUT: the caller's array; RK: the same after the last stage, or null
    int dtype = BZ_C128;
    int *flag = nullptr;             // raised by a NaN or Inf written to out
    // RK: stage 1 .. 4 of a step (Sec. 5.2); k is the derivative at the stage's input
    double2 *f0 = nullptr, *fsum = nullptr, *fin64 = nullptr;
    float2 *fin = nullptr;
    int stage = 0;
    double dt = 0;
};
#ifdef __CUDACC__
__device__ __forceinline__ void sink_store(void *out, int dtype, int *flag, size_t i, double2 v) {
    if (dtype == BZ_C128) {
        ((double2 *)out)[i] = v;
        note_finite(v, flag);
    } else {
        const float2 w = make_float2((float)v.x, (float)v.y);
        ((float2 *)out)[i] = w;
        note_finite(w, flag);
    }
}
__device__ __forceinline__ void sink_put(const Sink &s, size_t i, double2 v) {
    if (s.mode == Sink::ACC) {
        s.acc[i] = v;
    } else if (s.mode == Sink::OUT) {
        sink_store(s.out, s.dtype, s.flag, i, v);
    } else {
        // the state f0 and the running combination f0 + dt/6 (k1 + 2 k2 + 2 k3 + k4) in FP64; the next stage's
        // input in FP32 (and FP64 for the h pass)
        const double2 a = s.f0[i];
        const double dt = s.dt;
        double2 y;
        if (s.stage == 1) {
            s.fsum[i] = make_double2(a.x + dt / 6.0 * v.x, a.y + dt / 6.0 * v.y);
            y = make_double2(a.x + 0.5 * dt * v.x, a.y + 0.5 * dt * v.y);
        } else if (s.stage == 2 || s.stage == 3) {
            const double2 u = s.fsum[i];
            s.fsum[i] = make_double2(u.x + dt / 3.0 * v.x, u.y + dt / 3.0 * v.y);
            const double c = s.stage == 2 ? 0.5 * dt : dt;
            y = make_double2(a.x + c * v.x, a.y + c * v.y);
        } else {
            const double2 u = s.fsum[i];
            y = make_double2(u.x + dt / 6.0 * v.x, u.y + dt / 6.0 * v.y);
            s.f0[i] = y;
            if (s.out) sink_store(s.out, s.dtype, s.flag, i, y);
        }
        s.fin[i] = make_float2((float)y.x, (float)y.y);
        if (s.fin64) s.fin64[i] = y;
    }
}
#endif

// Fourier modes of one field: N^3 (3D) or N^2 (2D).
inline size_t modes(const Plan &pl) { return (size_t)pl.N * pl.N * (pl.dim == 2 ? 1 : pl.N); }

// Brackets one launch with events when timing is on (events are pre-created).
inline void tm_begin(Plan &pl, cudaStream_t st) {
    if (pl.tm.on && pl.tm.used < pl.tm.kind.size()) cudaEventRecord(pl.tm.ev[2 * pl.tm.used], st);
}
inline void tm_end(Plan &pl, cudaStream_t st, int kind) {
    if (pl.tm.on && pl.tm.used < pl.tm.kind.size()) {
        cudaEventRecord(pl.tm.ev[2 * pl.tm.used + 1], st);
        pl.tm.kind[pl.tm.used++] = kind;
    }
}

// bz_quad.cpp
int gauss_legendre(int n, double a, double b, std::vector<double> &x, std::vector<double> &w);
bz_status build_terms(Plan &pl, const double *sphere_xyz, const double *sphere_w);
bz_status build_kernel_constants(Plan &pl);
void build_theta_rules(Plan &pl);

// bz_ftable.cu
bz_status ftable_build(Plan &pl);
bz_status ftable_entries(Plan &pl, int count, const int *k_idx, const int *term, double *out);

// bz_collide.cu
// Qhat = Q over terms [p0, p1) of fhat (device arrays of one dtype)
bz_status collide_range(Plan &pl, int p0, int p1, const void *fhat, void *Qhat, int dtype, cudaStream_t st,
                        int *launches);
// the input set by collide_range or rk4_steps (pl.f32, pl.src), the result to the sink
bz_status collide_core(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink);
inline Sink acc_sink(Plan &pl) {
    Sink s;
    s.acc = pl.acc;
    return s;
}
// pl.h = IFFT(fin) in FP32 (one plane pass and one pencil pass through pl.S; N = 32: k_pair3)
bz_status h_fp32(Plan &pl, const float2 *fin, cudaStream_t st);

// bz_fused.cu
// Arguments of the fused item kernel (see k_fused): item w = (instance w / nblk, term block
// w % nblk); instance b lives in array slot slots[b] (identity when slots is null).
struct ItemArgs {
    const float2 *fin = nullptr;     // [slots][N^3] FP32 inputs
    const float2 *tw = nullptr;      // [P][3][N]
    const float2 *alpha = nullptr;   // [P][N^3]
    const float *gsc = nullptr;      // [slots][N_rho] radial scale r_i^(gamma_b - gamma_plan), or null
    float2 *part = nullptr;          // [slots][nblk][N^3] per-item partial sums
    const float2 *hg = nullptr;      // [slots][N^3] h = IFFT(fhat), stored FP32; null: formed in the kernel in FP32
    const int *slots = nullptr;      // device [count] or null
    const int *count_dev = nullptr;  // device instance count, or null (use count)
    int count = 1, p0 = 0, p1 = 0, TB = 1, nblk = 0, M = 1, N_rho = 1;
    int real = 0;                    // BZ_DATA_REAL: p0, p1 count term pairs, alpha = the pair table
    const float2 *cpair = nullptr;   // BZ_DATA_REAL: [pairs][3][N][N] Nyquist-plane table C
    float2 *part_s = nullptr;        // BZ_DATA_REAL: [slots][nblk][3][N][N] per-item sums X
};
int fused_candidates(int N, int *cs, int forced);
cudaError_t fused_setup(int N, int C, int *G, bool real);
bz_status launch_fused(const Plan &pl, const ItemArgs &a, cudaStream_t st);
// bz_hff.cu: h[slot] = IFFT(f[slot]), stored FP32, for the active slots (N <= 32); formed in double-float
// arithmetic (HFF_PAIRS: about 47 bits), in FP64 (where BZ_H_FP64 is asked for) or in FP32 (N = 32).  Kernel
// launches of one hff_launch:
enum { HFF_FP32 = 0, HFF_PAIRS = 1, HFF_FP64 = 2 };
inline int hff_launches(int N) { return N <= 16 ? 1 : 2; }
// fsym (BZ_DATA_REAL, N a power of two): transform the Hermitian, Nyquist-free part of f and
// store that part in FP32 to fsym; col (N = 32): in the layouts of k_col32 (fsym [k3 < 16][k1][k2], h packed
// floats [j3][j1][j2]; the same stride of N^3 float2 per slot) or, without fsym, of k_cube32 (fcopy
// [k3][k1][k2], h [j3][j1][j2]).  fcopy (complex data): f in FP32.  scr: 16 N^3 bytes per slot
// (N = 24, 32).
bz_status hff_launch(int N, int bits, const void *f, int dtype, const int *slots, const int *count_dev, int count,
                     double2 *scr, float2 *h, cudaStream_t st, float2 *fsym = nullptr, bool col = false,
                     float2 *fcopy = nullptr);
// fcopy (complex data, c128): where f goes in FP32, or null
bz_status hff_launch_2d(int N, int bits, const void *f, int dtype, float2 *h, float2 *fcopy, cudaStream_t st);
bz_status collide_fused(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink);
// bz_real.cu (BZ_DATA_REAL): the pair table from alpha (after ftable_build); pl.fsym from a
// c64 / c128 array
bz_status build_pair_table(Plan &pl);
bz_status sym_input(Plan &pl, const void *f, int dtype, cudaStream_t st);
// sink <- Q from the nblk item sums of pl.part (V) and pl.part_s (X): one kernel
bz_status reduce_sym(Plan &pl, int nblk, cudaStream_t st, const Sink &sink);
// chunked pipeline: sink <- Q from pl.acc (V, FP64; may be the sink) with pl.acc_s (X)
bz_status sym_output(Plan &pl, cudaStream_t st, const Sink &sink);

// bz_pair3.cu (BZ_DATA_REAL, N = 32): resident clusters and launch of k_pair3
cudaError_t pair3_setup(int *G);
bz_status launch_pair3(const Plan &pl, const ItemArgs &a, cudaStream_t st);

// bz_col32.cu (BZ_DATA_REAL, N = 32): one CTA per SM; items count terms.  The table from pl.alpha; sink <- the
// sum of nblk items
constexpr size_t kCol32Part = (size_t)18 * 32 * 32;     // float2 per item's sums
cudaError_t col32_setup(int *G);
bz_status launch_col32(const Plan &pl, const ItemArgs &a, cudaStream_t st);
bz_status col32_table(Plan &pl);
bz_status reduce_col(Plan &pl, int nblk, cudaStream_t st, const Sink &sink);

// bz_batch.cu: terms per item of a batch of one-term-per-SM items; asked <= 0: chosen
int one_sm_terms(bool real, int P, int capacity, int asked, int G);

// bz_cube32.cu (complex data, N = 32): as above; items' sums are N^3
cudaError_t cube32_setup(int *G);
bz_status launch_cube32(const Plan &pl, const ItemArgs &a, cudaStream_t st);
bz_status cube32_table(Plan &pl);
bz_status reduce_cube(Plan &pl, int nblk, cudaStream_t st, const Sink &sink);

// bz_mixed.cu (BZ_PREC_BF16X3, N = 32)
cudaError_t mixed_setup(int N, int *G);
bz_status mixed_upload(uint4 **wimg);
bz_status launch_mixed(const Plan &pl, const ItemArgs &a, cudaStream_t st);
// one bounded wait that nothing completes, giving up after `limit` clocks (bz_plan_wait_selftest)
bz_status wait_selftest(const Plan &pl, long long limit, cudaStream_t st);
cudaError_t collide_set_attributes(int N);
void reduce_parts(const float2 *part, int nblk, int n, const Sink &sink, cudaStream_t st);
int chunk_terms_for(int N);          // after collide_set_attributes(N)
int supported_N(int N);

// bz_lines.cu: the chunked pipeline at N = 48 and 64; terms (pairs) of a chunk, running sums of a lane
int lines_chunk(int N);
int lines_splits(int N);
inline bool lines_N(int N) { return N == 48 || N == 64; }
cudaError_t lines_set_attributes(int N);
bz_status collide_lines(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink);

// bz_2d.cu (dim = 2)
cudaError_t setup_2d(Plan &pl);                       // persistent grid size (pl.fused_G)
bz_status collide_2d(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink);

// bz_inhom.cu: free streaming of nx cells (bz_transport_x)
bz_status transport_x(int N, double L, int nx, double Lx, void *f, int dtype, double t, cudaStream_t st);

// bz_rk.cu
bz_status rk4_steps(Plan &pl, void *fhat, int dtype, double dt, int nsteps, cudaStream_t st,
                    int *launches);
bz_status moments(Plan &pl, const void *fhat, int dtype, double out[5], cudaStream_t st);

}  // namespace bz

#define BZ_CUDA_TRY(expr)                                   \
    do {                                                    \
        cudaError_t _e = (expr);                            \
        if (_e != cudaSuccess) return BZ_ERR_CUDA;          \
    } while (0)
