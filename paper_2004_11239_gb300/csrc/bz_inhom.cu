// Free streaming df/dt + v_1 df/dx = 0 of nx cells of Fourier coefficients (bz_transport_x).
//
// With f(x_c, v) = sum_k fhat_c(k) exp(i pi k.v / L) the exact solution f(x - v_1 t, v) at the
// velocity nodes needs the values along v_1 only: for each (k2, k3), the nx x N array
// fhat_c(k1, k2, k3) is transformed over the cells (x-DFT), over k1 to the node values
// f(v_1j) = sum_k1 (-1)^k1 fhat(k1) exp(2 pi i k1 j / N) (the factor (-1)^k1 = exp(-i pi k1)
// from the grid origin -L), multiplied by exp(-2 pi i kappa v_1j t / Lx), and transformed back.
// One CTA per (k2, k3); the array sits in shared memory between the passes, a line takes eight
// lanes (bz_line8.cuh) or, in FP64 from N = 24 and 16 cells on, one thread.  complex128 cells are computed in FP64, complex64 ones in double-float (the
// stored result has the error of its rounding; an FP64 instruction of a warp takes 68 clocks of a
// scheduler), whose exponents are those of FP32: a CTA brings its largest component near 1 by a power
// of two first, or the sums over the lines could leave the range that the cells are in.  The phases are
// products of two tables of powers of exp(2 pi i t L / (Lx N)), 49 FP64 sincospi a CTA.
#include <cmath>

#include "bz_internal.h"
#include "bz_line8.cuh"

namespace bz {

namespace {

// exp(i m theta) = a[m / 32] b[m mod 32] for |m| <= 512
struct Phases {
    double2 a[17], b[32];
};
__device__ __forceinline__ void load_c(const void *f, size_t i, cd &v) {
    const double2 u = ((const double2 *)f)[i];
    v = {u.x, u.y};
}
__device__ __forceinline__ void load_c(const void *f, size_t i, ffc &v) {
    const float2 u = ((const float2 *)f)[i];
    v = {{u.x, 0.f}, {u.y, 0.f}};
}
__device__ __forceinline__ void store_c(void *f, size_t i, cd v) { ((double2 *)f)[i] = make_double2(v.x, v.y); }
__device__ __forceinline__ void store_c(void *f, size_t i, ffc v) { ((float2 *)f)[i] = round2(v); }
// The bits of the larger |component|, and x times a power of two (cd needs no scaling)
__device__ __forceinline__ unsigned top_bits(ffc v) {
    return max(__float_as_uint(v.x.h) & 0x7fffffffu, __float_as_uint(v.y.h) & 0x7fffffffu);
}
__device__ __forceinline__ cd times2(cd v, float) { return v; }
__device__ __forceinline__ ffc times2(ffc v, float s) { return {{v.x.h * s, v.x.l * s}, {v.y.h * s, v.y.l * s}}; }
__device__ __forceinline__ void from_d(double2 u, cd &v) { v = {u.x, u.y}; }
__device__ __forceinline__ void from_d(double2 u, ffc &v) { v = {split(u.x), split(u.y)}; }
__device__ __forceinline__ cd times(cd v, double s) { return scale(v, s); }
__device__ __forceinline__ ffc times(ffc v, double s) { return scale(v, split(s)); }

__device__ __forceinline__ void load_phases(Phases &ph, double tau) {
    for (int e = threadIdx.x; e < 49; e += blockDim.x) {
        const int m = e < 32 ? e : 32 * (e - 32);
        double sn, cs;
        sincospi(2.0 * tau * m, &sn, &cs);
        if (e < 32) ph.b[e] = make_double2(cs, sn);
        else ph.a[e - 32] = make_double2(cs, sn);
    }
}

// Threads: 8 lanes a line, max(N, NX) lines.  C = cd (complex128 cells) or ffc (complex64).
// Bound by FP64 issue (cd) or by latency (ffc).  N = 16, 32 cells of complex64: 11 us (10 without the scaling);
// one line a thread in FP64 with a sincospi per value took 65.
template <int N, int NX, class C>
__global__ void __launch_bounds__(8 * (N > NX ? N : NX)) k_transport(void *f, double tau) {
    constexpr int R = N / 8, RX = NX / 8, WARPS = (N > NX ? N : NX) / 4;
    constexpr bool SCALE = std::is_same<C, ffc>::value;
    __shared__ C s[NX][N + 1];
    __shared__ Phases ph;
    __shared__ unsigned s_top[WARPS];
    const size_t n3 = (size_t)N * N * N;
    const size_t at = blockIdx.x;                            // k2 N + k3
    const int tid = threadIdx.x, line = tid / 8;
    load_phases(ph, tau);
    const LineFF<NX, C> X(tid & 7);
    const bool col = line < N;                               // whole warps: N and NX are multiples of 4
    C x[RX];
    if (col) {                                               // column k1 = line over the cells
        #pragma unroll
        for (int m = 0; m < RX; ++m) {
            load_c(f, (X.l + 8 * m) * n3 + (size_t)line * N * N + at, x[m]);
            x[m] = conj(x[m]);                               // forward by the inverse: conj, transform, conj
        }
    }
    float up = 1.f;                                          // 2^e and 2^-e of the array's largest component
    if constexpr (SCALE) {
        unsigned top = 0;
        #pragma unroll
        for (int m = 0; m < RX; ++m) top = max(top, col ? top_bits(x[m]) : 0u);
        top = __reduce_max_sync(0xffffffffu, top);
        if ((tid & 31) == 0) s_top[tid >> 5] = top;
        __syncthreads();
        #pragma unroll
        for (int w = 0; w < WARPS; ++w) top = max(top, s_top[w]);
        const unsigned e = min(max(top >> 23, 1u), 253u);    // both powers stay normal
        up = __uint_as_float(e << 23);
        const float down = __uint_as_float((254u - e) << 23);
        #pragma unroll
        for (int m = 0; m < RX; ++m) x[m] = times2(x[m], down);
    }
    if (col) {
        X(x);                                                // cells -> x-modes kappa
        #pragma unroll
        for (int r = 0; r < RX; ++r) s[r + RX * X.q][line] = conj(x[r]);
    }
    __syncthreads();
    if (line < NX) {                                         // x-mode row over k1
        const LineFF<N, C> F(tid & 7);
        C y[R];
        #pragma unroll
        for (int m = 0; m < R; ++m) {
            y[m] = s[line][F.l + 8 * m];
            if (F.l & 1) y[m] = neg(y[m]);                   // (-1)^k1
        }
        F(y);                                                // k1 -> node values f(v_1j)
        // phase exp(-2 pi i kappa v_1j t / Lx), v_1j = -L + 2 L j / N: exp(i kappa (N - 2 j) theta)
        const int kappa = line < NX / 2 ? line : line - NX;
        #pragma unroll
        for (int r = 0; r < R; ++r) {
            const int j = r + R * F.q, m = kappa * (N - 2 * j), am = m < 0 ? -m : m;
            C a, b;
            from_d(ph.a[am >> 5], a);
            from_d(ph.b[am & 31], b);
            a = mul(a, b);
            y[r] = conj(mul(y[r], m < 0 ? conj(a) : a));
        }
        // node values -> k1: y[r] sits at j = r + R q of lane bitrev; back to j = l + 8 m through shared memory
        __syncwarp();
        #pragma unroll
        for (int r = 0; r < R; ++r) s[line][r + R * F.q] = y[r];
        __syncwarp();
        #pragma unroll
        for (int m = 0; m < R; ++m) y[m] = s[line][F.l + 8 * m];
        F(y);
        __syncwarp();
        const double inv = 1.0 / ((double)N * NX);           // both inverse normalisations
        #pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r + R * F.q;
            s[line][k] = times(conj(y[r]), (k & 1) ? -inv : inv);
        }
    }
    __syncthreads();
    if (col) {
        #pragma unroll
        for (int m = 0; m < RX; ++m) x[m] = s[X.l + 8 * m][line];
        X(x);                                                // x-modes -> cells
        #pragma unroll
        for (int r = 0; r < RX; ++r) store_c(f, (r + RX * X.q) * n3 + (size_t)line * N * N + at, times2(x[r], up));
    }
}

// The same with a whole line to a thread, complex128 cells: fewer FP64 operations (a 32-point line takes about 13 a
// point, 17 over eight lanes), which bound the longer lines; the short ones are latency.  us with a line over
// eight lanes / to a thread: N = 32: 58 / 90 (8 cells), 116 / 105 (16), 179 / 127 (24), 235 / 143 (32);
// N = 24: 27 / 43, 52 / 51, 78 / 64, 103 / 74; N = 16, 32 cells: 35 / 49.
template <int N, int NX>
__global__ void __launch_bounds__(N > NX ? N : NX) k_transport_line(double2 *f, double tau) {
    __shared__ double2 s[NX][N + 1];
    __shared__ Phases ph;
    const size_t n3 = (size_t)N * N * N, at = blockIdx.x;    // at: k2 N + k3
    const int tid = threadIdx.x;
    load_phases(ph, tau);
    if (tid < N) {                                           // column k1 = tid over the cells
        double2 x[NX];
        #pragma unroll
        for (int c = 0; c < NX; ++c) x[c] = f[c * n3 + (size_t)tid * N * N + at];
        fft_inplace<NX, -1>(x);                              // cells -> x-modes kappa
        #pragma unroll
        for (int c = 0; c < NX; ++c) s[c][tid] = x[c];
    }
    __syncthreads();
    if (tid < NX) {                                          // x-mode row over k1
        double2 y[N];
        #pragma unroll
        for (int i = 0; i < N; ++i) y[i] = i & 1 ? cneg(s[tid][i]) : s[tid][i];
        fft_inplace<N, +1>(y);                               // k1 -> node values
        const int kappa = tid < NX / 2 ? tid : tid - NX;
        #pragma unroll
        for (int j = 0; j < N; ++j) {
            const int m = kappa * (N - 2 * j), am = m < 0 ? -m : m;
            double2 w = cmul(ph.a[am >> 5], ph.b[am & 31]);
            if (m < 0) w.y = -w.y;
            y[j] = cmul(y[j], w);
        }
        fft_inplace<N, -1>(y);                               // node values -> k1
        const double inv = 1.0 / ((double)N * NX);           // both inverse normalisations
        #pragma unroll
        for (int i = 0; i < N; ++i) s[tid][i] = cscale(y[i], i & 1 ? -inv : inv);
    }
    __syncthreads();
    if (tid < N) {
        double2 x[NX];
        #pragma unroll
        for (int c = 0; c < NX; ++c) x[c] = s[c][tid];
        fft_inplace<NX, +1>(x);                              // x-modes -> cells
        #pragma unroll
        for (int c = 0; c < NX; ++c) f[c * n3 + (size_t)tid * N * N + at] = x[c];
    }
}

template <int N, int NX> bz_status run(void *f, int dtype, double L, double Lx, double t, cudaStream_t st) {
    const double tau = t * L / (Lx * N);
    constexpr int threads = 8 * (N > NX ? N : NX);
    if constexpr (N >= 24 && NX >= 16) {
        if (dtype == BZ_C128) k_transport_line<N, NX><<<N * N, N > NX ? N : NX, 0, st>>>((double2 *)f, tau);
    } else {
        if (dtype == BZ_C128) k_transport<N, NX, cd><<<N * N, threads, 0, st>>>(f, tau);
    }
    if (dtype == BZ_C64) k_transport<N, NX, ffc><<<N * N, threads, 0, st>>>(f, tau);
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

template <int N> bz_status run_nx(int nx, void *f, int dtype, double L, double Lx, double t, cudaStream_t st) {
    switch (nx) {
        case 8: return run<N, 8>(f, dtype, L, Lx, t, st);
        case 16: return run<N, 16>(f, dtype, L, Lx, t, st);
        case 24: return run<N, 24>(f, dtype, L, Lx, t, st);
        case 32: return run<N, 32>(f, dtype, L, Lx, t, st);
    }
    return BZ_ERR_UNSUPPORTED;
}

}  // namespace

bz_status transport_x(int N, double L, int nx, double Lx, void *f, int dtype, double t, cudaStream_t st) {
    switch (N) {
        case 8: return run_nx<8>(nx, f, dtype, L, Lx, t, st);
        case 16: return run_nx<16>(nx, f, dtype, L, Lx, t, st);
        case 24: return run_nx<24>(nx, f, dtype, L, Lx, t, st);
        case 32: return run_nx<32>(nx, f, dtype, L, Lx, t, st);
    }
    return BZ_ERR_UNSUPPORTED;
}

}  // namespace bz

extern "C" bz_status bz_transport_x(int N, double L, int nx, double Lx, void *fcells, int dtype, double t,
                                    void *stream) {
    if (!fcells || !(L > 0) || !(Lx > 0) || !std::isfinite(t)) return BZ_ERR_ARG;
    if (dtype != BZ_C64 && dtype != BZ_C128) return BZ_ERR_ARG;
    return bz::transport_x(N, L, nx, Lx, fcells, dtype, t, (cudaStream_t)stream);
}
