// The chunked pipeline at N = 48 and 64 (Sec. 4, eq. realQ): lines, planes, lines.
//
// A chunk of T terms (BZ_DATA_REAL: term pairs) goes through three kernels over a scratch S[T][N^3]
// that stays in L2:
//   k_line_inv  lines along axis 1:  S = IFFT_1(beta fhat); a CTA keeps its lines of fhat in
//               registers and runs them through several terms
//   k_plane     planes j1:           S = FFT_23( h . IFFT_23(S) ) in shared memory, four of the six
//               one-axis transforms with one read and one write of the field
//   k_line_fwd  lines along axis 1:  sum += alpha . FFT_1(S), the sum over the chunk's terms in
//               registers (FP32, Kahan-compensated in term order, carried from chunk to chunk)
// so a term moves 4 fields through L2 (the order plane, pencil, plane, reduce moved 6) and the
// weights are the only traffic from HBM.  Measured, a collide before and now: N = 64 real, 192 pairs
// 616 -> 535 us; complex, 192 terms 563 -> 467; N = 48 real, 288 pairs 431 -> 355.  A chunk's kernels take 10 to 30 us
// each, the plane pass at a third of the FP32 rate with three warps a scheduler, the accumulating
// pass at 3 TB/s of loads; the two streams overlap them to about 0.6 of their sum.  Tried: planes
// as 8 x 8 by 512 threads (30 us a chunk of 19 against 28), planes landing through cp.async (33),
// 8-byte cp.async in the accumulating pass (65 against 24).  In the line passes a transform of N = A B points takes A
// threads with B points each (64 = 8 x 8, 48 = 4 x 12): n = A n1 + n2, k = k1 + B k2,
//   X[k1 + B k2] = sum_n2 W_A^(n2 k2) [ W_N^(n2 k1) sum_n1 x[A n1 + n2] W_B^(n1 k1) ];
// thread n2 transforms over n1; after an exchange through shared memory thread c transforms
// over n2 for its k1 = c, c + A, ... and holds the indices A n1 + c again.
#include <algorithm>

#include "bz_cluster.cuh"
#include "bz_fft.cuh"
#include "bz_internal.h"

namespace bz {

namespace {

template <int N> struct LP {
    static constexpr int A = N == 64 ? 8 : 4, B = N / A;
    static constexpr int N2 = N * N;
    static constexpr size_t N3 = (size_t)N * N * N;
    static constexpr int PPC = N == 64 ? 1 : 2;            // planes per CTA of k_plane
    static constexpr int TP = N * PPC, TL = 32 * A;        // threads of a k_plane CTA, of 32 lines
    static constexpr size_t PLANE_SMEM = (size_t)PPC * N * (N + 1) * sizeof(float2);
    static constexpr size_t FWD_SMEM = 4 * (size_t)N * 32 * sizeof(float2);   // two stages of (field, weights)
    static constexpr int EXTRA = 2 * N / 32;               // CTAs of the Nyquist lines (k_line_fwd)
    // Splits of a chunk's terms in k_line_fwd (CTAs of one wave), groups of them in k_line_inv, terms of a
    // chunk.  The scratch of both streams has to stay in the L2 of one die: measured at N = 64, 192 pairs
    // (12: 548 us, 14: 547, 16: 556, 19: 570), at N = 48, 288 pairs (22: 400, 30: 362, 36: 370).
    static constexpr int SPLITS = N == 64 ? 2 : 3, GROUPS = 4, CHUNK = N == 64 ? 14 : 30;
};

// x[k1] *= W_N^(SIGN n2 k1); w: the roots exp(+2 pi i j / N)
template <int N, int SIGN, class W> __device__ __forceinline__ void twiddle(float2 (&x)[LP<N>::B], int n2, const W *w) {
    #pragma unroll
    for (int k1 = 1; k1 < LP<N>::B; ++k1) {
        float2 v = w[n2 * k1];
        if (SIGN < 0) v.y = -v.y;
        x[k1] = cmul(x[k1], v);
    }
}
// get(k1, n2): the exchanged values; x[m + (B / A) k2] = X at index A (m + (B / A) k2) + c
template <int N, int SIGN, class Get> __device__ __forceinline__ void stage2(float2 (&x)[LP<N>::B], int c, Get get) {
    constexpr int A = LP<N>::A, B = LP<N>::B;
    #pragma unroll
    for (int m = 0; m < B / A; ++m) {
        float2 z[A];
        #pragma unroll
        for (int n2 = 0; n2 < A; ++n2) z[n2] = get(c + A * m, n2);
        fft_inplace<A, SIGN>(z);
        #pragma unroll
        for (int k2 = 0; k2 < A; ++k2) x[m + (B / A) * k2] = z[k2];
    }
}

// One transform along axis 1 of 32 lines (lane = line, warp = role): tile [N][32], free when called.
template <int N, int SIGN> __device__ __forceinline__ void line_fft(float2 (&x)[LP<N>::B], float2 *tile, int role, int lane) {
    constexpr int A = LP<N>::A, B = LP<N>::B;
    fft_inplace<B, SIGN>(x);
    twiddle<N, SIGN>(x, role, c_tw.v + tw_off<N>());       // warp-uniform: constant-bank broadcasts
    #pragma unroll
    for (int k1 = 0; k1 < B; ++k1) tile[(A * k1 + role) * 32 + lane] = x[k1];
    __syncthreads();
    stage2<N, SIGN>(x, role, [&](int k1, int n2) { return tile[(A * k1 + n2) * 32 + lane]; });
}

// 32 lines (k2, k3) per CTA, terms t0 .. t0 + per of the chunk; their twiddles are staged in shared
// memory at the start.  Bound by the latency of the exchange and by the stores to L2.
template <int N, bool PAIR>
__global__ void __launch_bounds__(LP<N>::TL, N == 64 ? 4 : 6)
k_line_inv(const float2 *__restrict__ f, const float2 *__restrict__ tw, float2 *__restrict__ S, int p0, int T, int per,
           int use_tw, const float *__restrict__ gsc, int M) {
    using P = LP<N>;
    constexpr int A = P::A, B = P::B, NT = (PAIR ? 6 : 3) * N;
    extern __shared__ float2 lsm[];
    float2 *tile = lsm, *stw = lsm + 2 * N * 32;           // two exchange tiles, [per][NT]
    const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
    const int g = blockIdx.x * 32 + lane, k2 = g / N, k3 = g % N;
    const int t0 = blockIdx.y * per, t1 = min(T, t0 + per);
    if (use_tw) {
        const float2 *w = tw + (size_t)(p0 + t0) * NT;
        for (int i = 2 * threadIdx.x; i < (t1 - t0) * NT; i += 2 * P::TL) cp_async16(stw + i, w + i);
        cp_async_commit();
    }
    float2 y[B];
    #pragma unroll
    for (int i = 0; i < B; ++i) y[i] = f[(size_t)(A * i + role) * P::N2 + g];
    cp_async_wait_all();
    __syncthreads();
    for (int t = t0; t < t1; ++t) {
        float2 x[B];
        if (use_tw) {
            // beta(k1, k2, k3) = b1(k1) b2(k2) b3(k3) per term; a pair takes b + i b'
            const float2 *w = stw + (t - t0) * NT;
            float2 a = cmul(w[N + k2], w[2 * N + k3]), b = make_float2(0.f, 0.f);
            if constexpr (PAIR) b = cmul(w[4 * N + k2], w[5 * N + k3]);
            if (gsc) {                                     // a batch slot's radial scale (a pair shares its node)
                const float sc = gsc[(PAIR ? 2 * (p0 + t) : p0 + t) / M];
                a = cscale(a, sc);
                b = cscale(b, sc);
            }
            #pragma unroll
            for (int i = 0; i < B; ++i) {
                float2 u = cmul(a, w[A * i + role]);
                if constexpr (PAIR) {
                    const float2 v = cmul(b, w[3 * N + A * i + role]);
                    u = make_float2(u.x - v.y, u.y + v.x);
                }
                x[i] = cmul(y[i], u);
            }
        } else {
            #pragma unroll
            for (int i = 0; i < B; ++i) x[i] = y[i];
        }
        line_fft<N, +1>(x, tile + ((t - t0) & 1) * N * 32, role, lane);   // two tiles: the barrier inside frees the other
        float2 *o = S + (size_t)t * P::N3 + g;
        #pragma unroll
        for (int i = 0; i < B; ++i) o[(size_t)(A * i + role) * P::N2] = x[i];
    }
}

// Planes j1 of one term, PPC to a CTA: a thread holds a whole line (columns along axis 2, then rows along
// axis 3), so four transforms take two exchanges.  h is kept as [j1][j3][j2], the order the rows
// read it in.  MODE 0: h = IFFT_23(S) (complex); 1: its real part as packed floats; 2: S = FFT_23(h
// IFFT_23(S)), h complex; 3: h real.  Bound by FP32 issue at three or four warps a scheduler.
template <int N, int MODE>
__global__ void __launch_bounds__(LP<N>::TP, N == 64 ? 6 : 5)
k_plane(float2 *__restrict__ S, const float2 *__restrict__ h, float2 *__restrict__ out) {
    using P = LP<N>;
    constexpr int LD = N + 1;
    extern __shared__ float2 tile[];
    const int c = threadIdx.x % N, pi = threadIdx.x / N, j1 = blockIdx.x * P::PPC + pi;
    float2 *s = tile + pi * N * LD;
    float2 *pl = S + (size_t)blockIdx.y * P::N3 + (size_t)j1 * P::N2 + c;
    float2 x[N];
    #pragma unroll
    for (int i = 0; i < N; ++i) x[i] = pl[i * N];
    fft_inplace<N, +1>(x);                                 // k2 -> j2 of column k3 = c
    #pragma unroll
    for (int i = 0; i < N; ++i) s[i * LD + c] = x[i];
    __syncthreads();
    #pragma unroll
    for (int i = 0; i < N; ++i) x[i] = s[c * LD + i];
    fft_inplace<N, +1>(x);                                 // k3 -> j3 of row j2 = c
    const size_t ho = (size_t)j1 * P::N2 + c;
    if constexpr (MODE < 2) {
        #pragma unroll
        for (int i = 0; i < N; ++i) {
            if constexpr (MODE == 0) out[ho + i * N] = x[i];
            else ((float *)out)[ho + i * N] = x[i].x;
        }
        return;
    }
    #pragma unroll
    for (int i = 0; i < N; ++i) {
        if constexpr (MODE == 3) x[i] = cscale(x[i], __ldg((const float *)h + ho + i * N));
        else x[i] = cmul(x[i], __ldg(h + ho + i * N));
    }
    fft_inplace<N, -1>(x);                                 // j3 -> k3
    #pragma unroll
    for (int i = 0; i < N; ++i) s[c * LD + i] = x[i];      // the thread's own row
    __syncthreads();
    #pragma unroll
    for (int i = 0; i < N; ++i) x[i] = s[i * LD + c];
    fft_inplace<N, -1>(x);                                 // j2 -> k2
    #pragma unroll
    for (int i = 0; i < N; ++i) pl[i * N] = x[i];
}

// Kahan-compensated FP32 sum of one component.
__device__ __forceinline__ void kahan(float &s, float &c, float v) {
    const float y = v - c, t = s + y;
    c = (t - s) - y;
    s = t;
}

// 32 lines (k2, k3) per CTA, terms t = blockIdx.y, + splits, ... of the chunk.  state [splits][N^3]
// (s.x, s.y, c.x, c.y) is the running sum of the split's terms (first: starts at zero).  PAIR: the terms'
// products X = C Z on the Nyquist planes go to xs [pairs][3][N][N] (families k1 = -N/2 [k2][k3], k2 = -N/2
// [k1][k3], k3 = -N/2 [k1][k2]), the first from here, the others from EXTRA further CTAs a term, which
// transform their 2 N lines again: kept beside the sums they would cost every CTA its registers, and
// summed by a few CTAs over all terms they take longer than the rest of the launch (69 us against 24).
// A warp copies its own rows (k1 = A i + role, 32 lines of 8 bytes) one term ahead and past L1; once they
// are in registers the exchange runs through the field's places: each warp writes its own.
// Bound by the loads: 8 N^3 bytes of scratch from L2 and as many of weights from HBM a term.
template <int N, bool PAIR>
__global__ void __launch_bounds__(LP<N>::TL, N == 64 ? 3 : 4)
k_line_fwd(const float2 *__restrict__ S, const float2 *__restrict__ wtab, const float2 *__restrict__ cpair,
           float4 *__restrict__ state, float2 *__restrict__ xs, int p0, int T, int first) {
    using P = LP<N>;
    constexpr int A = P::A, B = P::B;
    extern __shared__ float2 lsm[];                        // two stages of (field, weights)
    const int lane = threadIdx.x & 31, role = threadIdx.x >> 5, splits = gridDim.y;
    if constexpr (PAIR) {
        if (blockIdx.x >= P::N2 / 32) {                    // one term of 32 Nyquist lines
            const int e = blockIdx.x - P::N2 / 32, t = e / P::EXTRA * splits + blockIdx.y;
            if (t >= T) return;
            const int u = e % P::EXTRA * 32 + lane, fam = 1 + u / N, v = u % N;
            const float2 *in = S + (size_t)t * P::N3 + (fam == 1 ? (N / 2) * N + v : v * N + N / 2);
            const size_t o = ((size_t)(p0 + t) * 3 + fam) * P::N2 + v;
            float2 x[B], al[B];
            #pragma unroll
            for (int i = 0; i < B; ++i) x[i] = in[(size_t)(A * i + role) * P::N2];
            #pragma unroll
            for (int i = 0; i < B; ++i) al[i] = __ldcs(cpair + o + (A * i + role) * N);
            line_fft<N, -1>(x, lsm, role, lane);
            #pragma unroll
            for (int i = 0; i < B; ++i) xs[o + (A * i + role) * N] = cmul(x[i], al[i]);
            return;
        }
    }
    const int g0 = blockIdx.x * 32, g = g0 + lane;
    const float2 *w0 = wtab + (size_t)p0 * P::N3 + g0;
    float4 *st = state + (size_t)blockIdx.y * P::N3 + g;
    float4 s[B];
    #pragma unroll
    for (int i = 0; i < B; ++i) s[i] = first ? make_float4(0.f, 0.f, 0.f, 0.f) : st[(A * i + role) * P::N2];
    auto fetch = [&](int t, int buf) {
        if (t < T) {
            float2 *d = lsm + buf * 2 * N * 32;
            const float2 *in = S + (size_t)t * P::N3 + g0, *wi = w0 + (size_t)t * P::N3;
            #pragma unroll
            for (int i = 0; i < B / 2; ++i) {              // two rows at a time: 16 lanes each
                const int k = A * (2 * i + lane / 16) + role, e = 2 * (lane % 16);
                cp_async16(d + k * 32 + e, in + k * P::N2 + e);
                cp_async16(d + (N + k) * 32 + e, wi + k * P::N2 + e);
            }
        }
        cp_async_commit();
    };
    fetch(blockIdx.y, 0);
    int it = 0;
    for (int t = blockIdx.y; t < T; t += splits, ++it) {
        if (it) __syncthreads();                           // the other stage's exchange is over
        fetch(t + splits, (it + 1) & 1);
        const size_t xo = (size_t)(p0 + t) * 3 * P::N2 + g;
        float2 cz = make_float2(0.f, 0.f);
        if (PAIR && role == 0) cz = __ldcs(cpair + xo);    // index N/2 = A (N / 2A) + 0
        cp_async_wait_1();
        __syncwarp();
        float2 x[B], al[B];
        float2 *tile = lsm + (it & 1) * 2 * N * 32;
        const float2 *d = tile + role * 32 + lane;
        #pragma unroll
        for (int i = 0; i < B; ++i) x[i] = d[A * i * 32];
        __syncwarp();
        line_fft<N, -1>(x, tile, role, lane);
        #pragma unroll
        for (int i = 0; i < B; ++i) al[i] = d[(N + A * i) * 32];
        #pragma unroll
        for (int i = 0; i < B; ++i) {
            const float2 z = cmul(x[i], al[i]);
            kahan(s[i].x, s[i].z, z.x);
            kahan(s[i].y, s[i].w, z.y);
        }
        if (PAIR && role == 0) xs[xo] = cmul(x[N / (2 * A)], cz);
    }
    #pragma unroll
    for (int i = 0; i < B; ++i) st[(A * i + role) * P::N2] = s[i];
}

// acc[e] = sum over the units u of xs[u][e], n entries each: 32 entries x 8 slices to a block, slice j adds u = u0 +
// j, + 8, ... (compensated), then the slices in order.
__global__ void __launch_bounds__(256) k_x_sum(const float2 *__restrict__ xs, int u0, int u1, int n, double2 *__restrict__ acc) {
    __shared__ float4 red[8][32];
    const int kk = threadIdx.x % 32, sl = threadIdx.x / 32, e = blockIdx.x * 32 + kk;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    #pragma unroll 4
    for (int u = u0 + sl; u < u1; u += 8) {
        const float2 v = __ldcs(xs + (size_t)u * n + e);
        kahan(s.x, s.z, v.x);
        kahan(s.y, s.w, v.y);
    }
    red[sl][kk] = s;
    __syncthreads();
    if (sl) return;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    #pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float4 q = red[j][kk];
        kahan(a.x, a.z, q.x);
        kahan(a.y, a.w, q.y);
        kahan(a.x, a.z, -q.z);
        kahan(a.y, a.w, -q.w);
    }
    acc[e] = make_double2((double)a.x - (double)a.z, (double)a.y - (double)a.w);
}

// sink(i) = the sum of the n_states running sums in order, compensated in FP32 and turned into FP64 once
// (FP64 additions of every state took 26 us at N = 64).
__global__ void k_state_sum(const float4 *__restrict__ state, int n_states, int n, Sink sink) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < n_states; ++k) {
        const float4 v = __ldcs(state + (size_t)k * n + i);
        kahan(a.x, a.z, v.x);
        kahan(a.y, a.w, v.y);
        kahan(a.x, a.z, -v.z);
        kahan(a.y, a.w, -v.w);
    }
    sink_put(sink, i, make_double2((double)a.x - (double)a.z, (double)a.y - (double)a.w));
}

template <int N> cudaError_t attrs() {
    const void *k[4] = {(const void *)k_plane<N, 0>, (const void *)k_plane<N, 1>, (const void *)k_plane<N, 2>,
                        (const void *)k_plane<N, 3>};
    cudaError_t e = cudaSuccess;
    auto smem = [&](const void *p, size_t bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(p, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(p, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    };
    for (const void *p : k) smem(p, LP<N>::PLANE_SMEM);
    smem((const void *)k_line_fwd<N, false>, LP<N>::FWD_SMEM);
    smem((const void *)k_line_fwd<N, true>, LP<N>::FWD_SMEM);
    smem((const void *)k_line_inv<N, false>, 227 * 1024);
    smem((const void *)k_line_inv<N, true>, 227 * 1024);
    return e;
}

template <int N, bool REAL> bz_status run(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink) {
    using P = LP<N>;
    const int u0 = REAL ? p0 / 2 : p0, u1 = REAL ? p1 / 2 : p1;
    const int n3 = (int)P::N3, ns = REAL ? 3 * P::N2 : 0;
    if (REAL && ((p0 | p1) & 1)) return BZ_ERR_ARG;
    int nl = 0;
    auto inv_smem = [](int per) { return (size_t)(2 * N * 32 + per * (REAL ? 6 : 3) * N) * sizeof(float2); };
    tm_begin(pl, st);
    const float2 *f = pl.f32;
    if (REAL) {
        const bz_status s = sym_input(pl, pl.src, pl.src_dtype, st);
        if (s != BZ_OK) return s;
        f = pl.fsym;
        ++nl;
    }
    k_line_inv<N, false><<<dim3(P::N2 / 32, 1), P::TL, inv_smem(0), st>>>(f, pl.tw, pl.S, 0, 1, 1, 0, nullptr, 1);
    k_plane<N, REAL ? 1 : 0><<<dim3(N / P::PPC, 1), P::TP, P::PLANE_SMEM, st>>>(pl.S, nullptr, pl.h);
    tm_end(pl, st, TK_OTHER);
    nl += 2;
    const int nchunks = (u1 - u0 + pl.chunk - 1) / pl.chunk;
    // lanes: as many streams as chunks, up to 1 + pl.xn
    const int lanes = 1 + (pl.xn < nchunks - 1 ? pl.xn : (nchunks > 1 ? nchunks - 1 : 0));
    if (lanes > 1) {
        BZ_CUDA_TRY(cudaEventRecord(pl.ev_fork, st));
        for (int e = 0; e + 1 < lanes; ++e) BZ_CUDA_TRY(cudaStreamWaitEvent(pl.xst[e], pl.ev_fork, 0));
    }
    for (int c0 = u0, i = 0; c0 < u1; c0 += pl.chunk, ++i) {
        const int T = u1 - c0 < pl.chunk ? u1 - c0 : pl.chunk, ln = i % lanes;
        cudaStream_t cs = ln ? pl.xst[ln - 1] : st;
        float2 *S = ln ? pl.xS[ln - 1] : pl.S;
        float4 *state = pl.lstate + (size_t)ln * P::SPLITS * P::N3;
        const int per = std::min((T + P::GROUPS - 1) / P::GROUPS, 16);   // their twiddles are staged
        tm_begin(pl, cs);
        k_line_inv<N, REAL><<<dim3(P::N2 / 32, (T + per - 1) / per), P::TL, inv_smem(per), cs>>>(f, pl.tw, S, c0, T, per, 1, pl.gsc_cur, pl.M);
        tm_end(pl, cs, TK_PENCIL);
        tm_begin(pl, cs);
        k_plane<N, REAL ? 3 : 2><<<dim3(N / P::PPC, T), P::TP, P::PLANE_SMEM, cs>>>(S, pl.h, nullptr);
        tm_end(pl, cs, TK_PLANE_INV);
        tm_begin(pl, cs);
        const int extra = REAL ? P::EXTRA * ((T + P::SPLITS - 1) / P::SPLITS) : 0;
        k_line_fwd<N, REAL><<<dim3(P::N2 / 32 + extra, P::SPLITS), P::TL, P::FWD_SMEM, cs>>>(
            S, REAL ? pl.apair : pl.alpha, pl.cpair, state, pl.xs, c0, T, i < lanes);
        tm_end(pl, cs, TK_REDUCE);
        nl += 3;
    }
    for (int e = 0; e + 1 < lanes; ++e) {
        BZ_CUDA_TRY(cudaEventRecord(pl.xev_join[e], pl.xst[e]));
        BZ_CUDA_TRY(cudaStreamWaitEvent(st, pl.xev_join[e], 0));
    }
    tm_begin(pl, st);
    k_state_sum<<<(n3 + 255) / 256, 256, 0, st>>>(pl.lstate, nchunks > 0 ? lanes * P::SPLITS : 0, n3,
                                                 REAL ? acc_sink(pl) : sink);
    ++nl;
    if (REAL) {
        k_x_sum<<<ns / 32, 256, 0, st>>>(pl.xs, u0, u1, ns, pl.acc_s);
        ++nl;
        const bz_status s = sym_output(pl, st, sink);
        if (s != BZ_OK) return s;
        ++nl;
    }
    tm_end(pl, st, TK_OTHER);
    BZ_CUDA_TRY(cudaGetLastError());
    if (launches) *launches += nl;
    return BZ_OK;
}

}  // namespace

cudaError_t lines_set_attributes(int N) { return N == 64 ? attrs<64>() : attrs<48>(); }
int lines_chunk(int N) { return N == 64 ? LP<64>::CHUNK : LP<48>::CHUNK; }
int lines_splits(int N) { return N == 64 ? LP<64>::SPLITS : LP<48>::SPLITS; }

bz_status collide_lines(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink) {
    if (pl.N == 64) return pl.real ? run<64, true>(pl, p0, p1, st, launches, sink) : run<64, false>(pl, p0, p1, st, launches, sink);
    return pl.real ? run<48, true>(pl, p0, p1, st, launches, sink) : run<48, false>(pl, p0, p1, st, launches, sink);
}

}  // namespace bz
