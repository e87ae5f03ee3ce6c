// The 2D operator (Sec. 4 with d = 2; Sec. 4.1 (i)) on an N x N grid, N <= 64.
//
// A term's field is a slot of N threads, one line each, with [N][N + 1] values of shared memory; a CTA of
// 128 threads holds 128 / N slots, each with a block of terms of its own.  Per term (twiddles
// beta_p per axis, alpha_p = c_p F / N^2):
//   columns (thread = k2):  x = beta_p fhat over k1, IFFT over k1 -> S            (sync)
//   rows    (thread = j1):  IFFT over k2, times h, FFT over j2 -> S              (sync)
//   columns (thread = k2):  FFT over j1, acc += alpha_p x  (acc[., k2] is the thread's own)
// A column pass writes and reads only its own column of S, so the next term's first pass
// needs no barrier; the others are between the threads of a slot (two warps at N = 64, one or a part
// of one below).  The sums stay in registers, at N = 64 in tensor memory (128 words a thread), which
// lets two CTAs of four warps share an SM (three would spill: 85 us against 54); kept in shared memory they
// left room for six warps.  A
// CTA adds its slots' sums, and k_reduce_parts the CTAs', in a fixed order.  h = IFFT(fhat) is
// formed beforehand in double-float arithmetic (bz_hff.cu), stored FP32 as [j2][j1].
// Bound by FP32 issue and latency at eight warps an SM (N = 64).  Measured at N = 64, P = 2048: 54 us, and 74 with
// the sums in shared memory and h read by rows (32 sectors a load).
#include "bz_fft.cuh"
#include "bz_internal.h"
#include "bz_tmem.cuh"

namespace bz {

namespace {

constexpr int T2 = 128;
template <int N> struct D2 {
    static constexpr int LD = N + 1, SLOTS = T2 / N;
    static constexpr bool TM = N == 64;                   // sums in tensor memory
    static constexpr size_t SMEM = (size_t)SLOTS * N * LD * sizeof(float2);
    static constexpr int CTAS = N == 64 ? 2 : (N == 32 ? 3 : (N == 16 ? 5 : 8));   // per SM
};

// Slots blk = blockIdx.x * SLOTS + slot < nslots; slot blk takes the terms p0 + [blk, blk + 1) (p1 - p0) / nslots.
template <int N>
__global__ void __launch_bounds__(T2, D2<N>::CTAS)
k_collide_2d(const float2 *__restrict__ fin, const float2 *__restrict__ h, const float2 *__restrict__ tw,
             const float2 *__restrict__ alpha, float2 *__restrict__ part, int p0, int p1, int nslots) {
    using D = D2<N>;
    constexpr int LD = D::LD, N2 = N * N, NA = D::TM ? 1 : N;
    extern __shared__ float2 s2[];
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, slot = tid / N, c = tid % N, blk = blockIdx.x * D::SLOTS + slot;
    float2 *S = s2 + (size_t)slot * N * LD;
    uint32_t tl = 0;
    float2 acc[NA];
    #pragma unroll
    for (int i = 0; i < NA; ++i) acc[i] = make_float2(0.f, 0.f);
    if constexpr (D::TM) {
        if (tid < 32) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;\n"
                         ::"r"((uint32_t)__cvta_generic_to_shared(&s_tmem)) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        }
        tfence_before();
        __syncthreads();
        tfence_after();
        tl = s_tmem + ((uint32_t)(tid & ~31) << 16);
        float z[16];
        #pragma unroll
        for (int i = 0; i < 16; ++i) z[i] = 0.f;
        #pragma unroll
        for (int g = 0; g < 8; ++g) t_st16(tl + 16 * g, z);
        t_wait_st();
    }
    auto slot_sync = [&] {
        if constexpr (N == 64) asm volatile("bar.sync %0, 64;\n" ::"r"(1 + slot) : "memory");
        else __syncwarp();
    };
    const int nt = p1 - p0;
    const int t0 = p0 + (int)((long long)blk * nt / nslots), t1 = p0 + (int)((long long)(blk + 1) * nt / nslots);
    const int most = (nt + nslots - 1) / nslots;              // the same count of rounds for every slot of a warp
    for (int it = 0; it < most; ++it) {
        // a slot with nothing left repeats a term without adding it (its lanes share the warp's barriers)
        const bool on = blk < nslots && t0 + it < t1;
        if (D::TM && !on) break;                          // (N = 64: a slot is whole warps with a barrier of its own)
        const int p = on ? t0 + it : p0;
        const float2 *twp = tw + (size_t)p * 3 * N;           // [axis][m]; the third axis is unused in 2D
        const float2 *al = alpha + (size_t)p * N2;
        if (c == 0)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(al), "r"((uint32_t)(N2 * sizeof(float2))) : "memory");
        al += c;
        const float2 t2 = __ldg(twp + N + c);
        float2 x[N];
        #pragma unroll
        for (int i = 0; i < N; ++i) x[i] = cmul(fin[i * N + c], cmul(__ldg(twp + i), t2));
        fft_inplace<N, +1>(x);                               // k1 -> j1
        #pragma unroll
        for (int i = 0; i < N; ++i) S[i * LD + c] = x[i];
        slot_sync();
        #pragma unroll
        for (int j = 0; j < N; ++j) x[j] = S[c * LD + j];
        fft_inplace<N, +1>(x);                               // k2 -> j2 (row j1 = c)
        #pragma unroll
        for (int j = 0; j < N; ++j) x[j] = cmul(x[j], __ldg(h + j * N + c));
        fft_inplace<N, -1>(x);                               // j2 -> k2
        #pragma unroll
        for (int j = 0; j < N; ++j) S[c * LD + j] = x[j];
        slot_sync();
        #pragma unroll
        for (int i = 0; i < N; ++i) x[i] = S[i * LD + c];
        fft_inplace<N, -1>(x);                               // j1 -> k1 (column k2 = c)
        if constexpr (D::TM) {
            #pragma unroll
            for (int g = 0; g < 16; ++g) {
                float2 w[4];
                #pragma unroll
                for (int u = 0; u < 4; ++u)              // volatile: all 64 loaded at once would spill
                    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];\n" : "=f"(w[u].x), "=f"(w[u].y) : "l"(al + (4 * g + u) * N));
                float s[8];
                t_ld8(tl + 8 * g, s);
                t_wait_ld();
                #pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 z = x[4 * g + u];
                    s[2 * u] = fmaf(z.x, w[u].x, fmaf(-z.y, w[u].y, s[2 * u]));
                    s[2 * u + 1] = fmaf(z.x, w[u].y, fmaf(z.y, w[u].x, s[2 * u + 1]));
                }
                t_st8(tl + 8 * g, s);
            }
            t_wait_st();
        } else if (on) {
            #pragma unroll
            for (int i = 0; i < N; ++i) {
                const float2 w = __ldg(al + i * N);
                acc[i].x = fmaf(x[i].x, w.x, fmaf(-x[i].y, w.y, acc[i].x));
                acc[i].y = fmaf(x[i].x, w.y, fmaf(x[i].y, w.x, acc[i].y));
            }
        }
    }
    // the CTA's sum over its slots, compensated, in slot order
    if constexpr (D::TM) {
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            float s[16];
            t_ld16(tl + 16 * g, s);
            t_wait_ld();
            #pragma unroll
            for (int u = 0; u < 8; ++u) S[(8 * g + u) * LD + c] = make_float2(s[2 * u], s[2 * u + 1]);
        }
        tfence_before();
    } else {
        #pragma unroll
        for (int i = 0; i < N; ++i) S[i * LD + c] = acc[i];
    }
    __syncthreads();
    if constexpr (D::TM) {
        if (tid < 32)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;\n" ::"r"(s_tmem) : "memory");
    }
    float2 *out = part + (size_t)blockIdx.x * N2;
    for (int e = tid; e < N2; e += T2) {
        float2 s = make_float2(0.f, 0.f), k = s;
        #pragma unroll
        for (int j = 0; j < D::SLOTS; ++j) {
            const float2 v = s2[(size_t)j * N * LD + (e / N) * LD + e % N];
            const float yx = v.x - k.x, yy = v.y - k.y, tx = s.x + yx, ty = s.y + yy;
            k = make_float2((tx - s.x) - yx, (ty - s.y) - yy);
            s = make_float2(tx, ty);
        }
        out[e] = s;
    }
}

// pl.fused_G: CTAs that are resident at once
template <int N> cudaError_t setup_n(Plan &pl) {
    const cudaError_t e = cudaFuncSetAttribute(k_collide_2d<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D2<N>::SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    pl.fused_G = D2<N>::CTAS * sms;
    pl.fused_C = 1;
    return sms > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

template <int N> bz_status run_n(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink) {
    using D = D2<N>;
    const int nt = p1 - p0, most = pl.fused_G * D::SLOTS, nslots = nt < most ? nt : most;
    const int ctas = (nslots + D::SLOTS - 1) / D::SLOTS;
    tm_begin(pl, st);
    const bz_status hs = hff_launch_2d(N, pl.h_fp64, pl.src, pl.src_dtype, pl.h, pl.fcopy, st);
    if (hs != BZ_OK) return hs;
    tm_end(pl, st, TK_OTHER);
    tm_begin(pl, st);
    if (ctas > 0)
        k_collide_2d<N><<<ctas, T2, D::SMEM, st>>>(pl.f32, pl.h, pl.tw, pl.alpha, pl.part, p0, p1, nslots);
    tm_end(pl, st, TK_FUSED);
    tm_begin(pl, st);
    reduce_parts(pl.part, ctas, N * N, sink, st);
    tm_end(pl, st, TK_REDUCE);
    BZ_CUDA_TRY(cudaGetLastError());
    if (launches) *launches += ctas > 0 ? 3 : 2;
    return BZ_OK;
}

}  // namespace

cudaError_t setup_2d(Plan &pl) {
    switch (pl.N) {
        case 8: return setup_n<8>(pl);
        case 16: return setup_n<16>(pl);
        case 32: return setup_n<32>(pl);
        case 64: return setup_n<64>(pl);
    }
    return cudaErrorInvalidValue;
}

bz_status collide_2d(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink) {
    switch (pl.N) {
        case 8: return run_n<8>(pl, p0, p1, st, launches, sink);
        case 16: return run_n<16>(pl, p0, p1, st, launches, sink);
        case 32: return run_n<32>(pl, p0, p1, st, launches, sink);
        case 64: return run_n<64>(pl, p0, p1, st, launches, sink);
    }
    return BZ_ERR_UNSUPPORTED;
}

}  // namespace bz
