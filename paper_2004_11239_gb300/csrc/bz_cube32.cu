// Complex collide at N = 32 with one term's whole field on one SM: k_col32's passes (bz_col32.cu) for a
// full spectrum.
//
// The field is 32 columns k3 of 32 x 32 modes, 256 KB; shared memory holds 16 columns.  Along axis 3 the
// even and odd nodes separate: with e(k3) = x(k3) + x(k3 + 16) and o(k3) = (x(k3) - x(k3 + 16)) W32^k3, k3 < 16,
// the nodes j3 = 2m are the 16-point transform of e and j3 = 2m + 1 that of o; back, E and O of the two halves of
// the product with h give U(k3) = E + W32^-k3 O and U(k3 + 16) = E - W32^-k3 O.  Warp w owns the columns w and
// w + 16, whose combinations are its own, so the halves go through shared memory one after the other while
// the one not there waits in tensor memory in the lane that needs it again:
//   P1, P2 for column w (to tensor memory), then for w + 16; e to shared memory, o to tensor memory
//   -- barrier --  P3: two rows a thread, 16 points: inverse, h at the even nodes, forward, in place
//   -- barrier --  E to tensor memory, o to shared memory
//   -- barrier --  P3 with h at the odd nodes
//   -- barrier --  U of column w, P4, P5; U of column w + 16 (kept in tensor memory), P4, P5
// The sums of column w stay in tensor memory (64 words a thread, as the waiting half: all of it), those of
// column w + 16 in the item's place of the partial sums, which is in L2.  Input [k3][k1][k2], h and its product
// [j3][j1][j2], table and sums [k3][k1][k2].
// Measured at P = 1024: 179 us, k_fused (8-CTA clusters) 302.  A term takes 52 k clocks, some 28 k of them issue
// slots; bound as k_col32 by issue, the block barriers (four a term) and L2 latency (1 MB a term: fhat, h,
// weights and the second column's sums).
#include "bz_cluster.cuh"
#include "bz_fft.cuh"
#include "bz_internal.h"
#include "bz_tmem.cuh"

namespace bz {

namespace {

constexpr int QN = 32, QW = 16, QT = 32 * QW, QLD = QN + 1, QP = QN * QLD, Q2 = QN * QN;
constexpr size_t Q_SMEM = ((size_t)QW * QP + 2 * 3 * QN) * sizeof(float2);   // columns, the twiddles of two terms
constexpr uint32_t TQ_ACC = 0, TQ_HOLD = 256;                              // tensor-memory columns

__global__ void __launch_bounds__(QT, 1) k_cube32(ItemArgs a) {
    constexpr int N = QN;
    extern __shared__ __align__(16) float2 qsm[];
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    float2 *my = qsm + w * QP;                             // the warp's column: [j1 or k1][j2 or k2]
    float2 *stw = qsm + QW * QP;                           // twiddles, two buffers of [3][N]
    if (w == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n"
                     ::"r"((uint32_t)__cvta_generic_to_shared(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tfence_before();
    __syncthreads();
    tfence_after();
    const uint32_t tl = s_tmem + ((uint32_t)(32 * (w & 3)) << 16) + 64 * (w >> 2);
    constexpr size_t N3 = (size_t)N * N * N;
    const int count = a.count_dev ? *a.count_dev : a.count;
    const int nitems = count * a.nblk;
    float2 *rows = qsm + (2 * w) * QLD + lane;             // P3: rows (2w, lane) and (2w + 1, lane)
    const float2 wt = c_tw.v[tw_off<32>() + w];            // W32^w

    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const int b = it / a.nblk, blk = it % a.nblk;
        const int slot = a.slots ? a.slots[b] : b;
        const int t0 = a.p0 + blk * a.TB, t1 = min(a.p1, t0 + a.TB);
        const float2 *fin = a.fin + (size_t)slot * N3 + w * Q2 + lane;
        const float2 *hp = a.hg + (size_t)slot * N3 + 2 * w * N + lane;      // h of row (2w, lane), [j3] at stride N^2
        float2 *out = a.part + ((size_t)slot * a.nblk + blk) * N3 + w * Q2 + lane;
        {
            float v[8];
            #pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = 0.f;
            #pragma unroll
            for (int g = 0; g < 8; ++g) t_st8(tl + TQ_ACC + 8 * g, v);
            t_wait_st();
        }
        auto fetch_tw = [&](int p, int buf) {
            if (tid < 3 * N / 2) cp_async16(stw + buf * 3 * N + 2 * tid, a.tw + (size_t)p * 3 * N + 2 * tid);
            cp_async_commit();
        };
        __syncthreads();                                   // the previous item is done with the twiddles
        fetch_tw(t0, 0);
        cp_async_wait_all();
        __syncthreads();
        for (int p = t0; p < t1; ++p) {
            const float2 *tab = a.alpha + (size_t)p * N3 + w * Q2 + lane;
            if (tid == 0)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(a.alpha + (size_t)p * N3),
                             "r"((uint32_t)(N3 * sizeof(float2))) : "memory");
            const float2 *tws = stw + ((p - t0) & 1) * 3 * N;
            float2 x[N];
            #pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                // P1, P2 of column w + 16 half
                const float2 *f = fin + half * QW * Q2;
                #pragma unroll
                for (int i = 0; i < N; ++i) x[i] = f[i * N];
                float2 t23 = cmul(tws[N + lane], tws[2 * N + w + QW * half]);
                if (a.gsc) t23 = cscale(t23, a.gsc[(size_t)slot * a.N_rho + p / a.M]);
                #pragma unroll
                for (int i = 0; i < N; ++i) x[i] = cmul(x[i], cmul(t23, tws[i]));
                fft_inplace<N, +1>(x);                     // k1 -> j1
                __syncwarp();                              // the column's rows have been read (second half)
                #pragma unroll
                for (int i = 0; i < N; ++i) my[i * QLD + lane] = x[i];
                __syncwarp();
                #pragma unroll
                for (int i = 0; i < N; ++i) x[i] = my[lane * QLD + i];
                fft_inplace<N, +1>(x);                     // k2 -> j2
                if (half == 0) {
                    #pragma unroll
                    for (int g = 0; g < 8; ++g) t_st8(tl + TQ_HOLD + 8 * g, (const float *)(x + 4 * g));
                    t_wait_st();
                }
            }
            // e to the column (the thread's own row), o to tensor memory
            #pragma unroll
            for (int g = 0; g < 8; ++g) {
                float2 v[4];
                t_ld8(tl + TQ_HOLD + 8 * g, (float *)v);
                t_wait_ld();
                #pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 s = v[u], d = x[4 * g + u];
                    my[lane * QLD + 4 * g + u] = cadd(s, d);
                    v[u] = cmul(csub(s, d), wt);
                }
                t_st8(tl + TQ_HOLD + 8 * g, (const float *)v);
            }
            t_wait_st();
            __syncthreads();
            #pragma unroll 1
            for (int odd = 0; odd < 2; ++odd) {
                // P3: row (2w + r, lane), nodes j3 = 2m + odd
                #pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    float2 y[QW];
                    float2 *ro = rows + r * QLD;
                    const float2 *h = hp + r * N + odd * Q2;
                    #pragma unroll
                    for (int k = 0; k < QW; ++k) y[k] = ro[k * QP];
                    float2 hv[QW];
                    #pragma unroll
                    for (int m = 0; m < QW; ++m) hv[m] = h[2 * m * Q2];
                    fft_inplace<QW, +1>(y);
                    #pragma unroll
                    for (int m = 0; m < QW; ++m) y[m] = cmul(y[m], hv[m]);
                    fft_inplace<QW, -1>(y);
                    #pragma unroll
                    for (int k = 0; k < QW; ++k) ro[k * QP] = y[k];
                }
                if (odd) break;
                if (p + 1 < t1) fetch_tw(p + 1, (p + 1 - t0) & 1);
                __syncthreads();
                // E to tensor memory, o to the column: the thread's own row
                #pragma unroll
                for (int g = 0; g < 8; ++g) {
                    float2 v[4], e[4];
                    t_ld8(tl + TQ_HOLD + 8 * g, (float *)v);
                    t_wait_ld();
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        e[u] = my[lane * QLD + 4 * g + u];
                        my[lane * QLD + 4 * g + u] = v[u];
                    }
                    t_st8(tl + TQ_HOLD + 8 * g, (const float *)e);
                }
                t_wait_st();
                __syncthreads();
            }
            cp_async_wait_all();                           // the next twiddles
            __syncthreads();
            // U(w) = E + W^-w O, and U(w + 16) = E - W^-w O to tensor memory
            #pragma unroll
            for (int g = 0; g < 8; ++g) {
                float2 v[4];
                t_ld8(tl + TQ_HOLD + 8 * g, (float *)v);
                t_wait_ld();
                #pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 o = cmul(my[lane * QLD + 4 * g + u], make_float2(wt.x, -wt.y));
                    x[4 * g + u] = cadd(v[u], o);
                    v[u] = csub(v[u], o);
                }
                t_st8(tl + TQ_HOLD + 8 * g, (const float *)v);
            }
            t_wait_st();
            #pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                if (half) {
                    #pragma unroll
                    for (int g = 0; g < 8; ++g) t_ld8(tl + TQ_HOLD + 8 * g, (float *)(x + 4 * g));
                    t_wait_ld();
                    __syncwarp();                          // the column's reads of the first half are done
                }
                // P4, P5 of column w + 16 half
                fft_inplace<N, -1>(x);                     // j2 -> k2
                #pragma unroll
                for (int i = 0; i < N; ++i) my[lane * QLD + i] = x[i];
                __syncwarp();
                #pragma unroll
                for (int i = 0; i < N; ++i) x[i] = my[i * QLD + lane];
                const float2 *tp = tab + half * QW * Q2;
                float2 *op = out + QW * Q2;                // sums of column w + 16
                float2 an[4];
                #pragma unroll
                for (int u = 0; u < 4; ++u) an[u] = __ldg(tp + u * N);
                fft_inplace<N, -1>(x);                     // j1 -> k1
                #pragma unroll
                for (int g = 0; g < 8; ++g) {
                    float2 al[4];
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) al[u] = an[u];
                    if (g < 7) {
                        #pragma unroll
                        for (int u = 0; u < 4; ++u) an[u] = __ldg(tp + (4 * (g + 1) + u) * N);
                    }
                    float2 s[4];
                    if (half == 0) {
                        t_ld8(tl + TQ_ACC + 8 * g, (float *)s);
                        t_wait_ld();
                    } else {
                        #pragma unroll
                        for (int u = 0; u < 4; ++u) s[u] = p == t0 ? make_float2(0.f, 0.f) : op[(4 * g + u) * N];
                    }
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float2 z = x[4 * g + u];
                        s[u].x = fmaf(z.x, al[u].x, fmaf(-z.y, al[u].y, s[u].x));
                        s[u].y = fmaf(z.x, al[u].y, fmaf(z.y, al[u].x, s[u].y));
                    }
                    if (half == 0) {
                        t_st8(tl + TQ_ACC + 8 * g, (const float *)s);
                    } else {
                        #pragma unroll
                        for (int u = 0; u < 4; ++u) op[(4 * g + u) * N] = s[u];
                    }
                }
                if (half == 0) t_wait_st();
            }
            __syncwarp();                                  // the column is free again
        }
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            float2 s[4];
            t_ld8(tl + TQ_ACC + 8 * g, (float *)s);
            t_wait_ld();
            #pragma unroll
            for (int u = 0; u < 4; ++u) out[(4 * g + u) * N] = s[u];
        }
    }
    tfence_before();
    __syncthreads();
    if (w == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(s_tmem) : "memory");
}

// [rows][k1][k2][k3] -> [rows][k3][k1][k2]: one block per (row, k1).
__global__ void __launch_bounds__(256) k_cube_table(const float2 *__restrict__ in, float2 *__restrict__ out) {
    __shared__ float2 t[QN][QLD];
    const int k1 = blockIdx.x;
    const size_t row = (size_t)blockIdx.y * QN * Q2;
    for (int e = threadIdx.x; e < Q2; e += 256) t[e / QN][e % QN] = in[row + k1 * Q2 + e];   // [k2][k3]
    __syncthreads();
    for (int e = threadIdx.x; e < Q2; e += 256) out[row + (e / QN) * Q2 + k1 * QN + e % QN] = t[e % QN][e / QN];
}

// sink = the sum over the G items (block of 32 elements x 8 slices, compensated, as the other reductions).
__global__ void __launch_bounds__(256) k_reduce_cube(const float2 *__restrict__ part, int G, Sink sink) {
    __shared__ float4 red[8][32];
    const int kk = threadIdx.x % 32, sl = threadIdx.x / 32;
    const int e = blockIdx.x * 32 + kk;                    // [k3][k1][k2]
    auto add = [](float4 &s, float vr, float vi) {
        const float yr = vr - s.z, yi = vi - s.w, tr = s.x + yr, ti = s.y + yi;
        s.z = (tr - s.x) - yr;
        s.w = (ti - s.y) - yi;
        s.x = tr;
        s.y = ti;
    };
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    #pragma unroll 4
    for (int g = sl; g < G; g += 8) {
        const float2 v = __ldcs(part + (size_t)g * QN * Q2 + e);
        add(s, v.x, v.y);
    }
    red[sl][kk] = s;
    __syncthreads();
    if (sl) return;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    #pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 q = red[u][kk];
        add(t, q.x, q.y);
        add(t, -q.z, -q.w);
    }
    sink_put(sink, (size_t)(e % Q2) * QN + e / Q2,
             make_double2((double)t.x - (double)t.z, (double)t.y - (double)t.w));
}

}  // namespace

cudaError_t cube32_setup(int *G) {
    *G = 0;
    const cudaError_t e = cudaFuncSetAttribute(k_cube32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q_SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0;
    cudaGetDevice(&dev);
    return cudaDeviceGetAttribute(G, cudaDevAttrMultiProcessorCount, dev);
}

bz_status launch_cube32(const Plan &pl, const ItemArgs &a, cudaStream_t st) {
    if (pl.N != QN || a.real || !a.hg) return BZ_ERR_UNSUPPORTED;
    k_cube32<<<pl.fused_G, QT, Q_SMEM, st>>>(a);
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

bz_status cube32_table(Plan &pl) {
    for (int p0 = 0; p0 < pl.P; p0 += 32768) {
        const int n = pl.P - p0 < 32768 ? pl.P - p0 : 32768;
        k_cube_table<<<dim3(QN, n), 256>>>(pl.alpha + (size_t)p0 * QN * Q2, pl.acol + (size_t)p0 * QN * Q2);
    }
    BZ_CUDA_TRY(cudaGetLastError());
    BZ_CUDA_TRY(cudaDeviceSynchronize());
    return BZ_OK;
}

bz_status reduce_cube(Plan &pl, int nblk, cudaStream_t st, const Sink &sink) {
    k_reduce_cube<<<QN * Q2 / 32, 256, 0, st>>>(pl.part, nblk, sink);
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

}  // namespace bz
