// Real-data collide at N = 32 with one term's whole field on one SM (BZ_DATA_REAL).
//
// For real f every product h g_p is a real field, so a term needs half of the spectrum: the
// columns k3 = 0 .. 16 of 32 x 32 (k1, k2) modes.  Columns 0 and 16 are transforms of real planes
// and share one complex column (V0 + i V16), which leaves 16 columns = 128 KB: shared memory of one
// CTA.  16 warps, warp w owns column w:
//   P1  lane = k2:  x = beta_p fhat over k1 (loaded from L2), inverse over k1
//   P2  lane = j1:  inverse over k2                      (transpose inside the warp's own column)
//   -- block barrier --
//   P3  thread = two rows (j1, j2): their 2 x 16 half-spectra as one complex line of 32, inverse
//       over k3, times the real h of each row, forward over j3, two half-spectra back in place
//   -- block barrier --
//   P4  lane = j1:  forward over j2                      (the warp's own column again)
//   P5  lane = k2:  forward over j1, times alpha_p, added to the thread's sums
// Two block barriers a term; between them a warp runs P4, P5, P1, P2 on its own, so the loads of
// one warp overlap the arithmetic of another.  The real h of the thread's two rows (64 words) and
// the sums of its 32 modes (64 words) stay in tensor memory: 512 threads x 128 words = all of it,
// and the one CTA of an SM is the only user.
//
// Weights: table [P][18][32][32] -- columns k3 = 0 .. 15, column 16, and for the modes -k whose
// weight is not the conjugate of alpha(k) (k1 or k2 = -N/2, k3 = 17 .. 31) the rows
// conj alpha(-k) of k = (16, k2, k3) and k = (k1, 16, k3), k3 = 1 .. 15; an item's sums have the
// same layout.  Off those Q(-k) = conj Q(k) (Q is eq. realQ of the Hermitian, Nyquist-free part of
// fhat, every mode kept).  k_reduce_col adds the items and writes the full grid.
//
// The cluster kernels (k_pair3, k_fused) exchange a pair's 256 KB twice through distributed shared
// memory, whose rate bounds them: 32 and 51 resident clusters took the same time per pair.
// Measured at P = 1024 (one collide's terms): 92 us, k_pair3 155 us; 16 instances of P = 384: 474 us
// against 861.  What bounds it: instruction issue and the two barriers.  A term takes about 25 k
// clocks, of which 15 k are issue slots (FP32 four fifths of them); 4 k go to the barriers and
// the shared-memory bursts behind them, the rest to the latency of L2 loads and tensor memory
// with four warps a scheduler.  Measured without gain: fhat in shared memory or loaded a phase
// ahead, half of the weights staged there, longer look-ahead (96 - 101 us; the registers spill).
#include "bz_cluster.cuh"
#include "bz_fft.cuh"
#include "bz_internal.h"
#include "bz_tmem.cuh"

namespace bz {

namespace {

constexpr int CN = 32, CW = 16, CT = 32 * CW, CLD = CN + 1, CP = CN * CLD, C2 = CN * CN;
// columns, W of the packed column, sums of columns 0 and 16, the twiddles of two terms
constexpr size_t C_SMEM = ((size_t)CW * CP + 3 * C2 + 2 * 3 * CN) * sizeof(float2);
static_assert(C_SMEM <= 227 * 1024, "one CTA per SM");
constexpr uint32_t TC_ACC = 0, TC_H = 256;                             // tensor-memory columns

__global__ void __launch_bounds__(CT, 1) k_col32(ItemArgs a) {
    constexpr int N = CN;
    extern __shared__ __align__(16) float2 csm[];
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    float2 *my = csm + w * CP;                             // column w: [j1 or k1][j2 or k2]
    float2 *wst = csm + CW * CP;                           // W(k1, k2) of the packed column, last term
    float2 *accp = wst + C2;                               // sums of columns 0 and 16, [2][k1][k2]
    float2 *stw = accp + 2 * C2;                           // twiddles, two buffers of [3][N]
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
    const float2 *rows = csm + (2 * w) * CLD + lane;       // P3: rows (2w, lane) and (2w + 1, lane)

    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const int b = it / a.nblk, blk = it % a.nblk;
        const int slot = a.slots ? a.slots[b] : b;
        const int t0 = a.p0 + blk * a.TB, t1 = min(a.p1, t0 + a.TB);
        const float2 *fin = a.fin + (size_t)slot * N3 + w * C2 + lane;       // [k3][k1][k2]
        {
            // h [j3][j1][j2] (packed floats), halved: the half-spectra of two rows come out of one
            // line as Z(k3) +- conj Z(-k3)
            const float *h = (const float *)(a.hg + (size_t)slot * N3) + 2 * w * N + lane;
            float v[16];
            #pragma unroll
            for (int g = 0; g < 4; ++g) {
                #pragma unroll
                for (int u = 0; u < 8; ++u) {
                    v[2 * u] = 0.5f * h[(8 * g + u) * C2];
                    v[2 * u + 1] = 0.5f * h[(8 * g + u) * C2 + N];
                }
                t_st16(tl + TC_H + 16 * g, v);
            }
            #pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = 0.f;
            #pragma unroll
            for (int g = 0; g < 4; ++g) t_st16(tl + TC_ACC + 16 * g, v);
            t_wait_st();
        }
        // the packed column: W of a term is shared, and every thread adds four of its modes to the
        // sums (k1 = 2w, 2w + 1 of columns 0 and 16) while the next term is in P3
        #pragma unroll
        for (int u = 0; u < 4; ++u) accp[(u & 1) * C2 + (2 * w + (u >> 1)) * N + lane] = make_float2(0.f, 0.f);
        float2 pk[4];                                      // their weights, loaded ahead
        auto load_packed = [&](int p) {
            const float2 *tab = a.alpha + (size_t)p * 18 * C2 + 2 * w * N + lane;
            #pragma unroll
            for (int u = 0; u < 4; ++u) pk[u] = __ldg(tab + (u >> 1) * CW * C2 + (u & 1) * N);
        };
        auto add_packed = [&]() {
            #pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k1 = 2 * w + u;
                const float2 A0 = pk[u], A16 = pk[2 + u];
                const float2 z = wst[k1 * N + lane], y = wst[((N - k1) % N) * N + (N - lane) % N];
                const float2 z0 = make_float2(z.x + y.x, z.y - y.y), z16 = make_float2(z.y + y.y, y.x - z.x);
                float2 *q0 = accp + k1 * N + lane, *q1 = q0 + C2;
                float2 q = *q0;
                q.x = fmaf(z0.x, A0.x, fmaf(-z0.y, A0.y, q.x));
                q.y = fmaf(z0.x, A0.y, fmaf(z0.y, A0.x, q.y));
                *q0 = q;
                q = *q1;
                q.x = fmaf(z16.x, A16.x, fmaf(-z16.y, A16.y, q.x));
                q.y = fmaf(z16.x, A16.y, fmaf(z16.y, A16.x, q.y));
                *q1 = q;
            }
        };
        float2 x1 = make_float2(0.f, 0.f), x2 = make_float2(0.f, 0.f);
        auto fetch_tw = [&](int p, int buf) {
            if (tid < 3 * N / 2)
                cp_async16(stw + buf * 3 * N + 2 * tid, a.tw + (size_t)p * 3 * N + 2 * tid);
            cp_async_commit();
        };
        fetch_tw(t0, 0);
        cp_async_wait_all();
        __syncthreads();
        for (int p = t0; p < t1; ++p) {
            const float2 *tab = a.alpha + (size_t)p * 18 * C2;
            if (tid == 0)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(tab),
                             "r"((uint32_t)(18 * C2 * sizeof(float2))) : "memory");
            float2 x[N];
            // P1
            {
                #pragma unroll
                for (int i = 0; i < N; ++i) x[i] = i == N / 2 ? make_float2(0.f, 0.f) : fin[i * N];
                const float2 *tws = stw + ((p - t0) & 1) * 3 * N;
                float2 t23 = cmul(tws[N + lane], tws[2 * N + w]);
                if (a.gsc) t23 = cscale(t23, a.gsc[(size_t)slot * a.N_rho + p / a.M]);
                #pragma unroll
                for (int i = 0; i < N; ++i)
                    if (i != N / 2) x[i] = cmul(x[i], cmul(t23, tws[i]));
                fft_inplace<N, +1>(x);                     // k1 -> j1
                #pragma unroll
                for (int i = 0; i < N; ++i) my[i * CLD + lane] = x[i];
            }
            __syncwarp();
            // P2
            #pragma unroll
            for (int i = 0; i < N; ++i) x[i] = my[lane * CLD + i];
            fft_inplace<N, +1>(x);                         // k2 -> j2
            #pragma unroll
            for (int i = 0; i < N; ++i) my[lane * CLD + i] = x[i];
            if (p > t0) load_packed(p - 1);
            __syncthreads();
            if (p > t0) add_packed();
            if (p + 1 < t1) fetch_tw(p + 1, (p + 1 - t0) & 1);
            // P3: A = row (2w, lane), B = row (2w + 1, lane); x(k3) = A + i B with A(-k3) = conj A(k3)
            {
                #pragma unroll
                for (int k = 0; k < CW; ++k) {
                    const float2 A = rows[k * CP], B = rows[k * CP + CLD];
                    if (k == 0) {
                        x[0] = make_float2(A.x, B.x);
                        x[N / 2] = make_float2(0.f, 0.f);
                    } else {
                        x[k] = make_float2(A.x - B.y, A.y + B.x);
                        x[N - k] = make_float2(A.x + B.y, B.x - A.y);
                    }
                }
                fft_inplace<N, +1>(x);                     // k3 -> j3: (row A, row B)
                #pragma unroll
                for (int g = 0; g < 4; ++g) {
                    float h[16];
                    t_ld16(tl + TC_H + 16 * g, h);
                    t_wait_ld();
                    #pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        x[8 * g + u].x *= h[2 * u];
                        x[8 * g + u].y *= h[2 * u + 1];
                    }
                }
                fft_inplace<N, -1>(x);                     // j3 -> k3
                float2 *ro = const_cast<float2 *>(rows);
                ro[0] = make_float2(x[0].x, x[N / 2].x);   // columns 0 and 16 (both real) as one
                ro[CLD] = make_float2(x[0].y, x[N / 2].y);
                #pragma unroll
                for (int k = 1; k < CW; ++k) {
                    const float2 z = x[k], y = x[N - k];
                    ro[k * CP] = make_float2(z.x + y.x, z.y - y.y);
                    ro[k * CP + CLD] = make_float2(z.y + y.y, y.x - z.x);
                }
            }
            cp_async_wait_all();                           // the next twiddles
            __syncthreads();
            // P4; the warps w / 4 = 0 .. 3 start one after another, each once the one before has its line,
            // or the four warps of a scheduler would wait for their loads and weights all at once
            if (w >= 4) asm volatile("bar.sync %0, 256;\n" ::"r"(w >> 2) : "memory");
            #pragma unroll
            for (int i = 0; i < N; ++i) x[i] = my[lane * CLD + i];
            if (w < 12) asm volatile("bar.arrive %0, 256;\n" ::"r"((w >> 2) + 1) : "memory");
            fft_inplace<N, -1>(x);                         // j2 -> k2
            #pragma unroll
            for (int i = 0; i < N; ++i) my[lane * CLD + i] = x[i];
            __syncwarp();
            // P5: the weights are loaded one chunk of four ahead, the first during the transform
            #pragma unroll
            for (int i = 0; i < N; ++i) x[i] = my[i * CLD + lane];
            if (w == 0) {
                fft_inplace<N, -1>(x);                     // j1 -> k1
                #pragma unroll
                for (int i = 0; i < N; ++i) wst[i * N + lane] = x[i];
                continue;
            }
            const float2 *tp = tab + w * C2 + lane;
            float2 an[4];
            #pragma unroll
            for (int u = 0; u < 4; ++u) an[u] = __ldg(tp + u * N);
            fft_inplace<N, -1>(x);                         // j1 -> k1
            // the second weights of k = (16, lane, w) and k = (lane, 16, w)
            const float2 e1 = __ldg(tab + 17 * C2 + w * N + lane), e2 = __ldg(tab + 17 * C2 + (CW + w) * N + lane);
            __syncwarp();                                  // every lane has read its column
            if (lane == N / 2) {
                #pragma unroll
                for (int i = 0; i < N; ++i) my[i] = x[i];
            }
            __syncwarp();
            const float2 xu = my[lane], xv = x[N / 2];
            #pragma unroll
            for (int g = 0; g < 8; ++g) {
                float2 al[4];
                #pragma unroll
                for (int u = 0; u < 4; ++u) al[u] = an[u];
                if (g < 7) {
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) an[u] = __ldg(tp + (4 * (g + 1) + u) * N);
                }
                float s[8];
                t_ld8(tl + TC_ACC + 8 * g, s);
                t_wait_ld();
                #pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 z = x[4 * g + u];
                    s[2 * u] = fmaf(z.x, al[u].x, fmaf(-z.y, al[u].y, s[2 * u]));
                    s[2 * u + 1] = fmaf(z.x, al[u].y, fmaf(z.y, al[u].x, s[2 * u + 1]));
                }
                t_st8(tl + TC_ACC + 8 * g, s);
            }
            x1.x = fmaf(xv.x, e1.x, fmaf(-xv.y, e1.y, x1.x));
            x1.y = fmaf(xv.x, e1.y, fmaf(xv.y, e1.x, x1.y));
            x2.x = fmaf(xu.x, e2.x, fmaf(-xu.y, e2.y, x2.x));
            x2.y = fmaf(xu.x, e2.y, fmaf(xu.y, e2.x, x2.y));
            __syncwarp();                                  // row 0 of the column is free again
            t_wait_st();
        }
        load_packed(t1 - 1);
        __syncthreads();                                   // W of the last term
        add_packed();
        float2 *out = a.part + ((size_t)slot * a.nblk + blk) * 18 * C2;
        if (w != 0) {
            #pragma unroll
            for (int g = 0; g < 4; ++g) {
                float s[16];
                t_ld16(tl + TC_ACC + 16 * g, s);
                t_wait_ld();
                #pragma unroll
                for (int u = 0; u < 8; ++u) out[w * C2 + (8 * g + u) * N + lane] = make_float2(s[2 * u], s[2 * u + 1]);
            }
        }
        #pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = (2 * w + (u >> 1)) * N + lane;
            out[(u & 1) * CW * C2 + e] = accp[(u & 1) * C2 + e];
        }
        out[17 * C2 + w * N + lane] = x1;
        out[17 * C2 + (CW + w) * N + lane] = x2;
    }
    tfence_before();
    __syncthreads();
    if (w == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(s_tmem) : "memory");
}

// The table of k_col32 from alpha [P][k1][k2][k3]: one block per (term, k1), transposed through
// shared memory; the rows of conj alpha(-k) by the block of k1 = 16.
__global__ void __launch_bounds__(256) k_col_table(const float2 *__restrict__ alpha, float2 *__restrict__ tab) {
    __shared__ float2 t[CN][CLD];
    const int k1 = blockIdx.x, tid = threadIdx.x;
    const float2 *al = alpha + (size_t)blockIdx.y * CN * C2;
    float2 *o = tab + (size_t)blockIdx.y * 18 * C2;
    for (int e = tid; e < C2; e += 256) t[e / CN][e % CN] = al[k1 * C2 + e];     // [k2][k3]
    __syncthreads();
    for (int e = tid; e < 17 * CN; e += 256) o[(e / CN) * C2 + k1 * CN + e % CN] = t[e % CN][e / CN];
    if (k1 != CN / 2) return;
    for (int e = tid; e < 2 * CW * CN; e += 256) {
        const int k3 = (e / CN) % CW, u = e % CN, m = (CN - u) % CN;
        float2 v = make_float2(0.f, 0.f);
        if (k3 > 0) {
            // k = (16, u, k3) or (u, 16, k3): alpha at -k
            v = e < CW * CN ? t[m][CN - k3] : al[(size_t)m * C2 + (CN / 2) * CN + CN - k3];
            v.y = -v.y;
        }
        o[17 * C2 + e] = v;
    }
}

// Kahan-compensated FP32 sum (as the other reductions).
struct KahanC {
    float sr = 0.f, si = 0.f, cr = 0.f, ci = 0.f;
    __device__ __forceinline__ void add(float vr, float vi) {
        const float yr = vr - cr, yi = vi - ci;
        const float tr = sr + yr, ti = si + yi;
        cr = (tr - sr) - yr;
        ci = (ti - si) - yi;
        sr = tr;
        si = ti;
    }
};

// Where element e of an item's sums ([18][32][32]) goes: mode i (natural order), or -1; and the
// mode j that takes its conjugate, or -1.
__device__ __forceinline__ void col_modes(int e, int &i, int &j) {
    const int c = e / C2, u = (e / CN) % CN, v = e % CN;
    i = j = -1;
    if (c < 17) {                                          // (k1, k2, k3) = (u, v, c)
        i = (u * CN + v) * CN + c;
        if (c > 0 && c < CW && u != CW && v != CW) j = (((CN - u) % CN) * CN + (CN - v) % CN) * CN + CN - c;
    } else {
        const int k3 = u % CW, m = (CN - v) % CN;
        if (k3 == 0) return;
        if (u < CW) j = (CW * CN + m) * CN + CN - k3;      // k = (16, v, k3)
        else if (v != CW) j = (m * CN + CW) * CN + CN - k3;   // k = (v, 16, k3); (16, 16, k3) is above
    }
}

// sink = the sum over the G items on the full grid: block of 32 elements x 8 slices, slice s adds
// items s, s + 8, ..., then the slices in order (compensated).
__global__ void __launch_bounds__(256) k_reduce_col(const float2 *__restrict__ part, int G, Sink sink) {
    __shared__ float4 red[8][32];
    const int kk = threadIdx.x % 32, sl = threadIdx.x / 32;
    const int e = blockIdx.x * 32 + kk;
    KahanC s;
    #pragma unroll 4
    for (int g = sl; g < G; g += 8) {
        const float2 v = __ldcs(part + (size_t)g * 18 * C2 + e);
        s.add(v.x, v.y);
    }
    red[sl][kk] = make_float4(s.sr, s.si, s.cr, s.ci);
    __syncthreads();
    if (sl) return;
    KahanC t;
    #pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 q = red[u][kk];
        t.add(q.x, q.y);
        t.add(-q.z, -q.w);
    }
    const double2 v = make_double2((double)t.sr - (double)t.cr, (double)t.si - (double)t.ci);
    int i, j;
    col_modes(e, i, j);
    if (i >= 0) sink_put(sink, i, v);
    if (j >= 0) sink_put(sink, j, make_double2(v.x, -v.y));
}

}  // namespace

cudaError_t col32_setup(int *G) {
    *G = 0;
    cudaError_t e = cudaFuncSetAttribute(k_col32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C_SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0;
    cudaGetDevice(&dev);
    return cudaDeviceGetAttribute(G, cudaDevAttrMultiProcessorCount, dev);
}

bz_status launch_col32(const Plan &pl, const ItemArgs &a, cudaStream_t st) {
    if (pl.N != CN || !a.real || !a.hg) return BZ_ERR_UNSUPPORTED;
    k_col32<<<pl.fused_G, CT, C_SMEM, st>>>(a);
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

bz_status col32_table(Plan &pl) {
    for (int p0 = 0; p0 < pl.P; p0 += 32768) {
        const int n = pl.P - p0 < 32768 ? pl.P - p0 : 32768;
        k_col_table<<<dim3(CN, n), 256>>>(pl.alpha + (size_t)p0 * CN * C2, pl.acol + (size_t)p0 * 18 * C2);
    }
    BZ_CUDA_TRY(cudaGetLastError());
    BZ_CUDA_TRY(cudaDeviceSynchronize());
    return BZ_OK;
}

bz_status reduce_col(Plan &pl, int nblk, cudaStream_t st, const Sink &sink) {
    k_reduce_col<<<18 * C2 / 32, 256, 0, st>>>(pl.part, nblk, sink);
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

}  // namespace bz
