// The fused per-term pipeline (N <= 32): launch configuration, cluster-size setup and the
// fixed-order reduction of the items' partial sums.  The kernel itself is in
// bz_fused_kernel.cuh.
#include "bz_fused_kernel.cuh"

namespace bz {

// sink(k) = sum over g of part[g][k] with a fixed shape: thread (kk, s) of a 32 x 8 block sums
// g = s, s + 8, ... for mode k = 32 blockIdx.x + kk with Kahan compensation in FP32, then the
// eight slices are added in order s = 0..7 (compensated).  FP32 pipes only.
struct Kahan2 {
    float sr = 0.f, si = 0.f, cr = 0.f, ci = 0.f;
    __device__ __forceinline__ void add(float vr, float vi) {
        float yr = vr - cr, yi = vi - ci;
        float tr = sr + yr, ti = si + yi;
        cr = (tr - sr) - yr;
        ci = (ti - si) - yi;
        sr = tr;
        si = ti;
    }
};

__global__ void __launch_bounds__(256) k_reduce_parts(const float2 *__restrict__ part, int G, int n3, Sink sink) {
    __shared__ float4 red[8][32];
    const int kk = threadIdx.x % 32, sl = threadIdx.x / 32;
    const int k = blockIdx.x * 32 + kk;
    Kahan2 s;
    if (k < n3) {
        for (int g = sl; g < G; g += 8) {
            float2 v = part[(size_t)g * n3 + k];
            s.add(v.x, v.y);
        }
    }
    red[sl][kk] = make_float4(s.sr, s.si, s.cr, s.ci);
    __syncthreads();
    if (sl == 0 && k < n3) {
        Kahan2 t;
        #pragma unroll
        for (int u = 0; u < 8; ++u) {
            float4 q = red[u][kk];
            t.add(q.x, q.y);
            t.add(-q.z, -q.w);
        }
        sink_put(sink, k, make_double2((double)t.sr - (double)t.cr, (double)t.si - (double)t.ci));
    }
}

template <int N, int C, bool SC, bool R> static cudaError_t set_smem() {
    return cudaFuncSetAttribute(k_fused<N, C, SC, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)FK<N, C, R>::SMEM);
}

// Resident clusters (C > 1) or CTAs (C = 1) of the kernel that a plan of this form runs.
// The pair form (R) exists where the lanes of a plane share a warp (32 % N == 0).
template <int N> constexpr bool pair_form() { return 32 % N == 0; }

template <int N, int C, bool R> static cudaError_t occupancy(int *G) {
    using K = FK<N, C, R>;
    const void *kern;
    if constexpr (R) kern = (const void *)k_fused<N, C, false, true>;
    else kern = (const void *)k_fused<N, C, true, false>;
    cudaError_t e = cudaSuccess;
    if (C == 1) {
        int per_sm = 0, dev = 0, sms = 0;
        if constexpr (K::TM) per_sm = K::MIN_BLOCKS;         // (the query reports one CTA for kernels that allocate tensor memory)
        else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, K::THREADS, K::SMEM);
        if (e != cudaSuccess) return e;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        *G = per_sm * sms;
    } else {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C * 64);
        cfg.blockDim = dim3(K::THREADS);
        cfg.dynamicSmemBytes = K::SMEM;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(G, kern, &cfg);
        if (e != cudaSuccess) return e;
    }
    return *G > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

template <int N, int C> static cudaError_t setup_nc(int *G, bool real) {
    cudaError_t e = set_smem<N, C, false, false>();
    if (e == cudaSuccess) e = set_smem<N, C, true, false>();
    if (e != cudaSuccess) return e;
    if constexpr (pair_form<N>()) {
        if (real) {
            e = set_smem<N, C, false, true>();
            if (e == cudaSuccess) e = set_smem<N, C, true, true>();
            return e == cudaSuccess ? occupancy<N, C, true>(G) : e;
        }
    } else {
        if (real) return cudaErrorInvalidValue;
    }
    return occupancy<N, C, false>(G);
}

// Cluster sizes compiled for each N (the plan times them and keeps the fastest).  N = 16 takes
// one CTA unless two are asked for: 7.8 us at P = 192 against 8.6 for a single collide, and for 32
// instances of P = 192, 98 us against 154.
int fused_candidates(int N, int *cs, int forced) {
    switch (N) {
        case 8: cs[0] = 1; return 1;
        case 16: cs[0] = forced == 2 ? 2 : 1; return 1;
        case 24: cs[0] = 2; cs[1] = 3; return 2;
        case 32: cs[0] = 4; cs[1] = 8; return 2;
    }
    return 0;
}

// Resident clusters for (N, C) (0 when the fused path does not apply); real: the term-pair
// kernel of BZ_DATA_REAL.
cudaError_t fused_setup(int N, int C, int *G, bool real) {
    *G = 0;
    if (N == 8 && C == 1) return setup_nc<8, 1>(G, real);
    if (N == 16 && C == 1) return setup_nc<16, 1>(G, real);
    if (N == 16 && C == 2) return setup_nc<16, 2>(G, real);
    if (N == 24 && C == 2) return setup_nc<24, 2>(G, real);
    if (N == 24 && C == 3) return setup_nc<24, 3>(G, real);
    if (N == 32 && C == 4) return setup_nc<32, 4>(G, real);
    if (N == 32 && C == 8) return setup_nc<32, 8>(G, real);
    return cudaErrorInvalidValue;
}

template <int N, int C, bool SC, bool R> static bz_status launch_nc(int G, const ItemArgs &a, cudaStream_t st) {
    using K = FK<N, C, R>;
    if (C == 1) {
        k_fused<N, C, SC, R><<<G, K::THREADS, K::SMEM, st>>>(a);
    } else {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(G * C);
        cfg.blockDim = dim3(K::THREADS);
        cfg.dynamicSmemBytes = K::SMEM;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        BZ_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_fused<N, C, SC, R>, a));
    }
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

template <int N, int C> static bz_status launch_sc(int G, const ItemArgs &a, cudaStream_t st) {
    if (a.real) {
        if constexpr (pair_form<N>()) return a.gsc ? launch_nc<N, C, true, true>(G, a, st) : launch_nc<N, C, false, true>(G, a, st);
        else return BZ_ERR_UNSUPPORTED;
    }
    return a.gsc ? launch_nc<N, C, true, false>(G, a, st) : launch_nc<N, C, false, false>(G, a, st);
}

bz_status launch_fused(const Plan &pl, const ItemArgs &a, cudaStream_t st) {
    const int N = pl.N, C = pl.fused_C;
    if (pl.precision == BZ_PREC_BF16X3) return a.real ? BZ_ERR_UNSUPPORTED : launch_mixed(pl, a, st);
    if (pl.col32) return launch_col32(pl, a, st);
    if (pl.cube32) return launch_cube32(pl, a, st);
    if (pl.pair3 && a.real) return launch_pair3(pl, a, st);
    if (N == 8 && C == 1) return launch_sc<8, 1>(pl.fused_G, a, st);
    if (N == 16 && C == 1) return launch_sc<16, 1>(pl.fused_G, a, st);
    if (N == 16 && C == 2) return launch_sc<16, 2>(pl.fused_G, a, st);
    if (N == 24 && C == 2) return launch_sc<24, 2>(pl.fused_G, a, st);
    if (N == 24 && C == 3) return launch_sc<24, 3>(pl.fused_G, a, st);
    if (N == 32 && C == 4) return launch_sc<32, 4>(pl.fused_G, a, st);
    if (N == 32 && C == 8) return launch_sc<32, 8>(pl.fused_G, a, st);
    return BZ_ERR_UNSUPPORTED;
}

// sink(k) = sum over the nblk item partials of part (fixed order, compensated).
void reduce_parts(const float2 *part, int nblk, int n, const Sink &sink, cudaStream_t st) {
    k_reduce_parts<<<(n + 31) / 32, 256, 0, st>>>(part, nblk, n, sink);
}

// Whether a k_cube32 plan runs n terms of one instance on k_fused's 8-CTA clusters: while there is a cluster for each,
// they take 8.6 us where k_cube32 takes 23.  Measured, a whole collide, k_cube32 / clusters: n = 8 48 / 31 us, 32
// 49 / 33.  (Two rounds of clusters would still win a little, 49 / 45 at n = 72, but a plan's batches are on
// k_cube32, and a batch and a collide of the same terms then differ by the rounding of two kernels.)
static bool few_terms(const Plan &pl, int n) { return pl.cube32 && n > 0 && n < pl.few_G; }

// One instance (pl.f32), terms [p0, p1): one block of terms per resident cluster, then the
// fixed-order sum of the blocks into the sink.  BZ_DATA_REAL: the input is first reduced to
// its Hermitian, Nyquist-free part, the blocks are of term pairs [p0 / 2, p1 / 2), and the sum
// is symmetrised at the end.
bz_status collide_fused(Plan &pl, int p0, int p1, cudaStream_t st, int *launches, const Sink &sink) {
    const int n3 = pl.N * pl.N * pl.N;
    ItemArgs a;
    a.fin = pl.f32; a.tw = pl.tw; a.alpha = pl.alpha; a.part = pl.part; a.hg = pl.h;
    a.count = 1; a.p0 = p0; a.p1 = p1; a.M = pl.M; a.N_rho = pl.N_rho;
    int nl = 0;
    bz_status s = BZ_OK;
    const bool few = few_terms(pl, p1 - p0), cube = pl.cube32 && !few;
    if (cube) {
        a.fin = pl.fcol; a.alpha = pl.acol; a.hg = (const float2 *)pl.hcol;
    }
    if (pl.real) {
        if ((p0 | p1) & 1) return BZ_ERR_ARG;
        if (!pl.h_fp64 && !pl.col32) {
            // h formed in FP32 in the kernel from the symmetrised copy (the h pass writes it otherwise)
            tm_begin(pl, st);
            s = sym_input(pl, pl.src, pl.src_dtype, st);
            if (s != BZ_OK) return s;
            tm_end(pl, st, TK_OTHER);
            ++nl;
        }
        a.fin = pl.fsym; a.alpha = pl.apair; a.real = 1; a.cpair = pl.cpair; a.part_s = pl.part_s;
        a.p0 = p0 / 2; a.p1 = p1 / 2;
        if (pl.col32) {
            a.fin = pl.fcol; a.alpha = pl.acol; a.hg = (const float2 *)pl.hcol;
            a.p0 = p0; a.p1 = p1;                         // one term at a time
        }
    }
    const int nt = a.p1 - a.p0, G = few ? pl.few_G : pl.fused_G;
    a.TB = nt > 0 ? (nt + G - 1) / G : 1;
    a.nblk = nt > 0 ? (nt + a.TB - 1) / a.TB : 0;
    if (pl.h_fp64 || pl.col32) {
        tm_begin(pl, st);
        s = hff_launch(pl.N, pl.h_fp64, pl.src, pl.src_dtype, nullptr, nullptr, 1, pl.scr64,
                       pl.col32 || cube ? (float2 *)pl.hcol : pl.h, st,
                       pl.col32 ? pl.fcol : (pl.real ? pl.fsym : nullptr), pl.col32 || cube,
                       cube ? pl.fcol : pl.fcopy);
        if (s != BZ_OK) return s;
        tm_end(pl, st, TK_OTHER);
        nl += hff_launches(pl.N);
    } else if (pl.pair3) {
        // this kernel reads h: formed in FP32 from the symmetrised input by one plane pass and one pencil
        // pass of the chunked pipeline
        tm_begin(pl, st);
        s = h_fp32(pl, pl.fsym, st);
        if (s != BZ_OK) return s;
        tm_end(pl, st, TK_OTHER);
        nl += 2;
    } else {
        a.hg = nullptr;                                   // h formed in FP32 in the item prologue
    }
    tm_begin(pl, st);
    s = few ? launch_sc<32, 8>(G, a, st) : launch_fused(pl, a, st);
    if (s != BZ_OK) return s;
    tm_end(pl, st, TK_FUSED);
    tm_begin(pl, st);
    if (pl.real) {
        s = pl.col32 ? reduce_col(pl, a.nblk, st, sink) : reduce_sym(pl, a.nblk, st, sink);   // sums of the blocks, symmetrised
        if (s != BZ_OK) return s;
    } else if (cube) {
        s = reduce_cube(pl, a.nblk, st, sink);
        if (s != BZ_OK) return s;
    } else {
        reduce_parts(pl.part, a.nblk, n3, sink, st);
    }
    tm_end(pl, st, TK_REDUCE);
    BZ_CUDA_TRY(cudaGetLastError());
    nl += 2;
    if (launches) *launches += nl;
    return BZ_OK;
}

}  // namespace bz
