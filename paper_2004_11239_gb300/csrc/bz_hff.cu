// h = IFFT(fhat) stored FP32: the shared inverse transform of the fused pipelines (N = 8, 16, 24, 32) and of
// the 2D operator (N = 8, 16, 32, 64), in double-float arithmetic; in FP64 for BZ_H_FP64, in FP32 for the
// BZ_H_FP32 of k_col32 (ffc, cd, cf of bz_line8.cuh).
//
// FP32 transforms leave a noise floor of about eps max|h| over the whole grid, and the product
// h g_p turns that floor into errors where g_p is large and h is small; forming h with more bits
// removes that half of the rounding error (the per-term g_p stay FP32).  A number here is an
// unevaluated sum hi + lo of two floats (Dekker 1971; Knuth's TwoSum, FMA-based TwoProduct), about
// 47 significant bits on the FP32 pipes.  This part runs an FP64 instruction of a warp in 68
// clocks of its scheduler: an FP64 addition costs what 64 FP32 operations do, a double-float one 11.
// The stored h has the error of its rounding to FP32 either way (relative 2-norm 2.0e-8 .. 3.8e-8 at
// N = 8 .. 64, equal to the rounded FP64 transform's in every digit printed).
// Bound by latency for one instance, by FP32 issue in a batch.  Measured, all launches of one h, against
// the FP64 kernels before: N = 16 4.5 us (12.0), N = 24 6.3 us (39), N = 32 real 9 - 10 us (14.4); 251
// instances of N = 16 27 us (202), 16 of N = 32 real 22 us (138).
//
// A line of N = 8 R points takes 8 lanes with R points each (x[l + 8 m] in lane l): an R-point
// transform over m in registers, the twiddle W_N^(l r), and an 8-point transform over the lanes
// (radix 2 by shuffles, bit-reversed lanes), which leaves X[r + R q] in the lane of q = bitrev(l).
//   N = 24, 32: one CTA per plane k1 (axes 3 and 2 through shared memory), then lines along axis 1;
//   N = 8, 16:  a cluster of 8 CTAs per instance, R planes each; axis 1 gathers from the cluster;
//   2D:         a cluster of 8 CTAs, R rows each; axis 1 gathers from the cluster.
#include <cooperative_groups.h>

#include "bz_cluster.cuh"
#include "bz_internal.h"
#include "bz_line8.cuh"

namespace bz {

namespace {

__device__ __forceinline__ void from(double2 v, ffc &c) { c = {split(v.x), split(v.y)}; }
__device__ __forceinline__ void from(double2 v, cd &c) { c = {v.x, v.y}; }
__device__ __forceinline__ void from(double2 v, cf &c) { c = {(float)v.x, (float)v.y}; }
__device__ __forceinline__ void from(float2 v, ffc &c) { c = {{v.x, 0.f}, {v.y, 0.f}}; }
__device__ __forceinline__ void from(float2 v, cd &c) { c = {v.x, v.y}; }
__device__ __forceinline__ void from(float2 v, cf &c) { c = {v.x, v.y}; }
template <class C> using Packed = decltype(pack(C()));
__device__ __forceinline__ float4 shfl(float4 t, int s) {
    return make_float4(__shfl_sync(0xffffffffu, t.x, s), __shfl_sync(0xffffffffu, t.y, s),
                       __shfl_sync(0xffffffffu, t.z, s), __shfl_sync(0xffffffffu, t.w, s));
}
__device__ __forceinline__ double2 shfl(double2 t, int s) {
    return make_double2(__shfl_sync(0xffffffffu, t.x, s), __shfl_sync(0xffffffffu, t.y, s));
}
__device__ __forceinline__ float2 shfl(float2 t, int s) {
    return make_float2(__shfl_sync(0xffffffffu, t.x, s), __shfl_sync(0xffffffffu, t.y, s));
}
// 16 bytes of a cluster's shared memory
__device__ __forceinline__ float4 ld_cluster(const float4 *at, uint32_t rank) {
    const uint32_t ad = dsmem_addr(at, rank);
    float4 t;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(ad) : "memory");
    return t;
}
__device__ __forceinline__ double2 ld_cluster(const double2 *at, uint32_t rank) {
    const uint32_t ad = dsmem_addr(at, rank);
    double2 t;
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];\n" : "=d"(t.x), "=d"(t.y) : "r"(ad) : "memory");
    return t;
}

// fcopy: the entry rounded to FP32 is stored there too
template <class C> __device__ __forceinline__ C load_h(const void *f, int dtype, size_t i, float2 *fcopy = nullptr) {
    C c;
    if (dtype == BZ_C128) {
        const double2 v = ((const double2 *)f)[i];
        if (fcopy) fcopy[i] = make_float2((float)v.x, (float)v.y);
        from(v, c);
    } else {
        const float2 v = ((const float2 *)f)[i];
        if (fcopy) fcopy[i] = v;
        from(v, c);
    }
    return c;
}

struct HArgs {
    const void *f;             // [slots][N^3] (c64 / c128)
    int dtype;
    const int *slots, *count_dev;
    void *scr;                 // [slots][N^3] of 16 bytes between the two launches (N = 24, 32)
    float2 *h;                 // [slots][N^3]
    float2 *fout;              // real data: the Hermitian, Nyquist-free part in FP32, or null
    float2 *fcopy;             // complex data: f in FP32, or null
    int col;                   // fout [k3 < 16][k1][k2] and h packed floats [j3][j1][j2] (k_col32), or fcopy [k3][k1][k2]
                               // and h [j3][j1][j2] (k_cube32)
};

// fhat(k) of the instance, or (fout) its Hermitian part, zero where an index is N / 2, which is also
// stored.
template <int N, class C> __device__ __forceinline__ C input(const HArgs &a, size_t vol, int k1, int k2, int k3) {
    const size_t i = vol + ((size_t)k1 * N + k2) * N + k3;
    if (!a.fout) {
        if (!a.col) return load_h<C>(a.f, a.dtype, i, a.fcopy);
        a.fcopy[vol + ((size_t)k3 * N + k1) * N + k2] =
            a.dtype == BZ_C128 ? make_float2((float)((const double2 *)a.f)[i].x, (float)((const double2 *)a.f)[i].y)
                               : ((const float2 *)a.f)[i];
        return load_h<C>(a.f, a.dtype, i);
    }
    constexpr int H = N / 2;
    C v;
    from(make_float2(0.f, 0.f), v);
    if (k1 != H && k2 != H && k3 != H) {
        const size_t m = vol + ((size_t)((N - k1) % N) * N + (N - k2) % N) * N + (N - k3) % N;
        if (std::is_same<C, cf>::value && a.dtype == BZ_C128) {   // rounded once
            const double2 p = ((const double2 *)a.f)[i], q = ((const double2 *)a.f)[m];
            from(make_double2(0.5 * (p.x + q.x), 0.5 * (p.y - q.y)), v);
        } else {
            v = half(add(load_h<C>(a.f, a.dtype, i), conj(load_h<C>(a.f, a.dtype, m))));
        }
    }
    if (!a.col) a.fout[i] = round2(v);
    else if (k3 < H) a.fout[vol + ((size_t)k3 * N + k1) * N + k2] = round2(v);
    return v;
}

// Axes 3 and 2 of the R planes k1 = k10 .. into s[R][N][N + 1] ([k1][j2][j3]); 8 N threads a plane.
template <int N, class C>
__device__ __forceinline__ void planes_h(const HArgs &a, const LineFF<N, C> &F, size_t vol, int k10, Packed<C> *s) {
    constexpr int R = N / 8, LD = N + 1;
    const int pl = threadIdx.x / (8 * N), line = threadIdx.x / 8 % N;
    Packed<C> *sp = s + pl * N * LD;
    C v[R];
    #pragma unroll
    for (int m = 0; m < R; ++m) v[m] = input<N, C>(a, vol, k10 + pl, line, F.l + 8 * m);
    F(v);                                                 // k3 -> j3 of row k2 = line
    #pragma unroll
    for (int r = 0; r < R; ++r) sp[line * LD + r + R * F.q] = pack(v[r]);
    __syncthreads();
    #pragma unroll
    for (int m = 0; m < R; ++m) v[m] = unpack(sp[(F.l + 8 * m) * LD + line]);
    F(v);                                                 // k2 -> j2 of column j3 = line
    __syncthreads();
    #pragma unroll
    for (int r = 0; r < R; ++r) sp[(r + R * F.q) * LD + line] = pack(v[r]);
    __syncthreads();
}

// N = 24, 32: the plane k1 = blockIdx.x of instance blockIdx.y to scr ([k1][j2][j3]; col: [k1][j3][j2]).
template <int N, class C> __global__ void __launch_bounds__(8 * N) k_hff_plane(HArgs a) {
    __shared__ Packed<C> s[N * (N + 1)];
    if (a.count_dev && (int)blockIdx.y >= *a.count_dev) return;
    const size_t vol = (size_t)(a.slots ? a.slots[blockIdx.y] : blockIdx.y) * N * N * N;
    const int k1 = blockIdx.x;
    planes_h<N, C>(a, LineFF<N, C>(threadIdx.x & 7), vol, k1, s);
    Packed<C> *o = (Packed<C> *)a.scr + vol + (size_t)k1 * N * N;
    for (int e = threadIdx.x; e < N * N; e += 8 * N)
        o[e] = a.col ? s[(e % N) * (N + 1) + e / N] : s[(e / N) * (N + 1) + e % N];
}
// The same plane by a cluster of 4 CTAs (N = 32, FP64): 8 rows, then 8 columns a CTA.  FP64 issue bounds this form, and
// 32 planes would leave it to 32 SMs: a complex collide of 16 terms took 51 us so, 42 on 128.
template <class C> __global__ void __launch_bounds__(64) k_hff_plane4(HArgs a) {
    constexpr int N = 32, R = N / 8, LD = N + 1;
    __shared__ Packed<C> s[8 * LD];                       // [k2 - 8 c][j3]
    if (a.count_dev && (int)blockIdx.y >= *a.count_dev) return;          // uniform over the cluster
    const size_t vol = (size_t)(a.slots ? a.slots[blockIdx.y] : blockIdx.y) * N * N * N;
    const int c = (int)cooperative_groups::this_cluster().block_rank(), k1 = blockIdx.x / 4, line = threadIdx.x / 8;
    const LineFF<N, C> F(threadIdx.x & 7);
    C v[R];
    #pragma unroll
    for (int m = 0; m < R; ++m) v[m] = input<N, C>(a, vol, k1, 8 * c + line, F.l + 8 * m);
    F(v);                                                 // k3 -> j3 of row k2 = 8 c + line
    #pragma unroll
    for (int r = 0; r < R; ++r) s[line * LD + r + R * F.q] = pack(v[r]);
    cooperative_groups::this_cluster().sync();
    const int j3 = 8 * c + line;
    #pragma unroll
    for (int m = 0; m < R; ++m) v[m] = unpack(ld_cluster(&s[F.l * LD + j3], (uint32_t)m));   // k2 = l + 8 m
    F(v);                                                 // k2 -> j2 of column j3
    Packed<C> *o = (Packed<C> *)a.scr + vol + (size_t)k1 * N * N;
    #pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j2 = r + R * F.q;
        o[a.col ? j3 * N + j2 : j2 * N + j3] = pack(v[r]);
    }
    cooperative_groups::this_cluster().sync();               // no CTA leaves while its rows are read
}
// The lines along axis 1: (u, v) = (j2, j3), or (j3, j2) for col; PARTS CTAs to a u.
template <int N, class C, int PARTS> __global__ void __launch_bounds__(8 * N / PARTS) k_hff_line(HArgs a) {
    constexpr int R = N / 8;
    if (a.count_dev && (int)blockIdx.y >= *a.count_dev) return;
    const size_t vol = (size_t)(a.slots ? a.slots[blockIdx.y] : blockIdx.y) * N * N * N;
    // four adjacent lines of a warp, eight lanes each
    const int w = (threadIdx.x >> 5) + N / 4 / PARTS * (blockIdx.x % PARTS), u = blockIdx.x / PARTS;
    const int v0 = 4 * w + (threadIdx.x & 3);
    // lanes of a line are 4 apart so that its four neighbours' elements are adjacent in memory; the
    // shuffles want them in one group of 8: transposed on the way in and out by a shuffle
    const int lane = threadIdx.x & 31, l8 = lane >> 2, src = (lane & 7) * 4 + (lane >> 3), back = (lane & 3) * 8 + l8;
    const LineFF<N, C> F(lane & 7);
    const Packed<C> *in = (const Packed<C> *)a.scr + vol + (size_t)u * N + v0;
    C v[R];
    #pragma unroll
    for (int m = 0; m < R; ++m) v[m] = unpack(shfl(in[(size_t)(l8 + 8 * m) * N * N], src));
    F(v);
    const int q = ((l8 & 1) << 2) | (l8 & 2) | (l8 >> 2);  // of the lane that wrote this thread's value
    #pragma unroll
    for (int r = 0; r < R; ++r) {
        const float2 t = shfl(round2(v[r]), back);
        const int j1 = r + R * q;
        if (a.col && a.fout) ((float *)(a.h + vol))[((size_t)u * N + j1) * N + v0] = t.x;
        else if (a.col) a.h[vol + ((size_t)u * N + j1) * N + v0] = t;
        else a.h[vol + ((size_t)j1 * N + u) * N + v0] = t;
    }
}

// N = 8, 16: one cluster of 8 CTAs per instance.
template <int N, class C> __global__ void __launch_bounds__(N * N) k_hff_cube(HArgs a) {
    constexpr int R = N / 8, LD = N + 1;
    __shared__ Packed<C> s[R * N * LD];
    if (a.count_dev && (int)blockIdx.y >= *a.count_dev) return;          // uniform over the cluster
    const size_t vol = (size_t)(a.slots ? a.slots[blockIdx.y] : blockIdx.y) * N * N * N;
    const int c = (int)cooperative_groups::this_cluster().block_rank();
    const LineFF<N, C> F(threadIdx.x & 7);
    planes_h<N, C>(a, F, vol, R * c, s);
    cooperative_groups::this_cluster().sync();
    // lines (j2, j3), j2 = R c .. R c + R - 1
    const int j2 = R * c + threadIdx.x / (8 * N), j3 = threadIdx.x / 8 % N;
    C v[R];
    #pragma unroll
    for (int m = 0; m < R; ++m) {
        const int k1 = F.l + 8 * m;
        v[m] = unpack(ld_cluster(&s[(k1 % R) * N * LD + j2 * LD + j3], (uint32_t)(k1 / R)));
    }
    F(v);
    #pragma unroll
    for (int r = 0; r < R; ++r) a.h[vol + ((size_t)(r + R * F.q) * N + j2) * N + j3] = round2(v[r]);
    cooperative_groups::this_cluster().sync();               // no CTA leaves while its planes are read
}

// 2D: one cluster of 8 CTAs, rows k1 = R c ..
template <int N, class C> __global__ void __launch_bounds__(N < 32 ? 32 : N) k_hff_2d(const void *f, int dtype, float2 *h, float2 *fcopy) {
    constexpr int R = N / 8, LD = N + 1;
    __shared__ Packed<C> s[R * LD];
    const int c = (int)cooperative_groups::this_cluster().block_rank();
    const LineFF<N, C> F(threadIdx.x & 7);
    const int i = threadIdx.x / 8 < R ? threadIdx.x / 8 : R - 1;         // spare lanes repeat the last line
    C v[R];
    #pragma unroll
    for (int m = 0; m < R; ++m) v[m] = load_h<C>(f, dtype, (size_t)(R * c + i) * N + F.l + 8 * m, fcopy);
    F(v);                                                    // k2 -> j2
    #pragma unroll
    for (int r = 0; r < R; ++r) s[i * LD + r + R * F.q] = pack(v[r]);
    cooperative_groups::this_cluster().sync();
    #pragma unroll
    for (int m = 0; m < R; ++m) {
        const int k1 = F.l + 8 * m;
        v[m] = unpack(ld_cluster(&s[(k1 % R) * LD + R * c + i], (uint32_t)(k1 / R)));
    }
    F(v);                                                    // k1 -> j1 of column j2 = R c + i
    #pragma unroll
    for (int r = 0; r < R; ++r) h[(size_t)(R * c + i) * N + r + R * F.q] = round2(v[r]);   // [j2][j1]
    cooperative_groups::this_cluster().sync();
}

template <int CS = 8, class... P, class... A>
cudaError_t launch_clusters(void (*k)(P...), dim3 grid, int threads, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

template <class C> cudaError_t launch_n(int N, int count, const HArgs &a, cudaStream_t st) {
    switch (N) {
        case 8: return launch_clusters(k_hff_cube<8, C>, dim3(8, count), 64, st, a);
        case 16: return launch_clusters(k_hff_cube<16, C>, dim3(8, count), 256, st, a);
        case 24:
            k_hff_plane<24, C><<<dim3(24, count), 192, 0, st>>>(a);
            k_hff_line<24, C, 1><<<dim3(24, count), 192, 0, st>>>(a);
            return cudaGetLastError();
        case 32:
            if constexpr (std::is_same<C, cd>::value) {
                const cudaError_t e = launch_clusters<4>(k_hff_plane4<C>, dim3(4 * 32, count), 64, st, a);
                if (e != cudaSuccess) return e;
                k_hff_line<32, C, 4><<<dim3(4 * 32, count), 64, 0, st>>>(a);
            } else {
                k_hff_plane<32, C><<<dim3(32, count), 256, 0, st>>>(a);
                k_hff_line<32, C, 1><<<dim3(32, count), 256, 0, st>>>(a);
            }
            return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
}

template <class C> cudaError_t launch_2d(int N, const void *f, int dtype, float2 *h, float2 *fcopy, cudaStream_t st) {
    switch (N) {
        case 8: return launch_clusters(k_hff_2d<8, C>, dim3(8), 32, st, f, dtype, h, fcopy);
        case 16: return launch_clusters(k_hff_2d<16, C>, dim3(8), 32, st, f, dtype, h, fcopy);
        case 32: return launch_clusters(k_hff_2d<32, C>, dim3(8), 32, st, f, dtype, h, fcopy);
        case 64: return launch_clusters(k_hff_2d<64, C>, dim3(8), 64, st, f, dtype, h, fcopy);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

bz_status hff_launch(int N, int bits, const void *f, int dtype, const int *slots, const int *count_dev, int count,
                     double2 *scr, float2 *h, cudaStream_t st, float2 *fsym, bool col, float2 *fcopy) {
    if (count <= 0) return BZ_OK;
    if ((N != 8 && N != 16 && N != 24 && N != 32) || (col && (N != 32 || !(fsym || fcopy))) || (fsym && N == 24) ||
        (bits == HFF_FP32 && N != 32))
        return BZ_ERR_UNSUPPORTED;
    const HArgs a = {f, dtype, slots, count_dev, scr, h, fsym, fcopy, col};
    if (bits == HFF_FP64) BZ_CUDA_TRY(launch_n<cd>(N, count, a, st));
    else if (bits == HFF_PAIRS) BZ_CUDA_TRY(launch_n<ffc>(N, count, a, st));
    else {
        k_hff_plane<32, cf><<<dim3(32, count), 256, 0, st>>>(a);
        k_hff_line<32, cf, 1><<<dim3(32, count), 256, 0, st>>>(a);
    }
    BZ_CUDA_TRY(cudaGetLastError());
    return BZ_OK;
}

bz_status hff_launch_2d(int N, int bits, const void *f, int dtype, float2 *h, float2 *fcopy, cudaStream_t st) {
    if (N != 8 && N != 16 && N != 32 && N != 64) return BZ_ERR_UNSUPPORTED;
    BZ_CUDA_TRY(bits == HFF_FP64 ? launch_2d<cd>(N, f, dtype, h, fcopy, st) : launch_2d<ffc>(N, f, dtype, h, fcopy, st));
    return BZ_OK;
}

}  // namespace bz
