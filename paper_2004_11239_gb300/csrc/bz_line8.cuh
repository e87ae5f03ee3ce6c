// Transforms of N = 8 R points over 8 lanes, R points each, in double-float (ffc: pairs of FP32, about 47
// significant bits), FP64 (cd) or FP32 (cf) arithmetic.
//
// x[l + 8 m] in lane l -> X[r + R q] in the lane of q = bitrev(l): an R-point transform over m in
// registers, the twiddle W_N^(l r), and an 8-point transform over the lanes (radix 2 by shuffles).
#pragma once

#include <type_traits>

#include "bz_fft.cuh"
#include "bz_internal.h"

namespace bz {

struct ff { float h, l; };
struct ffc { ff x, y; };

struct alignas(16) RootFF { float xh, xl, yh, yl; };
struct RootTable { RootFF v[192]; };
constexpr RootTable make_roots() {
    RootTable t{};
    for (int j = 0; j < 192; ++j) {
        const TwCS c = unit_root(j, 192);
        t.v[j].xh = (float)c.c;
        t.v[j].xl = (float)(c.c - (double)(float)c.c);
        t.v[j].yh = (float)c.s;
        t.v[j].yl = (float)(c.s - (double)(float)c.s);
    }
    return t;
}
static __device__ const RootTable g_roots = make_roots();

struct alignas(16) RootD { double x, y; };
struct RootTableD { RootD v[192]; };
constexpr RootTableD make_rootsd() {
    RootTableD t{};
    for (int j = 0; j < 192; ++j) {
        const TwCS c = unit_root(j, 192);
        t.v[j].x = c.c;
        t.v[j].y = c.s;
    }
    return t;
}
static __device__ const RootTableD g_rootsd = make_rootsd();

struct cd { double x, y; };
struct cf { float x, y; };

// exp(+2 pi i j / N)
template <int N, class C> __device__ __forceinline__ C root(int j) {
    if constexpr (std::is_same<C, cd>::value) {
        const double2 v = __ldg((const double2 *)g_rootsd.v + (j % N) * (192 / N));
        return {v.x, v.y};
    } else {
        const float4 v = __ldg((const float4 *)g_roots.v + (j % N) * (192 / N));
        if constexpr (std::is_same<C, cf>::value) return {v.x, v.z};
        else return {{v.x, v.y}, {v.z, v.w}};
    }
}

// The _rn intrinsics keep the compiler from contracting or reordering the error-free steps.
__device__ __forceinline__ ff fadd(ff a, ff b) {
    const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
    float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    const float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ ff fneg(ff a) { return {-a.h, -a.l}; }
// a b + sign c d, sign = +-1
template <int SIGN> __device__ __forceinline__ ff fdot(ff a, ff b, ff c, ff d) {
    const float p = __fmul_rn(a.h, b.h), q0 = __fmul_rn(c.h, d.h), q = SIGN > 0 ? q0 : -q0;
    float pe = __fmaf_rn(a.h, b.h, -p), qe = __fmaf_rn(c.h, d.h, -q0);
    pe = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, pe));
    qe = __fmaf_rn(c.h, d.l, __fmaf_rn(c.l, d.h, qe));
    const float s = __fadd_rn(p, q), t = __fsub_rn(s, p);
    float e = __fadd_rn(__fsub_rn(p, __fsub_rn(s, t)), __fsub_rn(q, t));
    e = __fadd_rn(e, SIGN > 0 ? __fadd_rn(pe, qe) : __fsub_rn(pe, qe));
    const float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ ffc add(ffc a, ffc b) { return {fadd(a.x, b.x), fadd(a.y, b.y)}; }
__device__ __forceinline__ ffc neg(ffc a) { return {fneg(a.x), fneg(a.y)}; }
__device__ __forceinline__ ffc sub(ffc a, ffc b) { return add(a, neg(b)); }
__device__ __forceinline__ ffc mul(ffc a, ffc w) { return {fdot<-1>(a.x, w.x, a.y, w.y), fdot<1>(a.x, w.y, a.y, w.x)}; }
__device__ __forceinline__ ffc times_i(ffc a) { return {fneg(a.y), a.x}; }
__device__ __forceinline__ ffc half(ffc a) { return {{0.5f * a.x.h, 0.5f * a.x.l}, {0.5f * a.y.h, 0.5f * a.y.l}}; }
__device__ __forceinline__ ffc conj(ffc a) { return {a.x, fneg(a.y)}; }
__device__ __forceinline__ ffc scale(ffc a, ff s) {
    const ff z = {0.f, 0.f};
    return {fdot<1>(a.x, s, z, z), fdot<1>(a.y, s, z, z)};
}
__device__ __forceinline__ cd add(cd a, cd b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cd neg(cd a) { return {-a.x, -a.y}; }
__device__ __forceinline__ cd sub(cd a, cd b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cd mul(cd a, cd w) { return {fma(a.x, w.x, -a.y * w.y), fma(a.x, w.y, a.y * w.x)}; }
__device__ __forceinline__ cd times_i(cd a) { return {-a.y, a.x}; }
__device__ __forceinline__ cd half(cd a) { return {0.5 * a.x, 0.5 * a.y}; }
__device__ __forceinline__ cd conj(cd a) { return {a.x, -a.y}; }
__device__ __forceinline__ cd scale(cd a, double s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ cf add(cf a, cf b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cf neg(cf a) { return {-a.x, -a.y}; }
__device__ __forceinline__ cf sub(cf a, cf b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cf mul(cf a, cf w) { return {fmaf(a.x, w.x, -a.y * w.y), fmaf(a.x, w.y, a.y * w.x)}; }
__device__ __forceinline__ cf times_i(cf a) { return {-a.y, a.x}; }
__device__ __forceinline__ cf half(cf a) { return {0.5f * a.x, 0.5f * a.y}; }
__device__ __forceinline__ cf conj(cf a) { return {a.x, -a.y}; }
__device__ __forceinline__ cf scale(cf a, float s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ float4 pack(ffc a) { return make_float4(a.x.h, a.x.l, a.y.h, a.y.l); }
__device__ __forceinline__ ffc unpack(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ float2 round2(ffc a) { return make_float2(a.x.h, a.y.h); }   // |lo| <= ulp(hi) / 2
__device__ __forceinline__ double2 pack(cd a) { return make_double2(a.x, a.y); }
__device__ __forceinline__ cd unpack(double2 v) { return {v.x, v.y}; }
__device__ __forceinline__ float2 round2(cd a) { return make_float2((float)a.x, (float)a.y); }
__device__ __forceinline__ float2 pack(cf a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ cf unpack(float2 v) { return {v.x, v.y}; }
__device__ __forceinline__ float2 round2(cf a) { return make_float2(a.x, a.y); }

// A double as hi + lo by its bits (no FP64 instruction): hi the leading 24 bits of the mantissa, lo the
// other 29.  Below the FP32 range 0, above it and for Inf / NaN the FP32 infinity or NaN.
__device__ __forceinline__ ff split(double d) {
    const unsigned hw = (unsigned)__double2hiint(d), lw = (unsigned)__double2loint(d);
    const unsigned e = (hw >> 20) & 0x7ffu, sign = hw & 0x80000000u;
    if (e <= 1023u - 127u) return {__uint_as_float(sign), 0.f};
    if (e >= 1023u + 128u)
        return {__uint_as_float(sign | 0x7f800000u | (e == 0x7ffu && ((hw & 0xfffffu) | lw) ? 0x400000u : 0u)), 0.f};
    const unsigned ef = (e - 896u) << 23;
    const float h = __uint_as_float(sign | ef | ((hw & 0xfffffu) << 3) | (lw >> 29));
    const float l = __fmul_rn((float)(lw & 0x1fffffffu) * 0x1p-52f, __uint_as_float(sign | ef));
    const float s = __fadd_rn(h, l);                      // |lo| <= ulp(hi) / 2
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
// R-point transform in registers (sign +), natural order.
template <class C, int R> __device__ __forceinline__ void dft_reg(C (&v)[R]) {
    if constexpr (R == 2) {
        const C a = v[0];
        v[0] = add(a, v[1]);
        v[1] = sub(a, v[1]);
    } else if constexpr (R == 3) {
        // -1/2 and sqrt(3)/2 from the roots' table (exactly -1/2; sqrt(3)/2 to 48 bits)
        const C t = add(v[1], v[2]), d = sub(v[1], v[2]), m = sub(v[0], half(t));
        const C r = times_i(scale(d, root<3, C>(1).y));
        v[0] = add(v[0], t);
        v[1] = add(m, r);
        v[2] = sub(m, r);
    } else if constexpr (R == 4) {
        const C s0 = add(v[0], v[2]), d0 = sub(v[0], v[2]), s1 = add(v[1], v[3]), d1 = times_i(sub(v[1], v[3]));
        v[0] = add(s0, s1);
        v[2] = sub(s0, s1);
        v[1] = add(d0, d1);
        v[3] = sub(d0, d1);
    } else if constexpr (R == 8) {
        C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft_reg<C, 4>(e);
        dft_reg<C, 4>(o);
        o[1] = mul(o[1], root<8, C>(1));
        o[2] = times_i(o[2]);
        o[3] = mul(o[3], root<8, C>(3));
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = add(e[k], o[k]);
            v[k + 4] = sub(e[k], o[k]);
        }
    }
}

__device__ __forceinline__ ffc lane_xor(ffc a, int m) {
    return {{__shfl_xor_sync(0xffffffffu, a.x.h, m), __shfl_xor_sync(0xffffffffu, a.x.l, m)},
            {__shfl_xor_sync(0xffffffffu, a.y.h, m), __shfl_xor_sync(0xffffffffu, a.y.l, m)}};
}
__device__ __forceinline__ cf lane_xor(cf a, int m) {
    return {__shfl_xor_sync(0xffffffffu, a.x, m), __shfl_xor_sync(0xffffffffu, a.y, m)};
}
__device__ __forceinline__ cd lane_xor(cd a, int m) {
    return {__shfl_xor_sync(0xffffffffu, a.x, m), __shfl_xor_sync(0xffffffffu, a.y, m)};
}
// 8-point transform over 8 lanes (sign +): lane l ends with q = bitrev(l); w8 = W8^(l mod 4) where l >= 4,
// else 1.
template <class C> __device__ __forceinline__ C dft_lanes(C v, int l, C w8) {
    v = mul(add(lane_xor(v, 4), l & 4 ? neg(v) : v), w8);
    v = add(lane_xor(v, 2), l & 2 ? neg(v) : v);
    if ((l & 3) == 3) v = times_i(v);
    return add(lane_xor(v, 1), l & 1 ? neg(v) : v);
}

// The lane's twiddles, and one line: x[l + 8 m] in v[m] -> X[r + R q] in v[r].  Every lane of the warp takes part.
template <int N, class C = ffc> struct LineFF {
    static constexpr int R = N / 8;
    C w[R], w8;
    int l, q;
    __device__ __forceinline__ LineFF(int lane8) : l(lane8) {
        q = ((l & 1) << 2) | (l & 2) | (l >> 2);
        #pragma unroll
        for (int r = 1; r < R; ++r) w[r] = root<N, C>(l * r);
        w8 = root<8, C>(l & 4 ? l & 3 : 0);
    }
    __device__ __forceinline__ void operator()(C (&v)[R]) const {
        dft_reg<C, R>(v);
        #pragma unroll
        for (int r = 0; r < R; ++r) v[r] = dft_lanes(r ? mul(v[r], w[r]) : v[r], l, w8);
    }
};

}  // namespace bz
