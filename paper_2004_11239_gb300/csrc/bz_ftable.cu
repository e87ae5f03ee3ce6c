// Weight table F(k, r_i, qhat_j) on the GPU (Sec. 2.1 eq. FF, Sec. 4.1 split, 3D).
//
// With a = pi r / (2L), kappa = k.qhat, kperp = |k - kappa qhat|, x = a kappa, y = a kperp
// and g(t) = sin(t) b(cos t), the phi integral of eq. FF3D1 is exact (2 pi J0), so
//   F = 2 pi [ i x A1 - x^2 A2 / 2 - y^2 A3 / 4 ]                          (part I, [0, eps])
//     + 2 pi sum_n W_n [ (exp(i x c_n) - 1) J0(y s_n) + (J0(y s_n) - 1) ]   (part II, [eps, pi])
// with c_n = 1 - cos t_n, s_n = sin t_n, W_n = w_n g(t_n) from the host rule of the
// radial node.  The table stores alpha_p(k) = c_p F / N^3 in FP32 (the N^-3 of the
// forward transform folded in).
//
// Two evaluations of part II:
//   * single entries (bz_ftable_entries) sum the rule as written above, with CUDA's
//     double-precision j0; J0 - 1 uses its power series for small arguments.
//   * the plan's table takes the same sum through the addition theorem (Funk-Hecke): with
//     z = a |k|, chi the angle between k and qhat and exp(-i z khat.sigma) =
//     sum_l (2l + 1) (-i)^l j_l(z) P_l(khat.sigma),
//       part II = exp(i x) sum_{l >= 1} (2l + 1) (-i)^l j_l(z) mu_l P_l(cos chi),
//       mu_l = 2 pi sum_n W_n (P_l(cos t_n) - 1).
//     The rule enters through the mu_l only (one short sum per l on the host), j_l(z) depends on
//     (r_i, |k|^2) only (k_legendre_coef, one row per radial node and |k|^2), and an entry is a
//     Legendre series of about z + 25 terms of three operations (in double-float arithmetic up to 160
//     terms, in FP64 beyond), against a few hundred rule nodes of some hundred operations each.  The
//     mu_l come from the finest rule of the plan's nodes.  Measured over N = 8 .. 64, three
//     potentials and gammas: the FP32 table has the error against 64 bits that the direct FP64 sums gave
//     it, in the 2-norm, the largest entry and entry by entry.
#include <cmath>
#include <cstring>
#include <vector>

#include "bz_internal.h"
#include "bz_line8.cuh"

namespace bz {

namespace {

__device__ __forceinline__ double j0m1(double z) {
    if (fabs(z) < 0.25) {
        // J0(z) - 1 = sum_{m >= 1} (-(z/2)^2)^m / (m!)^2, Horner form to m = 8
        double u = -0.25 * z * z;
        double s = 1.0;
        #pragma unroll
        for (int m = 8; m >= 2; --m) s = 1.0 + s * u / ((double)m * (double)m);
        return u * s;
    }
    return j0(z) - 1.0;
}

// F for one (x, y) pair over one radial node's rule (nodes staged in shared memory).
__device__ __forceinline__ double2 f_value(double x, double y, const double *A, int n,
                                           const double *omc, const double *sn, const double *W) {
    double sr = -0.5 * x * x * A[1] - 0.25 * y * y * A[2];
    double si = x * A[0];
    for (int q = 0; q < n; ++q) {
        double jm1 = j0m1(y * sn[q]);
        double J = 1.0 + jm1;
        double sh, ch;
        sincos(0.5 * x * omc[q], &sh, &ch);
        // exp(i x c) - 1 = -2 sin^2(x c / 2) + i 2 sin(x c / 2) cos(x c / 2)
        sr += W[q] * (-2.0 * sh * sh * J + jm1);
        si += W[q] * (2.0 * sh * ch * J);
    }
    return make_double2(2.0 * M_PI * sr, 2.0 * M_PI * si);
}

struct TableArgs {
    int N, M, P, p0;
    int nin;                 // > 0: alpha is zero outside the signed range [-nin/2, nin/2) per axis
    double L, inv_n3;
    double A0, A1, A2;
    const double *term;      // [P][5]: r, q0, q1, q2, c
    const double *rule;      // concatenated omc | sn | W per radial node
    const int *rule_off;     // [N_rho + 1]
    float2 *alpha;           // [P][N^3]
    // 3D: the Legendre coefficients of radial nodes i0 .. (k_legendre_coef)
    int i0, g0, nkk, stride; // node of blockIdx.z = 0, term group of blockIdx.y = 0
    const double *coef;
    const int *cut;
    const double *g;         // [stride] g_l of the recurrence (double-float form: hi, lo as float2)
    // the double-float form
    const float2 *rk;        // [nkk] 1 / |k|
    const float2 *tq;        // [P][4] qhat, c_p / N^3
    const float4 *ph;        // [P][3][N] exp(i a qhat_d k)
};

// Coefficients of the Legendre series: row (radial node i, m = |k|^2) holds
// coef[l] = mu'_l j_l(z), z = pi r_i sqrt(m) / (2L), l = 0 .. cut - 1, where mu'_l carries (2l + 1), the
// sign of (-i)^l and the scale of the recurrence's polynomials; cut (even) drops the tail below
// 2^-60 of the row's largest.  j_l by downward recurrence from lmax (where |j_l| < 1e-22 for the
// largest z, or from the l where that holds for this z), normalised by sum (2l + 1) j_l^2 = 1 with
// the sign of j_0 = sin z / z or j_1.  One thread per row.
// Double-float form (dblf): entries as (hi, lo) float2, and ahead of them kRowHead with part I in the same
// variables, x = z c, y^2 = z^2 (1 - c^2): w0 + w1 c^2 + i w2 c; and z.
constexpr int kRowHead = 4;
struct CoefArgs {
    int i0, ni, nkk, stride, lmax, dblf;
    double A0, A1, A2;
    double L;
    const double *r;         // [N_rho] radial nodes
    const double *mu;        // [lmax + 1]
    double *coef;            // [ni][nkk][stride]
    int *cut;                // [ni][nkk]
};

__global__ void __launch_bounds__(64) k_legendre_coef(CoefArgs a) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= a.nkk) return;
    const size_t row = (size_t)blockIdx.y * a.nkk + m;
    const double z = M_PI * a.r[a.i0 + blockIdx.y] * sqrt((double)m) / (2.0 * a.L);
    double *c = a.coef + row * a.stride + (a.dblf ? kRowHead : 0);
    auto pair = [](double v) {
        const float h = (float)v;
        return make_float2(h, (float)(v - (double)h));
    };
    if (a.dblf) {
        float2 *w = (float2 *)(c - kRowHead);
        w[0] = pair(-0.5 * M_PI * z * z * a.A2);
        w[1] = pair(-2.0 * M_PI * z * z * (0.5 * a.A1 - 0.25 * a.A2));
        w[2] = pair(2.0 * M_PI * z * a.A0);
        w[3] = pair(z);
    }
    if (!(z > 0.0)) {                                     // k = 0: F = 0
        a.cut[row] = 0;
        return;
    }
    // |j_l(z)| <= z^l / (2l + 1)!!: the first l where this is below 1e-22 of j_1's scale
    int top = 1;
    const double lz = log(z);
    for (double lb = 0.0; top < a.lmax; ++top) {
        lb += lz - log(2.0 * top + 3.0);
        if (top > z && lb < -50.7) break;
    }
    const double iz = 1.0 / z;
    double f2 = 0.0, f1 = 1e-30, norm = 0.0;              // f_{l+1}, f_l
    for (int l = top; l >= 0; --l) {
        if (l < a.stride) c[l] = f1;
        norm += (2.0 * l + 1.0) * f1 * f1;
        const double f0 = (2.0 * l + 1.0) * iz * f1 - f2;
        f2 = f1;
        f1 = f0;
    }
    double sz, cz;
    sincos(z, &sz, &cz);
    const double j0 = sz * iz, j1 = z < 0.1 ? z / 3.0 : (j0 - cz) * iz;
    const double g0 = c[0], g1 = c[1];
    double sc = 1.0 / sqrt(norm);
    if (fabs(j0) > fabs(j1) ? (j0 < 0.0) != (g0 < 0.0) : (j1 < 0.0) != (g1 < 0.0)) sc = -sc;
    double big = 0.0;
    c[0] = 0.0;
    for (int l = 1; l <= top; ++l) {
        const double v = a.mu[l] * sc * c[l];
        c[l] = v;
        big = fmax(big, fabs(v));
    }
    int n = top;
    while (n > 1 && fabs(c[n]) < 0x1p-60 * big) --n;
    if ((n & 1) == 0) c[n + 1] = 0.0;                     // pairs (even, odd); stride >= lmax + 2
    a.cut[row] = (n | 1) + 1;
    if (a.dblf)
        for (int l = 0; l <= (n | 1); ++l) ((float2 *)c)[l] = pair(c[l]);
}

// Thread: one mode k (of each pair k, -k) and up to kLegTerms terms of one radial node, sharing the
// coefficient row.  The polynomials are 2^l times the monic Legendre ones, q_{l+1} = 2c q_l -
// g_l q_{l-1}, g_l = 4 l^2 / (4 l^2 - 1): two FP64 operations a step and a third for the sum; no
// over- or underflow for any l.  FP64 bound (this part runs about two FP64 lanes per clock and SM).
// Measured at N = 32, P = 384 (R = 6, s = 1/2): 4.6 ms; the direct sum over the rule took 578 ms.  It serves
// series longer than kFfSeries, where the double-float form below has fewer bits to spare.
constexpr int kLegTerms = 4;

__global__ void __launch_bounds__(128) ftable_kernel(TableArgs a) {
    extern __shared__ double sg[];                        // g_l, l = 0 .. lmax + 1
    for (int t = threadIdx.x; t < a.stride; t += blockDim.x) sg[t] = a.g[t];
    __syncthreads();
    const int N = a.N, n3 = N * N * N;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n3) return;
    const int il = blockIdx.z, j0 = (a.g0 + blockIdx.y) * kLegTerms;
    const int p0 = (a.i0 + il) * a.M + j0, np = min(kLegTerms, a.M - j0);
    int i1 = idx / (N * N), i2 = (idx / N) % N, i3 = idx % N;
    int k1 = i1 < N / 2 ? i1 : i1 - N;
    int k2 = i2 < N / 2 ? i2 : i2 - N;
    int k3 = i3 < N / 2 ? i3 : i3 - N;
    // F(-k) = conj F(k) (eq. FF): the entry of the smaller index of each pair (k, -k) is computed
    // and written to both; modes with a Nyquist component (-N/2) have no partner.
    const bool nyq = k1 == -N / 2 || k2 == -N / 2 || k3 == -N / 2;
    int midx = -1;
    if (!nyq) {
        midx = (((-k1 + N) % N) * N + ((-k2 + N) % N)) * N + ((-k3 + N) % N);
        if (midx < idx) return;                           // written by the partner's thread
    }
    // padded plans: only the modes of the caller's grid carry a weight (both members of the pair
    // are tested: -k leaves the range when a component of k is -nin/2)
    const int h = a.nin / 2;
    const bool in_k = a.nin == 0 || (k1 >= -h && k1 < h && k2 >= -h && k2 < h && k3 >= -h && k3 < h);
    const bool in_m = midx >= 0 && (a.nin == 0 || (-k1 >= -h && -k1 < h && -k2 >= -h && -k2 < h && -k3 >= -h && -k3 < h));
    if (!in_k && !in_m) {
        for (int u = 0; u < np; ++u) {
            a.alpha[(size_t)(p0 + u) * n3 + idx] = make_float2(0.f, 0.f);
            if (midx > idx) a.alpha[(size_t)(p0 + u) * n3 + midx] = make_float2(0.f, 0.f);
        }
        return;
    }
    const int kk = k1 * k1 + k2 * k2 + k3 * k3;
    const double ik = kk > 0 ? 1.0 / sqrt((double)kk) : 0.0;
    double kap[kLegTerms], c2[kLegTerms], q0[kLegTerms], q1[kLegTerms], sr[kLegTerms], si[kLegTerms];
    #pragma unroll
    for (int u = 0; u < kLegTerms; ++u) {
        const double *tp = a.term + 5 * (size_t)(p0 + (u < np ? u : 0));
        kap[u] = k1 * tp[1] + k2 * tp[2] + k3 * tp[3];
        c2[u] = 2.0 * fmin(1.0, fmax(-1.0, kap[u] * ik));
        q0[u] = 1.0;                                      // q_0
        q1[u] = c2[u];                                    // q_1 = 2 c
        sr[u] = si[u] = 0.0;
    }
    const size_t row = (size_t)il * a.nkk + kk;
    const double2 *c = (const double2 *)(a.coef + row * a.stride);
    const int cut = a.cut[row];
    for (int l = 0; l < cut; l += 2) {
        const double2 cl = c[l / 2];
        const double ga = sg[l + 1], gb = sg[l + 2];
        #pragma unroll
        for (int u = 0; u < kLegTerms; ++u) {
            sr[u] = fma(cl.x, q0[u], sr[u]);
            si[u] = fma(cl.y, q1[u], si[u]);
            q0[u] = fma(c2[u], q1[u], -ga * q0[u]);
            q1[u] = fma(c2[u], q0[u], -gb * q1[u]);
        }
    }
    for (int u = 0; u < np; ++u) {
        const double *tp = a.term + 5 * (size_t)(p0 + u);
        const double aa = M_PI * tp[0] / (2.0 * a.L);
        // x with the clamped cos chi: a point longer than 1 (a caller's rule, unit to a few digits) shifts it against
        // the j_l(a |k|), by a phase of z times the excess
        const double x = 0.5 * aa * c2[u] * (kk > 0 ? sqrt((double)kk) : 0.0);
        const double y2 = aa * aa * fmax((double)kk - kap[u] * kap[u], 0.0);
        double sx, cx;
        sincos(x, &sx, &cx);
        const double sc = tp[4] * a.inv_n3;
        const double fr = sc * (2.0 * M_PI * (-0.5 * x * x * a.A1 - 0.25 * y2 * a.A2) + (cx * sr[u] - sx * si[u]));
        const double fi = sc * (2.0 * M_PI * x * a.A0 + (cx * si[u] + sx * sr[u]));
        float2 *al = a.alpha + (size_t)(p0 + u) * n3;
        al[idx] = in_k ? make_float2((float)fr, (float)fi) : make_float2(0.f, 0.f);
        if (midx > idx) al[midx] = in_m ? make_float2((float)fr, (float)(-fi)) : make_float2(0.f, 0.f);
    }
}

// The same series in double-float arithmetic (pairs of FP32, about 47 bits; bz_line8.cuh): an FP64 instruction of a
// warp takes 68 clocks of a scheduler, a double-float product and sum 37 FP32 instructions.  No FP64 in
// the kernel: 1 / |k|, the axes' exp(i a qhat_d k_d) and part I's coefficients come from tables.  The
// table's error against 64 bits stays that of its FP32 rounding (2.6e-8).  Bound by FP32 issue.
// Measured at N = 32, P = 384: 0.80 ms and 0.20 for the rows, 4.6 in FP64 (plan creation 7.1 -> 2.9 ms; 46 s ->
// 91 ms at N = 64, P = 4096 since the direct sum).
__device__ __forceinline__ ff fmul(ff a, ff b) {
    const float p = __fmul_rn(a.h, b.h);
    const float e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
    const float h = __fadd_rn(p, e);
    return {h, __fsub_rn(e, __fsub_rn(h, p))};
}
__device__ __forceinline__ ff ld(float2 v) { return {v.x, v.y}; }

__global__ void k_axis_phases(int N, int M, double L, const double *__restrict__ term, float4 *__restrict__ ph) {
    const int p = blockIdx.x, d = threadIdx.x / N, i = threadIdx.x % N, k = i < N / 2 ? i : i - N;
    double sn, cs;
    sincos(M_PI * term[5 * p] / (2.0 * L) * term[5 * p + 1 + d] * k, &sn, &cs);
    const float c = (float)cs, s = (float)sn;
    ph[(size_t)p * 3 * N + threadIdx.x] = make_float4(c, (float)(cs - c), s, (float)(sn - s));
}

__global__ void __launch_bounds__(128) ftable_ff_kernel(TableArgs a) {
    extern __shared__ float2 sgf[];                       // g_l
    const int N = a.N, n3 = N * N * N;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    for (int t = threadIdx.x; t < a.stride; t += blockDim.x) sgf[t] = ((const float2 *)a.g)[t];
    __syncthreads();
    if (idx >= n3) return;
    const int il = blockIdx.z, j0 = (a.g0 + blockIdx.y) * kLegTerms;
    const int p0 = (a.i0 + il) * a.M + j0, np = min(kLegTerms, a.M - j0);
    const int i1 = idx / (N * N), i2 = (idx / N) % N, i3 = idx % N;
    const int k1 = i1 < N / 2 ? i1 : i1 - N, k2 = i2 < N / 2 ? i2 : i2 - N, k3 = i3 < N / 2 ? i3 : i3 - N;
    // pairs (k, -k) and the padded range as in ftable_kernel
    const bool nyq = k1 == -N / 2 || k2 == -N / 2 || k3 == -N / 2;
    int midx = -1;
    if (!nyq) {
        midx = (((-k1 + N) % N) * N + ((-k2 + N) % N)) * N + ((-k3 + N) % N);
        if (midx < idx) return;
    }
    const int h = a.nin / 2;
    const bool in_k = a.nin == 0 || (k1 >= -h && k1 < h && k2 >= -h && k2 < h && k3 >= -h && k3 < h);
    const bool in_m = midx >= 0 && (a.nin == 0 || (-k1 >= -h && -k1 < h && -k2 >= -h && -k2 < h && -k3 >= -h && -k3 < h));
    const int kk = k1 * k1 + k2 * k2 + k3 * k3;
    const size_t row = (size_t)il * a.nkk + kk;
    const float2 *rw = (const float2 *)(a.coef + row * a.stride);
    const float4 *c = (const float4 *)(rw + kRowHead);
    const int cut = in_k || in_m ? a.cut[row] : 0;
    const ff rk = ld(a.rk[kk]), zero = {0.f, 0.f};
    ff ch[kLegTerms], c2[kLegTerms], q0[kLegTerms], q1[kLegTerms], sr[kLegTerms], si[kLegTerms];
    float over[kLegTerms];                                // cos chi beyond 1 (a point longer than 1)
    #pragma unroll
    for (int u = 0; u < kLegTerms; ++u) {
        const float2 *tq = a.tq + 4 * (size_t)(p0 + (u < np ? u : 0));
        const ff f1 = {(float)k1, 0.f}, f2 = {(float)k2, 0.f}, f3 = {(float)k3, 0.f};
        ch[u] = fmul(fadd(fdot<1>(ld(tq[0]), f1, ld(tq[1]), f2), fmul(ld(tq[2]), f3)), rk);   // cos chi
        const float one = ch[u].h < 0.f ? -1.f : 1.f;
        over[u] = (ch[u].h - one) + ch[u].l;
        if (over[u] * one > 0.f) ch[u] = {one, 0.f};
        else over[u] = 0.f;
        c2[u] = {2.f * ch[u].h, 2.f * ch[u].l};
        q0[u] = {1.f, 0.f};
        q1[u] = c2[u];
        sr[u] = si[u] = zero;
    }
    for (int l = 0; l < cut; l += 2) {
        const float4 cl = c[l / 2];
        const ff ca = {cl.x, cl.y}, cb = {cl.z, cl.w}, ga = ld(sgf[l + 1]), gb = ld(sgf[l + 2]);
        #pragma unroll
        for (int u = 0; u < kLegTerms; ++u) {
            sr[u] = fadd(sr[u], fmul(ca, q0[u]));
            si[u] = fadd(si[u], fmul(cb, q1[u]));
            q0[u] = fdot<-1>(c2[u], q1[u], ga, q0[u]);
            q1[u] = fdot<-1>(c2[u], q0[u], gb, q1[u]);
        }
    }
    const ff w0 = ld(rw[0]), w1 = ld(rw[1]), w2 = ld(rw[2]);
    #pragma unroll
    for (int u = 0; u < kLegTerms; ++u) {
        if (u >= np) break;
        const float4 *ph = a.ph + (size_t)(p0 + u) * 3 * N;
        ffc e = mul(mul(unpack(ph[i1]), unpack(ph[N + i2])), unpack(ph[2 * N + i3]));
        if (over[u] != 0.f) {                             // the phase of the clamped cos chi: back by z over
            float sn, cs;
            sincosf(rw[3].x * over[u], &sn, &cs);
            e = mul(e, {{cs, 0.f}, {-sn, 0.f}});
        }
        ffc F = mul(e, {sr[u], si[u]});
        F.x = fadd(F.x, fadd(w0, fmul(w1, fmul(ch[u], ch[u]))));
        F.y = fadd(F.y, fmul(w2, ch[u]));
        const ff sc = ld(a.tq[4 * (size_t)(p0 + u) + 3]);
        const float fr = fmul(F.x, sc).h, fi = fmul(F.y, sc).h;
        float2 *al = a.alpha + (size_t)(p0 + u) * n3;
        al[idx] = in_k ? make_float2(fr, fi) : make_float2(0.f, 0.f);
        if (midx > idx) al[midx] = in_m ? make_float2(fr, -fi) : make_float2(0.f, 0.f);
    }
}

// 2D (Sec. 4.1 (i)): with x = a k.qhat, y = a k.qperp the odd terms cancel between parts I and
// III and part II folds onto [eps, pi], so
//   F = 2 [ i x A1 - x^2 A2 / 2 - y^2 A3 / 2 ] + 2 sum_n W_n [ (exp(i x c_n) - 1) cos(y s_n) + (cos(y s_n) - 1) ]
// with W_n = w_n b(t_n) (the circle's measure carries no sin t).
__device__ __forceinline__ double2 f_value_2d(double x, double y, const double *A, int n,
                                              const double *omc, const double *sn, const double *W) {
    double sr = -0.5 * x * x * A[1] - 0.5 * y * y * A[2];
    double si = x * A[0];
    for (int q = 0; q < n; ++q) {
        double sy, cy, sh, ch;
        sincos(0.5 * y * sn[q], &sy, &cy);
        const double cs = 1.0 - 2.0 * sy * sy;             // cos(y s), its deficit -2 sin^2(y s / 2)
        sincos(0.5 * x * omc[q], &sh, &ch);
        sr += W[q] * (-2.0 * sh * sh * cs - 2.0 * sy * sy);
        si += W[q] * (2.0 * sh * ch * cs);
    }
    return make_double2(2.0 * sr, 2.0 * si);
}

// 2D table: one thread per (mode of the N x N grid, term); alpha = c_p F / N^2.
__global__ void ftable2d_kernel(TableArgs a) {
    extern __shared__ double sm[];
    const int p = a.p0 + blockIdx.y;
    const int i = p / a.M;
    const int off = a.rule_off[i];
    const int n = a.rule_off[i + 1] - off;
    double *omc = sm, *sn = sm + n, *W = sm + 2 * n;
    const double *src = a.rule + 3 * (size_t)off;
    for (int t = threadIdx.x; t < 3 * n; t += blockDim.x) sm[t] = src[t];
    __syncthreads();
    const int N = a.N, n2 = N * N;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n2) return;
    const int i1 = idx / N, i2 = idx % N;
    const int k1 = i1 < N / 2 ? i1 : i1 - N;
    const int k2 = i2 < N / 2 ? i2 : i2 - N;
    const double *tp = a.term + 5 * (size_t)p;
    const double aa = M_PI * tp[0] / (2.0 * a.L);
    const double A[3] = {a.A0, a.A1, a.A2};
    const double2 F = f_value_2d(aa * (k1 * tp[1] + k2 * tp[2]), aa * (-k1 * tp[2] + k2 * tp[1]), A, n, omc, sn, W);
    const double sc = tp[4] * a.inv_n3;
    a.alpha[(size_t)p * n2 + idx] = make_float2((float)(sc * F.x), (float)(sc * F.y));
}

struct EntryArgs {
    int N, M, P, count, dim;
    double L;
    double A0, A1, A2;
    const double *term;
    const double *rule;
    const int *rule_off;
    const int *k_idx;
    const int *tsel;
    double *out;
};

// One thread per requested entry; rule read from global memory.
__global__ void fentries_kernel(EntryArgs a) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.count) return;
    const int N = a.N;
    int p = a.tsel[e];
    int i1 = a.k_idx[3 * e], i2 = a.k_idx[3 * e + 1], i3 = a.dim == 2 ? 0 : a.k_idx[3 * e + 2];
    if (p < 0 || p >= a.P || i1 < 0 || i1 >= N || i2 < 0 || i2 >= N || i3 < 0 || i3 >= N) {
        a.out[2 * e] = nan("");          // out-of-range request: no table access
        a.out[2 * e + 1] = nan("");
        return;
    }
    int i = p / a.M;
    int off = a.rule_off[i];
    int n = a.rule_off[i + 1] - off;
    const double *src = a.rule + 3 * (size_t)off;
    int k1 = i1 < N / 2 ? i1 : i1 - N;
    int k2 = i2 < N / 2 ? i2 : i2 - N;
    int k3 = i3 < N / 2 ? i3 : i3 - N;
    const double *tp = a.term + 5 * (size_t)p;
    double aa = M_PI * tp[0] / (2.0 * a.L);
    double A[3] = {a.A0, a.A1, a.A2};
    double2 F;
    if (a.dim == 2) {
        F = f_value_2d(aa * (k1 * tp[1] + k2 * tp[2]), aa * (-k1 * tp[2] + k2 * tp[1]), A, n, src, src + n, src + 2 * n);
    } else {
        double kap = k1 * tp[1] + k2 * tp[2] + k3 * tp[3];
        double kk = (double)k1 * k1 + (double)k2 * k2 + (double)k3 * k3;
        double kp2 = kk - kap * kap;
        double kp = kp2 > 0.0 ? sqrt(kp2) : 0.0;
        F = f_value(aa * kap, aa * kp, A, n, src, src + n, src + 2 * n);
    }
    a.out[2 * e] = F.x;
    a.out[2 * e + 1] = F.y;
}

}  // namespace

namespace {

// The 3D table: mu_l on the host, then per group of radial nodes the coefficient rows and the
// table entries.  A group's rows take at most kCoefBytes (at least one node).
constexpr size_t kCoefBytes = (size_t)64 << 20;
constexpr int kFfSeries = 160;

bz_status table3(Plan &pl, TableArgs a) {
    const int N = pl.N, nkk = 3 * (N / 2) * (N / 2) + 1;
    double rmax = 0.0;
    std::vector<double> r(pl.N_rho);
    for (int i = 0; i < pl.N_rho; ++i) {
        r[i] = pl.terms.r[(size_t)i * pl.M];
        rmax = r[i] > rmax ? r[i] : rmax;
    }
    // lmax: |j_l(z)| <= z^l / (2l + 1)!! < 1e-22 beyond it for every z of the plan
    const double zmax = M_PI * rmax * std::sqrt((double)(nkk - 1)) / (2.0 * pl.L);
    int lmax = 1;
    for (double lb = 0.0; !(lmax > zmax && lb < -50.7); ++lmax) lb += std::log(zmax) - std::log(2.0 * lmax + 3.0);
    // the double-float form up to l = kFfSeries: every plan whose R is within the box (N = 64: about 140)
    const bool dblf = lmax <= kFfSeries;
    const int stride = ((lmax + 4) & ~1) + (dblf ? kRowHead : 0);
    // mu'_l = 2 pi sum_n W_n (P_l(cos t_n) - 1) times (2l + 1), the sign of (-i)^l (the sum over odd l
    // is the imaginary part) and P_l / q_l; D_l = P_l - 1 by its own recurrence (no cancellation at
    // small angles), on the rule with the most nodes
    const ThetaRule *R = &pl.rules[0];
    for (const ThetaRule &q : pl.rules)
        if (q.W.size() > R->W.size()) R = &q;
    std::vector<double> mu(lmax + 1, 0.0);
    for (size_t n = 0; n < R->W.size(); ++n) {
        const double omc = R->omc[n], c = 1.0 - omc;
        double d0 = 0.0, d1 = -omc;                        // D_0, D_1
        for (int l = 1; l <= lmax; ++l) {
            mu[l] += R->W[n] * d1;
            const double d2 = ((2.0 * l + 1.0) * (c * d1 - omc) - l * d0) / (l + 1.0);
            d0 = d1;
            d1 = d2;
        }
    }
    double lead = 1.0;                                     // P_l / q_l = (2l)! / (4^l l!^2)
    for (int l = 1; l <= lmax; ++l) {
        lead *= (2.0 * l - 1.0) / (2.0 * l);
        const double sign = (l & 3) == 0 || (l & 3) == 3 ? 1.0 : -1.0;   // (-i)^l: -i, -1, i, 1
        mu[l] *= 2.0 * M_PI * (2.0 * l + 1.0) * sign * lead;
    }
    const size_t row = (size_t)nkk * stride * sizeof(double);
    int ni = (int)(kCoefBytes / row);
    const int groups = (pl.M + kLegTerms - 1) / kLegTerms;
    if (ni > 65535) ni = 65535;                            // gridDim limit
    if (ni < 1) ni = 1;
    if (ni > pl.N_rho) ni = pl.N_rho;
    const size_t gsm = (size_t)stride * sizeof(double);
    if (gsm > 48 * 1024)
        BZ_CUDA_TRY(cudaFuncSetAttribute(ftable_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm));
    // one upload: r, mu, g_l and, for the double-float form, 1 / |k| and the terms as (hi, lo)
    auto pair = [](double v) {
        const float f[2] = {(float)v, (float)(v - (double)(float)v)};
        double d;
        std::memcpy(&d, f, sizeof(d));
        return d;
    };
    std::vector<double> up(r);
    up.insert(up.end(), mu.begin(), mu.end());
    const size_t at_g = up.size();
    for (int t = 0; t < stride; ++t) {
        const double g = 4.0 * t * t / (4.0 * t * t - 1.0);
        up.push_back(dblf ? pair(g) : g);
    }
    const size_t at_rk = up.size(), at_tq = at_rk + (dblf ? nkk : 0);
    if (dblf) {
        for (int m = 0; m < nkk; ++m) up.push_back(pair(m ? 1.0 / std::sqrt((double)m) : 0.0));
        for (int p = 0; p < pl.P; ++p) {
            for (int d = 0; d < 3; ++d) up.push_back(pair(pl.terms.q[3 * (size_t)p + d]));
            up.push_back(pair(pl.terms.c[p] * a.inv_n3));
        }
    }
    const size_t head = (up.size() + 1) & ~(size_t)1;      // (the phases are 16-byte values)
    const size_t phases = dblf ? (size_t)pl.P * 3 * N * sizeof(float4) : 0;
    double *buf = nullptr;                                 // coefficient rows, the upload, phases, row lengths
    if (cudaMalloc(&buf, ni * row + head * sizeof(double) + phases + (size_t)ni * nkk * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return BZ_ERR_OOM;
    }
    double *coef = buf, *r_dev = coef + ni * row / sizeof(double), *mu_dev = r_dev + r.size();
    float4 *ph = (float4 *)(r_dev + head);
    int *cut = (int *)((char *)ph + phases);
    cudaError_t e = cudaMemcpy(r_dev, up.data(), up.size() * sizeof(double), cudaMemcpyHostToDevice);
    CoefArgs ca;
    ca.nkk = nkk; ca.stride = stride; ca.lmax = lmax; ca.L = pl.L; ca.r = r_dev; ca.mu = mu_dev; ca.coef = coef;
    ca.cut = cut; ca.dblf = dblf; ca.A0 = a.A0; ca.A1 = a.A1; ca.A2 = a.A2;
    a.nkk = nkk; a.stride = stride; a.coef = coef; a.cut = cut; a.g = r_dev + at_g;
    a.rk = (const float2 *)(r_dev + at_rk); a.tq = (const float2 *)(r_dev + at_tq); a.ph = ph;
    if (dblf) k_axis_phases<<<pl.P, 3 * N>>>(N, pl.M, pl.L, a.term, ph);
    for (int i0 = 0; e == cudaSuccess && i0 < pl.N_rho; i0 += ni) {
        const int n = pl.N_rho - i0 < ni ? pl.N_rho - i0 : ni;
        ca.i0 = a.i0 = i0;
        ca.ni = n;
        k_legendre_coef<<<dim3((nkk + 63) / 64, n), 64>>>(ca);
        for (a.g0 = 0; a.g0 < groups; a.g0 += 65535) {
            const int ng = groups - a.g0 < 65535 ? groups - a.g0 : 65535;
            const dim3 grid((N * N * N + 127) / 128, ng, n);
            if (dblf) ftable_ff_kernel<<<grid, 128, gsm>>>(a);
            else ftable_kernel<<<grid, 128, gsm>>>(a);
        }
        e = cudaGetLastError();
    }
    const cudaError_t es = cudaDeviceSynchronize();
    cudaFree(buf);
    return e == cudaSuccess && es == cudaSuccess ? BZ_OK : BZ_ERR_CUDA;
}

}  // namespace

// Uploads terms and theta rules; fills pl.alpha with c_p F / N^3 (FP32).
bz_status ftable_build(Plan &pl) {
    const int P = pl.P, N = pl.N;
    std::vector<double> term(5 * (size_t)P);
    for (int p = 0; p < P; ++p) {
        term[5 * p] = pl.terms.r[p];
        for (int d = 0; d < 3; ++d) term[5 * p + 1 + d] = pl.terms.q[3 * p + d];
        term[5 * p + 4] = pl.terms.c[p];
    }
    std::vector<double> rule;
    std::vector<int> off(pl.N_rho + 1, 0);
    pl.rule_max = 0;
    for (int i = 0; i < pl.N_rho; ++i) {
        const ThetaRule &R = pl.rules[i];
        int n = (int)R.W.size();
        off[i + 1] = off[i] + n;
        pl.rule_max = n > pl.rule_max ? n : pl.rule_max;
        rule.insert(rule.end(), R.omc.begin(), R.omc.end());
        rule.insert(rule.end(), R.sn.begin(), R.sn.end());
        rule.insert(rule.end(), R.W.begin(), R.W.end());
    }
    BZ_CUDA_TRY(cudaMalloc(&pl.term_dev, term.size() * sizeof(double)));
    BZ_CUDA_TRY(cudaMalloc(&pl.rule_buf, rule.size() * sizeof(double)));
    BZ_CUDA_TRY(cudaMalloc(&pl.rule_off, off.size() * sizeof(int)));
    BZ_CUDA_TRY(cudaMemcpy(pl.term_dev, term.data(), term.size() * sizeof(double), cudaMemcpyHostToDevice));
    BZ_CUDA_TRY(cudaMemcpy(pl.rule_buf, rule.data(), rule.size() * sizeof(double), cudaMemcpyHostToDevice));
    BZ_CUDA_TRY(cudaMemcpy(pl.rule_off, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice));

    const size_t smem = 3 * (size_t)pl.rule_max * sizeof(double);
    if (smem > 200 * 1024) return BZ_ERR_UNSUPPORTED;
    TableArgs a = {};
    a.N = N; a.M = pl.M; a.P = P; a.L = pl.L; a.nin = pl.Nin;
    a.inv_n3 = 1.0 / (double)modes(pl);      // the forward transform's N^-d
    a.A0 = pl.A[0]; a.A1 = pl.A[1]; a.A2 = pl.A[2];
    a.term = pl.term_dev; a.rule = pl.rule_buf; a.rule_off = pl.rule_off; a.alpha = pl.alpha;
    if (pl.dim != 2) return table3(pl, a);
    if (smem > 48 * 1024)
        BZ_CUDA_TRY(cudaFuncSetAttribute(ftable2d_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int n3 = (int)modes(pl), bs = 128;
    const int ychunk = 32768;   // gridDim.y limit
    for (int p0 = 0; p0 < P; p0 += ychunk) {
        a.p0 = p0;
        dim3 grid((n3 + bs - 1) / bs, (P - p0) < ychunk ? (P - p0) : ychunk);
        ftable2d_kernel<<<grid, bs, smem>>>(a);
        BZ_CUDA_TRY(cudaGetLastError());
    }
    BZ_CUDA_TRY(cudaDeviceSynchronize());
    return BZ_OK;
}

bz_status ftable_entries(Plan &pl, int count, const int *k_idx, const int *term, double *out) {
    if (count <= 0) return count == 0 ? BZ_OK : BZ_ERR_ARG;
    EntryArgs a;
    a.N = pl.Nin ? pl.Nin : pl.N;      // indices address the caller's grid
    a.M = pl.M; a.P = pl.P; a.count = count; a.L = pl.L; a.dim = pl.dim;
    a.A0 = pl.A[0]; a.A1 = pl.A[1]; a.A2 = pl.A[2];
    a.term = pl.term_dev; a.rule = pl.rule_buf; a.rule_off = pl.rule_off;
    a.k_idx = k_idx; a.tsel = term; a.out = out;
    fentries_kernel<<<(count + 127) / 128, 128>>>(a);
    BZ_CUDA_TRY(cudaGetLastError());
    BZ_CUDA_TRY(cudaDeviceSynchronize());
    return BZ_OK;
}

}  // namespace bz
