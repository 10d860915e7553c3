// tridiag.cuh -- eigenvalues and eigenvectors of the Lanczos matrix T (diagonal al[0..m),
// off-diagonal be[0..m-1)) in binary64, one CTA of TRI_NT threads per eigenpair.
//
// What bounds these kernels is the number of dependent binary64 instructions: the recurrences
// run over the m rows of T one after the other, and a warp's binary64 instruction occupies
// its quarter of the SM for 64 cycles however many lanes take part (a division is nine of
// them).  So
//   * the Sturm count uses the leading principal minors p_i (a three-term recurrence, three
//     instructions a row, no division) instead of their ratios;
//   * every pass cuts the bracket with 128 points at once, one a thread and one warp to each
//     quarter of the SM: 7 bits a pass;
//   * the first passes run in binary32, up to the width that its rounding allows;
//   * the eigenvector comes from the forward and the backward recurrence at once (two lanes),
//     joined at its largest component, instead of three serial solves with pivoting.
// The rows of T are loaded 32 at a time, one a lane, and handed round by shuffles, so m is
// not bounded by shared memory.  Measured on GB300 against bisection in one lane with
// divisions: 3 Ritz values at m = 40 in 50 instead of 1160 us, the convergence scan of all
// leading T_k, k <= 120, in 157 instead of 4070 us, the pick and eigenvector at m of about 80
// in 111 instead of 4780 us.
#pragma once

#include "hm_internal.cuh"

namespace hm {

constexpr int TRI_NT = 128;

template <class R>
__device__ __forceinline__ R tri_shfl(R v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// 2^k, -1022 <= k <= 1023
__device__ __forceinline__ double tri_pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }

// bits of the sign and exponent: the float itself, the high word of a double
__device__ __forceinline__ int tri_hi(float v) { return __float_as_int(v); }
__device__ __forceinline__ int tri_hi(double v) { return __double2hiint(v); }
__device__ __forceinline__ bool tri_zero(float v) { return (__float_as_int(v) << 1) == 0; }
__device__ __forceinline__ bool tri_zero(double v) { return ((__double2hiint(v) << 1) | __double2loint(v)) == 0; }
// v with its exponent field moved by k; zero when that leaves the normal numbers at the bottom
__device__ __forceinline__ float tri_scale(float v, int k) {
    const int h = __float_as_int(v), e = ((h >> 23) & 0xFF) + k;
    return e > 0 ? __int_as_float(h + (k << 23)) : 0.0f;
}
__device__ __forceinline__ double tri_scale(double v, int k) {
    const int h = __double2hiint(v), e = ((h >> 20) & 0x7FF) + k;
    return e > 0 ? __hiloint2double(h + (k << 20), __double2loint(v)) : 0.0;
}
template <class R> struct TriFmt;
template <> struct TriFmt<float> { static constexpr int MB = 23, EM = 0xFF, BIAS = 127, RUN = 4, TINY = -60; };
template <> struct TriFmt<double> { static constexpr int MB = 20, EM = 0x7FF, BIAS = 1023, RUN = 8, TINY = -100; };

// Gershgorin interval of T; called by whole warps, the same result in every lane
__device__ __forceinline__ void tri_gershgorin(int m, const double *al, const double *be, double *lo_, double *hi_) {
    double lo = 1e308, hi = -1e308;
    for (int i = threadIdx.x & 31; i < m; i += 32) {
        const double r = (i > 0 ? fabs(be[i - 1]) : 0.0) + (i < m - 1 ? fabs(be[i]) : 0.0);
        lo = fmin(lo, al[i] - r);
        hi = fmax(hi, al[i] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    *lo_ = lo;
    *hi_ = hi;
}

// Number of eigenvalues of s T below x, one x a lane (s: a power of two that brings the norm of
// T to about 1): sign changes of the leading minors p_i of s T - x, p_i = (s al_i - x) p_{i-1}
// - (s be_{i-1})^2 p_{i-2} (Givens 1954).  A minor that vanishes takes the sign opposite to
// its predecessor (the ratio form's rule of a tiny negative pivot).  p is brought back to
// [1, 2) every RUN rows (4 in binary32, 8 in binary64: a row may cost p a factor of the unit
// roundoff) by integer operations on its exponent.
template <class R>
__device__ __forceinline__ int tri_count(int m, const double *__restrict__ al, const double *__restrict__ be, double s,
                                         R x) {
    using F = TriFmt<R>;
    const int lane = threadIdx.x & 31;
    int cnt = 0;
    R p = R(1), pp = R(0);
    for (int i0 = 0; i0 < m; i0 += 32) {
        const int i = i0 + lane;
        const R a = i < m ? (R)(al[i] * s) : R(0);
        const R b = i > 0 && i < m ? (R)(be[i - 1] * s) : R(0);
        const R b2 = b * b;
        const int n = min(32, m - i0);
        for (int j0 = 0; j0 < n; j0 += F::RUN) {
#pragma unroll
            for (int jj = 0; jj < F::RUN; ++jj) {
                const int j = j0 + jj;
                const R t = tri_shfl(a, j) - x, c = tri_shfl(b2, j) * pp;
                if (j < n) {
                    R q = fma(t, p, -c);
                    if (tri_zero(q)) q = tri_scale(-p, F::TINY);
                    cnt += (int)((unsigned)(tri_hi(q) ^ tri_hi(p)) >> 31);
                    pp = p;
                    p = q;
                }
            }
            const int k = F::BIAS - ((tri_hi(p) >> F::MB) & F::EM);
            p = tri_scale(p, k);
            pp = tri_scale(pp, k);
        }
    }
    return cnt;
}

// e-th lowest eigenvalue (1-based): the Gershgorin interval cut in 129 parts a pass, until the
// bracket holds no further double.  The binary32 passes stop at a width of 2^-18 of the norm
// and the bracket is then widened by 2^-19: their rounding perturbs T by less than 20 2^-24.
// Called by all TRI_NT threads, the same result in every thread.
__device__ __forceinline__ double tri_eig(int m, const double *al, const double *be, int e) {
    double lo, hi;
    tri_gershgorin(m, al, be, &lo, &hi);
    const double bound = fmax(fabs(lo), fabs(hi));
    if (!(lo <= hi)) return 0.5 * (lo + hi);                  // no finite entry
    if (bound == 0.0) return 0.0;
    if (!(bound <= 1.7e308)) return __longlong_as_double(0x7ff8000000000000ll);
    const int ex = min(max(ilogb(bound), -1000), 1000);
    const double s = tri_pow2(-ex);
    const double pad = 2.0 * 2.220446049250313e-16 * bound * s;
    double a = lo * s - pad, c = hi * s + pad;
    const int t = threadIdx.x;
    {
        float fa = __double2float_rd(a), fc = __double2float_ru(c);
        for (int it = 0; it < 8 && fc - fa > 0x1p-18f; ++it) {
            const float w = (fc - fa) * (1.0f / (TRI_NT + 1));
            const int k = __syncthreads_count(tri_count<float>(m, al, be, s, fmaf(w, (float)(t + 1), fa)) < e);
            const float a2 = fmaf(w, (float)k, fa), c2 = fmaf(w, (float)(k + 1), fa);
            if (k < TRI_NT) fc = c2;
            if (k > 0) fa = a2;
        }
        a = fmax(a, (double)fa - 0x1p-19);
        c = fmin(c, (double)fc + 0x1p-19);
    }
    for (int it = 0; it < 16; ++it) {
        const double mid = 0.5 * (a + c);
        if (mid <= a || mid >= c) break;
        const double w = (c - a) * (1.0 / (TRI_NT + 1));
        const int k = __syncthreads_count(tri_count<double>(m, al, be, s, fma(w, (double)(t + 1), a)) < e);
        const double a2 = fma(w, (double)k, a), c2 = fma(w, (double)(k + 1), a);
        if (k < TRI_NT) c = fmin(c, c2);
        if (k > 0) a = fmax(a, a2);
    }
    return 0.5 * (a + c) * tri_pow2(ex);
}

// Eigenvector z (normalised) of T for its eigenvalue th; f, g: scratch of m doubles each.  Even
// lanes run f_{i+1} = ((th - al_i) f_i - be_{i-1} f_{i-1}) / be_i from f_0 = 1, odd lanes
// g_{i-1} = ((th - al_i) g_i - be_i g_{i+1}) / be_{i-1} from g_{m-1} = 1; each is stable while it
// grows, and they are joined at the row t with the smallest
//     gamma_t = al_t - th + be_{t-1} f_{t-1} / f_t + be_t g_{t+1} / g_t,
// the row of the largest component (Fernando 1997, twisted factorisation).  Returns the last
// component |z_{m-1}|; writes z when it is not NULL (its component t positive).  One whole warp.
__device__ __forceinline__ double tri_vec(int m, const double *al, const double *be, double th, double *z, double *f,
                                          double *g) {
    const int lane = threadIdx.x & 31;
    const bool odd = lane & 1;
    if (m <= 1) {
        if (z && lane == 0 && m == 1) z[0] = 1.0;
        return 1.0;
    }
    double v = 1.0, vp = 0.0;                                 // f_i (even lanes) / g_i (odd lanes)
    double *const arr = odd ? g : f;
    if (lane < 2) arr[odd ? m - 1 : 0] = 1.0;
    for (int i0 = 0; i0 < m - 1; i0 += 32) {
        const int i = i0 + lane, ib = m - 1 - i;              // row of the forward / backward step
        double c1f = 0.0, c2f = 0.0, c1b = 0.0, c2b = 0.0;
        if (i < m - 1) {
            const double rf = 1.0 / be[i], rb = 1.0 / be[ib - 1];
            c1f = (th - al[i]) * rf;
            c2f = i > 0 ? be[i - 1] * rf : 0.0;
            c1b = (th - al[ib]) * rb;
            c2b = ib < m - 1 ? be[ib] * rb : 0.0;
        }
        const int n = min(32, m - 1 - i0);
#pragma unroll 4
        for (int j = 0; j < n; ++j) {
            const double uf = tri_shfl(c1f, j), wf = tri_shfl(c2f, j), ub = tri_shfl(c1b, j), wb = tri_shfl(c2b, j);
            const double w = (odd ? wb : wf) * vp;
            const double nv = fma(odd ? ub : uf, v, -w);
            vp = v;
            v = nv;
            const int k = odd ? m - 2 - (i0 + j) : i0 + j + 1;
            if (lane < 2) arr[k] = v;
            if (((__double2hiint(v) >> 20) & 0x7FF) > 1023 + 400) {       // rare: keep the range
                v *= 0x1p-400;
                vp *= 0x1p-400;
                if (lane == 0) for (int q = 0; q <= k; ++q) f[q] *= 0x1p-400;
                if (lane == 1) for (int q = k; q < m; ++q) g[q] *= 0x1p-400;
            }
        }
    }
    __syncwarp();
    double best = 1e308;
    int t = 0;
    for (int i = lane; i < m; i += 32) {
        double gm = al[i] - th;
        if (i > 0) gm += be[i - 1] * f[i - 1] / f[i];
        if (i < m - 1) gm += be[i] * g[i + 1] / g[i];
        gm = fabs(gm);
        if (gm < best) { best = gm; t = i; }                  // NaN (a component underflowed) never wins
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double b2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int t2 = __shfl_xor_sync(0xffffffffu, t, o);
        if (b2 < best || (b2 == best && t2 < t)) { best = b2; t = t2; }
    }
    const double rf = 1.0 / f[t], rg = 1.0 / g[t];
    double ss = 0.0;
    for (int i = lane; i < m; i += 32) {
        const double zi = i <= t ? f[i] * rf : g[i] * rg;
        ss = fma(zi, zi, ss);
    }
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const double inv = 1.0 / sqrt(ss);
    if (z)
        for (int i = lane; i < m; i += 32) z[i] = (i <= t ? f[i] * rf : g[i] * rg) * inv;
    return fabs((t == m - 1 ? 1.0 : g[m - 1] * rg) * inv);
}

}  // namespace hm
