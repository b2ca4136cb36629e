// gf_simd.cuh -- small device helpers shared by the evaluation kernels:
// packed FP32 pair arithmetic, compensated sums, and the packed L2P sum with
// its recursion coefficients.  Everything sits in an unnamed namespace, so
// every translation unit that includes this header has its own copy of the
// coefficient tables and uploads it with its own upload_l2p_coefs().
#pragma once

#include <cmath>

#include "gf_internal.cuh"

namespace gf {
namespace {

template <class T>
struct __align__(16) Vec4 {
    T x, y, z, w;
};

template <class T>
__device__ __forceinline__ T rsqrt_t(T x);
template <>
__device__ __forceinline__ float rsqrt_t<float>(float x) {
    return rsqrtf(x);
}
template <>
__device__ __forceinline__ double rsqrt_t<double>(double x) {
    return rsqrt(x);
}

// Packed pairs of FP32 values (f32x2 arithmetic of sm_100 and later: one
// instruction does two FP32 operations, halving the issue slots of the
// near-field loop).
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void up2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// 1/sqrt(x) on the special-function unit, subnormal inputs read as zero
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

template <class T>
__device__ __forceinline__ void two_sum(T &hi, T &lo, T x) {
    const T s = hi + x;
    const T bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
}

// The L2P sums sum_{n<p, m} D_n^m conj(R_n^m(X)) of the gradient expansions
// (l2p_sum of fmm_math.cuh) with R_n^m = s_nm (x + iy)^m Q_n^m(z, r^2), Q real:
// Q_m^m = 1, Q_n = z Q_{n-1} - c_nm r^2 Q_{n-2}, c_nm = ((n-1)^2 - m^2) /
// ((2n-1)(2n-3)).  s_nm (and the factor 2 of the m > 0 terms) is in the staged
// coefficients, an order's sums are made with Q alone and turned by (x + iy)^m
// once: nine operations a term instead of twelve, and no square roots or
// divisions.  c_lq: -c_nm at n (n - 1) / 2 + m, m < n < kMaxP (zero at n = m + 1);
// l2p_scale: s_nm, twice it for m > 0, by real component.
__constant__ float c_lq[kMaxP * (kMaxP - 1) / 2 + 1];
__device__ float l2p_scale[kMaxP * kMaxP];

// For two points at once (packed pairs X, Y, Z).  D holds each scaled
// coefficient as a duplicated pair {d, d}.
__device__ __forceinline__ void l2p_sum2(int p, const float2 *Dx, const float2 *Dy, const float2 *Dz, uint64_t X,
                                         uint64_t Y, uint64_t Z, uint64_t &gx, uint64_t &gy, uint64_t &gz) {
    const uint64_t r2 = fma2(Z, Z, fma2(Y, Y, mul2(X, X)));
    const uint64_t NY = Y ^ 0x8000000080000000ull, one = pk2(1.f, 1.f);
    uint64_t wr = one, wi = 0;
    auto ld = [](const float2 *d, int k) { return *reinterpret_cast<const uint64_t *>(d + k); };
    gx = gy = gz = 0;
    for (int m = 0; m < p; ++m) {
        uint64_t Q = one, P = 0, xr = 0, xi = 0, yr = 0, yi = 0, zr = 0, zi = 0;
        for (int n = m; n < p; ++n) {
            if (n > m) {
                const float c = c_lq[n * (n - 1) / 2 + m];
                const uint64_t v = fma2(Z, Q, mul2(mul2(r2, pk2(c, c)), P));
                P = Q;
                Q = v;
            }
            const int k = n * n + (m == 0 ? 0 : 2 * m - 1);
            xr = fma2(ld(Dx, k), Q, xr);
            yr = fma2(ld(Dy, k), Q, yr);
            zr = fma2(ld(Dz, k), Q, zr);
            if (m > 0) {
                xi = fma2(ld(Dx, k + 1), Q, xi);
                yi = fma2(ld(Dy, k + 1), Q, yi);
                zi = fma2(ld(Dz, k + 1), Q, zi);
            }
        }
        gx = fma2(xr, wr, fma2(xi, wi, gx));
        gy = fma2(yr, wr, fma2(yi, wi, gy));
        gz = fma2(zr, wr, fma2(zi, wi, gz));
        const uint64_t nr = fma2(X, wr, mul2(NY, wi)), ni = fma2(X, wi, mul2(Y, wr));
        wr = nr;
        wi = ni;
    }
}

// l2p_sum2 for two packed pairs of points at once (four points): every
// coefficient is loaded once for both.
__device__ __forceinline__ void l2p_sum2x2(int p, const float2 *Dx, const float2 *Dy, const float2 *Dz,
                                           uint64_t X0, uint64_t Y0, uint64_t Z0, uint64_t X1, uint64_t Y1,
                                           uint64_t Z1, uint64_t g0[3], uint64_t g1[3]) {
    const uint64_t q0 = fma2(Z0, Z0, fma2(Y0, Y0, mul2(X0, X0)));
    const uint64_t q1 = fma2(Z1, Z1, fma2(Y1, Y1, mul2(X1, X1)));
    const uint64_t one = pk2(1.f, 1.f);
    uint64_t wr0 = one, wi0 = 0, wr1 = one, wi1 = 0;
    auto ld = [](const float2 *d, int k) { return *reinterpret_cast<const uint64_t *>(d + k); };
#pragma unroll
    for (int d = 0; d < 3; ++d) g0[d] = g1[d] = 0;
    for (int m = 0; m < p; ++m) {
        uint64_t Q0 = one, P0 = 0, Q1 = one, P1 = 0;
        uint64_t re0[3] = {0, 0, 0}, im0[3] = {0, 0, 0}, re1[3] = {0, 0, 0}, im1[3] = {0, 0, 0};
        for (int n = m; n < p; ++n) {
            if (n > m) {
                const float c = c_lq[n * (n - 1) / 2 + m];
                const uint64_t C = pk2(c, c);
                const uint64_t v0 = fma2(Z0, Q0, mul2(mul2(q0, C), P0)), v1 = fma2(Z1, Q1, mul2(mul2(q1, C), P1));
                P0 = Q0;
                Q0 = v0;
                P1 = Q1;
                Q1 = v1;
            }
            const int k = n * n + (m == 0 ? 0 : 2 * m - 1);
            const uint64_t dr[3] = {ld(Dx, k), ld(Dy, k), ld(Dz, k)};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                re0[d] = fma2(dr[d], Q0, re0[d]);
                re1[d] = fma2(dr[d], Q1, re1[d]);
            }
            if (m > 0) {
                const uint64_t di[3] = {ld(Dx, k + 1), ld(Dy, k + 1), ld(Dz, k + 1)};
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    im0[d] = fma2(di[d], Q0, im0[d]);
                    im1[d] = fma2(di[d], Q1, im1[d]);
                }
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            g0[d] = fma2(re0[d], wr0, fma2(im0[d], wi0, g0[d]));
            g1[d] = fma2(re1[d], wr1, fma2(im1[d], wi1, g1[d]));
        }
        const uint64_t N0 = Y0 ^ 0x8000000080000000ull, N1 = Y1 ^ 0x8000000080000000ull;
        uint64_t nr = fma2(X0, wr0, mul2(N0, wi0)), ni = fma2(X0, wi0, mul2(Y0, wr0));
        wr0 = nr;
        wi0 = ni;
        nr = fma2(X1, wr1, mul2(N1, wi1));
        ni = fma2(X1, wi1, mul2(Y1, wr1));
        wr1 = nr;
        wi1 = ni;
    }
}

// c[n (n - 1) / 2 + m] = -c_nm and sc[component] = the L2P scales, in FP64.
inline void l2p_tables(double *c, double *sc) {
    double sect = 1.0;
    for (int m = 0; m < kMaxP; ++m) {
        if (m > 0) sect *= -std::sqrt((2.0 * m - 1.0) / (2.0 * m));
        double v = m > 0 ? 2.0 * sect : sect;
        for (int n = m; n < kMaxP; ++n) {
            if (n > m) {
                v *= (2 * n - 1) / std::sqrt((double)((n + m) * (n - m)));
                c[n * (n - 1) / 2 + m] =
                    n > m + 1 ? -(double)((n - 1) * (n - 1) - m * m) / ((2 * n - 1) * (2 * n - 3)) : 0.0;
            }
            const int k = n * n + (m == 0 ? 0 : 2 * m - 1);
            sc[k] = v;
            if (m > 0) sc[k + 1] = v;
        }
    }
}

// The tables of l2p_sum2 for the current device.
inline gf_status upload_l2p_coefs() {
    double c[kMaxP * (kMaxP - 1) / 2 + 1] = {}, sc[kMaxP * kMaxP] = {};
    l2p_tables(c, sc);
    float cf[kMaxP * (kMaxP - 1) / 2 + 1], sf[kMaxP * kMaxP];
    for (size_t i = 0; i < sizeof(cf) / sizeof(cf[0]); ++i) cf[i] = (float)c[i];
    for (int i = 0; i < kMaxP * kMaxP; ++i) sf[i] = (float)sc[i];
    GF_CUDA(cudaMemcpyToSymbol(c_lq, cf, sizeof(cf)));
    GF_CUDA(cudaMemcpyToSymbol(l2p_scale, sf, sizeof(sf)));
    return GF_OK;
}

// ---------------------------------------------------------------- FP64 without the FP64 pipe
// FP64 arithmetic and conversions run at a small fraction of the FP32 rate
// on this GPU; these conversions use integer operations only.
// Sign, exponent and the top 23 mantissa bits of a double repacked as a
// float (truncation: relative error below 2^-23), integer operations only;
// false when the value is outside the normal FP32 range (zero excepted).
__device__ __forceinline__ bool trunc_f32(double x, float &f) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff) - 1023;
    if (e < -126 || e > 127) {
        f = 0.f;
        return (b << 1) == 0;
    }
    f = __uint_as_float((unsigned)((b >> 32) & 0x80000000ull) | ((unsigned)(e + 127) << 23) |
                        (unsigned)((b >> 29) & 0x7fffffull));
    return true;
}

// trunc(x 2^k) for |x 2^k| < 2^62, integer operations only.
__device__ __forceinline__ long long to_fix(double x, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;
    const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
    const int sh = e - 1075 + k;
    const long long v = sh >= 0 ? (long long)(m << sh) : (sh > -64 ? (long long)(m >> -sh) : 0);
    return (b >> 63) ? -v : v;
}

// |v| < 2^63 as a float, truncating, integer operations only.
__device__ __forceinline__ float fix_to_f32(long long v) {
    if (v == 0) return 0.f;
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << lz;   // leading one at bit 63
    return __uint_as_float((v < 0 ? 0x80000000u : 0u) | ((unsigned)(63 - lz + 127) << 23) |
                           (unsigned)((n >> 40) & 0x7fffffull));
}

// A double as a float by truncation, integer operations only: below the normal
// FP32 range zero, above it (and for NaN) infinity.
__device__ __forceinline__ float f32_trunc(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32), sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ff) - 1023;
    const unsigned mag = ((unsigned)(e + 127) << 23) | ((unsigned)(b >> 29) & 0x7fffffu);
    return __uint_as_float(sign | (e < -126 ? 0u : e > 127 ? 0x7f800000u : mag));
}

// A float as a double (subnormals read as zero; infinities and NaNs kept).
__device__ __forceinline__ double f32_to_f64(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xff;
    if (e == 0) return 0.0;
    if (e == 0xff)   // infinity or NaN
        return __longlong_as_double((long long)(((unsigned long long)(b >> 31) << 63) | 0x7ff0000000000000ull |
                                                ((unsigned long long)(b & 0x7fffffu) << 29)));
    return __longlong_as_double((long long)(((unsigned long long)(b >> 31) << 63) |
                                            ((unsigned long long)(e - 127 + 1023) << 52) |
                                            ((unsigned long long)(b & 0x7fffffu) << 29)));
}

// h + l as a double, |l| <= |h| (a compensated FP32 pair), with integer
// operations: the low part is added to the high part's bit pattern in units of
// its last place (exact but for bits below the double's last place, which are
// cut).  An FP64 addition takes as long as 64 of these instructions here.
__device__ __forceinline__ double pair_to_f64(float h, float l) {
    const float s = h + l, e = l - (s - h);
    const unsigned sb = __float_as_uint(s), eb = __float_as_uint(e);
    const int es = (int)((sb >> 23) & 0xff), ee = (int)((eb >> 23) & 0xff);
    if (es == 0 || es == 0xff) return f32_to_f64(s);
    unsigned long long v = ((unsigned long long)(es - 127 + 1023) << 52) | ((unsigned long long)(sb & 0x7fffffu) << 29);
    if (ee != 0) {
        const int sh = ee - es + 29;   // e = m 2^sh last places of s
        const unsigned m = (eb & 0x7fffffu) | 0x800000u;
        unsigned long long d = sh >= 0 ? (unsigned long long)m << min(sh, 30) : (sh > -32 ? (unsigned long long)(m >> -sh) : 0ull);
        const bool opp = ((sb ^ eb) >> 31) != 0;
        if (opp && (sb & 0x7fffffu) == 0) d <<= 1;   // below a power of two the places are half as wide
        v = opp ? v - d : v + d;
    }
    return __longlong_as_double((long long)(v | ((unsigned long long)(sb >> 31) << 63)));
}

// A scale factor x = (h + l) 2^e, h + l in [1, 2) to 2^-47, for compensated FP32
// results; |e| <= 800 (scale_pair: false beyond, or x not positive).
struct ScalePair {
    float h, l;
    int e;
};
// (h + l) x as a double
__device__ __forceinline__ double scaled_pair(float h, float l, ScalePair k) {
    const float p = h * k.h;
    const long long r = __double_as_longlong(pair_to_f64(p, fmaf(h, k.h, -p) + fmaf(h, k.l, l * k.h)));
    const int ex = (int)((r >> 52) & 0x7ff);
    return __longlong_as_double(ex == 0 || ex == 0x7ff ? r : r + ((long long)k.e << 52));
}
inline bool scale_pair(double x, ScalePair &k) {
    int e = 0;
    const double f = 2.0 * std::frexp(x, &e);   // x = f 2^(e - 1)
    k.h = (float)f;
    k.l = (float)(f - (double)k.h);
    k.e = e - 1;
    return f >= 1.0 && f < 2.0 && e > -800 && e < 800;
}

}  // namespace
}  // namespace gf
