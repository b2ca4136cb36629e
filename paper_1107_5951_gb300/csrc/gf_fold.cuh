// gf_fold.cuh -- mirror parities of expansion components and the staging of
// folded expansions in shared memory, shared by the translations between
// levels (gf_xlate.cu) and the SIMT M2L (gf_m2l.cu).  The symmetry itself is
// explained in gf_xlate.cu.
#pragma once

#include "gf_simd.cuh"

namespace gf {
namespace {

// Parity class of real component k (bit a: odd under the mirror of axis a).
// (sqrtf is exact enough for the degree: k + 1/2 is never a square.)
__device__ __forceinline__ int degree_of(int k) { return (int)sqrtf((float)k + 0.5f); }
__device__ __forceinline__ int parity_of(int k) {
    const int n = degree_of(k);
    const int ro = k - n * n, m = (ro + 1) >> 1, im = (ro > 0 && (ro & 1) == 0) ? 1 : 0;
    return ((m + im) & 1) | (im << 1) | (((n + m) & 1) << 2);
}

// In place: v[o] -> X_d = sum_o s_o(d) v[o] over the eight positions.
template <class T>
__device__ __forceinline__ void fold8(T (&v)[8]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (!((o >> a) & 1)) {
                const T lo = v[o], hi = v[o | (1 << a)];
                v[o] = hi + lo;
                v[o | (1 << a)] = hi - lo;
            }
}

// Shared-memory place of folded input j, class slot d, column c: columns in
// 16-byte groups, [j][group][slot][column of the group], so that the threads
// of a warp -- which read one group at up to eight different slots -- touch 128
// contiguous bytes.  The slot is XOR-ed with the group (and by the callers
// with a row number), which spreads the staging writes over the banks.
template <class T, int P>
struct Lay {
    static constexpr int G = P < 16 / (int)sizeof(T) ? P : 16 / (int)sizeof(T);   // columns per group
    static constexpr int NG = P / G;
    static __device__ __forceinline__ int at(int j, int d, int c) {
        const int q = c / G;
        return ((j * NG + q) * 8 + (d ^ (q & 7))) * G + c % G;
    }
};

// Sums of a thread's component for P columns; FP32 columns in packed pairs.
template <class T, int P>
struct Acc {
    static constexpr bool kPack = sizeof(T) == 4 && P > 1;
    static constexpr int G = Lay<T, P>::G;
    T v[kPack ? 1 : P];
    uint64_t w[kPack ? P / 2 : 1];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int c = 0; c < (kPack ? 1 : P); ++c) v[c] = T(0);
#pragma unroll
        for (int c = 0; c < (kPack ? P / 2 : 1); ++c) w[c] = 0;
    }
    // += t x[group q]
    __device__ __forceinline__ void add(int q, T t, const T *x) {
        if constexpr (kPack) {
            const uint64_t t2 = pk2(t, t);
            if constexpr (G == 4) {
                const ulonglong2 x4 = *reinterpret_cast<const ulonglong2 *>(x);
                w[2 * q] = fma2(t2, x4.x, w[2 * q]);
                w[2 * q + 1] = fma2(t2, x4.y, w[2 * q + 1]);
            } else {
                w[q] = fma2(t2, *reinterpret_cast<const uint64_t *>(x), w[q]);
            }
        } else if constexpr (G == 2) {
            const double2 x2 = *reinterpret_cast<const double2 *>(x);
            v[2 * q] = fma(t, (T)x2.x, v[2 * q]);
            v[2 * q + 1] = fma(t, (T)x2.y, v[2 * q + 1]);
        } else {
            v[q] = fma(t, x[0], v[q]);
        }
    }
    __device__ __forceinline__ T get(int c) const {
        if constexpr (kPack) {
            float a, b;
            up2(w[c / 2], a, b);
            return (c & 1) ? b : a;
        } else {
            return v[c];
        }
    }
};

// Four inputs [j0, j0 + 4) of a row as Tc (zeros when row < 0, and from K on:
// a row's padding may hold anything).
template <class Ts, class Tc>
__device__ __forceinline__ void load4(const Ts *in, int64_t row, int j0, int K, Tc (&v)[4]) {
    if constexpr (sizeof(Ts) == 4) {   // rows padded to 32 elements
        float4 x = row >= 0 ? __ldg(reinterpret_cast<const float4 *>(in + row + j0)) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (j0 + 4 > K) {
            x.w = 0.f;
            if (j0 + 2 >= K) x.z = 0.f;
            if (j0 + 1 >= K) x.y = 0.f;
        }
        v[0] = (Tc)x.x;
        v[1] = (Tc)x.y;
        v[2] = (Tc)x.z;
        v[3] = (Tc)x.w;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = row >= 0 && j0 + q < K ? (Tc)__ldg(in + row + j0 + q) : Tc(0);
    }
}

}  // namespace
}  // namespace gf
