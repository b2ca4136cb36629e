// gf_xlate.cu -- the translations between levels (M2M, L2L and their
// transposes) and the P2M of voxel leaves, folded by the mirror symmetry of
// the eight positions of a child in its parent.
//
// A mirror across a coordinate plane through the centre multiplies every real
// component of an expansion by +-1: component (n, m, Re / Im) by (-1)^m
// (x -> -x, Re; -(-1)^m for Im), by +1 / -1 (y -> -y, Re / Im) and by
// (-1)^(n + m) (z -> -z).  Its three signs form the component's parity class
// chi (one bit per axis, parity_of), and the operators of the eight child
// positions are mirror images of one of them,
//   T_o[i][j] = s_o(chi_i) s_o(chi_j) T_7[i][j],
// s_o(chi) = product over the axes on which position o lies on the negative
// side of (-1)^(bit of chi), T_7 the operator of the all-positive position.
// So the sum over the children of a parent needs one product instead of eight:
//   y[i] = sum_o sum_j T_o[i][j] x_o[j] = sum_j T_7[i][j] X_{chi_i ^ chi_j}[j],
//   X_d[j] = sum_o s_o(d) x_o[j]  (a Walsh-Hadamard transform of 8 values),
// and T_7 is triangular in the degree (an M2M output takes inputs of its
// degree and below, an L2L output of its degree and above), which halves the
// product again.  The same holds for the P2M: the 8^3 voxels below a parent of
// 4^3-voxel leaves, and the 4^3 voxels of a leaf, are eight mirrored octants,
// when the quadrature rule is its own mirror image.
//
// With a sixteenth of the arithmetic these stages need no tensor cores: the
// products run in FP32 (mixed precision, more exact than split TF32 operands)
// or FP64.  Small levels are bound by latency, large ones by the L1 data path
// and the children's rows.  Against batched 3xTF32 tensor-core products of all
// eight children (and unfolded FP64 sums): 464^3, p = 10, P2M 290 -> 213 us,
// the M2M of levels 5..2 225 -> 131 us, L2L 107 -> 69 us; 128^3, p = 14, FP64,
// P2M 1.37 -> 0.18 ms, M2M 13.3 -> 0.09 ms, L2L 1.7 -> 0.13 ms; 128^3, p = 12, 16
// models, M2M^T 3.1 -> 1.35 ms, L2L^T 3.0 -> 0.09 ms.
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "gf_fold.cuh"
#include "gf_m2l.cuh"

namespace gf {

namespace {

// s_o(chi) = -1 or +1
__device__ __forceinline__ bool mirror_neg(int chi, int o) { return __popc(chi & ~o & 7) & 1; }

// Threads of a block (FP64 sums take twice the registers).
template <class T>
constexpr int xlate_max() {
    return sizeof(T) == 8 ? 512 : 1024;
}

// Sums the blockDim.y partial sums of every (component, column), in order,
// through shared memory [column][part][component]; calls out(component,
// column, sum) once for each.  All threads call it after a __syncthreads()
// that ends the use of `red`.
template <class T, int P, class F>
__device__ __forceinline__ void merge_parts(const Acc<T, P> &acc, T *red, F out) {
    const int i = threadIdx.x, KT = blockDim.x, JS = blockDim.y;
#pragma unroll
    for (int c = 0; c < P; ++c) red[(c * JS + threadIdx.y) * KT + i] = acc.get(c);
    __syncthreads();
    for (int c = threadIdx.y; c < P; c += JS) {
        T s = red[c * JS * KT + i];
        for (int y = 1; y < JS; ++y) s += red[(c * JS + y) * KT + i];
        out(i, c, s);
    }
}

struct XArgs {
    const void *in;
    void *out;
    const void *tab;                // T_7, input component major [K][K]
    int K, ldk, B, kind;            // 0 M2M, 1 L2L, 2 M2M^T, 3 L2L^T
    uint32_t ncol;                  // output boxes times batch members
    int32_t plo[3], pn[3];          // M2M, M2M^T: parent block
    int32_t clo[3], cn[3];          // and child block
    const uint64_t *tkey;           // L2L: observer boxes of the level
    const int32_t *tparent;
    const int32_t *child;           // L2L^T: [box][8] child box or -1
    uint32_t *amax;                 // M2M: largest |output| of columns [alo, ahi) (float bits; may be null)
    uint32_t alo, ahi;
};

// Largest |v| over the warp's rows into *amax (NaN skipped, as fmaxf does).
__device__ __forceinline__ void amax_merge(uint32_t *amax, float am) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
    if ((threadIdx.x & 31) == 0 && am > 0.f) atomicMax(amax, __float_as_uint(am));
}

// Row of child o of column `col` (M2M: dense child block; L2L^T: the child
// table), or -1.
__device__ __forceinline__ int64_t child_row(const XArgs &a, uint32_t col, int o) {
    if (col >= a.ncol) return -1;
    const uint32_t box = col / (uint32_t)a.B, bb = col - box * a.B;
    if (a.kind == 0) {
        const uint32_t yz = box / (uint32_t)a.pn[0], px = box - yz * a.pn[0], pz = yz / (uint32_t)a.pn[1],
                       py = yz - pz * a.pn[1];
        const int32_t cx = 2 * ((int)px + a.plo[0]) + (o & 1) - a.clo[0],
                      cy = 2 * ((int)py + a.plo[1]) + ((o >> 1) & 1) - a.clo[1],
                      cz = 2 * ((int)pz + a.plo[2]) + (o >> 2) - a.clo[2];
        if (cx < 0 || cy < 0 || cz < 0 || cx >= a.cn[0] || cy >= a.cn[1] || cz >= a.cn[2]) return -1;
        return ((((int64_t)cz * a.cn[1] + cy) * a.cn[0] + cx) * a.B + bb) * a.ldk;
    }
    const int32_t ch = a.child[box * 8 + o];
    return ch >= 0 ? ((int64_t)ch * a.B + bb) * a.ldk : -1;
}

// Parent row and the child's position for column `col` of L2L / M2M^T (kShift: the
// column's own row, no signs).
template <bool kShift>
__device__ __forceinline__ int64_t parent_row(const XArgs &a, uint32_t col, int &o) {
    o = kShift ? 7 : 0;
    if (col >= a.ncol) return -1;
    if constexpr (kShift) return (int64_t)col * a.ldk;
    const uint32_t box = col / (uint32_t)a.B, bb = col - box * a.B;
    if (a.kind == 1) {
        o = (int)(a.tkey[box] & 7);
        return ((int64_t)a.tparent[box] * a.B + bb) * a.ldk;
    }
    const uint32_t yz = box / (uint32_t)a.cn[0], zc = yz / (uint32_t)a.cn[1];
    const int32_t x = a.clo[0] + (int)(box - yz * a.cn[0]), y = a.clo[1] + (int)(yz - zc * a.cn[1]), z = a.clo[2] + (int)zc;
    o = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
    return ((((int64_t)((z >> 1) - a.plo[2]) * a.pn[1] + (y >> 1) - a.plo[1]) * a.pn[0] + (x >> 1) - a.plo[0]) * a.B + bb) *
           a.ldk;
}

// Folded inputs of the block's P columns into shared memory (Lay): four
// inputs of one column per thread.  crow: [P][8] children's rows.
template <class Ts, class Tc, int P>
__device__ __forceinline__ void stage_fold(const XArgs &a, const int64_t *crow, Tc *xs, int tid, int nthr) {
    const Ts *in = reinterpret_cast<const Ts *>(a.in);
    const int ng = (a.K + 3) >> 2;
    for (int e = tid; e < ng * P; e += nthr) {
        const int c = e % P, g = e / P, j0 = 4 * g;
        Tc v[4][8];
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            Tc w[4];
            load4<Ts, Tc>(in, crow[c * 8 + o], j0, a.K, w);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q][o] = w[q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            fold8(v[q]);
            const int sw = parity_of(j0 + q) ^ (g & 7);
#pragma unroll
            for (int d = 0; d < 8; ++d) xs[Lay<Tc, P>::at(j0 + q, d ^ sw, c)] = v[q][d];
        }
    }
}

// Parent expansions of the block's P columns, their signs applied, as [j][P].
template <class Ts, class Tc, int P>
__device__ __forceinline__ void stage_spread(const XArgs &a, const int64_t *prow, const int *poct, Tc *xs, int tid,
                                             int nthr) {
    const Ts *in = reinterpret_cast<const Ts *>(a.in);
    const int ng = (a.K + 3) >> 2;
    for (int e = tid; e < ng * P; e += nthr) {
        const int c = e % P, j0 = 4 * (e / P);
        Tc v[4];
        load4<Ts, Tc>(in, prow[c], j0, a.K, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) xs[(j0 + q) * P + c] = mirror_neg(parity_of(j0 + q), poct[c]) ? -v[q] : v[q];
    }
}

// Children to parents (M2M; L2L^T), few columns or FP64: a block makes P
// columns (parent, batch member).  Thread (i, y) sums component i over every
// blockDim.y-th group of four inputs; the operator column of the thread
// streams from L1/L2 (coalesced over i) and serves the P columns.  Splitting
// the inputs over y shortens the chain of operator loads, which is what a
// level of a few hundred boxes takes its time for.
template <class Ts, class Tc, int P>
__global__ void __launch_bounds__(xlate_max<Tc>()) fold_kernel(XArgs a) {
    extern __shared__ __align__(16) unsigned char shraw[];
    Tc *xs = reinterpret_cast<Tc *>(shraw);   // folded inputs (Lay), then the partial sums
    __shared__ int64_t crow[P * 8];
    const int K = a.K, tid = threadIdx.y * blockDim.x + threadIdx.x, nthr = blockDim.x * blockDim.y;
    const uint32_t col0 = blockIdx.x * P;
    for (int e = tid; e < 8 * P; e += nthr) crow[e] = child_row(a, col0 + (e >> 3), e & 7);
    __syncthreads();
    stage_fold<Ts, Tc, P>(a, crow, xs, tid, nthr);
    __syncthreads();
    const int i = threadIdx.x, ic = min(i, K - 1);
    const int cls = parity_of(ic);
    // the warp's largest degree bounds its inputs (zero beyond a thread's own)
    const int n = degree_of(min(K - 1, i | 31));
    const int jmax = (n + 1) * (n + 1);
    const Tc *t = reinterpret_cast<const Tc *>(a.tab) + ic;
    Acc<Tc, P> acc;
    acc.zero();
    constexpr int G = Lay<Tc, P>::G, NG = Lay<Tc, P>::NG;
#pragma unroll 2
    for (int g = threadIdx.y; 4 * g < jmax; g += blockDim.y) {
        Tc tv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) tv[q] = 4 * g + q < jmax ? __ldg(t + (size_t)(4 * g + q) * K) : Tc(0);
        const int sl = cls ^ (g & 7);
#pragma unroll
        for (int u = 0; u < NG; ++u) {
            const Tc *x = xs + ((size_t)(4 * g * NG + u) * 8 + (sl ^ (u & 7))) * G;
#pragma unroll
            for (int q = 0; q < 4; ++q) acc.add(u, tv[q], x + q * 8 * P);
        }
    }
    __syncthreads();   // the folded inputs have been used
    float am = 0.f;
    Ts *out = reinterpret_cast<Ts *>(a.out);
    merge_parts<Tc, P>(acc, xs, [&](int k, int c, Tc sum) {
        const uint32_t col = col0 + c;
        if (col >= a.ncol) return;
        const Ts v = k < K ? (Ts)sum : Ts(0);
        if (k < a.ldk) out[(int64_t)col * a.ldk + k] = v;
        if (a.amax && col >= a.alo && col < a.ahi) am = fmaxf(am, fabsf((float)v));
    });
    if (a.amax) amax_merge(a.amax, am);
}

// Parents to children (L2L; M2M^T), added to the child's expansion, few
// columns or FP64: a block updates P columns (child, batch member) of any
// positions, thread (i, y) as above; the child's signs are applied to the
// staged parent expansion and to the result, so every column uses the same
// operator.
// kShift: the shift of a box's own expansion, stored (p2m_shift_run).
template <class Ts, class Tc, int P, bool kShift = false>
__global__ void __launch_bounds__(xlate_max<Tc>()) spread_kernel(XArgs a) {
    extern __shared__ __align__(16) unsigned char shraw[];
    Tc *xs = reinterpret_cast<Tc *>(shraw);   // [K rounded up to 4][P], then the partial sums
    __shared__ int64_t prow[P];
    __shared__ int poct[P];
    const int K = a.K, tid = threadIdx.y * blockDim.x + threadIdx.x, nthr = blockDim.x * blockDim.y;
    const uint32_t col0 = blockIdx.x * P;
    if (tid < P) prow[tid] = parent_row<kShift>(a, col0 + tid, poct[tid]);
    __syncthreads();
    stage_spread<Ts, Tc, P>(a, prow, poct, xs, tid, nthr);
    __syncthreads();
    const int i = threadIdx.x, ic = min(i, K - 1);
    const int cls = parity_of(ic);
    // the warp's inputs: from its lowest degree on (zero before a thread's own); kShift:
    // up to its highest
    const int n = kShift ? 0 : degree_of(min(K - 1, i & ~31));
    int jend = K;
    if constexpr (kShift) {
        const int top = degree_of(min(K - 1, i | 31)) + 1;
        jend = top * top;
    }
    const Tc *t = reinterpret_cast<const Tc *>(a.tab) + ic;
    Acc<Tc, P> acc;
    acc.zero();
    constexpr int G = Lay<Tc, P>::G, NG = Lay<Tc, P>::NG;
#pragma unroll 2
    for (int g = ((n * n) >> 2) + threadIdx.y; 4 * g < jend; g += blockDim.y) {
        Tc tv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) tv[q] = 4 * g + q < jend ? __ldg(t + (size_t)(4 * g + q) * K) : Tc(0);
#pragma unroll
        for (int u = 0; u < NG; ++u) {
            const Tc *x = xs + (size_t)4 * g * P + u * G;
#pragma unroll
            for (int q = 0; q < 4; ++q) acc.add(u, tv[q], x + q * P);
        }
    }
    __syncthreads();   // the staged inputs have been used
    Ts *out = reinterpret_cast<Ts *>(a.out);
    float am = 0.f;
    merge_parts<Tc, P>(acc, xs, [&](int k, int c, Tc sum) {
        if constexpr (kShift) {
            const uint32_t col = col0 + c;
            if (k >= a.ldk || col >= a.ncol) return;
            out[(int64_t)col * a.ldk + k] = k < K ? (Ts)sum : Ts(0);
            if (a.amax && k < K && col >= a.alo && col < a.ahi) am = fmaxf(am, fabsf((float)sum));
        } else {
            if (k >= K || col0 + c >= a.ncol) return;
            Ts *o = out + (int64_t)(col0 + c) * a.ldk + k;
            *o = (Ts)((Tc)*o + (mirror_neg(cls, poct[c]) ? -sum : sum));
        }
    });
    if constexpr (kShift)
        if (a.amax) amax_merge(a.amax, am);
}

// Parents to all their children (M2M^T) in FP64: with the inputs' classes kept
// apart, S_c[i] = sum over j of class c of T_7[i][j] x[j], child o takes
// s_o(chi_i) sum_c s_o(c) S_c[i]: one product and a transform of eight values
// serve the eight children.  Thread (i, y) sums classes y, y + blockDim.y, ...
// of component i for P parents.  Bound by the FP64 pipe; child by child
// (spread_kernel) 8,192 children at p = 12 took 295 us, now 102 us.
struct ClassPerm {
    const int *perm;   // components by class, ascending within one, -1: none
    int off[9];
};

template <class Ts, int P>
__global__ void __launch_bounds__(512) spread_all_kernel(XArgs a, ClassPerm cp) {
    extern __shared__ __align__(16) unsigned char shraw[];
    double *xs = reinterpret_cast<double *>(shraw);   // [K rounded up to 4][P], then [class][P][component]
    const int K = a.K, KT = blockDim.x, JS = blockDim.y, tid = threadIdx.y * KT + threadIdx.x, nthr = KT * JS;
    const uint32_t col0 = blockIdx.x * P;
    const Ts *in = reinterpret_cast<const Ts *>(a.in);
    const int ng = (K + 3) >> 2;
    for (int e = tid; e < ng * P; e += nthr) {
        const int c = e % P, j0 = 4 * (e / P);
        double v[4];
        load4<Ts, double>(in, col0 + c < a.ncol ? (int64_t)(col0 + c) * a.ldk : -1, j0, K, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) xs[(j0 + q) * P + c] = v[q];
    }
    __syncthreads();
    const int i = threadIdx.x, ic = min(i, K - 1);
    const int n = degree_of(min(K - 1, i & ~31));   // the warp's lowest degree
    const double *t = reinterpret_cast<const double *>(a.tab) + ic;
    constexpr int MC = 8;                           // classes per thread, at most
    double acc[MC][P];
#pragma unroll
    for (int m = 0; m < MC; ++m) {
#pragma unroll
        for (int c = 0; c < P; ++c) acc[m][c] = 0.0;
        const int cls = threadIdx.y + m * JS;
        if (cls >= 8) continue;
        int q = cp.off[cls];
        const int end = cp.off[cls + 1];
        while (q < end && __ldg(cp.perm + q) >= 0 && __ldg(cp.perm + q) < n * n) ++q;
#pragma unroll 4
        for (; q < end; ++q) {
            const int j = __ldg(cp.perm + q);
            if (j < 0) break;
            const double tv = __ldg(t + (size_t)j * K);
#pragma unroll
            for (int c = 0; c < P; ++c) acc[m][c] = fma(tv, xs[j * P + c], acc[m][c]);
        }
    }
    __syncthreads();   // the inputs have been used
#pragma unroll
    for (int m = 0; m < MC; ++m) {
        const int cls = threadIdx.y + m * JS;
        if (cls >= 8) continue;
#pragma unroll
        for (int c = 0; c < P; ++c) xs[(cls * P + c) * KT + i] = acc[m][c];
    }
    __syncthreads();
    if (i >= K) return;
    const int chi = parity_of(i);
    Ts *out = reinterpret_cast<Ts *>(a.out);
    for (int c = threadIdx.y; c < P; c += JS) {
        const uint32_t col = col0 + c;
        if (col >= a.ncol) continue;
        double v[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) v[d] = xs[(d * P + c) * KT + i];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
#pragma unroll
            for (int d = 0; d < 8; ++d)
                if (!((d >> ax) & 1)) {
                    const double even = v[d], odd = v[d | (1 << ax)];
                    v[d] = even - odd;
                    v[d | (1 << ax)] = even + odd;
                }
        const uint32_t box = col / (uint32_t)a.B, bb = col - box * a.B;
        const uint32_t yz = box / (uint32_t)a.pn[0], px = box - yz * a.pn[0], pz = yz / (uint32_t)a.pn[1],
                       py = yz - pz * a.pn[1];
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const int32_t cx = 2 * ((int)px + a.plo[0]) + (o & 1) - a.clo[0],
                          cy = 2 * ((int)py + a.plo[1]) + ((o >> 1) & 1) - a.clo[1],
                          cz = 2 * ((int)pz + a.plo[2]) + (o >> 2) - a.clo[2];
            if (cx < 0 || cy < 0 || cz < 0 || cx >= a.cn[0] || cy >= a.cn[1] || cz >= a.cn[2]) continue;
            Ts *d = out + ((((int64_t)cz * a.cn[1] + cy) * a.cn[0] + cx) * a.B + bb) * a.ldk + i;
            *d = (Ts)((double)*d + (mirror_neg(chi, o) ? -v[o] : v[o]));
        }
    }
}

// ---------------------------------------------------------------- many columns, FP32
// With thousands of columns the products are bound by reading operands out of
// shared memory and L1 (a 16-byte read per lane takes four cycles of the SM's
// 128-byte path, the eight multiply-adds that it feeds two), so a thread owns
// a tile: four components of one parity class (a quad; they share the folded
// inputs) times C columns.  Quads are ordered by degree, so that a warp's
// inputs stay bounded by the triangle.  The operator is stored [j][quad][4].
struct QuadArgs {
    const float *tq;      // [K rounded up to 4][4 nq], zero-padded
    const int *qk;        // [4 nq] component of each place, -1: none
    const int *info;      // [nq] class | lowest degree << 8 | highest degree << 16
    int nq;
};

// acc[o][pair] += t[o] x[pair] for C columns at x (16-byte groups `step` floats apart)
template <int C>
__device__ __forceinline__ void quad_fma(uint64_t (&acc)[4][C / 2], float4 t, const float *x, int step) {
    const uint64_t t0 = pk2(t.x, t.x), t1 = pk2(t.y, t.y), t2 = pk2(t.z, t.z), t3 = pk2(t.w, t.w);
#pragma unroll
    for (int u = 0; u < C / 4; ++u) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(x + u * step);
        acc[0][2 * u] = fma2(t0, v.x, acc[0][2 * u]);
        acc[0][2 * u + 1] = fma2(t0, v.y, acc[0][2 * u + 1]);
        acc[1][2 * u] = fma2(t1, v.x, acc[1][2 * u]);
        acc[1][2 * u + 1] = fma2(t1, v.y, acc[1][2 * u + 1]);
        acc[2][2 * u] = fma2(t2, v.x, acc[2][2 * u]);
        acc[2][2 * u + 1] = fma2(t2, v.y, acc[2][2 * u + 1]);
        acc[3][2 * u] = fma2(t3, v.x, acc[3][2 * u]);
        acc[3][2 * u + 1] = fma2(t3, v.y, acc[3][2 * u + 1]);
    }
}

// A thread's tile into rows os[col][ldk] (negated where neg(column) says so).
template <int C, class F>
__device__ __forceinline__ void quad_store(const uint64_t (&acc)[4][C / 2], const int *qk, float *os, int c0, int ldk,
                                           F neg) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const int k = qk[o];
        if (k < 0) continue;
#pragma unroll
        for (int u = 0; u < C / 2; ++u) {
            float x, y;
            up2(acc[o][u], x, y);
            os[(c0 + 2 * u) * ldk + k] = neg(c0 + 2 * u) ? -x : x;
            os[(c0 + 2 * u + 1) * ldk + k] = neg(c0 + 2 * u + 1) ? -y : y;
        }
    }
}

// Rows os[PB][ldk] (components from K on as zeros) to out, 16 bytes a thread,
// with the largest |value| of columns [alo, ahi).
__device__ __forceinline__ void rows_out(const float *os, float *out, uint32_t col0, uint32_t ncol, int PB, int K, int ldk,
                                         uint32_t *amax, uint32_t alo, uint32_t ahi) {
    float am = 0.f;
    const int n4 = ldk >> 2, nv = (int)min((uint32_t)PB, ncol - col0) * n4;
    for (int e = threadIdx.x; e < nv; e += blockDim.x) {
        const int c = e / n4, k = 4 * (e - c * n4);
        float4 v = *reinterpret_cast<const float4 *>(os + 4 * e);
        if (k >= K) v.x = 0.f;
        if (k + 1 >= K) v.y = 0.f;
        if (k + 2 >= K) v.z = 0.f;
        if (k + 3 >= K) v.w = 0.f;
        *reinterpret_cast<float4 *>(out + (int64_t)col0 * ldk + 4 * e) = v;
        if (amax && col0 + c >= alo && col0 + c < ahi)
            am = fmaxf(fmaxf(am, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
    }
    if (amax) amax_merge(amax, am);
}

constexpr int kFoldCols = 8, kSpreadCols = 32, kUpCols = 16;   // columns per block

__global__ void __launch_bounds__(160) fold_quad(XArgs a, QuadArgs q) {
    extern __shared__ __align__(16) unsigned char shraw[];
    float *xs = reinterpret_cast<float *>(shraw);   // folded inputs (Lay), then the rows
    __shared__ int64_t crow[kFoldCols * 8];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const uint32_t col0 = blockIdx.x * kFoldCols;
    for (int e = tid; e < 8 * kFoldCols; e += nthr) crow[e] = child_row(a, col0 + (e >> 3), e & 7);
    __syncthreads();
    stage_fold<float, float, kFoldCols>(a, crow, xs, tid, nthr);
    __syncthreads();
    const int on = tid < q.nq * (kFoldCols / 4), cg = on ? tid / q.nq : 0, quad = on ? tid - cg * q.nq : 0;
    const int info = q.info[quad], cls = info & 0xff;
    const int nmax = __reduce_max_sync(0xffffffffu, info >> 16), jmax = (nmax + 1) * (nmax + 1);
    uint64_t acc[4][2] = {};
    const float4 *t = reinterpret_cast<const float4 *>(q.tq) + quad;
#pragma unroll 2
    for (int g = 0; 4 * g < jmax; ++g) {
        const float *x = xs + ((4 * g * (kFoldCols / 4) + cg) * 8 + (cls ^ (g & 7) ^ cg)) * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u) quad_fma<4>(acc, __ldg(t + (4 * g + u) * q.nq), x + u * 8 * kFoldCols, 0);
    }
    __syncthreads();   // the folded inputs have been used
    if (on) quad_store<4>(acc, q.qk + 4 * quad, xs, 4 * cg, a.ldk, [](int) { return false; });
    __syncthreads();
    rows_out(xs, reinterpret_cast<float *>(a.out), col0, a.ncol, kFoldCols, a.K, a.ldk, a.amax, a.alo, a.ahi);
}

template <bool kShift>
__global__ void __launch_bounds__(320) spread_quad(XArgs a, QuadArgs q) {
    extern __shared__ __align__(16) unsigned char shraw[];
    float *xs = reinterpret_cast<float *>(shraw);   // [K rounded up to 4][kSpreadCols], then the rows
    __shared__ int64_t prow[kSpreadCols];
    __shared__ int poct[kSpreadCols];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const uint32_t col0 = blockIdx.x * kSpreadCols;
    if (tid < kSpreadCols) prow[tid] = parent_row<kShift>(a, col0 + tid, poct[tid]);
    __syncthreads();
    stage_spread<float, float, kSpreadCols>(a, prow, poct, xs, tid, nthr);
    __syncthreads();
    const int on = tid < q.nq * (kSpreadCols / 8), cg = on ? tid / q.nq : 0, quad = on ? tid - cg * q.nq : 0;
    const int info = q.info[quad], cls = info & 0xff;
    // inputs from the lowest output's degree on (kShift: up to the highest's)
    int g0 = 0, jend = a.K;
    if constexpr (kShift) {
        const int nmax = __reduce_max_sync(0xffffffffu, info >> 16);
        jend = (nmax + 1) * (nmax + 1);
    } else {
        const int nmin = __reduce_min_sync(0xffffffffu, (info >> 8) & 0xff);
        g0 = (nmin * nmin) >> 2;
    }
    uint64_t acc[4][4] = {};
    const float4 *t = reinterpret_cast<const float4 *>(q.tq) + quad;
#pragma unroll 2
    for (int g = g0; 4 * g < jend; ++g) {
        const float *x = xs + 4 * g * kSpreadCols + 8 * cg;
#pragma unroll
        for (int u = 0; u < 4; ++u) quad_fma<8>(acc, __ldg(t + (4 * g + u) * q.nq), x + u * kSpreadCols, 4);
    }
    __syncthreads();   // the staged inputs have been used
    if (on) quad_store<8>(acc, q.qk + 4 * quad, xs, 8 * cg, a.ldk, [&](int c) { return mirror_neg(cls, poct[c]); });
    __syncthreads();
    if constexpr (kShift) {
        rows_out(xs, reinterpret_cast<float *>(a.out), col0, a.ncol, kSpreadCols, a.K, a.ldk, a.amax, a.alo, a.ahi);
        return;
    }
    // rows added to the children's, 16 bytes a thread
    float *out = reinterpret_cast<float *>(a.out) + (int64_t)col0 * a.ldk;
    const int n4 = a.ldk >> 2, nv = (int)min((uint32_t)kSpreadCols, a.ncol - col0) * n4;
#pragma unroll 4
    for (int e = tid; e < nv; e += nthr) {
        const int k = 4 * (e % n4);
        const float4 v = *reinterpret_cast<const float4 *>(xs + 4 * e);
        float4 w = *reinterpret_cast<const float4 *>(out + 4 * e);
        if (k < a.K) w.x += v.x;
        if (k + 1 < a.K) w.y += v.y;
        if (k + 2 < a.K) w.z += v.z;
        if (k + 3 < a.K) w.w += v.w;
        *reinterpret_cast<float4 *>(out + 4 * e) = w;
    }
}

// ---------------------------------------------------------------- P2M
struct P2MArgs {
    const void *rho;                // up: the caller's grid [B][nz][ny][nx]
    const void *mass;               // leaf: [leaf][B][64]
    int64_t nvox;
    int32_t gn[3], voff[3];         // grid extent, its place in the tree (voxels)
    int32_t lo[3], n[3];            // up: the parents' block
    int64_t first;                  // leaf: first leaf
    uint32_t ncol;
    int B, K, ldk;
    const void *tab;                // [64][K]
    void *me;
    uint32_t *amax;                 // largest |output| of columns [alo, ahi)
    uint32_t alo, ahi;
    int *status;
};

// P2M into level L - 1, from the density grid: a block makes P columns
// (parent, batch member); a parent's 8^3 voxels are eight mirrored octants of
// 4^3, so after the fold a component takes 64 products (512 without).  A
// staging thread folds the four rows of eight voxels that mirror one (y, z)
// of the octant.
// kVec: FP32 grid whose rows and leaves are 4-voxel aligned (16-byte loads);
// otherwise voxel by voxel with bounds tests.
template <class T, bool kVec, int P>
__device__ __forceinline__ void stage_grid(const P2MArgs &a, int rho_f32, uint32_t col0, T *xs, int tid, int nthr) {
    bool bad = false;
    for (int e = tid; e < 16 * P; e += nthr) {
        const int c = e % P, yz = e / P, y = yz & 3, z = yz >> 2;
        const uint32_t col = col0 + c;
        const bool on = col < a.ncol;
        const uint32_t box = on ? col / (uint32_t)a.B : 0, bb = on ? col - box * a.B : 0;
        const uint32_t byz = box / (uint32_t)a.n[0], bz = byz / (uint32_t)a.n[1];
        const int32_t i0 = 8 * (a.lo[0] + (int)(box - byz * a.n[0])) - a.voff[0],
                      j0 = 8 * (a.lo[1] + (int)(byz - bz * a.n[1])) - a.voff[1], k0 = 8 * (a.lo[2] + (int)bz) - a.voff[2];
        T v[4][8];   // [x of the octant][position]
#pragma unroll
        for (int r = 0; r < 4; ++r) {   // row: bit 0 the y side, bit 1 the z side
            const int32_t j = j0 + ((r & 1) ? 4 + y : 3 - y), k = k0 + ((r >> 1) ? 4 + z : 3 - z);
            const bool in = on && j >= 0 && j < a.gn[1] && k >= 0 && k < a.gn[2];
            const int64_t base = (int64_t)bb * a.nvox + ((int64_t)k * a.gn[1] + j) * a.gn[0];
            T w[8];
            if constexpr (kVec) {
                const float *g = reinterpret_cast<const float *>(a.rho) + base;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int32_t i = i0 + 4 * h;
                    const float4 x = in && i >= 0 && i < a.gn[0] ? __ldg(reinterpret_cast<const float4 *>(g + i))
                                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
                    w[4 * h] = (T)x.x;
                    w[4 * h + 1] = (T)x.y;
                    w[4 * h + 2] = (T)x.z;
                    w[4 * h + 3] = (T)x.w;
                }
#pragma unroll
                for (int x = 0; x < 8; ++x) bad |= !isfinite(w[x]);
            } else {
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    const int32_t i = i0 + x;
                    w[x] = T(0);
                    if (in && i >= 0 && i < a.gn[0]) {
                        if (rho_f32) {
                            const float f = __ldg(reinterpret_cast<const float *>(a.rho) + base + i);
                            bad |= !isfinite(f);
                            w[x] = (T)f;
                        } else {
                            const double f = __ldg(reinterpret_cast<const double *>(a.rho) + base + i);
                            bad |= !isfinite(f);
                            w[x] = (T)f;
                        }
                    }
                }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                v[x][2 * r] = w[3 - x];
                v[x][2 * r + 1] = w[4 + x];
            }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            fold8(v[x]);
#pragma unroll
            for (int d = 0; d < 8; ++d) xs[Lay<T, P>::at(4 * yz + x, d ^ (yz & 7), c)] = v[x][d];
        }
    }
    if (bad) atomicOr(a.status, 1);
}

template <class T, bool kVec, int P>
__global__ void __launch_bounds__(xlate_max<T>()) p2m_up_fold(P2MArgs a, int rho_f32) {
    extern __shared__ __align__(16) unsigned char shraw[];
    T *xs = reinterpret_cast<T *>(shraw);   // folded densities (Lay), then the partial sums
    const int K = a.K, tid = threadIdx.y * blockDim.x + threadIdx.x, nthr = blockDim.x * blockDim.y;
    const uint32_t col0 = blockIdx.x * P;
    stage_grid<T, kVec, P>(a, rho_f32, col0, xs, tid, nthr);
    __syncthreads();
    const int i = threadIdx.x, ic = min(i, K - 1), cls = parity_of(ic);
    const T *t = reinterpret_cast<const T *>(a.tab) + ic;
    Acc<T, P> acc;
    acc.zero();
    constexpr int G = Lay<T, P>::G, NG = Lay<T, P>::NG;
#pragma unroll 2
    for (int g = threadIdx.y; g < 16; g += blockDim.y) {
        T tv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) tv[q] = __ldg(t + (size_t)(4 * g + q) * K);
        const int sl = cls ^ (g & 7);
#pragma unroll
        for (int u = 0; u < NG; ++u) {
            const T *x = xs + ((size_t)(4 * g * NG + u) * 8 + (sl ^ (u & 7))) * G;
#pragma unroll
            for (int q = 0; q < 4; ++q) acc.add(u, tv[q], x + q * 8 * P);
        }
    }
    __syncthreads();   // the folded densities have been used
    float am = 0.f;
    T *me = reinterpret_cast<T *>(a.me);
    merge_parts<T, P>(acc, xs, [&](int k, int c, T sum) {
        const uint32_t col = col0 + c;
        if (col >= a.ncol) return;
        const T v = k < K ? sum : T(0);
        if (k < a.ldk) me[(int64_t)col * a.ldk + k] = v;
        if (a.amax && col >= a.alo && col < a.ahi) am = fmaxf(am, fabsf((float)v));
    });
    if (a.amax) amax_merge(a.amax, am);
}

// The same for many columns in FP32, a quad of components times 8 columns per
// thread.
template <bool kVec>
__global__ void __launch_bounds__(160) p2m_up_quad(P2MArgs a, QuadArgs q, int rho_f32) {
    extern __shared__ __align__(16) unsigned char shraw[];
    float *xs = reinterpret_cast<float *>(shraw);   // folded densities (Lay), then the rows
    const int tid = threadIdx.x;
    const uint32_t col0 = blockIdx.x * kUpCols;
    stage_grid<float, kVec, kUpCols>(a, rho_f32, col0, xs, tid, blockDim.x);
    __syncthreads();
    const int on = tid < q.nq * (kUpCols / 8), cg = on ? tid / q.nq : 0, quad = on ? tid - cg * q.nq : 0;
    const int cls = q.info[quad] & 0xff;
    uint64_t acc[4][4] = {};
    const float4 *t = reinterpret_cast<const float4 *>(q.tq) + quad;
    const int s0 = 2 * cg;   // the thread's two 4-column groups: s0, s0 + 1
#pragma unroll 2
    for (int g = 0; g < 16; ++g) {
        const int sl = cls ^ (g & 7) ^ s0;   // s0 is even: group s0 + 1 sits at slot sl ^ 1
        const float *x = xs + ((4 * g * (kUpCols / 4) + s0) * 8 + sl) * 4;
        const int step = (8 + (sl ^ 1) - sl) * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u) quad_fma<8>(acc, __ldg(t + (4 * g + u) * q.nq), x + u * 8 * kUpCols, step);
    }
    __syncthreads();   // the folded densities have been used
    if (on) quad_store<8>(acc, q.qk + 4 * quad, xs, 8 * cg, a.ldk, [](int) { return false; });
    __syncthreads();
    rows_out(xs, reinterpret_cast<float *>(a.me), col0, a.ncol, kUpCols, a.K, a.ldk, a.amax, a.alo, a.ahi);
}

// P2M of the leaves [first, ...) from their 4^3 masses: eight mirrored
// octants of 2^3, eight products a component; a thread keeps its component's
// eight operator entries in registers.  Bound by writing the expansions.
constexpr int kLeafCols = 32;

template <class T>
__global__ void __launch_bounds__(320) p2m_leaf_fold(P2MArgs a) {
    using L = Lay<T, kLeafCols>;
    __shared__ __align__(16) T xs[8 * 8 * kLeafCols];
    const int K = a.K, tid = threadIdx.x;
    const uint32_t col0 = blockIdx.x * kLeafCols;
    const T *mass = reinterpret_cast<const T *>(a.mass) + (a.first * a.B + col0) * 64;
    for (int e = tid; e < 4 * kLeafCols; e += blockDim.x) {
        const int c = e % kLeafCols, yz = e / kLeafCols, y = yz & 1, z = yz >> 1;
        T v[2][8];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int yy = (r & 1) ? 2 + y : 1 - y, zz = (r >> 1) ? 2 + z : 1 - z;
            T w[4] = {T(0), T(0), T(0), T(0)};
            if (col0 + c < a.ncol) {
                const T *m = mass + (int64_t)c * 64 + (zz * 4 + yy) * 4;
                if constexpr (sizeof(T) == 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(m);
                    w[0] = x.x;
                    w[1] = x.y;
                    w[2] = x.z;
                    w[3] = x.w;
                } else {
#pragma unroll
                    for (int x = 0; x < 4; ++x) w[x] = m[x];
                }
            }
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                v[x][2 * r] = w[1 - x];
                v[x][2 * r + 1] = w[2 + x];
            }
        }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            fold8(v[x]);
#pragma unroll
            for (int d = 0; d < 8; ++d) xs[L::at(2 * yz + x, d ^ yz, c)] = v[x][d];
        }
    }
    __syncthreads();
    const int i = tid, ic = min(i, K - 1), cls = parity_of(ic);
    T t[8];
#pragma unroll
    for (int v = 0; v < 8; ++v)
        t[v] = __ldg(reinterpret_cast<const T *>(a.tab) +
                     (size_t)(((2 + (v >> 2)) * 4 + 2 + ((v >> 1) & 1)) * 4 + 2 + (v & 1)) * K + ic);
    float am = 0.f;
    T *me = reinterpret_cast<T *>(a.me) + a.first * a.B * a.ldk;
#pragma unroll 2
    for (int u = 0; u < L::NG; ++u) {
        Acc<T, L::G> acc;
        acc.zero();
#pragma unroll
        for (int v = 0; v < 8; ++v)
            acc.add(0, t[v], xs + ((v * L::NG + u) * 8 + (cls ^ (v >> 1) ^ (u & 7))) * L::G);
#pragma unroll
        for (int c = 0; c < L::G; ++c) {
            const uint32_t col = col0 + u * L::G + c;
            if (col >= a.ncol) break;
            const T v = i < K ? acc.get(c) : T(0);
            if (i < a.ldk) me[(int64_t)col * a.ldk + i] = v;
            if (a.amax && col >= a.alo && col < a.ahi) am = fmaxf(am, fabsf((float)v));
        }
    }
    if (a.amax) amax_merge(a.amax, am);
}

// Threads of a block: one per component, at least the row stride (padding is
// written as zeros).
inline int xlate_threads(int K, int ldk) { return (std::max(K, std::min(ldk, (K + 31) & ~31)) + 31) & ~31; }

// Input parts (blockDim.y): up to four.
template <class T>
dim3 xlate_block(int K, int ldk) {
    const int kt = xlate_threads(K, ldk);
    return dim3((unsigned)kt, (unsigned)std::min(4, xlate_max<T>() / kt));
}

// Columns per block: as many as leave a block for every SM (an operator
// element then serves that many columns), at most `most`.
inline int cols_per_block(int64_t ncol, int most) {
    int P = most;
    while (P > 1 && ncol < (int64_t)sm_count() * P) P >>= 1;
    return P;
}

// Shared memory: the staged inputs (`rows` of P columns), or the partial sums.
template <class T>
size_t xlate_smem(int rows, int P, dim3 blk) {
    return sizeof(T) * (size_t)P * std::max<size_t>(rows, (size_t)blk.x * blk.y);
}

// Whether `ncol` columns are enough for the tiled kernels: 32 for every SM.
// L2L of 12,500 columns, p = 12: split 57 us, tiled 42; M2M of 5,488: split 45,
// tiled 43; of 4,096: split 23 (L2L), below that the tiles leave SMs idle.
inline bool many_columns(int64_t ncol) { return ncol >= (int64_t)32 * sm_count(); }

QuadArgs quad_args(const Tables *T, const float *tq) {
    QuadArgs q;
    q.tq = tq;
    q.qk = T->quad_k;
    q.info = T->quad_info;
    q.nq = T->nquad;
    return q;
}

gf_status launch_fold_quad(const XArgs &a, const QuadArgs &q, cudaStream_t st) {
    const size_t shm = sizeof(float) * kFoldCols * std::max(8 * ((a.K + 3) & ~3), a.ldk);
    GF_TRY(ensure_smem(fold_quad, shm));
    fold_quad<<<ceil_div((int64_t)a.ncol, kFoldCols), (q.nq * (kFoldCols / 4) + 31) & ~31, shm, st>>>(a, q);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <bool kShift>
gf_status launch_spread_quad(const XArgs &a, const QuadArgs &q, cudaStream_t st) {
    const size_t shm = sizeof(float) * kSpreadCols * std::max((a.K + 3) & ~3, a.ldk);
    GF_TRY(ensure_smem(spread_quad<kShift>, shm));
    spread_quad<kShift><<<ceil_div((int64_t)a.ncol, kSpreadCols), (q.nq * (kSpreadCols / 8) + 31) & ~31, shm, st>>>(a, q);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class Ts, class Tc, int P>
gf_status launch_fold(const XArgs &a, cudaStream_t st) {
    const dim3 blk = xlate_block<Tc>(a.K, a.ldk);
    const size_t shm = xlate_smem<Tc>(8 * ((a.K + 3) & ~3), P, blk);
    GF_TRY((ensure_smem(fold_kernel<Ts, Tc, P>, shm)));
    fold_kernel<Ts, Tc, P><<<ceil_div((int64_t)a.ncol, P), blk, shm, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class Ts, class Tc, int P, bool kShift = false>
gf_status launch_spread(const XArgs &a, cudaStream_t st) {
    const dim3 blk = xlate_block<Tc>(a.K, a.ldk);
    const size_t shm = xlate_smem<Tc>((a.K + 3) & ~3, P, blk);
    GF_TRY((ensure_smem(spread_kernel<Ts, Tc, P, kShift>, shm)));
    spread_kernel<Ts, Tc, P, kShift><<<ceil_div((int64_t)a.ncol, P), blk, shm, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class Ts, int P>
gf_status launch_spread_all(const XArgs &a, const Tables *T, cudaStream_t st) {
    ClassPerm cp;
    cp.perm = T->cls_perm;
    for (int c = 0; c < 9; ++c) cp.off[c] = T->cls_off[c];
    const int kt = (a.K + 31) & ~31;
    const dim3 blk((unsigned)kt, kt <= 128 ? 4 : kt <= 256 ? 2 : 1);
    const size_t shm = sizeof(double) * P * std::max((size_t)8 * kt, (size_t)((a.K + 3) & ~3));
    GF_TRY((ensure_smem(spread_all_kernel<Ts, P>, shm)));
    spread_all_kernel<Ts, P><<<ceil_div((int64_t)a.ncol, P), blk, shm, st>>>(a, cp);
    GF_KERNEL_DONE();
    return GF_OK;
}

// The columns (from box `first`) of the output level's slabs that its M2L
// reads, when this forward's expansion writers take the M2L input maxima.
void amax_range(const FmmPlan *F, int l, int B, int64_t first, uint32_t *&amax, uint32_t &lo, uint32_t &hi) {
    const FmmLevel &lv = F->lev[l];
    const int64_t slab = lv.sn[0] * lv.sn[1];
    amax = F->amax_fused && lv.m2l_z1 >= lv.m2l_z0 ? F->tc_amax + l : nullptr;
    lo = amax ? (uint32_t)(std::max<int64_t>(0, lv.m2l_z0 * slab - first) * B) : 0;
    hi = amax ? (uint32_t)(std::max<int64_t>(0, (lv.m2l_z1 + 1) * slab - first) * B) : 0;
}

// Columns are indexed with 32 bits (a level's expansions would fill the
// device's memory long before).
gf_status check_columns(int64_t ncol, int level) {
    if (ncol <= (int64_t)0x7fffffff) return GF_OK;
    set_error("level %d holds too many expansions for one launch (%lld)", level, (long long)ncol);
    return GF_ERR_UNSUPPORTED;
}

}  // namespace

namespace {

// dst [(rows + 3) & ~3][4 nq] = the columns of src [rows][K] in quad order, zeros elsewhere
__global__ void permute_quads(const float *__restrict__ src, int rows, int K, const int *__restrict__ qk, int nq4,
                              float *__restrict__ dst) {
    const int j = blockIdx.x;
    for (int e = threadIdx.x; e < nq4; e += blockDim.x) {
        const int k = qk[e];
        dst[(size_t)j * nq4 + e] = j < rows && k >= 0 ? src[(size_t)j * K + k] : 0.f;
    }
}

}  // namespace

// The quad order of a degree and the FP32 operators in it.
gf_status xlate_prepare_tables(Tables *T, cudaStream_t st) {
    const int K = T->K;
    struct Quad {
        int cls, lo, hi, k[4];
    };
    std::vector<Quad> quads;
    for (int c = 0; c < 8; ++c) {
        int n = 0;
        for (int k = 0; k < K; ++k) {
            int deg = 0;
            while ((deg + 1) * (deg + 1) <= k) ++deg;
            const int ro = k - deg * deg, m = (ro + 1) >> 1, im = (ro > 0 && (ro & 1) == 0) ? 1 : 0;
            if ((((m + im) & 1) | (im << 1) | (((deg + m) & 1) << 2)) != c) continue;
            if (n % 4 == 0) quads.push_back(Quad{c, deg, deg, {-1, -1, -1, -1}});
            quads.back().k[n % 4] = k;
            quads.back().hi = deg;
            ++n;
        }
    }
    std::vector<int> perm;
    for (int c = 0; c < 8; ++c) {
        T->cls_off[c] = (int)perm.size();
        for (const Quad &q : quads)   // before the sort by degree: classes in turn, each a whole number of quads
            if (q.cls == c) perm.insert(perm.end(), q.k, q.k + 4);
    }
    T->cls_off[8] = (int)perm.size();
    GF_CUDA(cudaMalloc(&T->cls_perm, perm.size() * sizeof(int)));
    GF_TRY(upload_small(T->cls_perm, perm.data(), perm.size() * sizeof(int), st));
    std::stable_sort(quads.begin(), quads.end(), [](const Quad &x, const Quad &y) { return x.hi < y.hi; });
    T->nquad = (int)quads.size();
    std::vector<int> qk, info;
    for (const Quad &q : quads) {
        for (int o = 0; o < 4; ++o) qk.push_back(q.k[o]);
        info.push_back(q.cls | (q.lo << 8) | (q.hi << 16));
    }
    GF_CUDA(cudaMalloc(&T->quad_k, qk.size() * sizeof(int)));
    GF_CUDA(cudaMalloc(&T->quad_info, info.size() * sizeof(int)));
    GF_TRY(upload_small(T->quad_k, qk.data(), qk.size() * sizeof(int), st));
    GF_TRY(upload_small(T->quad_info, info.data(), info.size() * sizeof(int), st));
    const float *const tf[4] = {T->m2m_f, T->l2l_f, T->am2m_f, T->al2l_f};
    for (int kind = 0; kind < 4; ++kind)
        GF_TRY(xlate_quad_table(T, tf[kind] + (size_t)7 * K * K, K, &T->quad_f[kind], st));
    return GF_OK;
}

gf_status xlate_quad_table(const Tables *T, const float *src, int rows, float **dst, cudaStream_t st) {
    const int r4 = (rows + 3) & ~3, nq4 = 4 * T->nquad;
    if (cudaMalloc(dst, sizeof(float) * (size_t)r4 * nq4) != cudaSuccess) {
        cudaGetLastError();
        *dst = nullptr;
        set_error("cannot allocate an operator table");
        return GF_ERR_OOM;
    }
    permute_quads<<<r4, 128, 0, st>>>(src, rows, T->K, T->quad_k, nq4, *dst);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class Ts, class Tc>
gf_status translate_run(gf_plan_s *plan, int level, int kind, int B, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &lv = F->lev[level];
    const Tables *T = F->tab;
    XArgs a;
    memset(&a, 0, sizeof(a));
    a.K = F->K;
    a.ldk = F->KS;
    a.B = B;
    a.kind = kind;
    const double *const td[4] = {T->m2m_d, T->l2l_d, T->am2m_d, T->al2l_d};
    const float *const tf[4] = {T->m2m_f, T->l2l_f, T->am2m_f, T->al2l_f};
    const size_t t7 = (size_t)7 * F->K * F->K;
    a.tab = sizeof(Tc) == 8 ? (const void *)(td[kind] + t7) : (const void *)(tf[kind] + t7);
    const FmmLevel &up = kind == 0 || kind == 3 ? lv : F->lev[level - 1];
    const FmmLevel &dn = kind == 0 || kind == 3 ? F->lev[level + 1] : lv;
    for (int d = 0; d < 3; ++d) {
        a.plo[d] = (int32_t)up.slo[d];
        a.pn[d] = (int32_t)up.sn[d];
        a.clo[d] = (int32_t)dn.slo[d];
        a.cn[d] = (int32_t)dn.sn[d];
    }
    const int64_t ncol = (kind == 0 ? up.ns : kind == 1 ? dn.nt : kind == 2 ? dn.ns : up.nt) * B;
    if (ncol == 0) return GF_OK;
    GF_TRY(check_columns(ncol, level));
    a.ncol = (uint32_t)ncol;
    if (kind == 0) {
        a.in = dn.me;
        a.out = up.me;
        amax_range(F, level, B, 0, a.amax, a.alo, a.ahi);
    } else if (kind == 1) {
        a.in = up.le;
        a.out = dn.le;
        a.tkey = dn.tkey;
        a.tparent = dn.tparent;
    } else if (kind == 2) {
        a.in = up.me;
        a.out = dn.me;
    } else {
        a.in = dn.le;
        a.out = up.le;
        a.child = F->child[level];
    }
    if (sizeof(Ts) == 4 && sizeof(Tc) == 4 && many_columns(ncol)) {
        const QuadArgs q = quad_args(T, T->quad_f[kind]);
        return kind == 0 || kind == 3 ? launch_fold_quad(a, q, st) : launch_spread_quad<false>(a, q, st);
    }
    if (kind == 2 && sizeof(Tc) == 8) {   // by parents: every child of the dense blocks is updated
        const int64_t np = up.ns * B;
        a.ncol = (uint32_t)np;
        return np >= 2 * (int64_t)sm_count() ? launch_spread_all<Ts, 2>(a, T, st) : launch_spread_all<Ts, 1>(a, T, st);
    }
    if (kind == 0 || kind == 3) {
        switch (cols_per_block(ncol, sizeof(Tc) == 8 ? 4 : 8)) {
            case 1: return launch_fold<Ts, Tc, 1>(a, st);
            case 2: return launch_fold<Ts, Tc, 2>(a, st);
            case 4: return launch_fold<Ts, Tc, 4>(a, st);
            default: return launch_fold<Ts, Tc, 8>(a, st);
        }
    }
    switch (cols_per_block(ncol, sizeof(Tc) == 8 ? 8 : 16)) {
        case 1: return launch_spread<Ts, Tc, 1>(a, st);
        case 2: return launch_spread<Ts, Tc, 2>(a, st);
        case 4: return launch_spread<Ts, Tc, 4>(a, st);
        case 8: return launch_spread<Ts, Tc, 8>(a, st);
        default: return launch_spread<Ts, Tc, 16>(a, st);
    }
}

template gf_status translate_run<float, float>(gf_plan_s *, int, int, int, cudaStream_t);
template gf_status translate_run<float, double>(gf_plan_s *, int, int, int, cudaStream_t);
template gf_status translate_run<double, double>(gf_plan_s *, int, int, int, cudaStream_t);

bool p2m_fold_ok(const gf_plan_s *plan) {
    const FmmPlan *F = plan->fmm;
    if (F->points || F->b != 4 || !F->p2m_up_d) return false;
    return (plan->opt.reserved0 & GF_FLAG_SUM_AN) || rule_mirrors(plan->quad);   // (SUM-AN: exact voxel moments)
}

bool rule_mirrors(const QuadRule &q) {
    for (int a = 0; a < 3; ++a)   // the rule mirrored across axis a is the same set of nodes and weights
        for (int s = 0; s < q.nq; ++s) {
            bool found = false;
            for (int t = 0; t < q.nq && !found; ++t) {
                found = q.wn[t] == q.wn[s];
                for (int d = 0; d < 3; ++d) found = found && q.xi[t][d] == (d == a ? -q.xi[s][d] : q.xi[s][d]);
            }
            if (!found) return false;
        }
    return true;
}

static P2MArgs p2m_args(gf_plan_s *plan, int B, int level, int64_t first) {
    FmmPlan *F = plan->fmm;
    P2MArgs a;
    memset(&a, 0, sizeof(a));
    a.B = B;
    a.K = F->K;
    a.ldk = F->KS;
    a.me = F->lev[level].me;
    amax_range(F, level, B, first, a.amax, a.alo, a.ahi);
    if (F->shift_f[0]) {   // p2m_shift_run makes the expansions
        a.me = tc_split_rows(F, level);
        a.amax = nullptr;
    }
    a.status = plan->d_status;
    return a;
}

template <class T>
gf_status p2m_leaf_run(gf_plan_s *plan, int B, int64_t first, int64_t count, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    if (count <= 0) return GF_OK;
    P2MArgs a = p2m_args(plan, B, F->L, first);
    a.mass = F->mass;
    a.first = first;
    GF_TRY(check_columns(count * B, F->L));
    a.ncol = (uint32_t)(count * B);
    a.tab = sizeof(T) == 8 ? (const void *)F->p2m_d : (const void *)(F->shift_f[0] ? F->p2m_c_f : F->p2m_f);
    p2m_leaf_fold<T><<<ceil_div(a.ncol, kLeafCols), xlate_threads(a.K, a.ldk), 0, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class T>
gf_status p2m_up_run(gf_plan_s *plan, const void *rho, int rho_f32, int B, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &pa = F->lev[F->L - 1];
    P2MArgs a = p2m_args(plan, B, F->L - 1, 0);
    a.rho = rho;
    a.nvox = plan->nvox;
    bool vec = rho_f32 && ((uintptr_t)rho & 15) == 0;
    for (int d = 0; d < 3; ++d) {
        a.gn[d] = (int32_t)plan->grid.n[d];
        a.voff[d] = (int32_t)F->voff[d];
        a.lo[d] = (int32_t)pa.slo[d];
        a.n[d] = (int32_t)pa.sn[d];
    }
    // 16-byte loads of four voxels along x: rows of whole pieces, at whole pieces of the tree
    vec = vec && a.gn[0] % 4 == 0 && a.voff[0] % 4 == 0;
    GF_TRY(check_columns(pa.ns * B, F->L - 1));
    a.ncol = (uint32_t)(pa.ns * B);
    a.tab = sizeof(T) == 8 ? (const void *)F->p2m_up_d : (const void *)F->p2m_up_f;
    if (sizeof(T) == 4 && many_columns(a.ncol)) {
        const QuadArgs q = quad_args(F->tab, F->p2m_up_q);
        const size_t shm = sizeof(float) * kUpCols * std::max(64 * 8, a.ldk);
        const int threads = (q.nq * (kUpCols / 8) + 31) & ~31;
        const unsigned grid = ceil_div((int64_t)a.ncol, kUpCols);
        if (vec)
            p2m_up_quad<true><<<grid, threads, shm, st>>>(a, q, rho_f32);
        else
            p2m_up_quad<false><<<grid, threads, shm, st>>>(a, q, rho_f32);
        GF_KERNEL_DONE();
        return GF_OK;
    }
    const dim3 blk = xlate_block<T>(a.K, a.ldk);
#define GF_UP_LAUNCH(V, P)                                                                        \
    do {                                                                                          \
        const size_t shm = xlate_smem<T>(64 * 8, P, blk);                                         \
        GF_TRY((ensure_smem(p2m_up_fold<T, V, P>, shm)));                                         \
        p2m_up_fold<T, V, P><<<ceil_div((int64_t)a.ncol, P), blk, shm, st>>>(a, rho_f32);          \
    } while (0)
    if (vec)
        GF_UP_LAUNCH(true, 4);
    else
        GF_UP_LAUNCH(false, 4);
#undef GF_UP_LAUNCH
    GF_KERNEL_DONE();
    return GF_OK;
}

// A source moved by d moves its expansion by a triangular operator of d alone (the
// M2M without the change of scale), and every voxel moves by the same nodes: so the
// expansions of any rule are those of the voxel centres, which mirror, times one
// matrix, the nodes' weighted sum.  One node off the centre, 464^3, p = 10: the forward
// 3,022 us with the leaf P2M of every leaf (1,458 with a P2M on the tensor cores), now
// 1,463; 232^3 646 (543), now 460.
gf_status p2m_shift_run(gf_plan_s *plan, int B, int level, int64_t first, int64_t count, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    if (count <= 0) return GF_OK;
    const int which = level == F->L ? 0 : 1;
    const int64_t at = first * B * F->KS;
    XArgs a;
    memset(&a, 0, sizeof(a));
    a.in = tc_split_rows(F, level) + at;
    a.out = (float *)F->lev[level].me + at;
    a.tab = F->shift_f[which];
    a.K = F->K;
    a.ldk = F->KS;
    a.B = B;
    GF_TRY(check_columns(count * B, level));
    a.ncol = (uint32_t)(count * B);
    amax_range(F, level, B, first, a.amax, a.alo, a.ahi);
    if (many_columns(a.ncol)) return launch_spread_quad<true>(a, quad_args(F->tab, F->shift_q[which]), st);
    switch (cols_per_block(a.ncol, 16)) {
        case 1: return launch_spread<float, float, 1, true>(a, st);
        case 2: return launch_spread<float, float, 2, true>(a, st);
        case 4: return launch_spread<float, float, 4, true>(a, st);
        case 8: return launch_spread<float, float, 8, true>(a, st);
        default: return launch_spread<float, float, 16, true>(a, st);
    }
}

template gf_status p2m_leaf_run<float>(gf_plan_s *, int, int64_t, int64_t, cudaStream_t);
template gf_status p2m_leaf_run<double>(gf_plan_s *, int, int64_t, int64_t, cudaStream_t);
template gf_status p2m_up_run<float>(gf_plan_s *, const void *, int, int, cudaStream_t);
template gf_status p2m_up_run<double>(gf_plan_s *, const void *, int, int, cudaStream_t);

}  // namespace gf
