// gf_points.cu -- weighted point sources: the quadrature points of deformed
// hexahedral cells (the general SUM-G1 of Sec. 2.1, integrated in reference
// coordinates with the Jacobian of each cell's map) and scattered density
// points with their volumes (Sec. 4: the FMM takes a random point
// distribution once each point carries the volume of its Voronoi cell).
//
// Source s sits at x_s with volume weight a_s and samples density c(s) =
// s / per_cell; its mass is rho_{c(s)} a_s and the field is Eq. 7 over the
// sources,
//
//   g(r) = G sum_s rho_{c(s)} a_s (r - x_s) / |r - x_s|^3,
//
// by direct summation (FP64 with compensated tile sums; mixed precision with
// positions split into an exact integer part and a fraction of a fixed
// quantum) or by the FMM.  The FMM's tree is uniform: the leaf side is chosen
// from the sources' extent so that about kPointsPerLeaf sources share a leaf
// when they fill it; the sources are sorted by the linear index of their leaf
// in the dense block of source leaves, and every leaf records its first
// sorted source.  The observer tree, M2M, M2L, L2L and L2P are those of the
// voxel FMM (in leaf units: the plan's length unit is the leaf side), so
// only the P2M (harmonics of each point) and the near field (each
// neighbour leaf's points) are specific to points.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <vector>

#include "fmm_math.cuh"
#include "gf_fmm.cuh"
#include "gf_pair.cuh"
#include "gf_prim.cuh"
#include "gf_simd.cuh"

namespace gf {
namespace {

constexpr double kPointsPerLeaf = 48.0;

// ---------------------------------------------------------------- hexahedra
// Quadrature point q of cell c: the trilinear image of the reference node
// xi_q, and its volume weight 8 (w_q / sum w) |det dx/dxi| (corner a = i +
// 2 j + 4 k of the cell at reference signs (2i - 1, 2j - 1, 2k - 1)).
__global__ void hex_sources_kernel(const double *__restrict__ verts, int64_t ncell, QuadRule qr,
                                   double *__restrict__ x, double *__restrict__ a) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ncell * qr.nq) return;
    const int64_t c = s / qr.nq;
    const int q = (int)(s - c * qr.nq);
    const double *X = verts + 24 * c;
    const double e0 = qr.xi[q][0], e1 = qr.xi[q][1], e2 = qr.xi[q][2];
    double p[3] = {0.0, 0.0, 0.0};
    double J[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const double s0 = (k & 1) ? 1.0 : -1.0, s1 = (k & 2) ? 1.0 : -1.0, s2 = (k & 4) ? 1.0 : -1.0;
        const double f0 = 1.0 + s0 * e0, f1 = 1.0 + s1 * e1, f2 = 1.0 + s2 * e2;
        const double N = 0.125 * f0 * f1 * f2;
        const double d0 = 0.125 * s0 * f1 * f2, d1 = 0.125 * f0 * s1 * f2, d2 = 0.125 * f0 * f1 * s2;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double v = X[3 * k + d];
            p[d] += N * v;
            J[d][0] += d0 * v;
            J[d][1] += d1 * v;
            J[d][2] += d2 * v;
        }
    }
    const double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                       J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                       J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
    for (int d = 0; d < 3; ++d) x[3 * s + d] = p[d];
    a[s] = 8.0 * qr.wn[q] * fabs(det);
}

// The same in FP32 relative to the cell's first corner, for mixed-precision
// plans: the corners' FP64 differences, rounded to FP32, give the trilinear
// image of each node and its Jacobian as tensor products (along xi, then eta,
// then zeta), and the image is added back to the first corner in FP64.  FP64 is
// slow on this GPU, so of its instructions only those additions are used (three
// a corner, three a node); conversions are integer operations.
//
// A block takes 32 cells: a thread per corner makes the differences (in shared
// memory), then a thread per node the image and weight; nodes leave through
// shared memory so that a warp's 32 of them are written as one piece.  Bound by
// the instruction issue and the integer pipe.  2^22 cells of 8 nodes: a thread
// per cell, reading and writing 192 bytes apart from lane to lane, in 64-bit
// fixed point 1,056 us; the same arithmetic in this layout 720 us; now 498 us.
struct HexRuleF {
    int nq;
    float xi[kMaxQuad][3];
    float w8[kMaxQuad];   // 8 w_q / sum(w)
};

constexpr int kHexCells = 32;
constexpr int kHexStride = 28;   // floats per cell: 16-byte pieces an odd number apart

__global__ void __launch_bounds__(kHexCells * 8)
hex_sources_fix(const double *__restrict__ verts, int64_t ncell, const __grid_constant__ HexRuleF qr,
                double *__restrict__ x, double *__restrict__ a) {
    __shared__ __align__(16) float sD[kHexCells * kHexStride];   // [cell][d][corner]
    __shared__ double sX[kHexCells][3];
    __shared__ float4 rule[kMaxQuad];   // xi, w8
    __shared__ double stage[kHexCells / 4][96];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t c0 = (int64_t)blockIdx.x * kHexCells;
    const int cells = (int)min((int64_t)kHexCells, ncell - c0);
    if (tid < qr.nq) rule[tid] = make_float4(qr.xi[tid][0], qr.xi[tid][1], qr.xi[tid][2], qr.w8[tid]);
    {
        const int cell = tid >> 3, v = tid & 7;
        const double *X = verts + 24 * (c0 + min(cell, cells - 1)) + 3 * v;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double x0 = __shfl_sync(0xffffffffu, X[d], lane & ~7);
            sD[cell * kHexStride + d * 8 + v] = f32_trunc(X[d] - x0);
            if (v == 0) sX[cell][d] = x0;
        }
    }
    __syncthreads();
    const int total = cells * qr.nq;
    double *out = stage[warp];
    for (int s0 = warp * 32; s0 < total; s0 += kHexCells * 8) {
        const int s = min(s0 + lane, total - 1);
        const int cell = s / qr.nq;
        const float4 ru = rule[s - cell * qr.nq];
        const float f0 = 0.5f * (1.f - ru.x), f1 = 0.5f * (1.f + ru.x);
        const float g0 = 0.5f * (1.f - ru.y), g1 = 0.5f * (1.f + ru.y);
        const float h0 = 0.5f * (1.f - ru.z), h1 = 0.5f * (1.f + ru.z);
        float J[3][3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float4 lo = *reinterpret_cast<const float4 *>(sD + cell * kHexStride + d * 8);
            const float4 hi = *reinterpret_cast<const float4 *>(sD + cell * kHexStride + d * 8 + 4);
            const float D[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            // along xi: e_jk and d/dxi for the four (eta, zeta) corners
            float e[4], ex[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                e[r] = f0 * D[2 * r] + f1 * D[2 * r + 1];
                ex[r] = 0.5f * (D[2 * r + 1] - D[2 * r]);
            }
            // along eta (r = j + 2 k)
            const float e0 = g0 * e[0] + g1 * e[1], e1 = g0 * e[2] + g1 * e[3];
            const float ex0 = g0 * ex[0] + g1 * ex[1], ex1 = g0 * ex[2] + g1 * ex[3];
            const float ey0 = 0.5f * (e[1] - e[0]), ey1 = 0.5f * (e[3] - e[2]);
            // along zeta
            const float p = h0 * e0 + h1 * e1;
            J[d][0] = h0 * ex0 + h1 * ex1;
            J[d][1] = h0 * ey0 + h1 * ey1;
            J[d][2] = 0.5f * (e1 - e0);
            out[3 * lane + d] = sX[cell][d] + f32_to_f64(p);
        }
        const float det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                          J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                          J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
        const int64_t first = c0 * qr.nq + s0;
        const int cnt = min(32, total - s0);
        if (lane < cnt) a[first + lane] = f32_to_f64(ru.w * fabsf(det));
        __syncwarp();
        for (int e = lane; e < 3 * cnt; e += 32) x[3 * first + e] = out[e];
        __syncwarp();
    }
}

// ---------------------------------------------------------------- direct
__device__ __forceinline__ double load_rho_p(const void *rho, int f32, int64_t i) {
    return f32 ? (double)__ldg(reinterpret_cast<const float *>(rho) + i) : __ldg(reinterpret_cast<const double *>(rho) + i);
}

// Tiles of 64 observers (two per lane); the warps of a cluster take the
// sources 32 at a time (gf_pair.cuh), each lane staging one with its mass
// rho_{c(s)} a_s of batch member blockIdx.y.  16 FP64 instructions a pair,
// bound by the FP64 pipe.
template <bool kSolo>
__global__ void __launch_bounds__(kSolo ? 32 : kPairThreads)
direct_points_f64(const double *__restrict__ obs, int64_t M, const double *__restrict__ src,
                  const double *__restrict__ wt, int64_t S, int per_cell, int64_t ncell, const void *__restrict__ rho,
                  int rho_f32, double G, double *__restrict__ g, double *__restrict__ gz, int *__restrict__ status) {
    __shared__ double2 red[kSolo ? 1 : (kPairWarps + 1) * 6 * 32];
    __shared__ __align__(16) double2 stage[kSolo ? 1 : kPairWarps][32][2];   // (x, y), (z, mass)
    const int C = kSolo ? 1 : (int)cooperative_groups::this_cluster().num_blocks();
    const int rank = kSolo ? 0 : (int)cooperative_groups::this_cluster().block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.y;
    const int64_t tile = blockIdx.x / C;
    double r[6], s[6], c[6], a[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
        const int64_t j = tile * 64 + (v / 3) * 32 + lane;
        r[v] = j < M ? obs[3 * j + v % 3] : 0.0;
        s[v] = c[v] = a[v] = 0.0;
    }
    bool bad = false;
    double2(*st)[2] = stage[warp];
    int since = 0;
    for (int64_t t0 = (int64_t)(rank * kPairWarps + warp) * 32; t0 < S; t0 += kSolo ? 32 : (int64_t)C * kPairThreads) {
        const int64_t i = t0 + lane;
        __syncwarp();
        if (i < S) {
            const double rv = load_rho_p(rho, rho_f32, (int64_t)b * ncell + i / per_cell);
            bad |= !isfinite(rv);
            st[lane][0] = make_double2(src[3 * i], src[3 * i + 1]);
            st[lane][1] = make_double2(src[3 * i + 2], rv * wt[i]);
        }
        __syncwarp();
        const int cnt = (int)min((int64_t)32, S - t0);
#pragma unroll 2
        for (int e = 0; e < cnt; ++e) {
            const double2 p = st[e][0], q = st[e][1];
#pragma unroll
            for (int u = 0; u < 6; u += 3) {
                const double dx = r[u] - p.x, dy = r[u + 1] - p.y, dz = r[u + 2] - q.x;
                const double k3 = inv_r3(fma(dx, dx, fma(dy, dy, dz * dz)), q.y);
                a[u] = fma(k3, dx, a[u]);
                a[u + 1] = fma(k3, dy, a[u + 1]);
                a[u + 2] = fma(k3, dz, a[u + 2]);
            }
        }
        since += cnt;
        if (since >= 256) {
            since = 0;
#pragma unroll
            for (int v = 0; v < 6; ++v) {
                two_sum_d(s[v], c[v], a[v]);
                a[v] = 0.0;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 6; ++v) two_sum_d(s[v], c[v], a[v]);
    if (bad && status && tile == 0) atomicOr(status, 1);
    auto put = [&](int v, int l, double tot) {
        const int64_t j = tile * 64 + (v / 3) * 32 + l;
        if (j < M) {
            if (g) g[((int64_t)b * M + j) * 3 + v % 3] = G * tot;
            if (gz && v % 3 == 2) gz[(int64_t)b * M + j] = G * tot;
        }
    };
    if constexpr (kSolo) {
#pragma unroll
        for (int v = 0; v < 6; ++v) put(v, lane, s[v] + c[v]);
    } else {
        const double tot = cluster_total<6>(s, c, red);
        if (rank == 0 && threadIdx.x < 6 * 32) put(threadIdx.x >> 5, lane, tot);
    }
}

// Positions in units of the quantum q from the corner lo, split into an
// integer part (exact in FP32 below 2^24) and the fraction.
__global__ void split_points(const double *__restrict__ x, int64_t n, double lo0, double lo1, double lo2,
                             double inv_q, float *__restrict__ xi, float *__restrict__ xf) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double lo[3] = {lo0, lo1, lo2};
    for (int a = 0; a < 3; ++a) {
        const double u = (x[3 * j + a] - lo[a]) * inv_q;
        const double fl = floor(u);
        xi[3 * j + a] = (float)fl;
        xf[3 * j + a] = (float)(u - fl);
    }
}

// Mixed precision: the separation (ri - si) + (rf - sf) in quanta is an exact
// integer difference plus one rounding; FP32 pair terms, compensated FP32
// sums of about 256 sources, FP64 beyond.  Sources are staged as packed pairs
// (f32x2), so one instruction does two pairs of an observer.
template <bool kSolo>
__global__ void __launch_bounds__(kSolo ? 32 : kPairThreads)
direct_points_mixed(const float *__restrict__ oi, const float *__restrict__ of, int64_t M,
                    const float *__restrict__ si, const float *__restrict__ sf, const double *__restrict__ wt,
                    int64_t S, int per_cell, int64_t ncell, const void *__restrict__ rho, int rho_f32, float q,
                    double Gq, double *__restrict__ g, double *__restrict__ gz, int *__restrict__ status) {
    __shared__ double2 red[kSolo ? 1 : (kPairWarps + 1) * 6 * 32];
    // per pair of sources: integer parts {x0,x1, y0,y1}, {z0,z1, m0,m1}, fractions {x, y}, {z, -}
    __shared__ __align__(16) float stage[kSolo ? 1 : kPairWarps][16 * 16];
    const int C = kSolo ? 1 : (int)cooperative_groups::this_cluster().num_blocks();
    const int rank = kSolo ? 0 : (int)cooperative_groups::this_cluster().block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.y;
    const int64_t tile = blockIdx.x / C;
    uint64_t RI[6], RF[6], A[6];
    float h[6], l[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
        const int64_t j = tile * 64 + (v / 3) * 32 + lane;
        const float x = j < M ? oi[3 * j + v % 3] : 0.f, f = j < M ? of[3 * j + v % 3] : 0.f;
        RI[v] = pk2(x, x);
        RF[v] = pk2(f, f);
        A[v] = 0;
        h[v] = l[v] = 0.f;
    }
    bool bad = false;
    const double inv_q3 = 1.0 / ((double)q * (double)q * (double)q);
    float *st = stage[warp];
    auto merge = [&]() {
#pragma unroll
        for (int v = 0; v < 6; ++v) {
            float x0, x1;
            up2(A[v], x0, x1);
            two_sum(h[v], l[v], x0 + x1);
            A[v] = 0;
        }
    };
    int since = 0;
    for (int64_t t0 = (int64_t)(rank * kPairWarps + warp) * 32; t0 < S; t0 += kSolo ? 32 : (int64_t)C * kPairThreads) {
        const int64_t i = t0 + lane;
        __syncwarp();
        {
            float *rec = st + (lane >> 1) * 16 + (lane & 1);
            float v[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // past the end: massless
            if (i < S) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    v[d] = si[3 * i + d];
                    v[4 + d] = sf[3 * i + d];
                }
                const double r = load_rho_p(rho, rho_f32, (int64_t)b * ncell + i / per_cell);
                bad |= !isfinite(r);
                v[3] = (float)(r * wt[i] * inv_q3);   // mass in quantum units
            }
#pragma unroll
            for (int d = 0; d < 7; ++d) rec[2 * d] = v[d];
        }
        __syncwarp();
        const int cnt = (int)min((int64_t)32, S - t0);
#pragma unroll 2
        for (int e = 0; e < (cnt + 1) / 2; ++e) {
            const ulonglong2 p0 = *reinterpret_cast<const ulonglong2 *>(st + 16 * e),
                             p1 = *reinterpret_cast<const ulonglong2 *>(st + 16 * e + 4),
                             p2 = *reinterpret_cast<const ulonglong2 *>(st + 16 * e + 8);
            const uint64_t p3 = *reinterpret_cast<const uint64_t *>(st + 16 * e + 12);
#pragma unroll
            for (int u = 0; u < 6; u += 3) {
                const uint64_t dx = add2(sub2(RI[u], p0.x), sub2(RF[u], p2.x));
                const uint64_t dy = add2(sub2(RI[u + 1], p0.y), sub2(RF[u + 1], p2.y));
                const uint64_t dz = add2(sub2(RI[u + 2], p1.x), sub2(RF[u + 2], p3));
                const uint64_t R2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
                float r0, r1;
                up2(R2, r0, r1);
                const uint64_t Q = pk2(rsqrt_ftz(r0), rsqrt_ftz(r1));
                float k0, k1;
                up2(mul2(mul2(Q, Q), mul2(Q, p1.y)), k0, k1);
                // a source on the observer contributes nothing
                const uint64_t K = pk2(r0 > 1e-37f ? k0 : 0.f, r1 > 1e-37f ? k1 : 0.f);
                A[u] = fma2(K, dx, A[u]);
                A[u + 1] = fma2(K, dy, A[u + 1]);
                A[u + 2] = fma2(K, dz, A[u + 2]);
            }
        }
        since += cnt;
        if (since >= 256) {
            since = 0;
            merge();
        }
    }
    merge();
    if (bad && status && tile == 0) atomicOr(status, 1);
    double s[6], c[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
        s[v] = (double)h[v];
        c[v] = (double)l[v];
    }
    auto put = [&](int v, int l, double tot) {
        const int64_t j = tile * 64 + (v / 3) * 32 + l;
        if (j < M) {
            if (g) g[((int64_t)b * M + j) * 3 + v % 3] = Gq * tot;
            if (gz && v % 3 == 2) gz[(int64_t)b * M + j] = Gq * tot;
        }
    };
    if constexpr (kSolo) {
#pragma unroll
        for (int v = 0; v < 6; ++v) put(v, lane, s[v] + c[v]);
    } else {
        const double tot = cluster_total<6>(s, c, red);
        if (rank == 0 && threadIdx.x < 6 * 32) put(threadIdx.x >> 5, lane, tot);
    }
}

// ---------------------------------------------------------------- FMM set-up
struct PtGeo {
    double lo[3], inv_s;
    int64_t slo[3], sn[3];         // dense block of source leaves
    float lof[3], isf;             // FP32 copies for the fast key path
    int fixk;                      // fixed-point frame of the tree (< 0: not used)
    long long lofix[3], halfleaf_fix;
    float fix_to_leaf;
};

// Leaf coordinate of a source along one axis: floor((x - lo) / s) as
// evaluated in FP64 with one rounded subtraction and one rounded
// multiplication, clamped to the block.  FP32 gives the same floor unless
// the value is within a few FP32 roundings of an integer; FP64 is used only
// there.
__device__ __forceinline__ int leaf_coord(double v, const PtGeo &g, int a) {
    float xf;
    const bool fin = trunc_f32(v, xf);
    const float qf = (xf - g.lof[a]) * g.isf;
    const float fl = floorf(qf);
    const float dist = fminf(qf - fl, fl + 1.f - qf);
    const float tol = ((fabsf(xf) + fabsf(g.lof[a])) * fabsf(g.isf) + fabsf(qf) + 1.f) * 2e-6f;
    const int c0 = (int)g.slo[a], c1 = (int)(g.slo[a] + g.sn[a] - 1);   // below 2^kMaxLevels
    int c;
    if (!fin || !(dist > tol)) {
        const double f = floor(__dmul_rn(__dsub_rn(v, g.lo[a]), g.inv_s));
        c = (int)fmin(fmax(f, (double)c0), (double)c1);
    } else {
        c = (int)fl;
    }
    return min(max(c, c0), c1);
}

// Linear index of each source's leaf in the dense block (which has fewer than
// 2^32 leaves).
__global__ void point_keys(const double *__restrict__ x, int64_t S, PtGeo g, uint32_t *__restrict__ keys,
                           int *__restrict__ status) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    int c[3];
    for (int a = 0; a < 3; ++a) {
        const double v = x[3 * s + a];
        if ((((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ff) == 0x7ff) atomicOr(status + 2, 1);
        c[a] = leaf_coord(v, g, a) - (int)g.slo[a];
    }
    keys[s] = ((uint32_t)c[2] * (uint32_t)g.sn[1] + (uint32_t)c[1]) * (uint32_t)g.sn[0] + (uint32_t)c[0];
}

// Sorted sources: offset from the own leaf's centre and volume, leaf units.
// The leaf comes from the sorted key.  FP32: the offset as an exact
// fixed-point difference (the frame of the observers' offsets) scaled to
// leaf units; FP64: (x - lo) / s - (c + 1/2).
template <class T>
__global__ void point_gather(const double *__restrict__ x, const double *__restrict__ wt,
                             const int32_t *__restrict__ perm, const uint32_t *__restrict__ keys, int64_t S, PtGeo g,
                             double inv_s3, T *__restrict__ loc, int *__restrict__ status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S) return;
    const int64_t s = perm[i];
    const uint32_t key = keys[i], row = key / (uint32_t)g.sn[0], slab = row / (uint32_t)g.sn[1];
    const int64_t c[3] = {g.slo[0] + (int64_t)(key - row * (uint32_t)g.sn[0]),
                          g.slo[1] + (int64_t)(row - slab * (uint32_t)g.sn[1]), g.slo[2] + (int64_t)slab};
    for (int a = 0; a < 3; ++a) {
        if constexpr (sizeof(T) == 4) {
            if (g.fixk >= 0) {
                const long long d = to_fix(x[3 * s + a], g.fixk) - (g.lofix[a] + (2 * c[a] + 1) * g.halfleaf_fix);
                loc[4 * i + a] = fix_to_f32(d) * g.fix_to_leaf;
                continue;
            }
        }
        const double u = (x[3 * s + a] - g.lo[a]) * g.inv_s;
        loc[4 * i + a] = (T)(u - ((double)c[a] + 0.5));
    }
    const double v = wt[s] * inv_s3;
    if (!isfinite(v)) atomicOr(status + 3, 1);
    if constexpr (sizeof(T) == 4) {
        float f;
        trunc_f32(v, f);
        loc[4 * i + 3] = f;
    } else {
        loc[4 * i + 3] = v;
    }
}

// First sorted source of every dense leaf: leaf_beg[l] = number of sources
// whose key is below l (keys sorted), by a binary search per leaf.
__global__ void point_leaf_beg(const uint32_t *__restrict__ keys, int64_t S, int64_t nleaf,
                               int64_t *__restrict__ beg) {
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l > nleaf) return;
    int64_t lo = 0, hi = S;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (keys[mid] < (uint32_t)l)
            lo = mid + 1;
        else
            hi = mid;
    }
    beg[l] = lo;
}

// ---------------------------------------------------------------- FMM forward
template <class T>
__device__ __forceinline__ void ld_loc(const T *loc, int64_t i, T &x, T &y, T &z, T &w) {
    if constexpr (sizeof(T) == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(loc) + i);
        x = v.x;
        y = v.y;
        z = v.z;
        w = v.w;
    } else {
        const double2 a = __ldg(reinterpret_cast<const double2 *>(loc) + 2 * i);
        const double2 b = __ldg(reinterpret_cast<const double2 *>(loc) + 2 * i + 1);
        x = a.x;
        y = a.y;
        z = b.x;
        w = b.y;
    }
}

// Sorted masses in leaf units: m_i = rho_{c(perm_i)} v_i, [B][S].
template <class T>
__global__ void point_masses(const void *__restrict__ rho, int rho_f32, const int32_t *__restrict__ perm,
                             const T *__restrict__ loc, int64_t S, int per_cell, int64_t ncell,
                             T *__restrict__ m, int *__restrict__ status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S) return;
    const int b = (int)blockIdx.y;
    const int64_t e = (int64_t)b * S + i;
    const int64_t src = (int64_t)b * ncell + perm[i] / per_cell;
    if constexpr (sizeof(T) == 4) {
        if (rho_f32) {   // one rounding of the product, without the FP64 pipe
            const float r = ((const float *)rho)[src];
            if (!isfinite(r)) atomicOr(status, 1);
            m[e] = r * loc[4 * i + 3];
            return;
        }
    }
    const double r = load_rho_p(rho, rho_f32, src);
    if (!isfinite(r)) atomicOr(status, 1);
    m[e] = (T)(r * (double)loc[4 * i + 3]);
}

// P2M over the points of each leaf: ME_n^m = sum_i m_i conj(R_n^m(x_i - c)),
// x_i - c the point's offset from the leaf centre (leaf units).
//
// R_n^m = s_nm (x + iy)^m Q_n^m(z, r^2) with a real Q that starts at Q_m^m = 1
// and follows Q_n = z Q_{n-1} - c_nm r^2 Q_{n-2}, c_nm = ((n-1)^2 - m^2) /
// ((2n-1)(2n-3)) (the regular harmonics' recursion divided by its leading
// coefficients, whose product is s_nm), so a term costs three operations for
// Q and one for each real component, and s_nm is applied to the sums.
//
// What bounds it is the FP32 (FP64) issue rate, so nothing is spent on a sum
// across lanes: a lane owns two orders of one leaf, m <= p/2 and p + 1 - m (p
// even; none beside m = 0) or p - m (p odd) -- p + 1 or p + 2 terms whatever m,
// held in registers -- and walks over the leaf's points.  A warp
// takes 32 / GL leaves at once, GL >= p/2 + 1 lanes each; a leaf of more than
// kP2MBig points is taken by the whole warp, its lane groups' sums added at the
// end.  The points come through shared memory, one entry (FP32: a pair of
// points) made by each lane at a time: z and r^2, and the mass-weighted powers
// of x + iy, 16 bytes each, read back by the lanes of a leaf without bank
// conflicts (their orders are neighbours, entries an odd number of 16 bytes
// apart).  FP32 sums run over two points at once as packed pairs.
// A lane per point, with the harmonics summed over the warp through shared
// memory, took 3,254 us for 2^25 points in leaves of 48 at p = 12.
constexpr int kP2MWarps = 4;
constexpr int kP2MBig = 256;    // points from which a leaf takes the whole warp
constexpr int kP2MSeg = 1024;   // points of such a leaf summed before its row is updated
__constant__ double c_ps[(kMaxP + 1) * (kMaxP + 1)];   // s_nm by real component

__device__ __forceinline__ uint64_t v_mul(uint64_t a, uint64_t b) { return mul2(a, b); }
__device__ __forceinline__ uint64_t v_fma(uint64_t a, uint64_t b, uint64_t c) { return fma2(a, b, c); }
__device__ __forceinline__ double v_mul(double a, double b) { return a * b; }
__device__ __forceinline__ double v_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float v_sum(uint64_t v) {
    float l, h;
    up2(v, l, h);
    return l + h;
}
__device__ __forceinline__ double v_sum(double v) { return v; }
__device__ __forceinline__ void v_dup(float c, uint64_t &v) { v = pk2(c, c); }
__device__ __forceinline__ void v_dup(double c, double &v) { v = c; }

// 16-byte shared-memory entries an odd number apart from point to point
inline __host__ __device__ int p2m_stride(int p) { return (p + 2) | 1; }

// NS >= terms of a lane; SW <= p - p/2 + 1, the first term at which a
// lane can turn to its second order (selects are what the ALU does here).
template <class T, int GL, int NS, int SW>
__global__ void __launch_bounds__(kP2MWarps * 32, NS <= (sizeof(T) == 4 ? 13 : 11) ? 4 : 3)
point_p2m(const T *__restrict__ loc, const T *__restrict__ mass, const int64_t *__restrict__ leaf_beg, int64_t nleaf,
          int64_t S, int p, int B, int ldk, T *__restrict__ me, uint32_t *__restrict__ amax, int64_t amax_lo,
          int64_t amax_hi) {
    extern __shared__ __align__(16) unsigned char shraw[];
    constexpr int NG = 32 / GL, PT = sizeof(T) == 4 ? 2 : 1;
    constexpr int PTS = PT * GL;   // points a lane group stages at a time
    using V = std::conditional_t<sizeof(T) == 4, uint64_t, double>;
    struct __align__(16) V2 {
        V a, b;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = lane / GL, tk = lane % GL;
    const int K = (p + 1) * (p + 1), steps = p % 2 ? p + 2 : p + 1, stride = p2m_stride(p);
    V2 *sh = reinterpret_cast<V2 *>(shraw) + (size_t)warp * 32 * stride;
    V2 *own = sh + lane * stride;               // the entry this lane stages
    const V2 *grp_sh = sh + grp * GL * stride;
    // orders of this lane; lanes beyond p / 2 repeat the last one's, unwritten
    const int m1 = min(tk, p / 2), m2 = p % 2 ? p - m1 : min(p, p + 1 - m1);
    const int sw = p - m1 + 1;   // term sw is the first of order m2 (p even, m1 = 0: beyond the last)
    V nc[NS];   // -c_nm of each term
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const int m = i < sw ? m1 : m2, n = i < sw ? m1 + i : m2 + i - sw;
        const T c = n >= m + 2 ? T((n - 1) * (n - 1) - m * m) / T((2 * n - 1) * (2 * n - 3)) : T(0);
        v_dup(-c, nc[i]);
    }
    V one;
    v_dup(T(1), one);
    __shared__ T sc[(kMaxP + 1) * (kMaxP + 1)];
    for (int k = threadIdx.x; k < K; k += blockDim.x) sc[k] = (T)c_ps[k];
    __syncthreads();
    float big_in = 0.f;   // largest |component| written in [amax_lo, amax_hi)

    V ar[NS], ai[NS];
    // add the points base + ((c step + off) PTS + PT tk + e), c < nchunk, below end
    auto add_points = [&](int64_t base, int64_t end, int nchunk, int step, int off, const T *mb) {
        for (int c = 0; c < nchunk; ++c) {
            const int64_t first = base + (int64_t)(c * step + off) * PTS, i0 = first + PT * tk;
            T x[PT], y[PT], z[PT], q[PT], w;
#pragma unroll
            for (int e = 0; e < PT; ++e) {
                x[e] = y[e] = z[e] = q[e] = T(0);
                if (i0 + e < end) {
                    ld_loc(loc, i0 + e, x[e], y[e], z[e], w);
                    q[e] = mb[i0 + e];
                }
            }
            V X, Y, NY, Z, WR, WI;
            if constexpr (PT == 2) {
                X = pk2(x[0], x[1]);
                Y = pk2(y[0], y[1]);
                NY = pk2(-y[0], -y[1]);
                Z = pk2(z[0], z[1]);
                WR = pk2(q[0], q[1]);
                WI = 0;
            } else {
                X = x[0];
                Y = y[0];
                NY = -y[0];
                Z = z[0];
                WR = q[0];
                WI = 0.0;
            }
            __syncwarp();   // the entries of the chunk before have been read
            own[0] = V2{Z, v_fma(Z, Z, v_fma(Y, Y, v_mul(X, X)))};
            own[1] = V2{WR, WI};
            for (int m = 1; m <= p; ++m) {
                const V nr = v_fma(X, WR, v_mul(NY, WI)), ni = v_fma(X, WI, v_mul(Y, WR));
                WR = nr;
                WI = ni;
                own[1 + m] = V2{WR, WI};
            }
            __syncwarp();
            // entries that hold points, over the warp's leaves
            const int64_t rest = end - first;
            const int mine = rest <= 0 ? 0 : (int)((min(rest, (int64_t)PTS) + PT - 1) / PT);
            const int cnt = __reduce_max_sync(0xffffffffu, mine);
            for (int e = 0; e < cnt; ++e) {
                const V2 *pe = grp_sh + e * stride;
                const V2 zr = pe[0], w1 = pe[1 + m1], w2 = pe[1 + m2];
                V wr = w1.a, wi = w1.b, Q = one, P = zr.b;   // P is multiplied by 0 first
#pragma unroll
                for (int i = 0; i < NS; ++i) {
                    if (i > 0) {
                        if (i >= steps) break;
                        const V n = v_fma(zr.a, Q, v_mul(v_mul(nc[i], zr.b), P));
                        P = Q;
                        Q = n;
                        if (i >= SW && i == sw) {
                            Q = one;
                            wr = w2.a;
                            wi = w2.b;
                        }
                    }
                    ar[i] = v_fma(wr, Q, ar[i]);
                    ai[i] = v_fma(wi, Q, ai[i]);
                }
            }
        }
    };
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < NS; ++i) v_dup(T(0), ar[i]), v_dup(T(0), ai[i]);
    };
    // the sums into row `leaf` (whole: all lane groups' sums into it; add: on top of it)
    auto write = [&](int64_t leaf, int bb, bool whole, bool add, bool last) {
        T *dst = me + (leaf * B + bb) * ldk;
        const bool on = leaf < nleaf && tk <= p / 2 && (!whole || grp == 0);
        const bool in = amax && leaf >= amax_lo && leaf < amax_hi && last;
        auto put = [&](int k, T v) {
            const T r = add ? dst[k] + v : v;
            dst[k] = r;
            if (in) big_in = fmaxf(big_in, fabsf((float)r));
        };
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            if (i >= steps) break;
            T re = v_sum(ar[i]), im = v_sum(ai[i]);
            if (whole) {
#pragma unroll
                for (int o = GL; o < 32; o *= 2) {
                    re += __shfl_xor_sync(0xffffffffu, re, o);
                    im += __shfl_xor_sync(0xffffffffu, im, o);
                }
            }
            const int m = i < sw ? m1 : m2, n = i < sw ? m1 + i : m2 + i - sw;
            if (on) {
                const int k = n * n + (m == 0 ? 0 : 2 * m - 1);
                put(k, sc[k] * re);
                if (m > 0) put(k + 1, -sc[k] * im);   // conj
            }
        }
        if (leaf < nleaf && (!whole || grp == 0))
            for (int k = K + tk; k < ldk; k += GL) dst[k] = T(0);
    };

    const int64_t nwarp = (int64_t)gridDim.x * kP2MWarps;
    for (int64_t leaf0 = ((int64_t)blockIdx.x * kP2MWarps + warp) * NG; leaf0 < nleaf; leaf0 += nwarp * NG) {
        const int64_t leaf = leaf0 + grp;
        const int64_t i0 = leaf < nleaf ? leaf_beg[leaf] : 0, i1 = leaf < nleaf ? leaf_beg[leaf + 1] : 0;
        const bool any_big = __any_sync(0xffffffffu, i1 - i0 > kP2MBig);
        for (int bb = 0; bb < B; ++bb) {
            const T *mb = mass + (int64_t)bb * S;
            if (!any_big) {
                clear();
                const int n = __reduce_max_sync(0xffffffffu, (int)((i1 - i0 + PTS - 1) / PTS));
                add_points(i0, i1, n, 1, 0, mb);
                write(leaf, bb, false, false, true);
                continue;
            }
            for (int q = 0; q < NG; ++q) {
                const int64_t b0 = __shfl_sync(0xffffffffu, (long long)i0, q * GL);
                const int64_t b1 = __shfl_sync(0xffffffffu, (long long)i1, q * GL);
                if (leaf0 + q >= nleaf) break;
                for (int64_t s0 = b0;; s0 += kP2MSeg) {
                    const int64_t s1 = min(b1, s0 + kP2MSeg);
                    clear();
                    add_points(s0, s1, (int)((s1 - s0 + NG * PTS - 1) / (NG * PTS)), NG, grp, mb);
                    write(leaf0 + q, bb, true, s0 > b0, s1 == b1);
                    if (s1 == b1) break;
                }
            }
        }
    }
    if (amax) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) big_in = fmaxf(big_in, __shfl_xor_sync(0xffffffffu, big_in, o));
        if (lane == 0 && big_in > 0.f) atomicMax(amax, __float_as_uint(big_in));
    }
}

template <class T, int GL, int NS, int SW>
gf_status launch_point_p2m(const gf_plan_s *plan, int B, uint32_t *amax, int64_t lo, int64_t hi, cudaStream_t st) {
    const FmmPlan *F = plan->fmm;
    const PointSet &P = plan->pts;
    const FmmLevel &lv = F->lev[F->L];
    const size_t shm = (size_t)kP2MWarps * 32 * p2m_stride(F->p) * 16;
    GF_TRY((ensure_smem(point_p2m<T, GL, NS, SW>, shm)));
    const int64_t per_block = kP2MWarps * (32 / GL);
    const unsigned grid = (unsigned)std::min<int64_t>((lv.ns + per_block - 1) / per_block, 152 * 64);
    point_p2m<T, GL, NS, SW><<<grid, kP2MWarps * 32, shm, st>>>((const T *)P.loc, (const T *)F->mass, P.leaf_beg, lv.ns,
                                                            P.S, F->p, B, F->KS, (T *)lv.me, amax, lo, hi);
    GF_KERNEL_DONE();
    return GF_OK;
}

// Near field over the points of the 27 neighbour leaves + the L2P gradient
// of the leaf's local expansion + near + far in FP64, scattered to caller
// order.  One warp per work item (at most 64 observers of one leaf), two
// observers per lane.  A neighbour leaf's points are staged 64 at a time in
// the warp's shared-memory slice, as offsets from the item's leaf centre
// with their masses.  FP32: pairs of points as {x0,x1, y0,y1, z0,z1, m0,m1}
// and each observer duplicated, so one packed instruction does two pairs;
// the L2P evaluates the lane's two observers as one packed pair.
constexpr int kPtWarps = 4;
constexpr int kPtChunk = 64;

// Elements of a warp's slice (a multiple of 8): staged points, the three
// gradient expansions (FP32: duplicated pairs), 27 neighbour leaves (int64).
inline __host__ __device__ int pt_slice(int P2, int tsize) {
    const int dmul = tsize == 4 ? 2 : 1;
    return (4 * kPtChunk + 3 * dmul * P2 + 27 * (8 / tsize) + 7) & ~7;
}

struct PtEvalArgs {
    const int4 *items;
    int64_t n_items;
    const uint64_t *tkey;
    const int32_t *perm;
    const void *tloc;
    const void *loc;           // [S][4] sorted sources: offset from own leaf centre, volume
    const void *mass;          // [B][S] sorted masses (leaf units)
    const int64_t *leaf_beg;   // [nleaf + 1]
    const void *le;
    PtGeo g;
    int L, B, p, ldk;
    int64_t S, M;
    uint32_t part_lo, part_hi;
    double scale, eps2;
    double *gout, *gz;
};

template <class T>
__global__ void __launch_bounds__(kPtWarps * 32) point_eval(PtEvalArgs a) {
    extern __shared__ unsigned char shraw[];
    constexpr bool kF32 = sizeof(T) == 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P2 = a.p * a.p;
    T *wsh = reinterpret_cast<T *>(shraw) + (size_t)warp * pt_slice(P2, sizeof(T));
    T *Dx = wsh + 4 * kPtChunk, *Dy = Dx + (kF32 ? 2 : 1) * P2, *Dz = Dy + (kF32 ? 2 : 1) * P2;
    int64_t *nbl = reinterpret_cast<int64_t *>(Dz + (kF32 ? 2 : 1) * P2);
    const T *tloc = reinterpret_cast<const T *>(a.tloc);
    const T *loc = reinterpret_cast<const T *>(a.loc);
    const T *mass = reinterpret_cast<const T *>(a.mass);
    const T *le = reinterpret_cast<const T *>(a.le);
    const T eps2 = (T)a.eps2;
    for (int64_t it = (int64_t)blockIdx.x * kPtWarps + warp; it < a.n_items; it += (int64_t)gridDim.x * kPtWarps) {
        const int4 item = a.items[it];
        const int leaf = item.x;
        const uint64_t key = a.tkey[leaf];
        int64_t lc[3] = {0, 0, 0};
        for (int bit = 0; bit < 21; ++bit) {
            lc[0] |= (int64_t)((key >> (3 * bit)) & 1) << bit;
            lc[1] |= (int64_t)((key >> (3 * bit + 1)) & 1) << bit;
            lc[2] |= (int64_t)((key >> (3 * bit + 2)) & 1) << bit;
        }
        T tx[2], ty[2], tz[2];
        int tid[2];
        for (int w = 0; w < 2; ++w) {
            const int r = lane + 32 * w;
            tid[w] = r < item.z ? item.y + r : -1;
            const int64_t i = tid[w] >= 0 ? tid[w] : item.y;
            tx[w] = tloc[3 * i];
            ty[w] = tloc[3 * i + 1];
            tz[w] = tloc[3 * i + 2];
        }
        __syncwarp();
        if (lane < 27) {
            const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
            const int64_t sx_ = lc[0] + dx - a.g.slo[0], sy_ = lc[1] + dy - a.g.slo[1], sz_ = lc[2] + dz - a.g.slo[2];
            const bool in = sx_ >= 0 && sy_ >= 0 && sz_ >= 0 && sx_ < a.g.sn[0] && sy_ < a.g.sn[1] && sz_ < a.g.sn[2] &&
                            in_source_part(lc[0] + dx, lc[1] + dy, lc[2] + dz, a.L - 2, a.part_lo, a.part_hi);
            nbl[lane] = in ? (sz_ * a.g.sn[1] + sy_) * a.g.sn[0] + sx_ : -1;
        }
        __syncwarp();
        for (int bb = 0; bb < a.B; ++bb) {
            T hx[2] = {T(0), T(0)}, hy[2] = {T(0), T(0)}, hz[2] = {T(0), T(0)};
            T lx[2] = {T(0), T(0)}, ly[2] = {T(0), T(0)}, lz[2] = {T(0), T(0)};
            for (int nb = 0; nb < 27; ++nb) {
                const int64_t sl = nbl[nb];
                if (sl < 0) continue;
                const T ox = T(nb % 3 - 1), oy = T((nb / 3) % 3 - 1), oz = T(nb / 9 - 1);
                const int64_t i0 = a.leaf_beg[sl], i1 = a.leaf_beg[sl + 1];
                T px[2] = {T(0), T(0)}, py[2] = {T(0), T(0)}, pz[2] = {T(0), T(0)};
                uint64_t qx[2] = {0, 0}, qy[2] = {0, 0}, qz[2] = {0, 0};   // packed sums (FP32)
                for (int64_t c0 = i0; c0 < i1; c0 += kPtChunk) {
                    const int cnt = (int)min((int64_t)kPtChunk, i1 - c0);
                    __syncwarp();
                    for (int s = lane; s < cnt; s += 32) {
                        const int64_t i = c0 + s;
                        T x, y, z, w;
                        ld_loc(loc, i, x, y, z, w);
                        const T mq = mass[(int64_t)bb * a.S + i];
                        if constexpr (kF32) {
                            T *rec = wsh + (s >> 1) * 8 + (s & 1);
                            rec[0] = x + ox;
                            rec[2] = y + oy;
                            rec[4] = z + oz;
                            rec[6] = mq;
                        } else {
                            T *rec = wsh + 4 * s;
                            rec[0] = x + ox;
                            rec[1] = y + oy;
                            rec[2] = z + oz;
                            rec[3] = mq;
                        }
                    }
                    if constexpr (kF32) {
                        // an odd chunk ends with a massless point far away
                        if ((cnt & 1) && lane == 0) {
                            T *rec = wsh + (cnt >> 1) * 8 + 1;
                            rec[0] = rec[2] = rec[4] = T(1.0e4);
                            rec[6] = T(0);
                        }
                        __syncwarp();
                        uint64_t TX[2], TY[2], TZ[2];
#pragma unroll
                        for (int w = 0; w < 2; ++w) {
                            TX[w] = pk2(tx[w], tx[w]);
                            TY[w] = pk2(ty[w], ty[w]);
                            TZ[w] = pk2(tz[w], tz[w]);
                        }
                        const int npair = (cnt + 1) >> 1;
#pragma unroll 2
                        for (int q = 0; q < npair; ++q) {
                            const ulonglong2 xy = *reinterpret_cast<const ulonglong2 *>(wsh + q * 8);
                            const ulonglong2 zw = *reinterpret_cast<const ulonglong2 *>(wsh + q * 8 + 4);
#pragma unroll
                            for (int w = 0; w < 2; ++w) {
                                const uint64_t DX = sub2(TX[w], xy.x), DY = sub2(TY[w], xy.y), DZ = sub2(TZ[w], zw.x);
                                const uint64_t R2 = fma2(DZ, DZ, fma2(DY, DY, mul2(DX, DX)));
                                float r0, r1;
                                up2(R2, r0, r1);
                                // a point on the observer contributes nothing
                                const float i0f = r0 > (float)eps2 ? rsqrt_ftz(r0) : 0.f;
                                const float i1f = r1 > (float)eps2 ? rsqrt_ftz(r1) : 0.f;
                                const uint64_t RI = pk2(i0f, i1f);
                                const uint64_t K3 = mul2(mul2(mul2(RI, RI), RI), zw.y);
                                qx[w] = fma2(K3, DX, qx[w]);
                                qy[w] = fma2(K3, DY, qy[w]);
                                qz[w] = fma2(K3, DZ, qz[w]);
                            }
                        }
                    } else {
                        __syncwarp();
                        for (int s = 0; s < cnt; ++s) {
                            const T ux = wsh[4 * s], uy = wsh[4 * s + 1], uz = wsh[4 * s + 2], mq = wsh[4 * s + 3];
#pragma unroll
                            for (int w = 0; w < 2; ++w) {
                                const T dx = tx[w] - ux, dy = ty[w] - uy, dz = tz[w] - uz;
                                const T r2 = dx * dx + dy * dy + dz * dz;
                                const T ri = r2 > eps2 ? rsqrt(r2) : T(0);
                                const T k3 = mq * ri * ri * ri;
                                px[w] += k3 * dx;
                                py[w] += k3 * dy;
                                pz[w] += k3 * dz;
                            }
                        }
                    }
                }
                if constexpr (kF32) {
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        float a0, a1;
                        up2(qx[w], a0, a1);
                        px[w] = a0 + a1;
                        up2(qy[w], a0, a1);
                        py[w] = a0 + a1;
                        up2(qz[w], a0, a1);
                        pz[w] = a0 + a1;
                    }
                }
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    two_sum(hx[w], lx[w], px[w]);
                    two_sum(hy[w], ly[w], py[w]);
                    two_sum(hz[w], lz[w], pz[w]);
                }
            }
            // far field: gradient of the leaf's local expansion
            __syncwarp();
            const T *Lc = le + ((int64_t)leaf * a.B + bb) * a.ldk;
            T fx[2], fy[2], fz[2];
            if constexpr (kF32) {
                float2 *Dx2 = reinterpret_cast<float2 *>(Dx), *Dy2 = reinterpret_cast<float2 *>(Dy),
                       *Dz2 = reinterpret_cast<float2 *>(Dz);
                for (int e = lane; e < P2; e += 32) {
                    float vx, vy, vz;
                    grad_coeff<float>(Lc, e, vx, vy, vz);
                    const float f2 = __ldg(l2p_scale + e);
                    Dx2[e] = make_float2(f2 * vx, f2 * vx);
                    Dy2[e] = make_float2(f2 * vy, f2 * vy);
                    Dz2[e] = make_float2(f2 * vz, f2 * vz);
                }
                __syncwarp();
                uint64_t FX, FY, FZ;
                l2p_sum2(a.p, Dx2, Dy2, Dz2, pk2(tx[0], tx[1]), pk2(ty[0], ty[1]), pk2(tz[0], tz[1]), FX, FY, FZ);
                up2(FX, fx[0], fx[1]);
                up2(FY, fy[0], fy[1]);
                up2(FZ, fz[0], fz[1]);
            } else {
                for (int e = lane; e < P2; e += 32) grad_coeff<T>(Lc, e, Dx[e], Dy[e], Dz[e]);
                __syncwarp();
                for (int w = 0; w < 2; ++w) l2p_sum<T>(a.p, Dx, Dy, Dz, tx[w], ty[w], tz[w], fx[w], fy[w], fz[w]);
            }
            for (int w = 0; w < 2; ++w) {
                if (tid[w] < 0) continue;
                const double gx = ((double)hx[w] + (double)lx[w] - (double)fx[w]) * a.scale;
                const double gy = ((double)hy[w] + (double)ly[w] - (double)fy[w]) * a.scale;
                const double gzv = ((double)hz[w] + (double)lz[w] - (double)fz[w]) * a.scale;
                const int64_t j = a.perm[tid[w]];
                if (a.gout) {
                    double *o = a.gout + ((int64_t)bb * a.M + j) * 3;
                    o[0] = gx;
                    o[1] = gy;
                    o[2] = gzv;
                }
                if (a.gz) a.gz[(int64_t)bb * a.M + j] = gzv;
            }
            __syncwarp();
        }
    }
}

// Near (observer, source) pairs of the FMM: observers of each observer leaf
// times the points of its neighbour leaves.
__global__ void point_count_near(const uint64_t *__restrict__ tkey, const int32_t *__restrict__ leaf_obs,
                                 int64_t ntl, const int64_t *__restrict__ leaf_beg, PtGeo g,
                                 unsigned long long *__restrict__ out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntl) return;
    const uint64_t key = tkey[t];
    int64_t lc[3] = {0, 0, 0};
    for (int bit = 0; bit < 21; ++bit) {
        lc[0] |= (int64_t)((key >> (3 * bit)) & 1) << bit;
        lc[1] |= (int64_t)((key >> (3 * bit + 1)) & 1) << bit;
        lc[2] |= (int64_t)((key >> (3 * bit + 2)) & 1) << bit;
    }
    unsigned long long src = 0;
    for (int nb = 0; nb < 27; ++nb) {
        const int64_t x = lc[0] + nb % 3 - 1 - g.slo[0], y = lc[1] + (nb / 3) % 3 - 1 - g.slo[1],
                      z = lc[2] + nb / 9 - 1 - g.slo[2];
        if (x < 0 || y < 0 || z < 0 || x >= g.sn[0] || y >= g.sn[1] || z >= g.sn[2]) continue;
        const int64_t l = (z * g.sn[1] + y) * g.sn[0] + x;
        src += (unsigned long long)(leaf_beg[l + 1] - leaf_beg[l]);
    }
    atomicAdd(out, src * (unsigned long long)(leaf_obs[t + 1] - leaf_obs[t]));
}

PtGeo pt_geo(const gf_plan_s *plan) {
    const FmmPlan *F = plan->fmm;
    PtGeo g;
    memset(&g, 0, sizeof(g));
    for (int a = 0; a < 3; ++a) {
        g.lo[a] = F->lo[a];
        g.lof[a] = (float)F->lo[a];
        g.slo[a] = F->lev[F->L].slo[a];
        g.sn[a] = F->lev[F->L].sn[a];
    }
    g.inv_s = F->inv_s;
    g.isf = (float)F->inv_s;
    g.fixk = -1;
    return g;
}

// The recursion tables of this file's kernels on the current device.
gf_status upload_point_tables(int device) {
    static std::mutex mu;
    static unsigned long long done = 0;
    std::lock_guard<std::mutex> lk(mu);
    if (device >= 0 && device < 64 && ((done >> device) & 1ull)) return GF_OK;
    // s_nm: prod_{j <= m} -sqrt((2j-1) / (2j)) for the sectoral steps, then
    // prod_{j = m+1..n} (2j-1) / sqrt((j+m)(j-m))
    double ps[(kMaxP + 1) * (kMaxP + 1)] = {};
    double sect = 1.0;
    for (int m = 0; m <= kMaxP; ++m) {
        if (m > 0) sect *= -std::sqrt((2.0 * m - 1.0) / (2.0 * m));
        double v = sect;
        for (int n = m; n <= kMaxP; ++n) {
            if (n > m) v *= (2 * n - 1) / std::sqrt((double)((n + m) * (n - m)));
            ps[n * n + (m == 0 ? 0 : 2 * m - 1)] = v;
        }
    }
    GF_CUDA(cudaMemcpyToSymbol(c_ps, ps, sizeof(ps)));
    GF_TRY(upload_l2p_coefs());
    if (device >= 0 && device < 64) done |= 1ull << device;
    return GF_OK;
}

}  // namespace

// ---------------------------------------------------------------- host side
gf_status hex_sources_run(const double *verts, int64_t ncell, const QuadRule &qr, int precision, double *x,
                          double *a, cudaStream_t st) {
    const int64_t n = ncell * qr.nq;
    if (n == 0) return GF_OK;
    if (precision == GF_PREC_MIXED) {
        HexRuleF rf;
        memset(&rf, 0, sizeof(rf));
        rf.nq = qr.nq;
        for (int q = 0; q < qr.nq; ++q) {
            for (int d = 0; d < 3; ++d) rf.xi[q][d] = (float)qr.xi[q][d];
            rf.w8[q] = (float)(8.0 * qr.wn[q]);
        }
        hex_sources_fix<<<ceil_div(ncell, kHexCells), kHexCells * 8, 0, st>>>(verts, ncell, rf, x, a);
    } else {
        hex_sources_kernel<<<ceil_div(n, 256), 256, 0, st>>>(verts, ncell, qr, x, a);
    }
    GF_KERNEL_DONE();
    return GF_OK;
}

gf_status points_prepare_direct(gf_plan_s *plan, const double *src, const double *wt, const double *obs,
                                cudaStream_t st) {
    PointSet &P = plan->pts;
    DeviceArena &A = plan->arena;
    const int64_t S = P.S, M = plan->M;
    GF_TRY(A.alloc_n(&P.x, std::max<int64_t>(3 * S, 1)));
    GF_TRY(A.alloc_n(&P.a, std::max<int64_t>(S, 1)));
    GF_TRY(A.alloc_n(&plan->d_obs, std::max<int64_t>(3 * M, 1)));
    if (S > 0) {
        GF_CUDA(cudaMemcpyAsync(P.x, src, sizeof(double) * 3 * S, cudaMemcpyDeviceToDevice, st));
        GF_CUDA(cudaMemcpyAsync(P.a, wt, sizeof(double) * S, cudaMemcpyDeviceToDevice, st));
    }
    if (M > 0) GF_CUDA(cudaMemcpyAsync(plan->d_obs, obs, sizeof(double) * 3 * M, cudaMemcpyDeviceToDevice, st));
    if (plan->opt.precision == GF_PREC_MIXED && S > 0 && M > 0) {
        // one quantum for sources and observers: 2^-22 of the joint extent
        double bs[12], bo[12], lo[3], hi[3];
        double *d_bb;
        GF_TRY(A.alloc_n(&d_bb, 24));
        GF_TRY(bbox3(P.x, S, d_bb, st));
        GF_TRY(bbox3(plan->d_obs, M, d_bb + 12, st));
        GF_CUDA(cudaMemcpyAsync(bs, d_bb, sizeof(bs), cudaMemcpyDeviceToHost, st));
        GF_CUDA(cudaMemcpyAsync(bo, d_bb + 12, sizeof(bo), cudaMemcpyDeviceToHost, st));
        GF_CUDA(cudaStreamSynchronize(st));
        double ext = 0.0;
        for (int d = 0; d < 3; ++d) {
            lo[d] = std::min(bs[d], bo[d]);
            hi[d] = std::max(bs[3 + d], bo[3 + d]);
            if (!isfinite(lo[d]) || !isfinite(hi[d])) {
                set_error("source and observer coordinates must be finite");
                return GF_ERR_INVALID_ARG;
            }
            ext = std::max(ext, hi[d] - lo[d]);
        }
        int e = 0;
        frexp(std::max(ext, 1e-300), &e);   // ext < 2^e
        P.q = ldexp(1.0, e - 22);
        GF_TRY(A.alloc_n(&P.xi, 3 * S));
        GF_TRY(A.alloc_n(&P.xf, 3 * S));
        GF_TRY(A.alloc_n(&P.oi, 3 * M));
        GF_TRY(A.alloc_n(&P.of, 3 * M));
        split_points<<<ceil_div(S, 256), 256, 0, st>>>(P.x, S, lo[0], lo[1], lo[2], 1.0 / P.q, P.xi, P.xf);
        GF_KERNEL_DONE();
        split_points<<<ceil_div(M, 256), 256, 0, st>>>(plan->d_obs, M, lo[0], lo[1], lo[2], 1.0 / P.q, P.oi,
                                                       P.of);
        GF_KERNEL_DONE();
    }
    return GF_OK;
}

gf_status points_direct_forward(gf_plan_s *plan, const void *rho, int rho_dtype, int B, double *g, double *gz,
                                cudaStream_t st) {
    const PointSet &P = plan->pts;
    const int64_t M = plan->M;
    if (M == 0) return GF_OK;
    const int f32 = rho_dtype == GF_DTYPE_F32;
    const int64_t tiles = (M + 63) / 64;
    const bool f64 = plan->opt.precision == GF_PREC_FP64 || P.S == 0;
    const int cl = pair_cluster(tiles, (P.S + 31) / 32, f64 ? PairCost{8.0, 8.0, 4.0} : PairCost{0.25, 5.0, 8.0});
    if (f64) {
        if (cl == 0)
            return pair_launch_solo(direct_points_f64<true>, tiles, B, st, plan->d_obs, M, P.x, P.a, P.S, P.per_cell,
                                    P.ncell, rho, f32, plan->G, g, gz, plan->d_status);
        return pair_launch(direct_points_f64<false>, tiles, B, cl, st, plan->d_obs, M, P.x, P.a, P.S, P.per_cell, P.ncell,
                           rho, f32, plan->G, g, gz, plan->d_status);
    }
    // mass and separations in quanta: g = G / q^2 * (quantum-unit sum)
    if (cl == 0)
        return pair_launch_solo(direct_points_mixed<true>, tiles, B, st, P.oi, P.of, M, P.xi, P.xf, P.a, P.S, P.per_cell,
                                P.ncell, rho, f32, (float)P.q, plan->G * P.q, g, gz, plan->d_status);
    return pair_launch(direct_points_mixed<false>, tiles, B, cl, st, P.oi, P.of, M, P.xi, P.xf, P.a, P.S, P.per_cell,
                       P.ncell, rho, f32, (float)P.q, plan->G * P.q, g, gz, plan->d_status);
}

gf_status points_fmm_create(gf_plan_s *plan, const double *src, const double *wt, const double *obs,
                            cudaStream_t st) {
    FmmPlan *F = new (std::nothrow) FmmPlan();
    if (!F) {
        set_error("host allocation failed");
        return GF_ERR_OOM;
    }
    plan->fmm = F;
    PointSet &P = plan->pts;
    const int64_t S = P.S, M = plan->M;
    F->p = plan->opt.p;
    F->K = (F->p + 1) * (F->p + 1);
    F->B = plan->opt.max_batch;
    F->nq = 1;
    F->mixed = plan->opt.precision == GF_PREC_MIXED;
    F->m2l_tc64 = !F->mixed && (plan->opt.reserved0 & GF_FLAG_M2L_TENSOR);
    F->b = 1;
    F->points = true;
    DeviceArena &A = plan->arena;
    // ---- extents of the sources and of the observers
    double bs[6] = {0, 0, 0, 0, 0, 0}, bo[6] = {0, 0, 0, 0, 0, 0};
    {
        double *d_bb;
        GF_TRY(A.alloc_n(&d_bb, 24));
        if (S > 0) GF_TRY(bbox3(src, S, d_bb, st));
        if (M > 0) GF_TRY(bbox3(obs, M, d_bb + 12, st));
        double h[24];
        GF_CUDA(cudaMemcpyAsync(h, d_bb, sizeof(h), cudaMemcpyDeviceToHost, st));
        GF_CUDA(cudaStreamSynchronize(st));
        for (int d = 0; d < 6; ++d) {
            if (S > 0) bs[d] = h[d];
            if (M > 0) bo[d] = h[12 + d];
            if (!isfinite(bs[d]) || !isfinite(bo[d])) {
                set_error("source and observer coordinates must be finite");
                return GF_ERR_INVALID_ARG;
            }
        }
        if (S == 0)
            for (int d = 0; d < 6; ++d) bs[d] = bo[d];
        if (M == 0)
            for (int d = 0; d < 6; ++d) bo[d] = bs[d];
    }
    // ---- leaf side: about kPointsPerLeaf sources per leaf of their extent
    double ext_s[3], ext_max = 0.0, vol = 1.0;
    for (int d = 0; d < 3; ++d) {
        ext_s[d] = bs[3 + d] - bs[d];
        ext_max = std::max(ext_max, ext_s[d]);
    }
    if (ext_max <= 0.0) ext_max = 1.0;
    int flat = 0;
    for (int d = 0; d < 3; ++d) {
        if (ext_s[d] > 1e-6 * ext_max)
            vol *= ext_s[d];
        else
            ++flat;
    }
    const double nleaf_want = std::max(1.0, (double)S / kPointsPerLeaf);
    double side = flat == 0 ? cbrt(vol / nleaf_want) : (flat == 1 ? sqrt(vol / nleaf_want) : vol / nleaf_want);
    side = std::max(side, ext_max * 1e-6);
    double bb[6];
    for (int d = 0; d < 3; ++d) {
        bb[d] = std::min(bs[d], bo[d]);
        bb[3 + d] = std::max(bs[3 + d], bo[3 + d]);
    }
    double root_ext = 0.0;
    for (int d = 0; d < 3; ++d) root_ext = std::max(root_ext, bb[3 + d] - bb[d]);
    // the root spans the joint extent plus the shift of its corner below
    const double span = root_ext + 1e-6 * side;
    int L = 2;
    while (L < kMaxLevels - 1 && side * (double)((int64_t)1 << L) < span) ++L;
    if (side * (double)((int64_t)1 << L) < span) side = span / (double)((int64_t)1 << L) * (1.0 + 1e-9);
    F->L = L;
    F->h = side;   // the plan's length unit is the leaf side
    F->s_leaf = side;
    F->inv_s = 1.0 / side;
    for (int d = 0; d < 3; ++d) {
        F->lo[d] = bb[d] - 1e-7 * side;   // strictly inside the root
        F->voff[d] = 0;
    }
    const int64_t top = ((int64_t)1 << L) - 1;
    int64_t slo[3], shi[3];
    for (int d = 0; d < 3; ++d) {
        slo[d] = std::min<int64_t>(top, std::max<int64_t>(0, (int64_t)floor((bs[d] - F->lo[d]) * F->inv_s)));
        shi[d] = std::min<int64_t>(top, std::max<int64_t>(slo[d], (int64_t)floor((bs[3 + d] - F->lo[d]) * F->inv_s)));
    }
    for (int l = 0; l <= L; ++l) {
        FmmLevel &lv = F->lev[l];
        lv.ns = 1;
        for (int d = 0; d < 3; ++d) {
            lv.slo[d] = slo[d] >> (L - l);
            lv.sn[d] = (shi[d] >> (L - l)) - lv.slo[d] + 1;
            lv.ns *= lv.sn[d];
        }
    }
    const int64_t nleaf = F->lev[L].ns;
    if (nleaf > ((int64_t)1 << 31)) {
        set_error("the sources' leaf block is too large (%lld leaves)", (long long)nleaf);
        return GF_ERR_UNSUPPORTED;
    }
    // ---- sources sorted by leaf, each leaf's first source
    GF_TRY(upload_point_tables(plan->device));
    PtGeo g = pt_geo(plan);
    double bb_root[6];
    for (int d = 0; d < 6; ++d) bb_root[d] = bb[d];
    g.fixk = fixed_point_frame(F, bb_root, g.lofix, &g.halfleaf_fix, &g.fix_to_leaf);
    const size_t rs = F->mixed ? sizeof(float) : sizeof(double);
    GF_TRY(A.alloc(&P.loc, rs * 4 * (size_t)std::max<int64_t>(S, 1)));
    GF_TRY(A.alloc_n(&P.perm, std::max<int64_t>(S, 1)));
    GF_TRY(A.alloc_n(&P.leaf_beg, nleaf + 1));
    if (S > 0) {
        if (nleaf >= (int64_t)1 << 32) {   // their expansions would fill many devices
            set_error("point sources: %lld leaves", (long long)nleaf);
            return GF_ERR_OOM;
        }
        uint32_t *keys, *keys2;
        int32_t *vals2;
        GF_TRY(A.alloc_n(&keys, S));
        GF_TRY(A.alloc_n(&keys2, S));
        GF_TRY(A.alloc_n(&vals2, S));
        void *scratch;
        GF_TRY(A.alloc(&scratch, sort_scratch_bytes(S)));
        int bits = 1;
        while (bits < 32 && ((int64_t)1 << bits) < nleaf) ++bits;
        point_keys<<<ceil_div(S, 256), 256, 0, st>>>(src, S, g, radix_sort_input(keys, keys2, bits), plan->d_status);
        GF_KERNEL_DONE();
        GF_TRY(radix_sort(keys, P.perm, keys2, vals2, S, bits, scratch, st));
        const double inv_s3 = F->inv_s * F->inv_s * F->inv_s;
        if (F->mixed)
            point_gather<float><<<ceil_div(S, 256), 256, 0, st>>>(src, wt, P.perm, keys, S, g, inv_s3,
                                                                  (float *)P.loc, plan->d_status);
        else
            point_gather<double><<<ceil_div(S, 256), 256, 0, st>>>(src, wt, P.perm, keys, S, g, inv_s3,
                                                                   (double *)P.loc, plan->d_status);
        GF_KERNEL_DONE();
        point_leaf_beg<<<ceil_div(nleaf + 1, 256), 256, 0, st>>>(keys, S, nleaf, P.leaf_beg);
        GF_KERNEL_DONE();
    } else {
        GF_CUDA(cudaMemsetAsync(P.leaf_beg, 0, sizeof(int64_t) * (nleaf + 1), st));
    }
    double oz[2] = {bo[2], bo[5]}, olo[3] = {bo[0], bo[1], bo[2]}, ohi[3] = {bo[3], bo[4], bo[5]};
    return fmm_observer_tree(plan, obs, oz, olo, ohi, bb, st);
}

template <class T>
gf_status points_masses(gf_plan_s *plan, const void *rho, int rho_dtype, int B, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const PointSet &P = plan->pts;
    if (P.S == 0) return GF_OK;
    point_masses<T><<<dim3(ceil_div(P.S, 256), (unsigned)B), 256, 0, st>>>(rho, rho_dtype == GF_DTYPE_F32, P.perm,
                                                                          (const T *)P.loc, P.S, P.per_cell, P.ncell,
                                                                          (T *)F->mass, plan->d_status);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class T>
gf_status points_p2m(gf_plan_s *plan, int B, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &lv = F->lev[F->L];
    // the rows whose largest component scales the leaf level's M2L inputs
    const int64_t slab = lv.sn[0] * lv.sn[1];
    const bool in = F->amax_fused && lv.m2l_z1 >= lv.m2l_z0;
    uint32_t *amax = in ? F->tc_amax + F->L : nullptr;
    const int64_t lo = in ? lv.m2l_z0 * slab : 0, hi = in ? (lv.m2l_z1 + 1) * slab : 0;
    // lanes per leaf: the power of two that holds the p/2 + 1 lanes' orders;
    // terms per lane in a few sizes (what a size has beyond them is skipped)
    const int p = F->p;
    if (p <= 7) return launch_point_p2m<T, 4, 9, 2>(plan, B, amax, lo, hi, st);
    if (p <= 10) return launch_point_p2m<T, 8, 11, 5>(plan, B, amax, lo, hi, st);
    if (p <= 12) return launch_point_p2m<T, 8, 13, 7>(plan, B, amax, lo, hi, st);
    if (p <= 15) return launch_point_p2m<T, 8, 17, 8>(plan, B, amax, lo, hi, st);
    return launch_point_p2m<T, 16, 17, 9>(plan, B, amax, lo, hi, st);
}

template <class T>
gf_status points_eval(gf_plan_s *plan, int B, double *g, double *gz, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const PointSet &P = plan->pts;
    if (F->n_items == 0) return GF_OK;
    PtEvalArgs a;
    a.items = F->items;
    a.n_items = F->n_items;
    a.tkey = F->lev[F->L].tkey;
    a.perm = F->perm;
    a.tloc = sizeof(T) == 8 ? (const void *)F->tloc_d : (const void *)F->tloc_f;
    a.loc = P.loc;
    a.mass = F->mass;
    a.leaf_beg = P.leaf_beg;
    a.le = F->lev[F->L].le;
    a.g = pt_geo(plan);
    a.L = F->L;
    a.B = B;
    a.p = F->p;
    a.ldk = F->KS;
    a.S = P.S;
    a.M = plan->M;
    a.part_lo = plan->part_lo;
    a.part_hi = plan->part_hi;
    a.scale = plan->G * F->h;
    a.eps2 = sizeof(T) == 8 ? 1e-24 : 1e-14;
    a.gout = g;
    a.gz = gz;
    const size_t shm = sizeof(T) * kPtWarps * (size_t)pt_slice(F->p * F->p, (int)sizeof(T));
    GF_TRY(ensure_smem(point_eval<T>, shm));
    const unsigned grid = (unsigned)std::min<int64_t>((F->n_items + kPtWarps - 1) / kPtWarps, 152 * 64);
    point_eval<T><<<grid, kPtWarps * 32, shm, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

template gf_status points_masses<float>(gf_plan_s *, const void *, int, int, cudaStream_t);
template gf_status points_masses<double>(gf_plan_s *, const void *, int, int, cudaStream_t);
template gf_status points_p2m<float>(gf_plan_s *, int, cudaStream_t);
template gf_status points_p2m<double>(gf_plan_s *, int, cudaStream_t);
template gf_status points_eval<float>(gf_plan_s *, int, double *, double *, cudaStream_t);
template gf_status points_eval<double>(gf_plan_s *, int, double *, double *, cudaStream_t);

gf_status points_count_near(gf_plan_s *plan, unsigned long long *d_out, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &leaf = F->lev[F->L];
    if (leaf.nt == 0) return GF_OK;
    point_count_near<<<ceil_div(leaf.nt, 256), 256, 0, st>>>(leaf.tkey, F->leaf_beg, leaf.nt, plan->pts.leaf_beg,
                                                            pt_geo(plan), d_out);
    GF_KERNEL_DONE();
    return GF_OK;
}

}  // namespace gf
