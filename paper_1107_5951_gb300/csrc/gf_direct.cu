// gf_direct.cu -- direct summation (Sec. 2.1, SUM-G1/SUM-G2) of Eq. 1 in
// its N-body form (Eq. 7): every observer against every voxel quadrature
// point.  Used as the exact path ("direct mode") and its transpose.
//
// Layout: forward, tiles of up to 64 observers whose sources are shared by
// the warps of a thread-block cluster (gf_pair.cuh); transpose, one thread per
// voxel, a block staging tiles of 256 observers in shared memory.
// FP64 path: source coordinates are formed with explicitly rounded
// operations in the same order as the plain definition, so coincidence
// decisions (r == x) are exact.  Mixed path: coordinates are carried as
// integer voxel index plus an FP32 fraction, so the separation of near pairs
// is formed to FP32 relative accuracy whatever the size of the domain.
#include <cuda.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "gf_internal.cuh"
#include "gf_pair.cuh"
#include "gf_simd.cuh"

namespace gf {
namespace {

constexpr int kTile = 256;

struct GridArgs {
    int64_t nx, ny, nz, nvox;
    double ox, oy, oz, hx, hy, hz, vol;
};

GridArgs grid_args(const gf_plan_s *p) {
    GridArgs a;
    a.nx = p->grid.n[0];
    a.ny = p->grid.n[1];
    a.nz = p->grid.n[2];
    a.nvox = a.nx * a.ny * a.nz;
    a.ox = p->grid.origin[0];
    a.oy = p->grid.origin[1];
    a.oz = p->grid.origin[2];
    a.hx = p->grid.h[0];
    a.hy = p->grid.h[1];
    a.hz = p->grid.h[2];
    a.vol = a.hx * a.hy * a.hz;
    return a;
}

__device__ __forceinline__ double load_rho(const void *rho, int f32, int64_t idx) {
    return f32 ? (double)__ldg(reinterpret_cast<const float *>(rho) + idx)
               : __ldg(reinterpret_cast<const double *>(rho) + idx);
}

// Neumaier step on (s, c) with addend x.
__device__ __forceinline__ void neumaier(double &s, double &c, double x) {
    double t = s + x;
    c += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
    s = t;
}

// Position of quadrature node q of voxel (i,j,k) in FP64, rounded exactly as
// centre = origin + (i + 1/2) h, node = centre + (h/2) xi.
__device__ __forceinline__ double node_coord(double o, double h, int64_t i, double xi) {
    double c = __dadd_rn(o, __dmul_rn((double)i + 0.5, h));
    return __dadd_rn(c, __dmul_rn(__dmul_rn(0.5, h), xi));
}

// Work units of the forward sums: the sources of one grid row (fixed j, k
// and rule node q) share y and z, so a row is cut into pieces of at most
// kRow voxels and a warp takes every W-th piece (W warps in the cluster).
// Within a piece only x moves: a pair costs one difference, one square
// (on top of the row's dy^2 + dz^2), the kernel value and two sums (of k and
// of k dx); the y and z components are the row's sum of k times dy, dz.
constexpr int kRow = 30;   // lanes 30 and 31 form the row's y and z

struct RowSplit {
    int clen, nch;       // voxels per piece, pieces per row
    int ax[3];           // the axes of a row, j and k
    int n[3];            // their voxels
    int64_t stride[3];   // and strides in the density array
    double o[3], h[3];   // the grid's origin and voxel size along them
};

// Rows along axis `row`, cut into pieces of equal length.
inline RowSplit row_split(const GridArgs &ga, int row) {
    const int64_t n[3] = {ga.nx, ga.ny, ga.nz}, stride[3] = {1, ga.nx, ga.nx * ga.ny};
    const double o[3] = {ga.ox, ga.oy, ga.oz}, h[3] = {ga.hx, ga.hy, ga.hz};
    RowSplit r;
    r.nch = (int)((n[row] + kRow - 1) / kRow);
    r.clen = (int)((n[row] + r.nch - 1) / r.nch);
    for (int d = 0; d < 3; ++d) {
        r.ax[d] = d == 0 ? row : (d - 1 < row ? d - 1 : d);
        r.n[d] = (int)n[r.ax[d]];
        r.stride[d] = stride[r.ax[d]];
        r.o[d] = o[r.ax[d]];
        r.h[d] = h[r.ax[d]];
    }
    return r;
}

// The split of the sources and the blocks per cluster (pair_cluster) of a forward
// sum; cost(clen): of a piece.  Rows run along x, unless its pieces would be less than
// half as long as another axis's (a column of voxels: 20 instructions for every voxel's
// own row) and the longer rows, which are fewer to share out, take less time: two
// densities of 6 x 12 x 29 voxels at 227 stations are 82 us along x, 156 along z.
template <class Cost>
inline RowSplit row_split(const GridArgs &ga, int64_t tiles, int nq, Cost cost, int *cluster) {
    RowSplit best = row_split(ga, 0);
    double us = 0.0;
    auto split = [&](const RowSplit &r, double *t) {
        return pair_cluster(tiles, (int64_t)r.nch * nq * r.n[1] * r.n[2], cost(r.clen), t);
    };
    *cluster = split(best, &us);
    const int cx = best.clen;
    for (int a = 1; a < 3; ++a) {
        const RowSplit r = row_split(ga, a);
        if (r.clen <= 2 * cx) continue;
        double t = 0.0;
        const int c = split(r, &t);
        if (t < us) {
            us = t;
            best = r;
            *cluster = c;
        }
    }
    return best;
}

// Piece (ch, q, j, k) of the flat index u = ((k ny + j) nq + q) nch + ch,
// advanced by a fixed step without divisions.
struct RowIter {
    int ch, q, j, k;
    int dch, dq, dj, dk;
    int nch, nq, ny;
    __device__ static void split(int64_t u, int nch, int nq, int ny, int &ch, int &q, int &j, int &k) {
        ch = (int)(u % nch);
        u /= nch;
        q = (int)(u % nq);
        u /= nq;
        j = (int)(u % ny);
        k = (int)(u / ny);
    }
    __device__ RowIter(int64_t u0, int64_t step, int nch_, int nq_, int ny_) : nch(nch_), nq(nq_), ny(ny_) {
        split(u0, nch, nq, ny, ch, q, j, k);
        split(step, nch, nq, ny, dch, dq, dj, dk);
    }
    __device__ void next() {
        ch += dch;
        q += dq;
        j += dj;
        k += dk;
        if (ch >= nch) {
            ch -= nch;
            ++q;
        }
        if (q >= nq) {
            q -= nq;
            ++j;
        }
        if (j >= ny) {
            j -= ny;
            ++k;
        }
    }
};

__device__ __forceinline__ const void *rho_of(const void *rho, int f32, int64_t off) {
    return f32 ? (const void *)((const float *)rho + off) : (const void *)((const double *)rho + off);
}

// Bound by the FP64 pipe: 11 instructions a pair and about 20 a piece of
// R x 16 pairs.  16^3 voxels, 2x2x2 rule, 4096 stations (134 M pairs):
// 41.6 -> 4.07 ms (16 blocks of 256 threads before; 2.5 ms at two FP64
// instructions a clock and SM).
template <int R, bool kSolo>
__global__ void __launch_bounds__(kSolo ? 32 : kPairThreads)
direct_fwd_f64(const double *__restrict__ obs, int64_t M, const void *__restrict__ rho, int rho_f32, GridArgs ga,
               RowSplit rs, const QuadRule *__restrict__ qr, double G, double *__restrict__ g,
               double *__restrict__ gz, int *__restrict__ status) {
    __shared__ double2 red[kSolo ? 1 : (kPairWarps + 1) * 3 * R * 32];
    __shared__ __align__(16) double2 row_s[kSolo ? 1 : kPairWarps][32];   // (x, mass) of the piece; entries 30, 31: y, z
    const int C = kSolo ? 1 : (int)cooperative_groups::this_cluster().num_blocks();
    const int rank = kSolo ? 0 : (int)cooperative_groups::this_cluster().block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.y;
    const int64_t tile = blockIdx.x / C;
    double rx[R], ry[R], rz[R];
    double s[3 * R], c[3 * R], a[3 * R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int64_t j = (tile * R + u) * 32 + lane;
        rx[u] = j < M ? obs[3 * j + rs.ax[0]] : 0.0;
        ry[u] = j < M ? obs[3 * j + rs.ax[1]] : 0.0;
        rz[u] = j < M ? obs[3 * j + rs.ax[2]] : 0.0;
    }
#pragma unroll
    for (int v = 0; v < 3 * R; ++v) s[v] = c[v] = a[v] = 0.0;
    const void *rho_b = rho_of(rho, rho_f32, b * ga.nvox);
    double2 *row = row_s[warp];
    bool bad = false;   // a non-finite density (reported through status[0])
    RowIter it(rank * kPairWarps + warp, kSolo ? 1 : (int64_t)C * kPairWarps, rs.nch, qr->nq, rs.n[1]);
    auto fetch = [&](double &rv) {
        const int64_t i = (int64_t)it.ch * rs.clen + lane;
        rv = 0.0;
        if (it.k < rs.n[2] && lane < rs.clen && i < rs.n[0])
            rv = load_rho(rho_b, rho_f32, it.k * rs.stride[2] + it.j * rs.stride[1] + i * rs.stride[0]);
    };
    double rv;
    fetch(rv);
    int since = 0;   // sources summed since the last merge into (s, c)
    while (it.k < rs.n[2]) {
        const int i0 = it.ch * rs.clen;
        const int cnt = min(rs.clen, rs.n[0] - i0);
        // one node coordinate per lane: x of the piece's voxels, y (lane 30), z (lane 31)
        const int ax = lane < kRow ? 0 : lane - (kRow - 1);
        const double co = ax == 0 ? rs.o[0] : ax == 1 ? rs.o[1] : rs.o[2], ch = ax == 0 ? rs.h[0] : ax == 1 ? rs.h[1] : rs.h[2];
        const int ci = ax == 0 ? i0 + lane : ax == 1 ? it.j : it.k, da = ax == 0 ? rs.ax[0] : ax == 1 ? rs.ax[1] : rs.ax[2];
        const double x = node_coord(co, ch, ci, qr->xi[it.q][da]);
        bad |= !isfinite(rv);
        const double m = __dmul_rn(__dmul_rn(rv, ga.vol), qr->wn[it.q]);
        __syncwarp();
        row[lane] = make_double2(x, m);
        it.next();
        fetch(rv);   // the next piece's densities, in flight during this one
        __syncwarp();
        const double y = row[kRow].x, z = row[kRow + 1].x;
        double dy[R], dz[R], yz[R], S[R], SX[R];
#pragma unroll
        for (int u = 0; u < R; ++u) {
            dy[u] = ry[u] - y;
            dz[u] = rz[u] - z;
            yz[u] = fma(dy[u], dy[u], dz[u] * dz[u]);
            S[u] = SX[u] = 0.0;
        }
#pragma unroll 2
        for (int e = 0; e < cnt; ++e) {
            const double2 v = row[e];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const double dx = rx[u] - v.x;
                const double k3 = inv_r3(fma(dx, dx, yz[u]), v.y);
                S[u] += k3;
                SX[u] = fma(k3, dx, SX[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < R; ++u) {
            a[3 * u + 0] += SX[u];
            a[3 * u + 1] = fma(S[u], dy[u], a[3 * u + 1]);
            a[3 * u + 2] = fma(S[u], dz[u], a[3 * u + 2]);
        }
        since += cnt;
        if (since >= 240) {
            since = 0;
#pragma unroll
            for (int v = 0; v < 3 * R; ++v) {
                two_sum_d(s[v], c[v], a[v]);
                a[v] = 0.0;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 3 * R; ++v) two_sum_d(s[v], c[v], a[v]);
    if (bad && status && tile == 0) atomicOr(status, 1);
    auto put = [&](int v, int l, double tot) {
        const int u = v / 3, d = v - 3 * u, da = d == 0 ? rs.ax[0] : d == 1 ? rs.ax[1] : rs.ax[2];
        const int64_t j = (tile * R + u) * 32 + l;
        if (j < M) {
            if (g) g[((int64_t)b * M + j) * 3 + da] = G * tot;
            if (gz && da == 2) gz[(int64_t)b * M + j] = G * tot;
        }
    };
    if constexpr (kSolo) {
#pragma unroll
        for (int v = 0; v < 3 * R; ++v) put(v, lane, s[v] + c[v]);
    } else {
        const double tot = cluster_total<3 * R>(s, c, red);
        if (rank == 0 && threadIdx.x < 3 * R * 32) put(threadIdx.x >> 5, lane, tot);
    }
}


// Mixed precision: positions in voxel units split into an integer part
// (held exactly in FP32, |i| < 2^24) and a fraction; the pair separation is
// (ri - si) + (rf - sf), exact integer difference plus one rounding.  A lane's
// two observers form one packed pair (f32x2), the masses are staged as
// duplicated pairs, and the integer difference steps by one along the row:
// 9 packed instructions and two reciprocal square roots for two pairs.  A
// piece's FP32 sums are scaled by the rule's weight and merged into a
// compensated FP32 pair about every 240 sources (the FP64 pipe is too slow
// for a merge per piece); the pairs' sums, the factors G and the voxel volume
// are FP64.  Bound by the special-function unit and the issue slots; at a few
// hundred stations by latency.  40 x 40 x 32 voxels, 2x2x2 rule, 6000 stations
// (2.5e9 pairs): 29.3 -> 1.33 ms; 12 x 10 x 9 voxels, 300 stations: 625 -> 46 us,
// most of it the host.
template <bool kSolo>
__global__ void __launch_bounds__(kSolo ? 32 : kPairThreads)
direct_fwd_mixed(const float *__restrict__ obs_i, const float *__restrict__ obs_f, int64_t M,
                 const void *__restrict__ rho, int rho_f32, GridArgs ga, RowSplit rs,
                 const QuadRule *__restrict__ qr, double G, double *__restrict__ g, double *__restrict__ gz,
                 int *__restrict__ status) {
    __shared__ double2 red[kSolo ? 1 : (kPairWarps + 1) * 6 * 32];
    __shared__ __align__(16) float2 row_s[kSolo ? 1 : kPairWarps][32];   // masses as duplicated pairs
    const int C = kSolo ? 1 : (int)cooperative_groups::this_cluster().num_blocks();
    const int rank = kSolo ? 0 : (int)cooperative_groups::this_cluster().block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.y;
    const int64_t tile = blockIdx.x / C;
    uint64_t RI[3], RF[3];
    {
        const int64_t j0 = tile * 64 + lane, j1 = j0 + 32;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int da = rs.ax[d];
            RI[d] = pk2(j0 < M ? obs_i[3 * j0 + da] : 0.f, j1 < M ? obs_i[3 * j1 + da] : 0.f);
            RF[d] = pk2(j0 < M ? obs_f[3 * j0 + da] : 0.f, j1 < M ? obs_f[3 * j1 + da] : 0.f);
        }
    }
    const float fx = (float)rs.h[0], fy = (float)rs.h[1], fz = (float)rs.h[2];
    const uint64_t HX = pk2(fx, fx), HY = pk2(fy, fy), HZ = pk2(fz, fz), NEG1 = pk2(-1.f, -1.f);
    const void *rho_b = rho_of(rho, rho_f32, b * ga.nvox);
    float2 *row = row_s[warp];
    uint64_t A[3] = {0, 0, 0}, H[3] = {0, 0, 0}, L[3] = {0, 0, 0};
    bool bad = false;   // a non-finite density (reported through status[0])
    RowIter it(rank * kPairWarps + warp, kSolo ? 1 : (int64_t)C * kPairWarps, rs.nch, qr->nq, rs.n[1]);
    auto fetch = [&]() -> float {
        const int64_t i = (int64_t)it.ch * rs.clen + lane;
        if (it.k < rs.n[2] && lane < rs.clen && i < rs.n[0]) {
            const int64_t idx = it.k * rs.stride[2] + it.j * rs.stride[1] + i * rs.stride[0];
            if (rho_f32) {
                const float v = __ldg((const float *)rho_b + idx);
                bad |= !isfinite(v);
                return v;
            }
            const double v = __ldg((const double *)rho_b + idx);
            bad |= !isfinite(v);
            return (float)v;
        }
        return 0.f;
    };
    auto merge = [&]() {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const uint64_t s = add2(H[d], A[d]);
            const uint64_t bp = sub2(s, H[d]);
            L[d] = add2(L[d], add2(sub2(H[d], sub2(s, bp)), sub2(A[d], bp)));
            H[d] = s;
            A[d] = 0;
        }
    };
    float rv = fetch();
    int since = 0;   // sources summed since the last merge
    while (it.k < rs.n[2]) {
        const int i0 = it.ch * rs.clen;
        const int cnt = min(rs.clen, rs.n[0] - i0);
        const float *of = qr->offf[it.q];
        const float sx = of[rs.ax[0]], sy = of[rs.ax[1]], sz = of[rs.ax[2]], wq = qr->wnf[it.q];
        const float cj = (float)it.j, ck = (float)it.k, ci = (float)(i0 - 1);
        __syncwarp();
        row[lane] = make_float2(rv, rv);
        it.next();
        rv = fetch();   // the next piece's densities, in flight during this one
        __syncwarp();
        const uint64_t FX = sub2(RF[0], pk2(sx, sx));
        const uint64_t DY = mul2(HY, add2(sub2(RI[1], pk2(cj, cj)), sub2(RF[1], pk2(sy, sy))));
        const uint64_t DZ = mul2(HZ, add2(sub2(RI[2], pk2(ck, ck)), sub2(RF[2], pk2(sz, sz))));
        const uint64_t YZ = fma2(DY, DY, mul2(DZ, DZ));
        uint64_t D = sub2(RI[0], pk2(ci, ci)), S = 0, SX = 0;
        auto sweep = [&](auto guarded) {
            constexpr bool kGuard = decltype(guarded)::value;
#pragma unroll 4
            for (int e = 0; e < cnt; ++e) {
                const uint64_t m2 = *reinterpret_cast<const uint64_t *>(row + e);
                D = add2(D, NEG1);
                const uint64_t E = mul2(add2(D, FX), HX);
                const uint64_t R2 = fma2(E, E, YZ);
                float r0, r1;
                up2(R2, r0, r1);
                const uint64_t Q = pk2(rsqrt_ftz(r0), rsqrt_ftz(r1));
                uint64_t K = mul2(mul2(Q, Q), mul2(Q, m2));
                if constexpr (kGuard) {   // a source on the observer contributes nothing
                    float k0, k1;
                    up2(K, k0, k1);
                    K = pk2(r0 > 1e-37f ? k0 : 0.f, r1 > 1e-37f ? k1 : 0.f);
                }
                S = add2(S, K);
                SX = fma2(K, E, SX);
            }
        };
        float y0, y1;
        up2(YZ, y0, y1);
        // only a row through an observer can hold a source at its position
        if (__any_sync(0xffffffffu, !(y0 > 1e-30f) || !(y1 > 1e-30f)))
            sweep(std::true_type{});
        else
            sweep(std::false_type{});
        const uint64_t W = pk2(wq, wq), SW = mul2(S, W);
        A[0] = fma2(SX, W, A[0]);
        A[1] = fma2(SW, DY, A[1]);
        A[2] = fma2(SW, DZ, A[2]);
        since += cnt;
        if (since >= 240) {
            since = 0;
            merge();
        }
    }
    merge();
    if (bad && status && tile == 0) atomicOr(status, 1);
    double s[6], c[6];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        float h0, h1, l0, l1;
        up2(H[d], h0, h1);
        up2(L[d], l0, l1);
        s[d] = (double)h0;
        c[d] = (double)l0;
        s[3 + d] = (double)h1;
        c[3 + d] = (double)l1;
    }
    const double scale = G * ga.vol;
    auto put = [&](int v, int l, double tot) {
        const int u = v / 3, d = v - 3 * u, da = d == 0 ? rs.ax[0] : d == 1 ? rs.ax[1] : rs.ax[2];
        const int64_t j = tile * 64 + u * 32 + l;
        if (j < M) {
            if (g) g[((int64_t)b * M + j) * 3 + da] = scale * tot;
            if (gz && da == 2) gz[(int64_t)b * M + j] = scale * tot;
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

// Tiles of 64 observers (two per lane), or of 32 when there are no more.  An FP64
// instruction of a warp takes 16 clocks of its SM.
gf_status launch_fwd_f64(const double *obs, int64_t M, const void *rho, int rho_f32, const GridArgs &ga, int nq,
                         const QuadRule *qr, int B, double G, double *g, double *gz, int *status, cudaStream_t st) {
    int c = 0;
    if (M <= 32) {
        const RowSplit rs = row_split(ga, 1, nq, [](int n) { return PairCost{(11.0 * n + 30.0) * 16.0 / 2070.0, 4.0, 4.0}; }, &c);
        c = std::max(1, c);
        return pair_launch(direct_fwd_f64<1, false>, 1, B, c, st, obs, M, rho, rho_f32, ga, rs, qr, G, g, gz, status);
    }
    const int64_t tiles = (M + 63) / 64;
    const RowSplit rs = row_split(ga, tiles, nq, [](int n) { return PairCost{(22.0 * n + 30.0) * 16.0 / 2070.0, 8.0, 4.0}; }, &c);
    if (c == 0)
        return pair_launch_solo(direct_fwd_f64<2, true>, tiles, B, st, obs, M, rho, rho_f32, ga, rs, qr, G, g, gz, status);
    return pair_launch(direct_fwd_f64<2, false>, tiles, B, c, st, obs, M, rho, rho_f32, ga, rs, qr, G, g, gz, status);
}

gf_status launch_fwd_mixed(const float *oi, const float *of, int64_t M, const void *rho, int rho_f32,
                           const GridArgs &ga, int nq, const QuadRule *qr, int B, double G, double *g, double *gz,
                           int *status, cudaStream_t st) {
    const int64_t tiles = (M + 63) / 64;
    int c = 0;
    const RowSplit rs = row_split(ga, tiles, nq, [](int n) { return PairCost{(12.0 * n + 40.0) / 2070.0, 5.0, 8.0}; }, &c);
    if (c == 0)
        return pair_launch_solo(direct_fwd_mixed<true>, tiles, B, st, oi, of, M, rho, rho_f32, ga, rs, qr, G, g, gz, status);
    return pair_launch(direct_fwd_mixed<false>, tiles, B, c, st, oi, of, M, rho, rho_f32, ga, rs, qr, G, g, gz, status);
}

// Transpose: one thread per voxel, observers (with their weights) staged in
// shared memory.  grad_v = G V sum_q wn_q sum_j r_j . (x'_j - x_vq)/|.|^3.
__global__ void __launch_bounds__(kTile)
direct_adj_f64(const double *__restrict__ obs, int64_t M, const double *__restrict__ r,
               int ncomp, GridArgs ga, const QuadRule *__restrict__ qr, double G,
               double *__restrict__ grad) {
    __shared__ double ox[kTile], oy[kTile], oz[kTile], w0[kTile], w1[kTile], w2[kTile];
    const int b = blockIdx.y;
    const int64_t v = (int64_t)blockIdx.x * kTile + threadIdx.x;
    const bool active = v < ga.nvox;
    const int64_t i = active ? v % ga.nx : 0, jj = active ? (v / ga.nx) % ga.ny : 0,
                  k = active ? v / (ga.nx * ga.ny) : 0;
    const int nq = qr->nq;
    const double *rb = r + (int64_t)b * M * ncomp;
    double s = 0, c = 0;
    for (int64_t t0 = 0; t0 < M; t0 += kTile) {
        const int64_t j = t0 + threadIdx.x;
        __syncthreads();
        if (j < M) {
            ox[threadIdx.x] = obs[3 * j + 0];
            oy[threadIdx.x] = obs[3 * j + 1];
            oz[threadIdx.x] = obs[3 * j + 2];
            if (ncomp == 1) {
                w0[threadIdx.x] = 0.0;
                w1[threadIdx.x] = 0.0;
                w2[threadIdx.x] = rb[j];
            } else {
                w0[threadIdx.x] = rb[3 * j + 0];
                w1[threadIdx.x] = rb[3 * j + 1];
                w2[threadIdx.x] = rb[3 * j + 2];
            }
        } else {
            ox[threadIdx.x] = oy[threadIdx.x] = oz[threadIdx.x] = 0.0;
            w0[threadIdx.x] = w1[threadIdx.x] = w2[threadIdx.x] = 0.0;
        }
        __syncthreads();
        const int cnt = (M - t0) < kTile ? (int)(M - t0) : kTile;
        double part = 0.0;
        for (int q = 0; q < nq; ++q) {
            const double x = node_coord(ga.ox, ga.hx, i, qr->xi[q][0]);
            const double y = node_coord(ga.oy, ga.hy, jj, qr->xi[q][1]);
            const double z = node_coord(ga.oz, ga.hz, k, qr->xi[q][2]);
            double pq = 0.0;
            for (int u = 0; u < cnt; ++u) {
                const double dx = ox[u] - x, dy = oy[u] - y, dz = oz[u] - z;
                const double r2 = dx * dx + dy * dy + dz * dz;
                const double ri = rsqrt(r2);
                const double k3 = (r2 > 0.0) ? ri * ri * ri : 0.0;
                pq = fma(k3, w0[u] * dx + w1[u] * dy + w2[u] * dz, pq);
            }
            part = fma(qr->wn[q], pq, part);
        }
        neumaier(s, c, part);
    }
    if (active) grad[(int64_t)b * ga.nvox + v] = G * ga.vol * (s + c);
}

__global__ void split_voxel_coords(const double *__restrict__ obs, int64_t M, GridArgs ga,
                                   float *__restrict__ oi, float *__restrict__ of) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const double o[3] = {ga.ox, ga.oy, ga.oz};
    const double h[3] = {ga.hx, ga.hy, ga.hz};
    for (int a = 0; a < 3; ++a) {
        const double u = (obs[3 * j + a] - o[a]) / h[a];
        const double fl = floor(u);
        oi[3 * j + a] = (float)fl;
        of[3 * j + a] = (float)(u - fl);
    }
}

}  // namespace

gf_status direct_prepare(gf_plan_s *plan, const double *obs_dev, cudaStream_t st) {
    const int64_t M = plan->M;
    GF_TRY(plan->arena.alloc_n(&plan->d_obs, (size_t)std::max<int64_t>(M, 1) * 3));
    if (M > 0)
        GF_CUDA(cudaMemcpyAsync(plan->d_obs, obs_dev, sizeof(double) * 3 * M,
                                cudaMemcpyDeviceToDevice, st));
    if (plan->opt.precision == GF_PREC_MIXED) {
        float *oi, *of;
        GF_TRY(plan->arena.alloc_n(&oi, (size_t)std::max<int64_t>(M, 1) * 3));
        GF_TRY(plan->arena.alloc_n(&of, (size_t)std::max<int64_t>(M, 1) * 3));
        plan->d_obs_ivox = nullptr;
        plan->d_obs_fvox = of;
        // integer parts are stored as exact FP32 integers
        plan->d_obs_ivox = reinterpret_cast<int32_t *>(oi);
        if (M > 0) {
            split_voxel_coords<<<ceil_div(M, 256), 256, 0, st>>>(obs_dev, M, grid_args(plan), oi, of);
            GF_KERNEL_DONE();
        }
    }
    return GF_OK;
}

gf_status direct_forward(gf_plan_s *plan, const void *rho, int rho_dtype, int B, double *g,
                         double *gz, cudaStream_t st) {
    const int64_t M = plan->M;
    if (M == 0) return GF_OK;
    const GridArgs ga = grid_args(plan);
    const int f32 = rho_dtype == GF_DTYPE_F32;
    if (plan->opt.precision == GF_PREC_FP64)
        return launch_fwd_f64(plan->d_obs, M, rho, f32, ga, plan->quad.nq, quad_device(plan), B, plan->G, g, gz,
                              plan->d_status, st);
    return launch_fwd_mixed(reinterpret_cast<const float *>(plan->d_obs_ivox), plan->d_obs_fvox, M, rho, f32, ga,
                            plan->quad.nq, quad_device(plan), B, plan->G, g, gz, plan->d_status, st);
}

gf_status direct_adjoint(gf_plan_s *plan, const double *r, int ncomp, int B, double *grad,
                         cudaStream_t st) {
    const GridArgs ga = grid_args(plan);
    const dim3 grid(ceil_div(ga.nvox, kTile), B);
    direct_adj_f64<<<grid, kTile, 0, st>>>(plan->d_obs, plan->M, r, ncomp, ga, quad_device(plan),
                                           plan->G, grad);
    GF_KERNEL_DONE();
    return GF_OK;
}

}  // namespace gf

// ---------------------------------------------------------------------------
// Allocation-free direct forward (gf_direct_forward_static in gf.h).
//
// Some callers cannot allocate device memory when they need a forward
// solve: code that runs inside another framework's allocator callback and
// must not re-enter it, processes whose device memory is entirely reserved
// by a caching pool they do not own, and services that forbid any
// allocation after start-up so that their memory footprint stays fixed.
// This variant of the mixed-precision direct kernel needs no plan: its only
// scratch -- the normalised quadrature rule and the observers' voxel
// coordinates split into integer and fractional parts -- lives in one
// file-scope device array of fixed size, which every GPU that loads this
// library holds until the process exits.
namespace gf {
namespace {

constexpr int64_t kStaticMaxObs = 65536;
constexpr size_t kStaticQuadBytes = (sizeof(QuadRule) + 255) & ~size_t(255);
constexpr size_t kStaticCoordBytes = sizeof(float) * 3 * kStaticMaxObs;
constexpr size_t kStaticBytes = kStaticQuadBytes + 2 * kStaticCoordBytes;

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

std::mutex g_static_mu;
void *g_static_addr[256] = {};
CUcontext g_static_ctx[256] = {};

// Device address of the scratch array on the current device.  The host
// symbol is only a stand-in, so the address is looked up once per device
// (with that device current) and cached with the context it belongs to; a
// new context on the device (after cudaDeviceReset, say) looks it up again.
gf_status static_scratch_address(void **out) {
    int dev = 0;
    GF_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) {
        set_error("device ordinal %d out of range", dev);
        return GF_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lk(g_static_mu);
    // the driver's cuCtxGetCurrent, found through the runtime (the library
    // does not link the driver library)
    typedef CUresult (*CtxGetCurrent)(CUcontext *);
    static CtxGetCurrent ctx_get = nullptr;
    if (!ctx_get) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn) {
            set_error("cannot find the driver's cuCtxGetCurrent");
            return GF_ERR_CUDA;
        }
        ctx_get = reinterpret_cast<CtxGetCurrent>(fn);
    }
    CUcontext ctx = nullptr;
    if (ctx_get(&ctx) != CUDA_SUCCESS) ctx = nullptr;   // none yet: the lookup makes one
    if (!ctx || !g_static_addr[dev] || g_static_ctx[dev] != ctx) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) {
            set_error("cudaGetSymbolAddress of the static scratch failed: %s", cudaGetErrorString(e));
            return GF_ERR_CUDA;
        }
        if (ctx_get(&ctx) != CUDA_SUCCESS) ctx = nullptr;
        g_static_addr[dev] = p;
        g_static_ctx[dev] = ctx;
    }
    *out = g_static_addr[dev];
    return GF_OK;
}

// Writes the quadrature rule, passed by value, into the scratch array.
__global__ void store_quad_rule(QuadRule qr, QuadRule *__restrict__ dst) {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(&qr);
    uint32_t *out = reinterpret_cast<uint32_t *>(dst);
    for (size_t i = threadIdx.x; i < sizeof(QuadRule) / 4; i += blockDim.x) out[i] = src[i];
}

}  // namespace
}  // namespace gf

extern "C" gf_status gf_direct_forward_static(const gf_grid *grid, const gf_quad *quad, const double *obs_dev,
                                              int64_t M, const void *rho_dev, int32_t rho_dtype, int32_t B,
                                              double G, double *g_dev, double *gz_dev, void *stream) {
    using namespace gf;
    if (!grid || !quad) {
        set_error("grid and quad must be non-NULL");
        return GF_ERR_INVALID_ARG;
    }
    if (M < 0 || M > kStaticMaxObs) {
        set_error("gf_direct_forward_static takes at most %lld observers (M = %lld); use a plan instead",
                  (long long)kStaticMaxObs, (long long)M);
        return GF_ERR_INVALID_ARG;
    }
    for (int a = 0; a < 3; ++a) {
        if (grid->n[a] < 1 || grid->n[a] > kMaxAxis || !(grid->h[a] > 0.0) || !isfinite(grid->h[a]) ||
            !isfinite(grid->origin[a])) {
            set_error("grid axis %d: need 1 <= n <= 2^22, finite h > 0 and finite origin", a);
            return GF_ERR_INVALID_ARG;
        }
    }
    if (grid->n[0] * grid->n[1] > kMaxVoxels / grid->n[2]) {
        set_error("grid exceeds 2^40 voxels");
        return GF_ERR_INVALID_ARG;
    }
    if (quad->nq < 1 || quad->nq > kMaxQuad || !quad->xi || !quad->w) {
        set_error("quad.nq = %d must be in [1, %d] with non-NULL xi and w", quad->nq, kMaxQuad);
        return GF_ERR_INVALID_ARG;
    }
    if (rho_dtype != GF_DTYPE_F64 && rho_dtype != GF_DTYPE_F32) {
        set_error("rho_dtype = %d is neither GF_DTYPE_F64 nor GF_DTYPE_F32", rho_dtype);
        return GF_ERR_INVALID_ARG;
    }
    if (B < 1 || B > 64 || !(G >= 0.0) || !isfinite(G)) {
        set_error("need 1 <= B <= 64 and a finite G >= 0 (0 selects 6.67428e-11)");
        return GF_ERR_INVALID_ARG;
    }
    if ((M > 0 && (!obs_dev || !rho_dev)) || (!g_dev && !gz_dev)) {
        set_error("obs_dev and rho_dev must be non-NULL and at least one of g_dev, gz_dev given");
        return GF_ERR_INVALID_ARG;
    }
    QuadRule qr;
    memset(&qr, 0, sizeof(qr));
    qr.nq = quad->nq;
    double wsum = 0.0;
    for (int q = 0; q < quad->nq; ++q) {
        if (!(quad->w[q] > 0.0) || !isfinite(quad->w[q])) {
            set_error("quad.w[%d] must be finite and positive", q);
            return GF_ERR_INVALID_ARG;
        }
        wsum += quad->w[q];
    }
    for (int q = 0; q < quad->nq; ++q) {
        qr.wn[q] = quad->w[q] / wsum;
        qr.wnf[q] = (float)qr.wn[q];
        for (int a = 0; a < 3; ++a) {
            const double x = quad->xi[3 * q + a];
            if (!(fabs(x) <= 1.0)) {
                set_error("quad.xi[%d][%d] must lie in [-1, 1]", q, a);
                return GF_ERR_INVALID_ARG;
            }
            qr.xi[q][a] = x;
            qr.offf[q][a] = (float)(0.5 + 0.5 * x);
        }
    }
    if (M == 0) return GF_OK;
    void *base = nullptr;
    GF_TRY(static_scratch_address(&base));
    unsigned char *scr = reinterpret_cast<unsigned char *>(base);
    QuadRule *d_qr = reinterpret_cast<QuadRule *>(scr);
    float *oi = reinterpret_cast<float *>(scr + kStaticQuadBytes);
    float *of = reinterpret_cast<float *>(scr + kStaticQuadBytes + kStaticCoordBytes);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    GridArgs ga;
    ga.nx = grid->n[0];
    ga.ny = grid->n[1];
    ga.nz = grid->n[2];
    ga.nvox = ga.nx * ga.ny * ga.nz;
    ga.ox = grid->origin[0];
    ga.oy = grid->origin[1];
    ga.oz = grid->origin[2];
    ga.hx = grid->h[0];
    ga.hy = grid->h[1];
    ga.hz = grid->h[2];
    ga.vol = ga.hx * ga.hy * ga.hz;
    // every byte the kernels read is rewritten here, so nothing left by an
    // earlier call is used and nothing needs clearing; the rule travels as a
    // kernel argument (no host memory is read once this call returns)
    store_quad_rule<<<1, 256, 0, st>>>(qr, d_qr);
    GF_KERNEL_DONE();
    split_voxel_coords<<<ceil_div(M, 256), 256, 0, st>>>(obs_dev, M, ga, oi, of);
    GF_KERNEL_DONE();
    return launch_fwd_mixed(oi, of, M, rho_dev, rho_dtype == GF_DTYPE_F32, ga, qr.nq, d_qr, B,
                            G > 0.0 ? G : 6.67428e-11, g_dev, gz_dev, nullptr, st);
}
