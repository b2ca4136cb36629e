// gf_fmm.cu -- the FMM of Sec. 2.3 on the GPU: operator tables, upward sweep
// (P2M, M2M), downward sweep (M2L over the interaction list, L2L) and field
// evaluation (L2P plus the near-field direct sum, Eq. 10).
//
// Every kernel here works in voxel units (h = 1); see gf_fmm.cuh.  The
// evaluation is two kernels: the near-field sum over the nearest-neighbour
// leaves, left per observer, and the local-expansion gradient with the
// near+far sum in FP64 and the scatter back to the caller's observer order.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "fmm_math.cuh"
#include "gf_fmm.cuh"
#include "gf_m2l.cuh"
#include "gf_simd.cuh"
#include "gf_pair.cuh"
#include "gf_sum_an.cuh"

namespace gf {

namespace {

struct LogFact {
    double v[kLogFactN];
};

LogFact host_logfact() {
    LogFact lf;
    for (int i = 0; i < kLogFactN; ++i) lf.v[i] = lgamma((double)i + 1.0);
    return lf;
}

// One block per operator: 343 M2L slots (the 27 near offsets stay unused),
// then 8 M2M and 8 L2L octants.  Entries are written transposed
// (input component major).
__global__ void build_ops(int p, int K, LogFact lf, double *__restrict__ m2l_d, float *__restrict__ m2l_f,
                          double *__restrict__ m2m_d, float *__restrict__ m2m_f, double *__restrict__ l2l_d,
                          float *__restrict__ l2l_f) {
    extern __shared__ double sh[];
    const int op = blockIdx.x;
    int kind;
    double d[3];
    double *od;
    float *of;
    int H;
    if (op < 343) {
        const int dx = op % 7 - 3, dy = (op / 7) % 7 - 3, dz = op / 49 - 3;
        if (max(abs(dx), max(abs(dy), abs(dz))) <= 1) return;
        kind = OP_M2L;
        d[0] = dx;
        d[1] = dy;
        d[2] = dz;
        H = 2 * p;
        od = m2l_d + (size_t)op * K * K;
        of = m2l_f + (size_t)op * K * K;
    } else {
        const int oct = (op - 343) & 7;
        kind = op < 351 ? OP_M2M : OP_L2L;
        d[0] = ((oct & 1) - 0.5) * 0.5;
        d[1] = (((oct >> 1) & 1) - 0.5) * 0.5;
        d[2] = (((oct >> 2) & 1) - 0.5) * 0.5;
        H = p;
        od = (kind == OP_M2M ? m2m_d : l2l_d) + (size_t)oct * K * K;
        of = (kind == OP_M2M ? m2m_f : l2l_f) + (size_t)oct * K * K;
    }
    const int nt = (H + 1) * (H + 2) / 2;
    double *re = sh, *im = sh + nt;
    if (threadIdx.x == 0) {
        if (kind == OP_M2L)
            irregular_harmonics<double>(H, d[0], d[1], d[2], re, im);
        else
            regular_harmonics<double>(H, d[0], d[1], d[2], re, im);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
        const int c = e / K, k = e - c * K;
        const double v = op_entry(kind, p, k, c, re, im, lf.v);
        od[e] = v;
        of[e] = (float)v;
    }
}

// P2M matrix with the quadrature folded in: P[v][k] = sum_q wn_q *
// (k-th real component of conj R((x_vq - c)/b)), x_vq - c in voxel units.
__global__ void build_p2m(int p, int K, int b, const QuadRule *__restrict__ qr, double *__restrict__ pd,
                          float *__restrict__ pf) {
    extern __shared__ double sh[];
    const int v = blockIdx.x;
    const int lx = v % b, ly = (v / b) % b, lz = v / (b * b);
    const int nt = (p + 1) * (p + 2) / 2;
    double *re = sh, *im = sh + nt, *acc = sh + 2 * nt;
    for (int k = threadIdx.x; k < K; k += blockDim.x) acc[k] = 0.0;
    __syncthreads();
    for (int q = 0; q < qr->nq; ++q) {
        if (threadIdx.x == 0) {
            const double y0 = (lx + 0.5 + 0.5 * qr->xi[q][0] - 0.5 * b) / b;
            const double y1 = (ly + 0.5 + 0.5 * qr->xi[q][1] - 0.5 * b) / b;
            const double y2 = (lz + 0.5 + 0.5 * qr->xi[q][2] - 0.5 * b) / b;
            regular_harmonics<double>(p, y0, y1, y2, re, im);
        }
        __syncthreads();
        const double w = qr->wn[q];
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            int n = (int)sqrt((double)k);
            while (n * n > k) --n;
            while ((n + 1) * (n + 1) <= k) ++n;
            const int ro = k - n * n, m = (ro + 1) / 2;
            const bool isim = ro > 0 && (ro % 2 == 0);
            acc[k] += isim ? -w * im[tri(n, m)] : w * re[tri(n, m)];
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        pd[(size_t)v * K + k] = acc[k];
        pf[(size_t)v * K + k] = (float)acc[k];
    }
}

// P2M into the parent level of the child at the all-positive position 7:
// Q[v][k] = sum_i P[v][i] T_7[i][k] (T_7 its M2M operator, input component
// major), the parent expansion of unit mass at voxel v of that child.  The
// other children's are its mirror images (gf_xlate.cu).  One block per voxel.
__global__ void compose_p2m_up(const double *__restrict__ P, const double *__restrict__ T7, int K,
                               double *__restrict__ Q, float *__restrict__ Qf) {
    const double *pv = P + (size_t)blockIdx.x * K;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        double s = 0.0;
        for (int i = 0; i < K; ++i) s += pv[i] * T7[(size_t)i * K + k];
        Q[(size_t)blockIdx.x * K + k] = s;
        Qf[(size_t)blockIdx.x * K + k] = (float)s;
    }
}

// Shift of an expansion by a rule's nodes, for a leaf (block 0) and its parent
// (block 1): S[c][k] = sum_q wn_q T_q[c][k], T_q the M2M by node q's offset from the
// voxel's centre without the M2M's change of scale (2^-degree of the input).
__global__ void build_shift(int p, int K, int b, const QuadRule *__restrict__ qr, LogFact lf, double *__restrict__ sd,
                            float *__restrict__ sf) {
    extern __shared__ double sh[];
    const double unit = 0.5 / ((double)b * (blockIdx.x + 1));
    const int nt = (p + 1) * (p + 2) / 2;
    double *re = sh, *im = sh + nt;
    double *out = sd + (size_t)blockIdx.x * K * K;
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) out[e] = 0.0;
    for (int q = 0; q < qr->nq; ++q) {
        __syncthreads();
        if (threadIdx.x == 0)
            regular_harmonics<double>(p, unit * qr->xi[q][0], unit * qr->xi[q][1], unit * qr->xi[q][2], re, im);
        __syncthreads();
        for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
            const int c = e / K;
            out[e] += qr->wn[q] * ldexp(op_entry(OP_M2M, p, e - c * K, c, re, im, lf.v), (int)sqrt(c + 0.5));
        }
    }
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) sf[(size_t)blockIdx.x * K * K + e] = (float)out[e];
}

// The P2M matrices of position 7 transposed for the adjoint, rows in class
// order: ut[c][v] = Q[v][perm_c], lt[c][v] = P[octant voxel v][perm_c] (zeros for
// perm_c = -1).  One block per row.
__global__ void transpose_p2m(const double *__restrict__ P, const double *__restrict__ Q, const int *__restrict__ perm,
                              int K, double *__restrict__ utd, float *__restrict__ utf, double *__restrict__ ltd,
                              float *__restrict__ ltf) {
    const int c = blockIdx.x, v = threadIdx.x, k = perm[c];
    const double q = k >= 0 ? Q[(size_t)v * K + k] : 0.0;
    utd[c * 64 + v] = q;
    utf[c * 64 + v] = (float)q;
    if (v < 8) {
        const double x =
            k >= 0 ? P[(size_t)(((2 + (v >> 2)) * 4 + 2 + ((v >> 1) & 1)) * 4 + 2 + (v & 1)) * K + k] : 0.0;
        ltd[c * 8 + v] = x;
        ltf[c * 8 + v] = (float)x;
    }
}

// P2M matrix of closed-form voxels (SUM-AN): P[v][k] = the k-th real component
// of conj R((x - c)/b) integrated over voxel v (unit volume in voxel units),
// by a Gauss-Legendre rule of m nodes per axis, exact for every regular solid
// harmonic of degree <= 2m - 1.
struct GaussLeg {
    int m;
    double x[16], w[16];   // nodes on [-1, 1], weights summing to 2
};

__global__ void build_p2m_exact(int p, int K, int b, GaussLeg gl, double *__restrict__ pd,
                                float *__restrict__ pf) {
    extern __shared__ double sh[];
    const int v = blockIdx.x;
    const int lx = v % b, ly = (v / b) % b, lz = v / (b * b);
    const int nt = (p + 1) * (p + 2) / 2;
    double *re = sh, *im = sh + nt, *acc = sh + 2 * nt;
    for (int k = threadIdx.x; k < K; k += blockDim.x) acc[k] = 0.0;
    __syncthreads();
    const int m = gl.m;
    for (int q = 0; q < m * m * m; ++q) {
        const int qi = q % m, qj = (q / m) % m, qk = q / (m * m);
        if (threadIdx.x == 0) {
            const double y0 = (lx + 0.5 + 0.5 * gl.x[qi] - 0.5 * b) / b;
            const double y1 = (ly + 0.5 + 0.5 * gl.x[qj] - 0.5 * b) / b;
            const double y2 = (lz + 0.5 + 0.5 * gl.x[qk] - 0.5 * b) / b;
            regular_harmonics<double>(p, y0, y1, y2, re, im);
        }
        __syncthreads();
        const double w = 0.125 * gl.w[qi] * gl.w[qj] * gl.w[qk];
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            int n = (int)sqrt((double)k);
            while (n * n > k) --n;
            while ((n + 1) * (n + 1) <= k) ++n;
            const int ro = k - n * n, mm = (ro + 1) / 2;
            const bool isim = ro > 0 && (ro % 2 == 0);
            acc[k] += isim ? -w * im[tri(n, mm)] : w * re[tri(n, mm)];
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        pd[(size_t)v * K + k] = acc[k];
        pf[(size_t)v * K + k] = (float)acc[k];
    }
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton's method on the
// three-term recurrence of the Legendre polynomials).
GaussLeg gauss_legendre(int m) {
    GaussLeg g;
    g.m = m;
    for (int i = 0; i < m; ++i) {
        double x = cos(M_PI * (i + 0.75) / (m + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int n = 2; n <= m; ++n) {
                const double pn = ((2.0 * n - 1.0) * x * p1 - (n - 1.0) * p0) / n;
                p0 = p1;
                p1 = pn;
            }
            const double pm = m == 1 ? x : p1, pm1 = m == 1 ? 1.0 : p0;
            dp = m * (x * pm - pm1) / (x * x - 1.0);
            const double dx = pm / dp;
            x -= dx;
            if (fabs(dx) < 1e-16) break;
        }
        g.x[i] = x;
        g.w[i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
    return g;
}

// ---------------------------------------------------------------- sources
struct Block3 {
    int64_t lo[3], n[3];
};

Block3 block_of(const FmmLevel &lv) {
    Block3 b;
    for (int a = 0; a < 3; ++a) {
        b.lo[a] = lv.slo[a];
        b.n[a] = lv.sn[a];
    }
    return b;
}

// Leaf-blocked densities: mass[leaf][bb][v] = rho of the grid voxel that
// sits at local position v of the leaf (0 outside the grid).  Flags any
// non-finite density in status[0].
template <class Tm>
__global__ void block_densities(const void *__restrict__ rho, int rho_f32, int64_t nx, int64_t ny, int64_t nz,
                                int64_t vx, int64_t vy, int64_t vz, Block3 blk, int b, int B,
                                Tm *__restrict__ mass, int *__restrict__ status) {
    const int64_t b3 = (int64_t)b * b * b;
    const int64_t total = blk.n[0] * blk.n[1] * blk.n[2] * B * b3;
    const int64_t nvox = nx * ny * nz;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = e % b3;
        const int64_t rest = e / b3;
        const int bb = (int)(rest % B);
        const int64_t leaf = rest / B;
        const int64_t Lx = blk.lo[0] + leaf % blk.n[0];
        const int64_t Ly = blk.lo[1] + (leaf / blk.n[0]) % blk.n[1];
        const int64_t Lz = blk.lo[2] + leaf / (blk.n[0] * blk.n[1]);
        const int64_t i = Lx * b + v % b - vx;
        const int64_t j = Ly * b + (v / b) % b - vy;
        const int64_t k = Lz * b + v / ((int64_t)b * b) - vz;
        Tm m = Tm(0);
        if (i >= 0 && i < nx && j >= 0 && j < ny && k >= 0 && k < nz) {
            const int64_t idx = (int64_t)bb * nvox + (k * ny + j) * nx + i;
            const double r = rho_f32 ? (double)reinterpret_cast<const float *>(rho)[idx]
                                     : reinterpret_cast<const double *>(rho)[idx];
            if (!isfinite(r)) atomicOr(status, 1);
            m = (Tm)r;
        }
        mass[e] = m;
    }
}

// P2M: ME[leaf][bb][k] = sum_v P[v][k] mass[leaf][bb][v].  A block handles
// kP2MLeaves leaves; each thread owns coefficients k, k + blockDim, ...
constexpr int kP2MLeaves = 4;

template <class T>
__global__ void __launch_bounds__(128)
p2m_kernel(const T *__restrict__ mass, const T *__restrict__ P, int64_t nleaf, int b3, int B, int K,
           int ldk, T *__restrict__ me) {
    extern __shared__ unsigned char shraw[];
    T *ms = reinterpret_cast<T *>(shraw);  // [kP2MLeaves*B][b3]
    const int64_t leaf0 = (int64_t)blockIdx.x * kP2MLeaves;
    const int nl = (int)std::min<int64_t>(kP2MLeaves, nleaf - leaf0);
    const int ncol = nl * B;
    for (int e = threadIdx.x; e < ncol * b3; e += blockDim.x) ms[e] = mass[leaf0 * B * b3 + e];
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        T acc[kP2MLeaves * 4];
        for (int c0 = 0; c0 < ncol; c0 += kP2MLeaves * 4) {
            const int cn = std::min(kP2MLeaves * 4, ncol - c0);
#pragma unroll
            for (int c = 0; c < kP2MLeaves * 4; ++c) acc[c] = T(0);
            for (int v = 0; v < b3; ++v) {
                const T pv = P[(size_t)v * K + k];
#pragma unroll
                for (int c = 0; c < kP2MLeaves * 4; ++c)
                    if (c < cn) acc[c] += pv * ms[(c0 + c) * b3 + v];
            }
#pragma unroll
            for (int c = 0; c < kP2MLeaves * 4; ++c)
                if (c < cn) me[(leaf0 * B + c0 + c) * ldk + k] = acc[c];
        }
    }
}

// Fused a0 + a3 for leaves of at most 4^3 voxels: a block takes a 4x4x4
// tile of leaves for one batch member, reads their densities straight from
// the caller's grid (rows of 4b contiguous voxels), writes the leaf-blocked
// copy used by the near field, and multiplies the 64 leaves' masses by the
// P2M matrix held in shared memory: ME[leaf][k] = sum_v P[v][k] mass[leaf][v].
// Thread (tl, tk) of 16 x 16 owns leaves 4tl..4tl+3 and coefficients
// tk + 16j, j < RPT.
constexpr int kFTile = 4;                       // leaves per tile edge
constexpr int kFLeaves = kFTile * kFTile * kFTile;
constexpr int kFPitch = kFLeaves + 4;           // padded row of the mass tile (bank spread)

__host__ __device__ inline int p2m_fused_pitch(int K) { return (K + 15) & ~15; }

template <class T>
__host__ __device__ inline size_t p2m_fused_smem(int b3, int K, int ldk) {
    const size_t in = (size_t)b3 * p2m_fused_pitch(K) + (size_t)b3 * kFPitch;
    const size_t out = (size_t)kFLeaves * ldk;
    return sizeof(T) * (in > out ? in : out);
}

template <class T, int BV, int RPT>
__global__ void __launch_bounds__(256)
p2m_fused(const void *__restrict__ rho, int rho_f32, int64_t nx, int64_t ny, int64_t nz, int64_t vx, int64_t vy,
          int64_t vz, Block3 blk, int B, const T *__restrict__ P, int K, int ldk, T *__restrict__ mass,
          T *__restrict__ me, int *__restrict__ status) {
    extern __shared__ unsigned char shraw[];
    constexpr int b3 = BV * BV * BV;
    constexpr int e4 = kFTile * BV;   // voxels per tile edge
    const int KP = p2m_fused_pitch(K);
    T *Ps = reinterpret_cast<T *>(shraw);   // [b3][KP]
    T *ms = Ps + (size_t)b3 * KP;           // [b3][kFPitch]: voxel-major, leaf-minor
    T *os = reinterpret_cast<T *>(shraw);   // [64][ldk] (after the product)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bb = blockIdx.y;
    const int64_t ntx = (blk.n[0] + kFTile - 1) / kFTile, nty = (blk.n[1] + kFTile - 1) / kFTile;
    const int64_t tile = blockIdx.x;
    const int64_t l0x = (tile % ntx) * kFTile, l0y = ((tile / ntx) % nty) * kFTile, l0z = tile / (ntx * nty) * kFTile;
    for (int v = warp; v < b3; v += 8)
        for (int k = lane; k < KP; k += 32) Ps[v * KP + k] = k < K ? P[(size_t)v * K + k] : T(0);
    // densities of the tile's (4b)^3 voxels, x fastest (coalesced rows)
    const int64_t nvox = nx * ny * nz;
    const int64_t gx0 = (blk.lo[0] + l0x) * BV - vx, gy0 = (blk.lo[1] + l0y) * BV - vy,
                  gz0 = (blk.lo[2] + l0z) * BV - vz;
    bool bad = false;
    for (int e = tid; e < e4 * e4 * e4; e += 256) {
        const int ix = e % e4, iy = (e / e4) % e4, iz = e / (e4 * e4);
        const int64_t i = gx0 + ix, j = gy0 + iy, k = gz0 + iz;
        T m = T(0);
        if (i >= 0 && i < nx && j >= 0 && j < ny && k >= 0 && k < nz) {
            const int64_t idx = (int64_t)bb * nvox + (k * ny + j) * nx + i;
            const double r = rho_f32 ? (double)reinterpret_cast<const float *>(rho)[idx]
                                     : reinterpret_cast<const double *>(rho)[idx];
            bad |= !isfinite(r);
            m = (T)r;
        }
        const int leaf = ((iz / BV) * kFTile + iy / BV) * kFTile + ix / BV;
        const int v = ((iz % BV) * BV + iy % BV) * BV + ix % BV;
        ms[v * kFPitch + leaf] = m;
    }
    if (bad) atomicOr(status, 1);
    __syncthreads();
    // leaf-blocked masses for the near field: mass[leaf][bb][v]
    for (int e = tid; e < kFLeaves * b3; e += 256) {
        const int leaf = e / b3, v = e % b3;
        const int64_t gx = l0x + leaf % kFTile, gy = l0y + (leaf / kFTile) % kFTile, gz = l0z + leaf / (kFTile * kFTile);
        if (gx >= blk.n[0] || gy >= blk.n[1] || gz >= blk.n[2]) continue;
        const int64_t gl = (gz * blk.n[1] + gy) * blk.n[0] + gx;
        mass[(gl * B + bb) * b3 + v] = ms[v * kFPitch + leaf];
    }
    const int tl = tid & 15, tk = tid >> 4;
    T acc[4][RPT];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < RPT; ++j) acc[i][j] = T(0);
#pragma unroll 4
    for (int v = 0; v < b3; ++v) {
        T m4[4];
        if constexpr (sizeof(T) == 4) {
            const float4 t4 = *reinterpret_cast<const float4 *>(ms + v * kFPitch + 4 * tl);
            m4[0] = t4.x;
            m4[1] = t4.y;
            m4[2] = t4.z;
            m4[3] = t4.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) m4[i] = ms[v * kFPitch + 4 * tl + i];
        }
        const T *pr = Ps + (size_t)v * KP + tk;
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const T pv = (tk + 16 * j < KP) ? pr[16 * j] : T(0);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i][j] += pv * m4[i];
        }
    }
    __syncthreads();   // Ps and ms are reused as the output staging area
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const int k = tk + 16 * j;
            if (k < ldk) os[(4 * tl + i) * ldk + k] = k < K ? acc[i][j] : T(0);
        }
    __syncthreads();
    for (int leaf = warp; leaf < kFLeaves; leaf += 8) {
        const int64_t gx = l0x + leaf % kFTile, gy = l0y + (leaf / kFTile) % kFTile, gz = l0z + leaf / (kFTile * kFTile);
        if (gx >= blk.n[0] || gy >= blk.n[1] || gz >= blk.n[2]) continue;
        const int64_t gl = (gz * blk.n[1] + gy) * blk.n[0] + gx;
        T *dst = me + (gl * B + bb) * ldk;
        for (int k = lane; k < ldk; k += 32) dst[k] = os[leaf * ldk + k];
    }
}

template <class T, int BV>
gf_status launch_p2m_fused_b(gf_plan_s *plan, const void *rho, int rho_f32, int B, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &lv = F->lev[F->L];
    const int K = F->K;
    const Block3 blk = block_of(lv);
    const int64_t tiles = ((blk.n[0] + kFTile - 1) / kFTile) * ((blk.n[1] + kFTile - 1) / kFTile) *
                          ((blk.n[2] + kFTile - 1) / kFTile);
    const size_t shm = p2m_fused_smem<T>(BV * BV * BV, K, F->KS);
    const T *P = sizeof(T) == 8 ? (const T *)F->p2m_d : (const T *)F->p2m_f;
    const dim3 grid((unsigned)tiles, (unsigned)B);
#define GF_P2M_LAUNCH(R)                                                                                    \
    do {                                                                                                    \
        GF_TRY(ensure_smem(p2m_fused<T, BV, R>, shm));                                                      \
        p2m_fused<T, BV, R><<<grid, 256, shm, st>>>(rho, rho_f32, plan->grid.n[0], plan->grid.n[1],          \
                                                    plan->grid.n[2], F->voff[0], F->voff[1], F->voff[2], blk, B, \
                                                    P, K, F->KS, (T *)F->mass, (T *)lv.me, plan->d_status); \
    } while (0)
    const int rpt = (p2m_fused_pitch(K) + 15) / 16;
    if (rpt <= 4)
        GF_P2M_LAUNCH(4);
    else if (rpt <= 8)
        GF_P2M_LAUNCH(8);
    else if (rpt <= 12)
        GF_P2M_LAUNCH(12);
    else
        GF_P2M_LAUNCH(20);
#undef GF_P2M_LAUNCH
    GF_KERNEL_DONE();
    return GF_OK;
}

// Leaf-blocked densities only (the P2M then runs on the tensor cores):
// thread x of block (y, z) copies the BV voxels of row (y, z) of leaf x --
// consecutive threads read consecutive voxels of the grid row and each
// writes one BV-wide piece of its leaf's mass row.  Grid: (ceil(nLx/128),
// nLy*BV, nLz*BV*B).
template <class T, int BV>
__global__ void __launch_bounds__(128)
block_rows(const void *__restrict__ rho, int rho_f32, int64_t nx, int64_t ny, int64_t nz, int64_t vx, int64_t vy,
           int64_t vz, Block3 blk, int64_t lz0, int64_t nlz, int B, T *__restrict__ mass, int *__restrict__ status) {
    constexpr int b3 = BV * BV * BV;
    const int64_t lx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (lx >= blk.n[0]) return;
    const int yv = blockIdx.y;
    const int64_t zb = blockIdx.z;
    const int64_t nzv = nlz * BV;
    const int zv = (int)(lz0 * BV + zb % nzv);   // voxel layer within the block
    const int bb = (int)(zb / nzv);
    const int64_t j = blk.lo[1] * BV + yv - vy, k = blk.lo[2] * BV + zv - vz;
    const int64_t i0 = (blk.lo[0] + lx) * BV - vx;
    const bool row_in = j >= 0 && j < ny && k >= 0 && k < nz;
    const int64_t base = (int64_t)bb * nx * ny * nz + (k * ny + j) * nx;
    T m[BV];
    bool bad = false;
#pragma unroll
    for (int x = 0; x < BV; ++x) {
        const int64_t i = i0 + x;
        T v = T(0);
        if (row_in && i >= 0 && i < nx) {
            const double r = rho_f32 ? (double)reinterpret_cast<const float *>(rho)[base + i]
                                     : reinterpret_cast<const double *>(rho)[base + i];
            bad |= !isfinite(r);
            v = (T)r;
        }
        m[x] = v;
    }
    if (bad) atomicOr(status, 1);
    const int64_t leaf = ((int64_t)(zv / BV) * blk.n[1] + yv / BV) * blk.n[0] + lx;
    T *dst = mass + (leaf * B + bb) * b3 + ((zv % BV) * BV + yv % BV) * BV;
    if constexpr (BV == 4 && sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(dst) = make_float4(m[0], m[1], m[2], m[3]);
    } else {
#pragma unroll
        for (int x = 0; x < BV; ++x) dst[x] = m[x];
    }
}

template <class T, int BV>
gf_status launch_blocking(gf_plan_s *plan, const void *rho, int rho_f32, int B, int64_t lz0, int64_t nlz,
                          cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const Block3 blk = block_of(F->lev[F->L]);
    if (nlz <= 0) return GF_OK;
    const int64_t gz = nlz * BV * B;
    if (blk.n[1] * BV > 65535 || gz > 65535) {
        set_error("leaf block too large for the density re-blocking grid");
        return GF_ERR_UNSUPPORTED;
    }
    const dim3 grid(ceil_div(blk.n[0], 128), (unsigned)(blk.n[1] * BV), (unsigned)gz);
    block_rows<T, BV><<<grid, 128, 0, st>>>(rho, rho_f32, plan->grid.n[0], plan->grid.n[1], plan->grid.n[2],
                                            F->voff[0], F->voff[1], F->voff[2], blk, lz0, nlz, B, (T *)F->mass,
                                            plan->d_status);
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class T>
gf_status launch_p2m_fused(gf_plan_s *plan, const void *rho, int rho_f32, int B, cudaStream_t st) {
    switch (plan->fmm->b) {
        case 1: return launch_p2m_fused_b<T, 1>(plan, rho, rho_f32, B, st);
        case 2: return launch_p2m_fused_b<T, 2>(plan, rho, rho_f32, B, st);
        case 3: return launch_p2m_fused_b<T, 3>(plan, rho, rho_f32, B, st);
        default: return launch_p2m_fused_b<T, 4>(plan, rho, rho_f32, B, st);
    }
}

// Whether the fused kernel applies (leaves of at most 4^3 voxels, tables
// that fit one block's shared memory).
template <class T>
bool p2m_fused_ok(const FmmPlan *F) {
    const int b3 = F->b * F->b * F->b;
    return F->b <= 4 && p2m_fused_pitch(F->K) <= 320 && p2m_fused_smem<T>(b3, F->K, F->KS) <= 200 * 1024;
}

// ---------------------------------------------------------------- evaluation
constexpr int kEvalWarps = 4;
constexpr int kEvalChunk = 64;
constexpr int kTPL = 2;            // targets per lane: a work item has <= 64 targets
constexpr int kSrcTable = 512;     // per-block table of a leaf's source offsets
constexpr int kMaxLat = 8;         // lattice planes per axis of a leaf (lattice near field)

constexpr int kLatGroups = 4;      // lattice form: lane groups sharing a small item

// Elements of one warp's shared-memory slice of the near-field kernel
// (a multiple of 8): 4 kEvalChunk staged source values (FP32: 8, the
// duplicated lattice weights of up to kLatGroups leaves) and 27
// neighbour-leaf entries (int64).
inline __host__ __device__ int eval_stage(int tsize) { return (tsize == 4 ? 2 : 1) * 4 * kEvalChunk; }
inline __host__ __device__ int eval_slice(int tsize) { return (eval_stage(tsize) + 27 * 8 / tsize + 7) & ~7; }

struct EvalArgs {
    int L;                       // leaf level
    uint32_t part_lo, part_hi;   // source partition (in_source_part)
    const int4 *items;
    int64_t n_items;
    unsigned long long *queue; // [0]: next item, [1]: warps done (zero between launches)
    void *nsum;                // [B][M][6] T: (hi, lo) of x, y, z per observer (key order)
    const uint64_t *tkey;      // leaf keys
    const int32_t *perm;
    const void *tloc;          // [M][3] T
    const void *mass;          // [ns_L][B][b3] T
    const void *le;            // [nt_L][B][ldk] T
    const QuadRule *qr;
    Block3 blk;                // leaf source block
    int b, nq, B, K, ldk, p;
    int64_t M;
    double scale;              // G * h
    double eps2;               // coincidence radius^2 (voxel units)
    int guard_all;             // quadrature nodes on voxel faces: every leaf may hold
                               // a source coincident with an observer (else only
                               // the observer's own leaf can)
    double *g, *gz;
    // Lattice form of a leaf's sources (rules that are tensor products of m
    // nodes per axis): the b^3 nq sources sit on N1^3 lattice points, N1 =
    // b m.  lat_c[a][i]: coordinate of lattice plane i along axis a from the
    // leaf centre (voxel units); lat_q[(ia % m) + m ((ib % m) + m (ic % m))]
    // is the rule's node at lattice point (ia, ib, ic).
    int lat_m;
    float lat_c[3][kMaxLat];
    int lat_q[kMaxQuad];
};

// Near field of the observers of one leaf, its sums (hi, lo) left in nsum for the
// far-field kernel, one warp per work
// item; warps take items from a queue (one atomic per item), so a warp that
// drew a short item takes the next one at once.  The sources of each
// neighbouring leaf are staged in the warp's shared-memory slice in chunks
// of 64 (position relative to the target leaf's centre, mass times
// quadrature weight) and every lane sweeps them for its two observers.
// Per-leaf partial sums are merged with TwoSum.  N1 > 0 (FP32, sources on
// an N1^3 lattice per leaf): the lattice form of the near field below; an
// item of at most 32 observers there splits its neighbour leaves over 2 or
// 4 groups of lanes that hold the same observers, and the groups' sums are
// merged by shuffles.
template <class T, int N1>
__global__ void __launch_bounds__(kEvalWarps * 32, sizeof(T) == 4 ? 5 : 1)   // FP32: 5 blocks (20 warps, 96 registers) per SM
eval_kernel(EvalArgs a) {
    extern __shared__ unsigned char shraw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b3 = a.b * a.b * a.b;
    const int nsrc = b3 * a.nq;
    // block-wide table: offset of source u (voxel u / nq, node u % nq) from
    // its leaf's centre, quadrature weight, voxel index
    Vec4<T> *tab = reinterpret_cast<Vec4<T> *>(shraw);
    int *tvox = reinterpret_cast<int *>(tab + kSrcTable);
    // per-warp slice, a multiple of 8 elements so every slice keeps the
    // alignment of the vector type: staged sources, the item's neighbour leaves
    constexpr bool kF32 = std::is_same<T, float>::value;
    const int wstride = eval_slice(sizeof(T));
    T *wsh = reinterpret_cast<T *>(tvox + kSrcTable) + (size_t)warp * wstride;
    Vec4<T> *src = reinterpret_cast<Vec4<T> *>(wsh);
    int64_t *nbl = reinterpret_cast<int64_t *>(wsh + eval_stage(sizeof(T)));
    const T *tloc = reinterpret_cast<const T *>(a.tloc);
    const T *mass = reinterpret_cast<const T *>(a.mass);
    const T half_b = T(0.5) * T(a.b);
    const T eps2 = (T)a.eps2;
    const bool use_tab = nsrc <= kSrcTable;
    if (N1 > 0) {
        // lattice point n = i + N1 (j + N1 k): its voxel and the rule's weight
        const int m = a.lat_m;
        for (int n = threadIdx.x; n < N1 * N1 * N1; n += blockDim.x) {
            const int i = n % N1, j = (n / N1) % N1, k = n / (N1 * N1);
            const int v = i / m + a.b * (j / m + a.b * (k / m));
            const int q = a.lat_q[i % m + m * (j % m + m * (k % m))];
            tab[n].w = (T)a.qr->wn[q];
            tvox[n] = v;
        }
    } else if (use_tab) {
        for (int u = threadIdx.x; u < nsrc; u += blockDim.x) {
            const int v = u / a.nq, q = u - v * a.nq;
            Vec4<T> e;
            e.x = T(v % a.b) + (T)(0.5 + 0.5 * a.qr->xi[q][0]) - half_b;
            e.y = T((v / a.b) % a.b) + (T)(0.5 + 0.5 * a.qr->xi[q][1]) - half_b;
            e.z = T(v / (a.b * a.b)) + (T)(0.5 + 0.5 * a.qr->xi[q][2]) - half_b;
            e.w = (T)a.qr->wn[q];
            tab[u] = e;
            tvox[u] = v;
        }
    }
    __syncthreads();
    // lattice form: this lane's two lattice points (weight, voxel)
    float lw0 = 0.f, lw1 = 0.f;
    int lv0 = 0, lv1 = 0;
    if (N1 > 0) {
        lw0 = (float)tab[lane].w;
        lw1 = (float)tab[lane + 32].w;
        lv0 = tvox[lane];
        lv1 = tvox[lane + 32];
    }
    for (;;) {
        int64_t it = 0;
        if (lane == 0) it = (int64_t)atomicAdd(a.queue, 1ull);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= a.n_items) break;
        const int4 item = a.items[it];
        const int leaf = item.x;
        // lattice form: lanes per group (gs) and groups (ns) for this item;
        // lane = grp * gs + r0 holds observers r0 and r0 + gs of the item
        int gs = 32;
        if constexpr (N1 > 0 && kF32) {
            const int np = (item.z + 1) >> 1;
            gs = np > 16 ? 32 : np > 8 ? 16 : 32 / kLatGroups;
        }
        const int ns = 32 / gs, grp = lane / gs, r0 = lane - grp * gs;
        int64_t lc[3] = {0, 0, 0};   // the leaf's box coordinates (near field only)
        {
            const uint64_t k = a.tkey[leaf];
            for (int bit = 0; bit < 21; ++bit) {
                lc[0] |= (int64_t)((k >> (3 * bit)) & 1) << bit;
                lc[1] |= (int64_t)((k >> (3 * bit + 1)) & 1) << bit;
                lc[2] |= (int64_t)((k >> (3 * bit + 2)) & 1) << bit;
            }
        }
        T tx[kTPL], ty[kTPL], tz[kTPL];
        int tid[kTPL];
#pragma unroll
        for (int u = 0; u < kTPL; ++u) {
            const int r = r0 + gs * u;
            tid[u] = r < item.z ? item.y + r : -1;
            const int64_t i = tid[u] >= 0 ? tid[u] : item.y;
            tx[u] = tloc[3 * i + 0];
            ty[u] = tloc[3 * i + 1];
            tz[u] = tloc[3 * i + 2];
        }
        // the item's neighbour leaves inside the source block, in the order of
        // nb = (dx + 1) + 3 (dy + 1) + 9 (dz + 1): source-block index * 32 + nb
        __syncwarp();
        int nv = 0;
        {
            bool in = false;
            int64_t sidx = 0;
            if (lane < 27) {
                const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
                const int64_t sx = lc[0] + dx - a.blk.lo[0], sy = lc[1] + dy - a.blk.lo[1],
                              sz = lc[2] + dz - a.blk.lo[2];
                in = sx >= 0 && sy >= 0 && sz >= 0 && sx < a.blk.n[0] && sy < a.blk.n[1] && sz < a.blk.n[2] &&
                     in_source_part(lc[0] + dx, lc[1] + dy, lc[2] + dz, a.L - 2, a.part_lo, a.part_hi);
                sidx = (sz * a.blk.n[1] + sy) * a.blk.n[0] + sx;
            }
            const unsigned vm = __ballot_sync(0xffffffffu, in);
            if (in) nbl[__popc(vm & ((1u << lane) - 1u))] = sidx * 32 + lane;
            nv = __popc(vm);
        }
        __syncwarp();
        for (int bb = 0; bb < a.B; ++bb) {
            T hx[kTPL], hy[kTPL], hz[kTPL], lx[kTPL], ly[kTPL], lz[kTPL];
#pragma unroll
            for (int u = 0; u < kTPL; ++u) hx[u] = hy[u] = hz[u] = lx[u] = ly[u] = lz[u] = T(0);
            // ---- near field: the leaf itself and its nearest neighbours (in the
            // lattice form, group grp takes entries grp, grp + ns, ...; a group
            // past the end computes entry c0's leaf and drops the result)
            for (int c0 = 0; c0 < nv; c0 += ns) {
                const bool act = c0 + grp < nv;
                const int64_t ent = nbl[act ? c0 + grp : c0];
                const int64_t sl = ent >> 5;
                const int nb = (int)(ent & 31);
                const int dx = nb % 3 - 1, dy = (nb / 3) % 3 - 1, dz = nb / 9 - 1;
                const T *ms = mass + (sl * a.B + bb) * b3;
                const T ox = T(dx * a.b), oy = T(dy * a.b), oz = T(dz * a.b);
                if constexpr (N1 > 0 && std::is_same<T, float>::value) {
                    // Lattice form.  With d = t - s and the sources on the planes
                    // x = X_i, y = Y_j, z = Z_k, the leaf's sum of w d / |d|^3 is
                    //   (sum_i dx_i Sx_i, sum_j dy_j Sy_j, sum_k dz_k Sz_k),
                    //   Sx_i = sum_{j,k} w_ijk |d_ijk|^-3  (Sy_j, Sz_k alike),
                    // so a source costs one add (|d|^2 from the squared plane
                    // distances), the reciprocal square root, three multiplies and
                    // three adds; the lane's two observers form one packed pair.
                    constexpr int N3 = N1 * N1 * N1;
                    __syncwarp();
                    float2 *wl = reinterpret_cast<float2 *>(wsh) + grp * N3;
                    static_assert(N1 == 4, "two lattice points per lane, rows of four");
                    if (gs == 32) {
                        const float w0 = lw0 * ms[lv0], w1 = lw1 * ms[lv1];
                        wl[lane] = make_float2(w0, w0);
                        wl[lane + 32] = make_float2(w1, w1);
                    } else {
                        for (int n = r0; n < N3; n += gs) {
                            const float w = (float)tab[n].w * ms[tvox[n]];
                            wl[n] = make_float2(w, w);
                        }
                    }
                    __syncwarp();
                    const uint64_t PX = pk2(tx[0], tx[1]), PY = pk2(ty[0], ty[1]), PZ = pk2(tz[0], tz[1]);
                    uint64_t X2[N1], Y2[N1], SX[N1], SY[N1];
#pragma unroll
                    for (int i = 0; i < N1; ++i) {
                        const float cx = a.lat_c[0][i] + ox, cy = a.lat_c[1][i] + oy;
                        const uint64_t ex = sub2(PX, pk2(cx, cx)), ey = sub2(PY, pk2(cy, cy));
                        X2[i] = mul2(ex, ex);
                        Y2[i] = mul2(ey, ey);
                        SX[i] = SY[i] = 0;
                    }
                    uint64_t QZ = 0;
                    // one z-plane of the lattice at a time (Sz_k is a single sum)
                    auto lattice = [&](auto guarded) {
                        constexpr bool kGuard = decltype(guarded)::value;
#pragma unroll 1
                        for (int k = 0; k < N1; ++k) {
                            const float cz = a.lat_c[2][k] + oz;
                            const uint64_t ez = sub2(PZ, pk2(cz, cz));
                            const uint64_t Z2 = mul2(ez, ez);
                            const uint64_t *wk = reinterpret_cast<const uint64_t *>(wl + N1 * N1 * k);
                            uint64_t SZ = 0;
#pragma unroll
                            for (int j = 0; j < N1; ++j) {
                                const uint64_t YZ = add2(Y2[j], Z2);
                                // the row's four terms: each into its Sx_i, their
                                // pairwise sum once into Sy_j and Sz (short chains)
                                uint64_t K3v[N1];
#pragma unroll
                                for (int i = 0; i < N1; ++i) {
                                    const uint64_t R2 = add2(X2[i], YZ);
                                    float r0, r1;
                                    up2(R2, r0, r1);
                                    float i0 = rsqrt_ftz(r0), i1 = rsqrt_ftz(r1);
                                    if constexpr (kGuard) {
                                        i0 = r0 > (float)eps2 ? i0 : 0.f;
                                        i1 = r1 > (float)eps2 ? i1 : 0.f;
                                    }
                                    const uint64_t RI = pk2(i0, i1);
                                    K3v[i] = mul2(mul2(RI, RI), mul2(RI, wk[i + N1 * j]));
                                    SX[i] = add2(SX[i], K3v[i]);
                                }
                                const uint64_t tj = add2(add2(K3v[0], K3v[1]), add2(K3v[2], K3v[3]));
                                SY[j] = add2(SY[j], tj);
                                SZ = add2(SZ, tj);
                            }
                            QZ = fma2(SZ, ez, QZ);
                        }
                    };
                    if (a.guard_all || __any_sync(0xffffffffu, nb == 13))
                        lattice(std::true_type{});
                    else
                        lattice(std::false_type{});
                    uint64_t QX = 0, QY = 0;
#pragma unroll
                    for (int i = 0; i < N1; ++i) {
                        const float cx = a.lat_c[0][i] + ox, cy = a.lat_c[1][i] + oy;
                        QX = fma2(SX[i], sub2(PX, pk2(cx, cx)), QX);
                        QY = fma2(SY[i], sub2(PY, pk2(cy, cy)), QY);
                    }
                    float gx[2], gy[2], gz[2];
                    up2(QX, gx[0], gx[1]);
                    up2(QY, gy[0], gy[1]);
                    up2(QZ, gz[0], gz[1]);
                    if (act) {
#pragma unroll
                        for (int u = 0; u < kTPL; ++u) {
                            two_sum(hx[u], lx[u], (T)gx[u]);
                            two_sum(hy[u], ly[u], (T)gy[u]);
                            two_sum(hz[u], lz[u], (T)gz[u]);
                        }
                    }
                    continue;
                }
                T px[kTPL], py[kTPL], pz[kTPL];
#pragma unroll
                for (int u = 0; u < kTPL; ++u) px[u] = py[u] = pz[u] = T(0);
                constexpr bool kPacked = std::is_same<T, float>::value;
                uint64_t qx[kTPL], qy[kTPL], qz[kTPL];   // packed partial sums (FP32)
#pragma unroll
                for (int u = 0; u < kTPL; ++u) qx[u] = qy[u] = qz[u] = 0;
                for (int c0 = 0; c0 < nsrc; c0 += kEvalChunk) {
                    const int cnt = min(kEvalChunk, nsrc - c0);
                    __syncwarp();
                    for (int s = lane; s < cnt; s += 32) {
                        const int u = c0 + s;
                        Vec4<T> e;
                        int v;
                        if (use_tab) {
                            e = tab[u];
                            v = tvox[u];
                        } else {
                            v = u / a.nq;
                            const int q = u - v * a.nq;
                            e.x = T(v % a.b) + (T)(0.5 + 0.5 * a.qr->xi[q][0]) - half_b;
                            e.y = T((v / a.b) % a.b) + (T)(0.5 + 0.5 * a.qr->xi[q][1]) - half_b;
                            e.z = T(v / (a.b * a.b)) + (T)(0.5 + 0.5 * a.qr->xi[q][2]) - half_b;
                            e.w = (T)a.qr->wn[q];
                        }
                        e.x += ox;
                        e.y += oy;
                        e.z += oz;
                        e.w *= ms[v];
                        if constexpr (kPacked) {
                            // pairs of sources as {x0,x1, y0,y1, z0,z1, w0,w1}
                            T *rec = wsh + (s >> 1) * 8 + (s & 1);
                            rec[0] = e.x;
                            rec[2] = e.y;
                            rec[4] = e.z;
                            rec[6] = e.w;
                        } else {
                            src[s] = e;
                        }
                    }
                    if constexpr (kPacked) {
                        // an odd chunk ends with a massless source far away
                        if ((cnt & 1) && lane == 0) {
                            T *rec = wsh + (cnt >> 1) * 8 + 1;
                            rec[0] = rec[2] = rec[4] = T(1.0e4);
                            rec[6] = T(0);
                        }
                        __syncwarp();
                        uint64_t TX[kTPL], TY[kTPL], TZ[kTPL];
#pragma unroll
                        for (int u = 0; u < kTPL; ++u) {
                            TX[u] = pk2(tx[u], tx[u]);
                            TY[u] = pk2(ty[u], ty[u]);
                            TZ[u] = pk2(tz[u], tz[u]);
                        }
                        const int npair = (cnt + 1) >> 1;
                        // Only the observer's own leaf (or any leaf, when nodes lie
                        // on voxel faces) can hold a source at the observer's
                        // position; elsewhere r2 > 0 and the coincidence test is
                        // dropped from the pair loop.
                        auto sweep = [&](auto guarded) {
                            constexpr bool kGuard = decltype(guarded)::value;
#pragma unroll 2
                            for (int q = 0; q < npair; ++q) {
                                const ulonglong2 xy = *reinterpret_cast<const ulonglong2 *>(wsh + q * 8);
                                const ulonglong2 zw = *reinterpret_cast<const ulonglong2 *>(wsh + q * 8 + 4);
#pragma unroll
                                for (int u = 0; u < kTPL; ++u) {
                                    const uint64_t DX = sub2(TX[u], xy.x), DY = sub2(TY[u], xy.y),
                                                   DZ = sub2(TZ[u], zw.x);
                                    const uint64_t R2 = fma2(DZ, DZ, fma2(DY, DY, mul2(DX, DX)));
                                    float r0, r1;
                                    up2(R2, r0, r1);
                                    float i0, i1;
                                    if constexpr (kGuard) {
                                        i0 = r0 > (float)eps2 ? rsqrt_ftz(r0) : 0.f;
                                        i1 = r1 > (float)eps2 ? rsqrt_ftz(r1) : 0.f;
                                    } else {
                                        i0 = rsqrt_ftz(r0);
                                        i1 = rsqrt_ftz(r1);
                                    }
                                    const uint64_t RI = pk2(i0, i1);
                                    const uint64_t K3 = mul2(mul2(mul2(RI, RI), RI), zw.y);
                                    qx[u] = fma2(K3, DX, qx[u]);
                                    qy[u] = fma2(K3, DY, qy[u]);
                                    qz[u] = fma2(K3, DZ, qz[u]);
                                }
                            }
                        };
                        if (a.guard_all || nb == 13)
                            sweep(std::true_type{});
                        else
                            sweep(std::false_type{});
                        continue;
                    }
                    __syncwarp();
#pragma unroll 4
                    for (int s = 0; s < cnt; ++s) {
                        const Vec4<T> e = src[s];
#pragma unroll
                        for (int u = 0; u < kTPL; ++u) {
                            const T ddx = tx[u] - e.x, ddy = ty[u] - e.y, ddz = tz[u] - e.z;
                            const T r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                            const T ri = r2 > eps2 ? rsqrt_t<T>(r2) : T(0);
                            const T k3 = e.w * (ri * ri * ri);
                            px[u] += k3 * ddx;
                            py[u] += k3 * ddy;
                            pz[u] += k3 * ddz;
                        }
                    }
                }
                if constexpr (kPacked) {
#pragma unroll
                    for (int u = 0; u < kTPL; ++u) {
                        float a0, a1;
                        up2(qx[u], a0, a1);
                        px[u] = a0 + a1;
                        up2(qy[u], a0, a1);
                        py[u] = a0 + a1;
                        up2(qz[u], a0, a1);
                        pz[u] = a0 + a1;
                    }
                }
#pragma unroll
                for (int u = 0; u < kTPL; ++u) {
                    two_sum(hx[u], lx[u], px[u]);
                    two_sum(hy[u], ly[u], py[u]);
                    two_sum(hz[u], lz[u], pz[u]);
                }
            }
            // the groups' sums of the same observers, merged into every group
            for (int o = gs; o < 32; o <<= 1) {
#pragma unroll
                for (int u = 0; u < kTPL; ++u) {
                    const T vx = __shfl_xor_sync(0xffffffffu, hx[u], o), wx = __shfl_xor_sync(0xffffffffu, lx[u], o);
                    const T vy = __shfl_xor_sync(0xffffffffu, hy[u], o), wy = __shfl_xor_sync(0xffffffffu, ly[u], o);
                    const T vz = __shfl_xor_sync(0xffffffffu, hz[u], o), wz = __shfl_xor_sync(0xffffffffu, lz[u], o);
                    two_sum(hx[u], lx[u], vx);
                    two_sum(hy[u], ly[u], vy);
                    two_sum(hz[u], lz[u], vz);
                    lx[u] += wx;
                    ly[u] += wy;
                    lz[u] += wz;
                }
            }
            T *ns = reinterpret_cast<T *>(a.nsum);
#pragma unroll
            for (int u = 0; u < kTPL; ++u) {
                if (tid[u] < 0 || grp != 0) continue;
                T *q = ns + ((int64_t)bb * a.M + tid[u]) * 6;
                q[0] = hx[u];
                q[1] = lx[u];
                q[2] = hy[u];
                q[3] = ly[u];
                q[4] = hz[u];
                q[5] = lz[u];
            }
        }
    }
    // the last warp out leaves the queue at zero for the next launch
    if (lane == 0) {
        __threadfence();
        if (atomicAdd(a.queue + 1, 1ull) == (unsigned long long)gridDim.x * kEvalWarps - 1) {
            a.queue[0] = 0;
            a.queue[1] = 0;
        }
    }
}

// Far field of the split evaluation in FP32 (after the near-field kernel
// has left each observer's compensated near sums in nsum): the L2P gradient
// of the leaf's local expansion, near + far, the scale and the scatter.  One
// warp takes up to 128 observers of one leaf, four per lane as two packed
// pairs that share every coefficient load; the warps take the evaluation
// items (64 observers each) from the queue and skip every second item of a
// leaf, which the warp holding the item before it covers.
// Bound by the FP32 pipe.  With the real recursion of l2p_sum2 (nine operations a
// term; the complex one took twelve) 2.1 M observers in 128^3 283 -> 227 us,
// 1024 x 1024 stations over 464^3 130 -> 101 us.
constexpr int kFarWarps = 4;
constexpr int kFarTargets = 128;
static_assert(kFarTargets == 2 * kTPL * 32, "two evaluation items per far item");
inline __host__ __device__ int far_slice(int P2) { return (6 * P2 + 7) & ~7; }   // floats per warp

__global__ void __launch_bounds__(kFarWarps * 32, 5) eval_far_kernel(EvalArgs a, const int32_t *__restrict__ leaf_beg) {
    extern __shared__ float fsh[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P2 = a.p * a.p;
    float2 *Dx2 = reinterpret_cast<float2 *>(fsh + (size_t)warp * far_slice(P2));
    float2 *Dy2 = Dx2 + P2, *Dz2 = Dy2 + P2;
    const float *tloc = reinterpret_cast<const float *>(a.tloc);
    const float *le = reinterpret_cast<const float *>(a.le);
    const float *ns = reinterpret_cast<const float *>(a.nsum);
    const float inv_b = 1.f / (float)a.b;
    const float far_sf = (float)(-1.0 / ((double)a.b * (double)a.b));
    for (;;) {
        int64_t it = 0;
        if (lane == 0) it = (int64_t)atomicAdd(a.queue, 1ull);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= a.n_items) break;
        const int4 item = a.items[it];
        const int leaf = item.x;
        const int lb = leaf_beg[leaf];
        if (((item.y - lb) / (kFarTargets / 2)) & 1) continue;   // covered with the item before it
        const int cnt = min(kFarTargets, leaf_beg[leaf + 1] - item.y);
        int tid[4];
        float tx[4], ty[4], tz[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = lane + 32 * u;
            tid[u] = r < cnt ? item.y + r : -1;
            const int64_t i = tid[u] >= 0 ? tid[u] : item.y;
            tx[u] = tloc[3 * i + 0] * inv_b;
            ty[u] = tloc[3 * i + 1] * inv_b;
            tz[u] = tloc[3 * i + 2] * inv_b;
        }
        for (int bb = 0; bb < a.B; ++bb) {
            const float *L = le + ((int64_t)leaf * a.B + bb) * a.ldk;
            __syncwarp();
            // duplicated pairs, scaled
            for (int e = lane; e < P2; e += 32) {
                float vx, vy, vz;
                grad_coeff<float>(L, e, vx, vy, vz);
                const float f2 = __ldg(l2p_scale + e);
                Dx2[e] = make_float2(f2 * vx, f2 * vx);
                Dy2[e] = make_float2(f2 * vy, f2 * vy);
                Dz2[e] = make_float2(f2 * vz, f2 * vz);
            }
            __syncwarp();
            uint64_t G0[3], G1[3] = {0, 0, 0};
            if (cnt > kFarTargets / 2)
                l2p_sum2x2(a.p, Dx2, Dy2, Dz2, pk2(tx[0], tx[1]), pk2(ty[0], ty[1]), pk2(tz[0], tz[1]),
                           pk2(tx[2], tx[3]), pk2(ty[2], ty[3]), pk2(tz[2], tz[3]), G0, G1);
            else   // at most 64 observers: one pair per lane
                l2p_sum2(a.p, Dx2, Dy2, Dz2, pk2(tx[0], tx[1]), pk2(ty[0], ty[1]), pk2(tz[0], tz[1]), G0[0], G0[1],
                         G0[2]);
            float fx[4], fy[4], fz[4];
            up2(G0[0], fx[0], fx[1]);
            up2(G0[1], fy[0], fy[1]);
            up2(G0[2], fz[0], fz[1]);
            up2(G1[0], fx[2], fx[3]);
            up2(G1[1], fy[2], fy[3]);
            up2(G1[2], fz[2], fz[3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (tid[u] < 0) continue;
                // near (hi + lo) + far as a compensated FP32 pair, then the pair's
                // sum and the scale in FP64 (integer conversions)
                const float *q = ns + ((int64_t)bb * a.M + tid[u]) * 6;
                float sx = q[0], ex = q[1], sy = q[2], ey = q[3], sz = q[4], ez = q[5];
                two_sum(sx, ex, far_sf * fx[u]);
                two_sum(sy, ey, far_sf * fy[u]);
                two_sum(sz, ez, far_sf * fz[u]);
                const double gx = (f32_to_f64(sx) + f32_to_f64(ex)) * a.scale;
                const double gy = (f32_to_f64(sy) + f32_to_f64(ey)) * a.scale;
                const double gzv = (f32_to_f64(sz) + f32_to_f64(ez)) * a.scale;
                const int64_t j = a.perm[tid[u]];
                if (a.g) {
                    double *o = a.g + ((int64_t)bb * a.M + j) * 3;
                    o[0] = gx;
                    o[1] = gy;
                    o[2] = gzv;
                }
                if (a.gz) a.gz[(int64_t)bb * a.M + j] = gzv;
            }
        }
    }
    // the last warp out leaves the queue at zero for the next launch
    if (lane == 0) {
        __threadfence();
        if (atomicAdd(a.queue + 1, 1ull) == (unsigned long long)gridDim.x * kFarWarps - 1) {
            a.queue[0] = 0;
            a.queue[1] = 0;
        }
    }
}

// Near field in FP64 of rules whose sources form a 4^3 lattice per leaf: the sums
// that eval_kernel makes.  The FP64 pipe takes two instructions a clock and SM,
// so their number is what counts: with the lattice sums of the FP32 form (|d|^2
// from the squared plane distances, rows added up before they are weighted) and
// inv_r3's seven, 10.3 per pair of observer and source against 23.  A block takes
// half a work item, an observer per lane; its warps share out the neighbour leaves
// and their compensated sums meet in shared memory in warp order, so that a few
// items are enough to keep many SMs busy (a warp per item left 16 of 152 busy for
// 0.8 ms under 64 x 64 stations).  65,536 observers over 128^3: 3,000 -> 1,715 us.
constexpr int kNear64Warps = 8;
// static shared memory: lattice planes, weights, voxels; masses and sums of each warp
constexpr size_t kNear64Static = 12 * 8 + 64 * 8 + 64 * 4 + kNear64Warps * (64 * 8 + 96 * 16);

__global__ void __launch_bounds__(kNear64Warps * 32) near_f64_kernel(EvalArgs a) {
    __shared__ double lat[3][4];                          // lattice planes from the leaf's centre (voxel units)
    __shared__ double lw[64];                             // the rule's weight at each lattice point
    __shared__ int lv[64];                                // its voxel
    __shared__ __align__(16) double wts[kNear64Warps][64];   // masses of the warp's leaf
    __shared__ double2 part[kNear64Warps][3][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b3 = a.b * a.b * a.b, m = a.lat_m;
    const double half_b = 0.5 * (double)a.b;
    if (threadIdx.x < 64) {
        const int n = threadIdx.x, i = n % 4, j = (n / 4) % 4, k = n / 16;
        lv[n] = i / m + a.b * (j / m + a.b * (k / m));
        lw[n] = a.qr->wn[a.lat_q[i % m + m * (j % m + m * (k % m))]];
    } else if (threadIdx.x < 76) {
        const int d = (threadIdx.x - 64) / 4, i = (threadIdx.x - 64) % 4;
        const int step = d == 0 ? 1 : d == 1 ? m : m * m;
        lat[d][i] = (double)(i / m) + (0.5 + 0.5 * a.qr->xi[a.lat_q[(i % m) * step]][d]) - half_b;
    }
    __syncthreads();
    const double *tloc = reinterpret_cast<const double *>(a.tloc);
    const double *mass = reinterpret_cast<const double *>(a.mass);
    double *ns = reinterpret_cast<double *>(a.nsum);
    const long long eps_bits = __double_as_longlong(a.eps2);
    const int64_t units = 2 * a.n_items;
    for (int64_t un = blockIdx.x; un < units; un += gridDim.x) {
        const int4 item = a.items[un >> 1];
        const int r0 = 32 * (int)(un & 1);
        if (r0 >= item.z) continue;   // the whole block
        const uint64_t key = a.tkey[item.x];
        const bool on = r0 + lane < item.z;
        const int64_t i0 = item.y + (on ? r0 + lane : r0);
        const double tx = tloc[3 * i0], ty = tloc[3 * i0 + 1], tz = tloc[3 * i0 + 2];
        int64_t slot = -1;   // lane nb: neighbour leaf nb
        {
            int64_t lc[3] = {0, 0, 0};
            for (int bit = 0; bit < a.L; ++bit)
                for (int d = 0; d < 3; ++d) lc[d] |= (int64_t)((key >> (3 * bit + d)) & 1) << bit;
            if (lane < 27) {
                const int64_t X = lc[0] + lane % 3 - 1, Y = lc[1] + (lane / 3) % 3 - 1, Z = lc[2] + lane / 9 - 1;
                const int64_t sx = X - a.blk.lo[0], sy = Y - a.blk.lo[1], sz = Z - a.blk.lo[2];
                if (sx >= 0 && sy >= 0 && sz >= 0 && sx < a.blk.n[0] && sy < a.blk.n[1] && sz < a.blk.n[2] &&
                    in_source_part(X, Y, Z, a.L - 2, a.part_lo, a.part_hi))
                    slot = (sz * a.blk.n[1] + sy) * a.blk.n[0] + sx;
            }
        }
        const unsigned have = __ballot_sync(0xffffffffu, slot >= 0);
        for (int bb = 0; bb < a.B; ++bb) {
            double h[3] = {0.0, 0.0, 0.0}, l[3] = {0.0, 0.0, 0.0};
            unsigned rest = have;
            for (int e = 0; rest; ++e) {
                const int nb = __ffs(rest) - 1;
                rest &= rest - 1;
                const int64_t sl = __shfl_sync(0xffffffffu, (long long)slot, nb);
                if (e % kNear64Warps != warp) continue;
                const double *ms = mass + (sl * a.B + bb) * b3;
                const double ox = (double)((nb % 3 - 1) * a.b), oy = (double)((nb / 3 % 3 - 1) * a.b),
                             oz = (double)((nb / 9 - 1) * a.b);
                __syncwarp();
                wts[warp][lane] = lw[lane] * ms[lv[lane]];
                wts[warp][lane + 32] = lw[lane + 32] * ms[lv[lane + 32]];
                __syncwarp();
                const bool guard = a.guard_all || nb == 13;   // a source may coincide with an observer
                double dx[4], dy[4], X2[4], Y2[4], SX[4], SY[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    dx[i] = tx - (lat[0][i] + ox);
                    dy[i] = ty - (lat[1][i] + oy);
                    X2[i] = dx[i] * dx[i];
                    Y2[i] = dy[i] * dy[i];
                    SX[i] = SY[i] = 0.0;
                }
                double gz = 0.0;
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    const double dz = tz - (lat[2][k] + oz), Z2 = dz * dz;
                    double SZ = 0.0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const double YZ = Y2[j] + Z2;
                        const double2 w01 = *reinterpret_cast<const double2 *>(&wts[warp][16 * k + 4 * j]);
                        const double2 w23 = *reinterpret_cast<const double2 *>(&wts[warp][16 * k + 4 * j + 2]);
                        const double w[4] = {w01.x, w01.y, w23.x, w23.y};
                        double K3[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const double r2 = X2[i] + YZ;
                            K3[i] = inv_r3(r2, w[i]);
                            if (guard) K3[i] = __double_as_longlong(r2) > eps_bits ? K3[i] : 0.0;
                            SX[i] += K3[i];
                        }
                        const double t = (K3[0] + K3[1]) + (K3[2] + K3[3]);
                        SY[j] += t;
                        SZ += t;
                    }
                    gz = fma(SZ, dz, gz);
                }
                double gx = 0.0, gy = 0.0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    gx = fma(SX[i], dx[i], gx);
                    gy = fma(SY[i], dy[i], gy);
                }
                two_sum(h[0], l[0], gx);
                two_sum(h[1], l[1], gy);
                two_sum(h[2], l[2], gz);
            }
            __syncthreads();   // the member before has been read
#pragma unroll
            for (int d = 0; d < 3; ++d) part[warp][d][lane] = make_double2(h[d], l[d]);
            __syncthreads();
            if (warp < 3) {
                double H = 0.0, C = 0.0;
#pragma unroll
                for (int w = 0; w < kNear64Warps; ++w) {
                    const double2 v = part[w][warp][lane];
                    two_sum(H, C, v.x);
                    C += v.y;
                }
                if (on) {
                    double *q = ns + ((int64_t)bb * a.M + i0) * 6 + 2 * warp;
                    q[0] = H;
                    q[1] = C;
                }
            }
        }
        __syncthreads();
    }
}

// Far field of the split evaluation in FP64: the L2P gradient of the leaf's local
// expansion, near + far, the scale and the scatter; a warp per half work item, an
// observer per lane.  With R_n^m = s_nm (x + iy)^m Q_n^m (z, r^2), Q real (the
// recursion of the points' P2M), the coefficients of the three gradient expansions
// are staged times s_nm and an order's sums are made with Q alone, three FP64
// instructions a term for Q and six for the sums, then turned by (x + iy)^m once.
// Bound by the FP64 pipe; a square root and a division for every term took 580 us
// for 65,536 observers at p = 14, now 184 us.
__constant__ double c_far_c[kMaxP * (kMaxP - 1) / 2 + 1];   // -((n-1)^2 - m^2) / ((2n-1)(2n-3)) at n (n-1) / 2 + m
__constant__ double c_far_s[kMaxP * kMaxP];   // s_nm by real component, twice it for m > 0
constexpr int kFar64Warps = 4;

__global__ void __launch_bounds__(kFar64Warps * 32) far_f64_kernel(EvalArgs a) {
    extern __shared__ __align__(16) unsigned char shraw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P2 = a.p * a.p;
    double *Dx = reinterpret_cast<double *>(shraw) + (size_t)warp * 3 * P2, *Dy = Dx + P2, *Dz = Dy + P2;
    const double *tloc = reinterpret_cast<const double *>(a.tloc);
    const double *le = reinterpret_cast<const double *>(a.le);
    const double *ns = reinterpret_cast<const double *>(a.nsum);
    const double inv_b = 1.0 / (double)a.b;
    const double far_s = -1.0 / ((double)a.b * (double)a.b);
    const int64_t units = 2 * a.n_items;
    for (int64_t un = (int64_t)blockIdx.x * kFar64Warps + warp; un < units; un += (int64_t)gridDim.x * kFar64Warps) {
        const int4 item = a.items[un >> 1];
        const int r0 = 32 * (int)(un & 1);
        if (r0 >= item.z) continue;
        const bool on = r0 + lane < item.z;
        const int64_t i0 = item.y + (on ? r0 + lane : r0);
        const double X = tloc[3 * i0] * inv_b, Y = tloc[3 * i0 + 1] * inv_b, Z = tloc[3 * i0 + 2] * inv_b;
        const double R2 = X * X + Y * Y + Z * Z;
        for (int bb = 0; bb < a.B; ++bb) {
            const double *L = le + ((int64_t)item.x * a.B + bb) * a.ldk;
            __syncwarp();
            for (int e = lane; e < P2; e += 32) {
                double vx, vy, vz;
                grad_coeff<double>(L, e, vx, vy, vz);
                const double sc = c_far_s[e];
                Dx[e] = sc * vx;
                Dy[e] = sc * vy;
                Dz[e] = sc * vz;
            }
            __syncwarp();
            double g[3] = {0.0, 0.0, 0.0}, wr = 1.0, wi = 0.0;
            for (int m = 0; m < a.p; ++m) {
                if (m > 0) {
                    const double nr = X * wr - Y * wi, ni = X * wi + Y * wr;
                    wr = nr;
                    wi = ni;
                }
                double Q = 1.0, P = 0.0;
                double re[3] = {0.0, 0.0, 0.0}, im[3] = {0.0, 0.0, 0.0};
                for (int n = m; n < a.p; ++n) {
                    if (n > m) {
                        // -((n-1)^2 - m^2) / ((2n-1)(2n-3)), zero at n = m + 1
                        const double v = fma(Z, Q, c_far_c[n * (n - 1) / 2 + m] * R2 * P);
                        P = Q;
                        Q = v;
                    }
                    const int k = n * n + (m == 0 ? 0 : 2 * m - 1);
                    re[0] = fma(Dx[k], Q, re[0]);
                    re[1] = fma(Dy[k], Q, re[1]);
                    re[2] = fma(Dz[k], Q, re[2]);
                    if (m > 0) {
                        im[0] = fma(Dx[k + 1], Q, im[0]);
                        im[1] = fma(Dy[k + 1], Q, im[1]);
                        im[2] = fma(Dz[k + 1], Q, im[2]);
                    }
                }
#pragma unroll
                for (int d = 0; d < 3; ++d) g[d] = fma(re[d], wr, fma(im[d], wi, g[d]));
            }
            if (!on) continue;
            const double *q = ns + ((int64_t)bb * a.M + i0) * 6;
            const double gx = (q[0] + (q[1] + far_s * g[0])) * a.scale, gy = (q[2] + (q[3] + far_s * g[1])) * a.scale,
                         gzv = (q[4] + (q[5] + far_s * g[2])) * a.scale;
            const int64_t j = a.perm[i0];
            if (a.g) {
                double *o = a.g + ((int64_t)bb * a.M + j) * 3;
                o[0] = gx;
                o[1] = gy;
                o[2] = gzv;
            }
            if (a.gz) a.gz[(int64_t)bb * a.M + j] = gzv;
        }
    }
}

constexpr int kAnNb = 12;                          // voxels per axis of the 27-leaf block of closed-form voxels
constexpr int kAnBlock = kAnNb * kAnNb * kAnNb;

// Near field of closed-form voxels (SUM-AN in the FMM) in FP32: the sums that
// eval_kernel makes, the far field following as for quadrature voxels.  One
// warp per half work item, an observer per lane; the densities of the item's 27
// neighbour leaves (a 12^3 voxel block, 4^3-voxel leaves) are staged in the
// warp's shared-memory slice.  The sums are those of an_near_block with radius 2:
// - Voxels beyond Chebyshev distance 2 of the observer's own: two voxels of a row
//   at a time as packed pairs.  With r^2 = x^2 + Y, Y, y and z constant on a row,
//   the midpoint rule and the cube's l = 4 term are x (A + B x^2) and, summed over
//   the row, y (sum A + y^2 sum B): 22 packed operations for two voxels.  The
//   voxels of the closed form get r^2 = 1e36, so that they add zero; rows of
//   leaves without sources are passed over.
// - The others in closed form on their 6^3 corner lattice, by offset from the
//   observer's voxel, so that the sign of every coordinate, and with it the form
//   of every logarithm, is the same across the warp; the corner weights of a row
//   are differences of column sums.
// Bound by the instruction issue, logarithms and arctangents above all.  One
// observer's voxels one by one, both forms and the L2P's square roots and
// divisions in one kernel, took 1,690 us for 512 x 512 stations over 128^3 voxels;
// now 600 us and 40 us of far field.
//
// Quotients and roots from the approximate reciprocals, refined by one Newton
// step on the residual (in the last place); operands are normal numbers here.
__device__ __forceinline__ float an_quot(float n, float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    const float q = n * r;
    return fmaf(fmaf(-q, d, n), r, q);
}
__device__ __forceinline__ float an_root(float x) {
    const float y = rsqrt_ftz(x), r = x * y;
    return x > 0.f ? fmaf(fmaf(-r, r, x), 0.5f * y, r) : 0.f;
}

// atan(n / d), d != 0, as the angle of the smaller to the larger of |n| and |d|:
// one division for both ranges.  On [0, 1] t + t s q(s), s = t^2, q of degree 8
// fitted to the smallest largest relative error (1.1e-8 in this form; evaluated in
// FP32, 1.2 units in the last place).
__device__ __forceinline__ float an_angle(float n, float d) {
    const float an = fabsf(n), ad = fabsf(d);
    const float t = an_quot(fminf(an, ad), fmaxf(an, ad)), s = t * t;
    float q = -0.0017539296532049775f;
    q = fmaf(q, s, 0.010726941749453545f);
    q = fmaf(q, s, -0.030804593116044998f);
    q = fmaf(q, s, 0.05755209922790527f);
    q = fmaf(q, s, -0.08377315104007721f);
    q = fmaf(q, s, 0.1094203069806099f);
    q = fmaf(q, s, -0.142619326710701f);
    q = fmaf(q, s, 0.1999826580286026f);
    q = fmaf(q, s, -0.3333328366279602f);
    float r = fmaf(q * s, t, t);
    if (an > ad) r = (1.57079637f - r) - 4.37113883e-8f;   // pi / 2 in two parts
    return __uint_as_float(__float_as_uint(r) ^ ((__float_as_uint(n) ^ __float_as_uint(d)) & 0x80000000u));
}

// ln(a + R), R = sqrt(a^2 + q); 0 when q is zero
__device__ __forceinline__ float an_ln_of(float a, float q, float R) {
    float x = a + R;
    if (a < 0.f) x = an_quot(q, R - a);
    return q > 0.f ? logf(x) : 0.f;
}

constexpr int kAnWarps = 4;
inline __host__ __device__ int near_an_slice() { return kAnBlock + 32; }   // floats: densities, 27 leaf numbers

__global__ void __launch_bounds__(kAnWarps * 32, 7) near_an_kernel(EvalArgs a) {
    extern __shared__ __align__(16) unsigned char shraw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *blk = reinterpret_cast<float *>(shraw) + (size_t)warp * near_an_slice();
    int *slots = reinterpret_cast<int *>(blk + kAnBlock);
    const float *tloc = reinterpret_cast<const float *>(a.tloc);
    const float *mass = reinterpret_cast<const float *>(a.mass);
    float *ns = reinterpret_cast<float *>(a.nsum);
    constexpr float c = 7.f / 192.f;
    const uint64_t c3 = pk2(3.f * c, 3.f * c), nc9 = pk2(-9.f * c, -9.f * c), one = pk2(1.f, 1.f), half = pk2(0.5f, 0.5f);
    const int64_t units = 2 * a.n_items;
    for (int64_t un = (int64_t)blockIdx.x * kAnWarps + warp; un < units; un += (int64_t)gridDim.x * kAnWarps) {
        const int4 item = a.items[un >> 1];
        const int r0 = 32 * (int)(un & 1);
        if (r0 >= item.z) continue;
        const int leaf = item.x;
        const uint64_t key = a.tkey[leaf];
        const bool on = r0 + lane < item.z;
        const int64_t i0 = item.y + (on ? r0 + lane : r0);
        // position in the block (own leaf at [4, 8)) and the voxel it is in
        const float tx = tloc[3 * i0] + 6.f, ty = tloc[3 * i0 + 1] + 6.f, tz = tloc[3 * i0 + 2] + 6.f;
        const int vi = min(max((int)floorf(tx), 2), kAnNb - 3), vj = min(max((int)floorf(ty), 2), kAnNb - 3),
                  vk = min(max((int)floorf(tz), 2), kAnNb - 3);
        uint32_t have;   // the neighbour leaves that hold sources
        int slot = -1;
        {
            int64_t lc[3] = {0, 0, 0};
            for (int bit = 0; bit < a.L; ++bit)
                for (int d = 0; d < 3; ++d) lc[d] |= (int64_t)((key >> (3 * bit + d)) & 1) << bit;
            if (lane < 27) {
                const int64_t X = lc[0] + lane % 3 - 1, Y = lc[1] + (lane / 3) % 3 - 1, Z = lc[2] + lane / 9 - 1;
                const int64_t sx = X - a.blk.lo[0], sy = Y - a.blk.lo[1], sz = Z - a.blk.lo[2];
                if (sx >= 0 && sy >= 0 && sz >= 0 && sx < a.blk.n[0] && sy < a.blk.n[1] && sz < a.blk.n[2] &&
                    in_source_part(X, Y, Z, a.L - 2, a.part_lo, a.part_hi))
                    slot = (int)((sz * a.blk.n[1] + sy) * a.blk.n[0] + sx);
            }
            have = __ballot_sync(0xffffffffu, slot >= 0);
            __syncwarp();   // the unit before has read its slots
            slots[lane] = slot;
        }
        uint64_t X2[6], XP[6];   // offsets along x of the row's pairs of voxels, and their squares
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            XP[q] = pk2(tx - (2 * q + 0.5f), tx - (2 * q + 1.5f));
            X2[q] = mul2(XP[q], XP[q]);
        }
        const uint32_t nearx = 0x1fu << (vi - 2);
        for (int bb = 0; bb < a.B; ++bb) {
            __syncwarp();
            // one 4-voxel row of a leaf per lane and step: rows (z, y) of 3 leaves
            for (int e = lane; e < 3 * kAnNb * kAnNb; e += 32) {
                const int xl = e % 3, yz = e / 3, y = yz % kAnNb, z = yz / kAnNb;
                const int l = (z >> 2) * 9 + (y >> 2) * 3 + xl;
                const int sl = slots[l];
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (sl >= 0)
                    v = __ldg(reinterpret_cast<const float4 *>(mass + ((int64_t)sl * a.B + bb) * 64) + (z & 3) * 4 + (y & 3));
                *reinterpret_cast<float4 *>(blk + yz * kAnNb + 4 * xl) = v;
            }
            __syncwarp();
            float sx = 0.f, ex = 0.f, sy = 0.f, ey = 0.f, sz = 0.f, ez = 0.f;
            for (int k = 0; k < kAnNb; ++k) {
                const float z = tz - (k + 0.5f), z2 = z * z;
                for (int j = 0; j < kAnNb; ++j) {
                    if (!(have >> ((k >> 2) * 9 + (j >> 2) * 3) & 7u)) continue;
                    const float y = ty - (j + 0.5f), y2 = y * y;
                    const float q2 = y2 + z2, q4 = y2 * y2 + z2 * z2;
                    const uint64_t Q2 = pk2(q2, q2), Q4 = pk2(q4, q4);
                    const uint32_t skip = max(abs(j - vj), abs(k - vk)) <= 2 ? nearx : 0u;
                    const bool any = __any_sync(0xffffffffu, skip != 0u);
                    const float4 *row = reinterpret_cast<const float4 *>(blk + (k * kAnNb + j) * kAnNb);
                    uint64_t SA = 0, SB = 0, GX = 0;
#pragma unroll
                    for (int q = 0; q < 6; q += 2) {
                        const float4 m4 = row[q / 2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint64_t M = h ? pk2(m4.z, m4.w) : pk2(m4.x, m4.y);
                            uint64_t R2 = add2(X2[q + h], Q2);
                            if (any) {
                                float ra, rb;
                                up2(R2, ra, rb);
                                R2 = pk2((skip >> (2 * (q + h))) & 1u ? 1e36f : ra,
                                         (skip >> (2 * (q + h))) & 2u ? 1e36f : rb);
                            }
                            float ra, rb;
                            up2(R2, ra, rb);
                            uint64_t I = pk2(rsqrt_ftz(ra), rsqrt_ftz(rb));
                            // one Newton step: I += I/2 (1 - R2 I^2)
                            const uint64_t E = fma2(mul2(R2 ^ 0x8000000080000000ull, I), I, one);
                            I = fma2(mul2(half, I), E, I);
                            const uint64_t I2 = mul2(I, I), I3 = mul2(I, I2), I9 = mul2(I3, mul2(I3, I3));
                            const uint64_t S4 = fma2(X2[q + h], X2[q + h], Q4);
                            // A = r^-3 + c r^-9 (3 r^2 - 9 S4 / r^2), B = 4 c r^-9 (its 4 c at the row's end)
                            const uint64_t A = fma2(I9, fma2(nc9, mul2(S4, I2), mul2(c3, R2)), I3);
                            const uint64_t MA = mul2(M, A), MB = mul2(M, I9);
                            SA = add2(SA, MA);
                            SB = add2(SB, MB);
                            GX = fma2(fma2(mul2(MB, pk2(4.f * c, 4.f * c)), X2[q + h], MA), XP[q + h], GX);
                        }
                    }
                    float lo, hi;
                    up2(SA, lo, hi);
                    const float sa = lo + hi;
                    up2(SB, lo, hi);
                    const float sb = 4.f * c * (lo + hi);
                    up2(GX, lo, hi);
                    two_sum(sx, ex, lo + hi);
                    two_sum(sy, ey, y * (sa + sb * y2));
                    two_sum(sz, ez, z * (sa + sb * z2));
                }
            }
            // closed form: corners v - 2 .. v + 3 of the 5^3 voxels around the observer's
            const float *own = blk + ((vk - 2) * kAnNb + vj - 2) * kAnNb + vi - 2;
            for (int K = 0; K < 6; ++K) {
                const float w = (float)(vk - 2 + K) - tz, w2 = w * w;
                float qp[5] = {0.f, 0.f, 0.f, 0.f, 0.f};   // column sums of the row before
                for (int J = 0; J < 6; ++J) {
                    float t[5];   // signed density sums of the corner row's 5 voxel columns
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const float up = K < 5 && J < 5 ? own[(K * kAnNb + J) * kAnNb + i] : 0.f;
                        const float dn = K > 0 && J < 5 ? own[((K - 1) * kAnNb + J) * kAnNb + i] : 0.f;
                        const float q = dn - up;
                        t[i] = q - qp[i];
                        qp[i] = q;
                    }
                    float gx = 0.f, gy = 0.f, gz = 0.f;
                    const float v = (float)(vj - 2 + J) - ty, v2 = v * v, qu = v2 + w2;
                    float tp = 0.f;
#pragma unroll 1   // the body is some 250 instructions: six copies overflow the instruction cache
                    for (int I = 0; I < 6; ++I) {
                        const float D = t[0] - tp;
                        tp = t[0];
#pragma unroll
                        for (int i = 0; i < 4; ++i) t[i] = t[i + 1];
                        t[4] = 0.f;
                        if (!__any_sync(0xffffffffu, D != 0.f)) continue;
                        const float u = (float)(vi - 2 + I) - tx, u2 = u * u;
                        const float R = an_root(u2 + qu);
                        const float Lu = an_ln_of(u, qu, R), Lv = an_ln_of(v, u2 + w2, R), Lw = an_ln_of(w, u2 + v2, R);
                        const float au = u != 0.f ? u * an_angle(v * w, u * R) : 0.f;
                        const float av = v != 0.f ? v * an_angle(w * u, v * R) : 0.f;
                        const float aw = w != 0.f ? w * an_angle(u * v, w * R) : 0.f;
                        gx += D * (v * Lw + w * Lv - au);
                        gy += D * (w * Lu + u * Lw - av);
                        gz += D * (u * Lv + v * Lu - aw);
                    }
                    two_sum(sx, ex, gx);
                    two_sum(sy, ey, gy);
                    two_sum(sz, ez, gz);
                }
            }
            if (on) {
                float *q = ns + ((int64_t)bb * a.M + i0) * 6;
                q[0] = sx;
                q[1] = ex;
                q[2] = sy;
                q[3] = ey;
                q[4] = sz;
                q[5] = ez;
            }
        }
    }
}

// Near field + far field of closed-form voxels in FP64: one warp
// per work item, two observers per lane.  The densities of the item's 27
// neighbour leaves (a 12^3 voxel block, 4^3-voxel leaves) are staged in the
// warp's shared-memory slice; each observer takes the voxels within
// Chebyshev distance RAD of its own voxel in closed form on their corner
// lattice and the others by the midpoint rule with a uniform cube's l = 4
// term (an_near_block); the far field is the L2P gradient of the leaf's
// local expansion (made from exact voxel moments).
inline __host__ __device__ int eval_an_slice(int P2) { return (kAnBlock + 3 * P2 + 27 * 2 + 7) & ~7; }

template <class T, int RAD>
__global__ void __launch_bounds__(kEvalWarps * 32) eval_an_kernel(EvalArgs a) {
    extern __shared__ unsigned char shraw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P2 = a.p * a.p;
    T *blk = reinterpret_cast<T *>(shraw) + (size_t)warp * eval_an_slice(P2);
    T *Dx = blk + kAnBlock, *Dy = Dx + P2, *Dz = Dy + P2;
    int64_t *nbl = reinterpret_cast<int64_t *>(Dz + P2 + ((P2 * 3 + kAnBlock) & 1));
    const T *tloc = reinterpret_cast<const T *>(a.tloc);
    const T *mass = reinterpret_cast<const T *>(a.mass);
    const T *le = reinterpret_cast<const T *>(a.le);
    const T inv_b = T(1) / T(a.b);
    const double far_s = -1.0 / ((double)a.b * (double)a.b);
    for (int64_t it = (int64_t)blockIdx.x * kEvalWarps + warp; it < a.n_items; it += (int64_t)gridDim.x * kEvalWarps) {
        const int4 item = a.items[it];
        const int leaf = item.x;
        const uint64_t key = a.tkey[leaf];
        int64_t lc[3] = {0, 0, 0};
        for (int bit = 0; bit < 21; ++bit) {
            lc[0] |= (int64_t)((key >> (3 * bit)) & 1) << bit;
            lc[1] |= (int64_t)((key >> (3 * bit + 1)) & 1) << bit;
            lc[2] |= (int64_t)((key >> (3 * bit + 2)) & 1) << bit;
        }
        T tx[kTPL], ty[kTPL], tz[kTPL];
        int tid[kTPL];
#pragma unroll
        for (int u = 0; u < kTPL; ++u) {
            const int r = lane + 32 * u;
            tid[u] = r < item.z ? item.y + r : -1;
            const int64_t i = tid[u] >= 0 ? tid[u] : item.y;
            tx[u] = tloc[3 * i + 0] + T(6);   // position in the block (own leaf at [4, 8))
            ty[u] = tloc[3 * i + 1] + T(6);
            tz[u] = tloc[3 * i + 2] + T(6);
        }
        __syncwarp();
        if (lane < 27) {
            const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
            const int64_t sx = lc[0] + dx - a.blk.lo[0], sy = lc[1] + dy - a.blk.lo[1], sz = lc[2] + dz - a.blk.lo[2];
            const bool in = sx >= 0 && sy >= 0 && sz >= 0 && sx < a.blk.n[0] && sy < a.blk.n[1] && sz < a.blk.n[2] &&
                            in_source_part(lc[0] + dx, lc[1] + dy, lc[2] + dz, a.L - 2, a.part_lo, a.part_hi);
            nbl[lane] = in ? (sz * a.blk.n[1] + sy) * a.blk.n[0] + sx : -1;
        }
        __syncwarp();
        for (int bb = 0; bb < a.B; ++bb) {
            for (int e = lane; e < kAnBlock; e += 32) {
                const int x = e % kAnNb, y = (e / kAnNb) % kAnNb, z = e / (kAnNb * kAnNb);
                const int64_t sl = nbl[(z >> 2) * 9 + (y >> 2) * 3 + (x >> 2)];
                blk[e] = sl >= 0 ? mass[(sl * a.B + bb) * 64 + ((z & 3) * 4 + (y & 3)) * 4 + (x & 3)] : T(0);
            }
            const T *L = le + ((int64_t)leaf * a.B + bb) * a.ldk;
            for (int e = lane; e < P2; e += 32) grad_coeff<T>(L, e, Dx[e], Dy[e], Dz[e]);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kTPL; ++u) {
                if (tid[u] < 0) continue;
                T gn[3];
                an_near_block<T>(blk, kAnNb, tx[u], ty[u], tz[u], gn, RAD);
                T fx, fy, fz;
                l2p_sum<T>(a.p, Dx, Dy, Dz, (tx[u] - T(6)) * inv_b, (ty[u] - T(6)) * inv_b, (tz[u] - T(6)) * inv_b,
                           fx, fy, fz);
                const double gx = ((double)gn[0] + far_s * (double)fx) * a.scale;
                const double gy = ((double)gn[1] + far_s * (double)fy) * a.scale;
                const double gzv = ((double)gn[2] + far_s * (double)fz) * a.scale;
                const int64_t j = a.perm[tid[u]];
                if (a.g) {
                    double *o = a.g + ((int64_t)bb * a.M + j) * 3;
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

// Adjoint tables: adj[slot][i*K + o] = fwd[mslot][o*K + i], where mslot is
// the slot of -offset for M2L and the same octant for M2M/L2L.
__global__ void transpose_ops(const double *__restrict__ fwd, double *__restrict__ adjd, float *__restrict__ adjf,
                              int K, int nslots, int negate) {
    const int slot = blockIdx.x;
    int mslot = slot;
    if (negate) {
        const int dx = slot % 7 - 3, dy = (slot / 7) % 7 - 3, dz = slot / 49 - 3;
        mslot = (-dz + 3) * 49 + (-dy + 3) * 7 + (-dx + 3);
    }
    const size_t KK = (size_t)K * K;
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
        const int i = e / K, o = e - i * K;
        const double v = fwd[(size_t)mslot * KK + (size_t)o * K + i];
        adjd[(size_t)slot * KK + e] = v;
        adjf[(size_t)slot * KK + e] = (float)v;
    }
    (void)nslots;
}

// The far field's tables for the current device.
gf_status upload_far_coefs() {
    double c[kMaxP * (kMaxP - 1) / 2 + 1] = {}, sc[kMaxP * kMaxP] = {};
    l2p_tables(c, sc);
    GF_CUDA(cudaMemcpyToSymbol(c_far_c, c, sizeof(c)));
    GF_CUDA(cudaMemcpyToSymbol(c_far_s, sc, sizeof(sc)));
    return GF_OK;
}

// ---------------------------------------------------------------- tables
std::mutex g_tab_mu;
std::vector<Tables *> g_tabs;

}  // namespace

gf_status get_tables(int device, int p, cudaStream_t st, const Tables **out) {
    std::lock_guard<std::mutex> lk(g_tab_mu);
    for (Tables *t : g_tabs)
        if (t->device == device && t->p == p) {
            *out = t;
            return GF_OK;
        }
    Tables *T = new Tables();
    T->device = device;
    T->p = p;
    T->K = (p + 1) * (p + 1);
    T->Kp = (T->K + 7) & ~7;
    const size_t KK = (size_t)T->K * T->K;
    // tables live for the life of the process: one set per (device, p)
    GF_CUDA(cudaMalloc(&T->m2l_d, 343 * KK * sizeof(double)));
    GF_CUDA(cudaMalloc(&T->m2l_f, 343 * KK * sizeof(float)));
    GF_CUDA(cudaMalloc(&T->m2m_d, 8 * KK * sizeof(double)));
    GF_CUDA(cudaMalloc(&T->l2l_d, 8 * KK * sizeof(double)));
    GF_CUDA(cudaMalloc(&T->m2m_f, 8 * KK * sizeof(float)));
    GF_CUDA(cudaMalloc(&T->l2l_f, 8 * KK * sizeof(float)));
    GF_CUDA(cudaMemsetAsync(T->m2l_d, 0, 343 * KK * sizeof(double), st));
    GF_CUDA(cudaMemsetAsync(T->m2l_f, 0, 343 * KK * sizeof(float), st));
    const int H = 2 * p;
    const size_t shm = sizeof(double) * (H + 1) * (H + 2);
    build_ops<<<343 + 16, 256, shm, st>>>(p, T->K, host_logfact(), T->m2l_d, T->m2l_f, T->m2m_d, T->m2m_f,
                                          T->l2l_d, T->l2l_f);
    GF_KERNEL_DONE();
    GF_CUDA(cudaMalloc(&T->am2l_d, 343 * KK * sizeof(double)));
    GF_CUDA(cudaMalloc(&T->am2l_f, 343 * KK * sizeof(float)));
    GF_CUDA(cudaMalloc(&T->am2m_d, 8 * KK * sizeof(double)));
    GF_CUDA(cudaMalloc(&T->am2m_f, 8 * KK * sizeof(float)));
    GF_CUDA(cudaMalloc(&T->al2l_d, 8 * KK * sizeof(double)));
    GF_CUDA(cudaMalloc(&T->al2l_f, 8 * KK * sizeof(float)));
    transpose_ops<<<343, 256, 0, st>>>(T->m2l_d, T->am2l_d, T->am2l_f, T->K, 343, 1);
    GF_KERNEL_DONE();
    transpose_ops<<<8, 256, 0, st>>>(T->m2m_d, T->am2m_d, T->am2m_f, T->K, 8, 0);
    GF_KERNEL_DONE();
    transpose_ops<<<8, 256, 0, st>>>(T->l2l_d, T->al2l_d, T->al2l_f, T->K, 8, 0);
    GF_KERNEL_DONE();
    GF_TRY(m2l_prepare_tables(T, st));
    GF_TRY(xlate_prepare_tables(T, st));
    GF_TRY(upload_l2p_coefs());
    GF_TRY(upload_far_coefs());
    GF_CUDA(cudaStreamSynchronize(st));
    g_tabs.push_back(T);
    *out = T;
    return GF_OK;
}

// P2M matrices, one per (device, p, leaf size, quadrature rule), cached for
// the life of the process like the operator tables: plans rebuilt for the
// same rule (a solve loop, a server) do not rebuild them.
struct P2MEntry {
    int device, p, b, nq;
    int exact;             // closed-form voxels: moments integrated exactly
    double xi[kMaxQuad][3], wn[kMaxQuad];
    double *pd = nullptr;
    float *pf = nullptr;
    double *ud = nullptr;  // 4^3-voxel leaves: P2M into the parent level from position 7 [64][K]
    float *uf = nullptr, *uq = nullptr;   // FP32 copy, and in quad order
    double *utd = nullptr, *ltd = nullptr;   // transposes in class order [K][64], [K][8]
    float *utf = nullptr, *ltf = nullptr;
    // rules that do not mirror: the shift by their nodes (leaf, parent) in FP64 and
    // FP32, in quad order, and the matrices of the voxel centres
    double *sd = nullptr;
    float *sf = nullptr, *sq[2] = {};
    P2MEntry *centre = nullptr;
};
std::mutex g_p2m_mu;
std::vector<P2MEntry *> g_p2m;

static void use_p2m(FmmPlan *F, const P2MEntry *e) {
    F->p2m_d = e->pd;
    F->p2m_f = e->pf;
    F->p2m_upt_d = e->utd;
    F->p2m_upt_f = e->utf;
    F->p2m_leaft_d = e->ltd;
    F->p2m_leaft_f = e->ltf;
    // the split inputs hold the centres' expansions until the M2L's input split
    const bool shift = e->centre && F->mixed && F->tab->m2l_tc;
    for (int i = 0; i < 2; ++i) {
        F->shift_f[i] = shift ? e->sf + (size_t)i * F->K * F->K : nullptr;
        F->shift_q[i] = shift ? e->sq[i] : nullptr;
    }
    if (shift) {
        e = e->centre;
        F->p2m_c_f = e->pf;
    }
    F->p2m_up_d = e->ud;
    F->p2m_up_f = e->uf;
    F->p2m_up_q = e->uq;
}

// The cached matrices of a rule, made when they are not there (qr: the rule on the
// device; null: the voxel's centre).  Called with g_p2m_mu held.
static gf_status find_p2m(const FmmPlan *F, int device, const QuadRule &q, const QuadRule *qr, int exact, cudaStream_t st,
                          P2MEntry **out) {
    for (P2MEntry *e : g_p2m)
        if (e->device == device && e->p == F->p && e->b == F->b && e->nq == q.nq && e->exact == exact &&
            !memcmp(e->xi, q.xi, sizeof(double) * 3 * q.nq) && !memcmp(e->wn, q.wn, sizeof(double) * q.nq)) {
            *out = e;
            return GF_OK;
        }
    const int b3 = F->b * F->b * F->b, K = F->K, KP = F->tab->cls_off[8];
    P2MEntry *centre = nullptr;
    if (F->b == 4 && !exact && !rule_mirrors(q)) {
        QuadRule c;
        memset(&c, 0, sizeof(c));
        c.nq = 1;
        c.wn[0] = 1.0;
        GF_TRY(find_p2m(F, device, c, nullptr, 0, st, &centre));
    }
    P2MEntry *e = new P2MEntry();
    e->device = device;
    e->p = F->p;
    e->b = F->b;
    e->nq = q.nq;
    e->exact = exact;
    e->centre = centre;
    memcpy(e->xi, q.xi, sizeof(double) * 3 * q.nq);
    memcpy(e->wn, q.wn, sizeof(double) * q.nq);
    if (cudaMalloc(&e->pd, sizeof(double) * b3 * K) != cudaSuccess ||
        cudaMalloc(&e->pf, sizeof(float) * b3 * K) != cudaSuccess ||
        (F->b == 4 && (cudaMalloc(&e->ud, sizeof(double) * b3 * K) != cudaSuccess ||
                       cudaMalloc(&e->uf, sizeof(float) * b3 * K) != cudaSuccess ||
                       cudaMalloc(&e->utd, sizeof(double) * b3 * KP) != cudaSuccess ||
                       cudaMalloc(&e->utf, sizeof(float) * b3 * KP) != cudaSuccess ||
                       cudaMalloc(&e->ltd, sizeof(double) * 8 * KP) != cudaSuccess ||
                       cudaMalloc(&e->ltf, sizeof(float) * 8 * KP) != cudaSuccess)) ||
        (centre && (cudaMalloc(&e->sd, sizeof(double) * 2 * K * K) != cudaSuccess ||
                    cudaMalloc(&e->sf, sizeof(float) * 2 * K * K) != cudaSuccess))) {
        cudaGetLastError();
        for (void *m : {(void *)e->pd, (void *)e->pf, (void *)e->ud, (void *)e->uf, (void *)e->utd, (void *)e->utf,
                        (void *)e->ltd, (void *)e->ltf, (void *)e->sd, (void *)e->sf})
            cudaFree(m);
        delete e;
        set_error("cannot allocate the P2M matrix");
        return GF_ERR_OOM;
    }
    const size_t shm = sizeof(double) * ((F->p + 1) * (F->p + 2) + K);
    if (exact || !qr) {
        // exact: degree <= p, ceil((p + 1) / 2) nodes per axis
        build_p2m_exact<<<b3, 128, shm, st>>>(F->p, K, F->b, gauss_legendre(exact ? (F->p + 2) / 2 : 1), e->pd, e->pf);
    } else {
        build_p2m<<<b3, 128, shm, st>>>(F->p, K, F->b, qr, e->pd, e->pf);
    }
    GF_KERNEL_DONE();
    if (e->ud) {
        compose_p2m_up<<<b3, 128, 0, st>>>(e->pd, F->tab->m2m_d + (size_t)7 * K * K, K, e->ud, e->uf);
        GF_KERNEL_DONE();
        GF_TRY(xlate_quad_table(F->tab, e->uf, b3, &e->uq, st));
        transpose_p2m<<<KP, 64, 0, st>>>(e->pd, e->ud, F->tab->cls_perm, K, e->utd, e->utf, e->ltd, e->ltf);
        GF_KERNEL_DONE();
    }
    if (centre) {
        build_shift<<<2, 256, shm, st>>>(F->p, K, F->b, qr, host_logfact(), e->sd, e->sf);
        GF_KERNEL_DONE();
        for (int i = 0; i < 2; ++i) GF_TRY(xlate_quad_table(F->tab, e->sf + (size_t)i * K * K, K, &e->sq[i], st));
    }
    GF_CUDA(cudaStreamSynchronize(st));   // other streams may use the cached matrix next
    g_p2m.push_back(e);
    *out = e;
    return GF_OK;
}

gf_status get_p2m(gf_plan_s *plan, cudaStream_t st) {
    std::lock_guard<std::mutex> lk(g_p2m_mu);
    P2MEntry *e = nullptr;
    GF_TRY(find_p2m(plan->fmm, plan->device, plan->quad, quad_device(plan),
                    (plan->opt.reserved0 & GF_FLAG_SUM_AN) ? 1 : 0, st, &e));
    use_p2m(plan->fmm, e);
    return GF_OK;
}

gf_status fmm_alloc_workspaces(gf_plan_s *plan, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    DeviceArena &A = plan->arena;
    const size_t rs = F->mixed ? sizeof(float) : sizeof(double);
    const int K = F->K, B = F->B;
    F->KS = (F->mixed || F->m2l_tc64) ? (K + 31) & ~31 : K;
    for (int l = 2; l <= F->L; ++l) {
        FmmLevel &lv = F->lev[l];
        GF_TRY(A.alloc(&lv.me, (size_t)std::max<int64_t>(lv.ns, 1) * B * F->KS * rs));
        GF_TRY(A.alloc(&lv.le, (size_t)std::max<int64_t>(lv.nt, 1) * B * F->KS * rs));
    }
    const int b3 = F->b * F->b * F->b;
    const int64_t nmass = F->points ? plan->pts.S : F->lev[F->L].ns * b3;
    GF_TRY(A.alloc(&F->mass, (size_t)std::max<int64_t>(nmass, 1) * B * rs));
    if (!F->points) GF_TRY(A.alloc(&F->nsum, (size_t)std::max<int64_t>(plan->M, 1) * B * 6 * rs));
    static bool il_ready[64] = {false};
    static std::mutex il_mu;
    {
        std::lock_guard<std::mutex> lk(il_mu);
        if (!il_ready[plan->device & 63]) {
            static signed char h_il[8][189][3];
            for (int c = 0; c < 8; ++c) il_offsets_host(c, h_il[c]);
            GF_TRY(m2l_upload_offsets(h_il));
            il_ready[plan->device & 63] = true;
        }
    }
    GF_TRY(get_tables(plan->device, F->p, st, &F->tab));
    if (!F->points) GF_TRY(get_p2m(plan, st));
    GF_TRY(m2l_tc_prepare(plan));
    return m2l_oz_prepare(plan);
}

// ---------------------------------------------------------------- forward
namespace {

// Lattice form of a leaf's sources for the near field: when the rule is a
// tensor product of m nodes per axis (the same nodes on every axis), the
// b^3 nq sources of a leaf sit on an N1^3 lattice, N1 = b m.  Fills the
// plane coordinates and the node map of `a` and returns N1, or 0 when the
// rule is not such a product or N1 is not the size the kernel handles (4).
static int lattice_of(const QuadRule &qr, int b, EvalArgs &a) {
    double nodes[kMaxQuad];
    int m = 0;
    for (int q = 0; q < qr.nq; ++q) {   // distinct x-nodes, ascending
        const double x = qr.xi[q][0];
        bool seen = false;
        for (int t = 0; t < m; ++t) seen = seen || nodes[t] == x;
        if (!seen) nodes[m++] = x;
    }
    std::sort(nodes, nodes + m);
    if (m * m * m != qr.nq || b * m != 4 || b * m > kMaxLat) return 0;
    int seen[kMaxQuad];
    for (int t = 0; t < qr.nq; ++t) seen[t] = 0;
    for (int q = 0; q < qr.nq; ++q) {
        int idx[3];
        for (int d = 0; d < 3; ++d) {
            idx[d] = -1;
            for (int t = 0; t < m; ++t)
                if (qr.xi[q][d] == nodes[t]) idx[d] = t;
            if (idx[d] < 0) return 0;
        }
        const int c = idx[0] + m * (idx[1] + m * idx[2]);
        if (seen[c]++) return 0;
        a.lat_q[c] = q;
    }
    a.lat_m = m;
    const float half_b = 0.5f * (float)b;
    for (int d = 0; d < 3; ++d)
        for (int i = 0; i < b * m; ++i)
            a.lat_c[d][i] = ((float)(i / m) + (float)(0.5 + 0.5 * nodes[i % m])) - half_b;
    return b * m;
}

// Arguments of the evaluation kernels; returns the lattice size N1 of the
// near field's lattice form (0: the generic source list).
template <class T>
int eval_setup(gf_plan_s *plan, int B, double *g, double *gz, EvalArgs &a) {
    const FmmPlan *F = plan->fmm;
    const int L = F->L;
    a.L = L;
    a.part_lo = plan->part_lo;
    a.part_hi = plan->part_hi;
    a.items = F->items;
    a.n_items = F->n_items;
    a.queue = F->eval_queue;
    a.nsum = F->nsum;
    a.tkey = F->lev[L].tkey;
    a.perm = F->perm;
    a.tloc = sizeof(T) == 8 ? (const void *)F->tloc_d : (const void *)F->tloc_f;
    a.mass = F->mass;
    a.le = F->lev[L].le;
    a.qr = quad_device(plan);
    a.blk = block_of(F->lev[L]);
    a.b = F->b;
    a.nq = F->nq;
    a.B = B;
    a.K = F->K;
    a.ldk = F->KS;
    a.p = F->p;
    a.M = plan->M;
    a.scale = plan->G * F->h;
    a.eps2 = sizeof(T) == 8 ? 1e-18 : 1e-12;
    a.guard_all = 0;
    for (int q = 0; q < plan->quad.nq; ++q)
        for (int d = 0; d < 3; ++d)
            if (fabs(plan->quad.xi[q][d]) >= 1.0) a.guard_all = 1;
    a.g = g;
    a.gz = gz;
    return lattice_of(plan->quad, F->b, a);
}

// Dynamic shared memory, at least shm, with which no more blocks of a launch fit one
// SM than an even spread over the SMs puts there (`stat`: the kernel's static part).
// The near field of a small model is a few dozen blocks that start as the M2L on
// the tensor cores leaves the SMs, and the first SMs to come free took as many as
// fitted while the others stood idle: 64^3 voxels under 128^2 stations, a 2x2x2 rule
// in 4^3-voxel leaves, 798 us where the same launches in line took 441; closed form
// 394 against 272; FP64 38.1 ms against 12.4; now 387, 213 us and 12.3 ms.  (Beside an
// M2L on the SIMT cores nothing is in the way, and an FP64 near field on every SM
// slows it.)
size_t spread_smem(bool spread, unsigned blocks, size_t shm, size_t stat) {
    if (!spread) return shm;
    constexpr size_t kSM = 228 * 1024, kBlock = 1024;   // an SM's; what a block takes beside its own
    const size_t per = (blocks + (unsigned)sm_count() - 1) / (unsigned)sm_count();
    const size_t want = (kSM / (per + 1) + 128) & ~(size_t)127;
    return std::max(shm, want > kBlock + stat ? want - kBlock - stat : 0);
}

// One evaluation kernel (mode 1: near field, 2: far field).  FP64 rules of a 4^3
// lattice per leaf and closed-form voxels have near fields of their own; the
// queued kernels run on the blocks that fit the device at once.
template <class T>
gf_status eval_launch(gf_plan_s *plan, EvalArgs a, int n1, int mode, cudaStream_t st) {
    const FmmPlan *F = plan->fmm;
    const bool spread = mode == 1 && m2l_fills_sms(plan, a.B);
    const unsigned grid = (unsigned)std::min<int64_t>((F->n_items + kEvalWarps - 1) / kEvalWarps, 152 * 64);
    const size_t shm = spread_smem(spread, grid, kSrcTable * (sizeof(Vec4<T>) + sizeof(int)) +
                                             sizeof(T) * kEvalWarps * eval_slice((int)sizeof(T)), 0);
    if (sizeof(T) == 4 && mode == 2) {
        const size_t fshm = sizeof(float) * kFarWarps * far_slice(F->p * F->p);
        GF_TRY((ensure_smem(eval_far_kernel, fshm)));
        const unsigned fg = (unsigned)std::min<int64_t>((F->n_items + kFarWarps - 1) / kFarWarps, 152 * 64);
        const unsigned rg = std::min<unsigned>(fg, resident_blocks(eval_far_kernel, kFarWarps * 32, fshm));
        eval_far_kernel<<<rg, kFarWarps * 32, fshm, st>>>(a, F->leaf_beg);
    } else if (sizeof(T) == 8 && mode == 2) {
        const size_t fshm = sizeof(double) * kFar64Warps * 3 * F->p * F->p;
        const unsigned fg = (unsigned)std::min<int64_t>((2 * F->n_items + kFar64Warps - 1) / kFar64Warps, 152 * 64);
        far_f64_kernel<<<fg, kFar64Warps * 32, fshm, st>>>(a);
    } else if (sizeof(T) == 8 && n1 == 4) {
        const unsigned ng = (unsigned)std::min<int64_t>(2 * F->n_items, 152 * 64);
        const size_t nshm = spread_smem(spread, ng, 0, kNear64Static);
        GF_TRY((ensure_smem(near_f64_kernel, nshm, kNear64Static)));
        near_f64_kernel<<<ng, kNear64Warps * 32, nshm, st>>>(a);
    } else if (sizeof(T) == 4 && (plan->opt.reserved0 & GF_FLAG_SUM_AN)) {
        const unsigned ag = (unsigned)std::min<int64_t>((2 * F->n_items + kAnWarps - 1) / kAnWarps, 152 * 64);
        const size_t ashm = spread_smem(spread, ag, sizeof(float) * kAnWarps * near_an_slice(), 0);
        GF_TRY((ensure_smem(near_an_kernel, ashm)));
        near_an_kernel<<<std::min<unsigned>(ag, resident_blocks(near_an_kernel, kAnWarps * 32, ashm)), kAnWarps * 32, ashm,
                         st>>>(a);
    } else if (sizeof(T) == 4 && n1 == 4) {
        GF_TRY((ensure_smem(eval_kernel<float, 4>, shm)));
        const unsigned rg = std::min<unsigned>(grid, resident_blocks(eval_kernel<float, 4>, kEvalWarps * 32, shm));
        eval_kernel<float, 4><<<rg, kEvalWarps * 32, shm, st>>>(a);
    } else {
        GF_TRY((ensure_smem(eval_kernel<T, 0>, shm)));
        const unsigned rg = std::min<unsigned>(grid, resident_blocks(eval_kernel<T, 0>, kEvalWarps * 32, shm));
        eval_kernel<T, 0><<<rg, kEvalWarps * 32, shm, st>>>(a);
    }
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class T>
gf_status run_forward(gf_plan_s *plan, const void *rho, int rho_dtype, int B, double *g, double *gz,
                      cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const int K = F->K, L = F->L;
    const int b3 = F->b * F->b * F->b;
    const bool pts = F->points;
    const bool fused = !pts && p2m_fused_ok<T>(F);
    const Block3 lb = block_of(F->lev[L]);
    // 4^3-voxel leaves: the folded P2M kernels, where the rule does not mirror on the
    // voxel centres with its shift after them
    const bool shift = F->shift_f[0] != nullptr;
    const bool fold = !pts && (p2m_fold_ok(plan) || shift) && lb.n[1] * 4 <= 65535 && lb.n[2] * 4 * B <= 65535;
    bool up = false;   // level L-1 expansions made straight from the density grid
    // the kernels that write each level's expansions (folded, or the points'
    // P2M) also take the largest |input| of the slabs its M2L reads, in place of a pass over
    // those rows before the M2L
    F->amax_fused = (fold || pts) && F->tc_amax != nullptr;
    if (F->amax_fused) GF_CUDA(cudaMemsetAsync(F->tc_amax, 0, (kMaxLevels + 1) * sizeof(uint32_t), st));
    if (pts) {
        // a0 + a3 for point sources: masses in leaf order, P2M over each leaf's points
        GF_TRY(points_masses<T>(plan, rho, rho_dtype, B, st));
        stage_mark(plan, 1, st);
        GF_TRY(points_p2m<T>(plan, B, st));
    } else if (fold) {
        // a0 + a3 (timed as P2M): leaf-blocked masses and leaf expansions, of
        // every leaf or -- when the expansions of level L-1 come straight from
        // the grid -- of the z-slabs that the leaf level's M2L (and so the near
        // field) reaches
        stage_mark(plan, 1, st);
        up = L - 1 > 2;   // level 2 keeps its FP64 M2M
        const FmmLevel &lf = F->lev[L];
        const int64_t z0 = up ? lf.m2l_z0 : 0;
        const int64_t nz = up ? std::max<int64_t>(0, lf.m2l_z1 - lf.m2l_z0 + 1) : lb.n[2];
        const int64_t slab = lb.n[0] * lb.n[1];
        GF_TRY((launch_blocking<T, 4>(plan, rho, rho_dtype == GF_DTYPE_F32, B, z0, nz, st)));
        GF_TRY(p2m_leaf_run<T>(plan, B, z0 * slab, nz * slab, st));
        if (up) GF_TRY(p2m_up_run<T>(plan, rho, rho_dtype == GF_DTYPE_F32, B, st));
        if (shift) {
            GF_TRY(p2m_shift_run(plan, B, L, z0 * slab, nz * slab, st));
            if (up) GF_TRY(p2m_shift_run(plan, B, L - 1, 0, F->lev[L - 1].ns, st));
        }
    } else if (fused) {
        stage_mark(plan, 1, st);
        GF_TRY(launch_p2m_fused<T>(plan, rho, rho_dtype == GF_DTYPE_F32, B, st));
    }
    // a0: leaf-blocked densities
    if (!fused && !fold && !pts) {
        const FmmLevel &lv = F->lev[L];
        const int64_t total = lv.ns * B * b3;
        const unsigned grid = (unsigned)std::min<int64_t>((total + 255) / 256, 152 * 16);
        block_densities<T><<<grid, 256, 0, st>>>(rho, rho_dtype == GF_DTYPE_F32, plan->grid.n[0], plan->grid.n[1],
                                                 plan->grid.n[2], F->voff[0], F->voff[1], F->voff[2],
                                                 block_of(lv), F->b, B, (T *)F->mass, plan->d_status);
        GF_KERNEL_DONE();
    }
    if (!fused && !fold && !pts) stage_mark(plan, 1, st);
    // a3: P2M at the leaves
    if (!fused && !fold && !pts) {
        const FmmLevel &lv = F->lev[L];
        const unsigned grid = ceil_div(lv.ns, kP2MLeaves);
        const size_t shm = sizeof(T) * kP2MLeaves * B * b3;
        const T *P = sizeof(T) == 8 ? (const T *)F->p2m_d : (const T *)F->p2m_f;
        GF_TRY(ensure_smem(p2m_kernel<T>, shm));
        p2m_kernel<T><<<grid, 128, shm, st>>>((const T *)F->mass, P, lv.ns, b3, B, K, F->KS, (T *)lv.me);
        GF_KERNEL_DONE();
    }
    stage_mark(plan, 2, st);
    // a4: M2M up to level 2.  In mixed precision the translation into the
    // top level (2) is done in FP64, the deeper ones in FP32.
    for (int l = up ? L - 2 : L - 1; l >= 2; --l) {
        if (sizeof(T) == 4 && l <= 2)
            GF_TRY((translate_run<T, double>(plan, l, 0, B, st)));
        else
            GF_TRY((translate_run<T, T>(plan, l, 0, B, st)));
    }
    stage_mark(plan, 3, st);
    // a7-a9 set up before the M2L: the near field of the evaluation only
    // reads the leaf masses, so it runs on the plan's second stream beside
    // the M2L and the L2L chain (from the M2L's launch on); the far field
    // (L2P, near + far in FP64, scatter) joins it once the L2L is done.
    // With stage timing on, both halves run in line on the forward's stream.
    const bool eval_on = !pts && F->n_items > 0;
    const bool an = (plan->opt.reserved0 & GF_FLAG_SUM_AN) != 0;
    EvalArgs ea;
    int n1 = 0;
    if (eval_on) n1 = eval_setup<T>(plan, B, g, gz, ea);
    const bool beside = eval_on && !(an && sizeof(T) == 8) && plan->side && !plan->timing;
    // a5/a6: M2L at every level (each overwrites its level's LE), then the
    // L2L chain from level 3 down, which adds each finished parent LE.
    GF_TRY(m2l_run<T>(plan, B, false, st, beside ? plan->ev_fork : nullptr));   // marks the input split's end (4)
    if (beside) {
        GF_CUDA(cudaStreamWaitEvent(plan->side, plan->ev_fork, 0));
        GF_TRY(eval_launch<T>(plan, ea, n1, 1, plan->side));
        GF_CUDA(cudaEventRecord(plan->ev_join, plan->side));
    }
    stage_mark(plan, 5, st);
    for (int l = 3; l <= L; ++l) {
        const FmmLevel &lv = F->lev[l];
        if (lv.nt == 0) continue;
        if (sizeof(T) == 4 && l - 1 <= 2)
            GF_TRY((translate_run<T, double>(plan, l, 1, B, st)));
        else
            GF_TRY((translate_run<T, T>(plan, l, 1, B, st)));
    }
    stage_mark(plan, 6, st);
    // a7-a9: near field + L2P + combine + scatter
    if (pts) {
        GF_TRY(points_eval<T>(plan, B, g, gz, st));
    } else if (eval_on && an && sizeof(T) == 8) {
        // closed-form voxels: radius 2 in FP32 (near_an_kernel), 4 in FP64 (the
        // closed form cancels like (d/h)^3, so the precision sets how far it is
        // used; beyond it the corrected midpoint rule errs like (h/d)^6)
        const unsigned grid = (unsigned)std::min<int64_t>((F->n_items + kEvalWarps - 1) / kEvalWarps, 152 * 64);
        const size_t shan = sizeof(T) * kEvalWarps * eval_an_slice(F->p * F->p) + 64;
        GF_TRY((ensure_smem(eval_an_kernel<double, 4>, shan)));
        eval_an_kernel<double, 4><<<grid, kEvalWarps * 32, shan, st>>>(ea);
        GF_KERNEL_DONE();
    } else if (eval_on) {
        if (beside)
            GF_CUDA(cudaStreamWaitEvent(st, plan->ev_join, 0));
        else
            GF_TRY(eval_launch<T>(plan, ea, n1, 1, st));
        GF_TRY(eval_launch<T>(plan, ea, n1, 2, st));
    }
    stage_mark(plan, 7, st);
    return GF_OK;
}

}  // namespace

gf_status fmm_forward(gf_plan_s *plan, const void *rho, int rho_dtype, int B, double *g, double *gz,
                      cudaStream_t st) {
    if (plan->M == 0) return GF_OK;
    if (plan->fmm->mixed) return run_forward<float>(plan, rho, rho_dtype, B, g, gz, st);
    return run_forward<double>(plan, rho, rho_dtype, B, g, gz, st);
}


}  // namespace gf
