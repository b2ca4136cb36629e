// gf_adjoint.cu -- the transpose of the FMM forward model.
//
// Eq. 1 is linear in the density, so the gradient of any misfit with respect
// to the voxel densities is the transpose of the forward operator applied to
// the misfit's derivative with respect to the outputs.  The forward operator
// is, per observer j,  g_j = G h (N rho + E L Mt P rho)_j  with N the near
// field, P the P2M matrix, Mt the M2M/M2L chain up to the leaf local
// expansions and E the L2P gradient.  This file applies, exactly,
//   grad = G h (N^T r + P^T Mt^T L^T E^T r):
//   E^T  -- each leaf's observers deposit r_j . grad(basis_k)(X_j) into a dual
//           local expansion (l2p_adj);
//   L^T  -- dual local expansions flow from children to parents (L2L^T);
//   M2L^T-- every source box collects T_{-o}^T times the dual local expansion
//           of the observer box at offset o, over its parity class's 189
//           offsets (the interaction-list rule is symmetric);
//   M2M^T-- dual multipole expansions flow from parents to children;
//   P^T, N^T -- dual multipole expansions are expanded back over the voxels
//           and the near-field sum is taken with the observers as sources.
// Under 4^3-voxel leaves and a mirror-symmetric rule the transposed P2M is
// folded like the forward one (gf_xlate.cu) and goes from level L - 1 straight
// to the voxels (p2m_transpose); the leaf level then holds only what its own
// M2L^T puts there -- in the few z-slabs that an interaction list reaches --
// and is added, with the near field (near_transpose), to those slabs.  Other
// plans bring the dual expansions down to every leaf (adj_eval).
// The plan's ME/LE/mass workspaces hold the dual quantities, so a plan's
// forward and adjoint calls must not overlap on the device.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "fmm_math.cuh"
#include "gf_fmm.cuh"
#include "gf_m2l.cuh"
#include "gf_pair.cuh"
#include "gf_simd.cuh"

namespace gf {
namespace {

__device__ __forceinline__ int64_t unmorton(uint64_t k, int s) {
    int64_t c = 0;
    for (int bit = 0; bit < 21; ++bit) c |= (int64_t)((k >> (3 * bit + s)) & 1) << bit;
    return c;
}

// observer box index over the widened source block of a level
__global__ void fill_imap(const uint64_t *__restrict__ tkey, int64_t nt, int64_t lo0, int64_t lo1, int64_t lo2,
                          int64_t n0, int64_t n1, int64_t n2, int32_t *__restrict__ imap) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    const uint64_t k = tkey[t];
    const int64_t x = unmorton(k, 0) - lo0, y = unmorton(k, 1) - lo1, z = unmorton(k, 2) - lo2;
    if (x >= 0 && y >= 0 && z >= 0 && x < n0 && y < n1 && z < n2) imap[(z * n1 + y) * n0 + x] = (int32_t)t;
}

// child[parent][position] for the observer boxes of the next level
__global__ void fill_child(const uint64_t *__restrict__ tkey, const int32_t *__restrict__ tparent, int64_t nt,
                           int32_t *__restrict__ child) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nt) return;
    child[(int64_t)tparent[c] * 8 + (int)(tkey[c] & 7)] = (int32_t)c;
}

// ---------------------------------------------------------------- E^T
// Recursion coefficients of the regular harmonics (the recursion of
// fmm_math.cuh): for m < n < kMaxP, t = n (n + 1) / 2 + m,
//   c_ha[t] = (2n - 1) / sqrt((n + m)(n - m)),
//   c_hb[t] = sqrt((n - 1 + m)(n - 1 - m)) / sqrt((n + m)(n - m)),
// c_hf[m] = -sqrt((2m - 1) / (2m)).
__constant__ double c_ha[kMaxP * (kMaxP + 1) / 2], c_hb[kMaxP * (kMaxP + 1) / 2], c_hf[kMaxP];
__constant__ float c_haf[kMaxP * (kMaxP + 1) / 2], c_hbf[kMaxP * (kMaxP + 1) / 2], c_hff[kMaxP];

template <class T>
__device__ __forceinline__ T hcoef(const double *d, const float *f, int i) {
    if constexpr (sizeof(T) == 4)
        return f[i];
    else
        return d[i];
}

// Dual local expansion of one observer leaf:
//   LE*_k = -(1/b^2) sum_j sum_a r_ja d(phi_k)/dX_a (X_j)
// phi_k the k-th real basis function of a local expansion (R_n^0, 2 Re R_n^m,
// 2 Im R_n^m) and X_j the observer's offset from the leaf centre in leaf
// units.  The derivatives of degree n are combinations of harmonics of degree
// n - 1 (fmm_math.cuh), so the observers are first summed into moments,
// W^c_k = sum_j r_jc R_k(X_j) for every weight column c (component and batch
// member) -- the harmonics of 32 observers at a time, made once for all
// columns, times their weights -- and the combination is taken once per leaf.
// One block per leaf; thread k of the sums holds up to CT columns.
// 1024 leaves of 64 observers, p = 12, 16 models: 452 -> 37 us (a block synchronised
// three times for every observer and took square roots per harmonic before).
template <class T, int CT>
__global__ void __launch_bounds__(256)
l2p_adj(const int32_t *__restrict__ leaf_beg, const int32_t *__restrict__ perm, const T *__restrict__ tloc,
        const double *__restrict__ r, int ncomp, int64_t M, int B, int p, int K, int ldk, int b,
        T *__restrict__ le) {
    extern __shared__ __align__(16) unsigned char shraw[];
    const int P2 = p * p, C = ncomp * B;
    T *H = reinterpret_cast<T *>(shraw);        // [32][P2 | 1] harmonics; then the moments [C][P2]
    T *rw = H + ((32 * (P2 | 1) + 3) & ~3);     // [32][CT] weights
    T *W = H;
    const int hs = P2 | 1;
    const int64_t t = blockIdx.x;
    const int j0 = leaf_beg[t], j1 = leaf_beg[t + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T inv_b = T(1) / T(b);
    T acc[CT];
#pragma unroll
    for (int c = 0; c < CT; ++c) acc[c] = T(0);
    for (int jj = j0; jj < j1; jj += 32) {
        const int cnt = min(32, j1 - jj);
        __syncthreads();   // the previous observers have been used
        for (int e = threadIdx.x; e < 32 * CT; e += blockDim.x) {
            const int j = e / CT, c = e - j * CT;
            T v = T(0);
            if (j < cnt && c < C) {
                const int64_t cj = perm[jj + j];
                const int bb = c / ncomp, a = c - bb * ncomp;
                v = (T)r[((int64_t)bb * M + cj) * ncomp + a];
            }
            rw[e] = v;
        }
        {   // lane's observer, columns m = warp, warp + 8, ... of its harmonics
            const int64_t j = jj + min(lane, cnt - 1);
            const T x = tloc[3 * j] * inv_b, y = tloc[3 * j + 1] * inv_b, z = tloc[3 * j + 2] * inv_b;
            const T r2 = x * x + y * y + z * z;
            T *h = H + lane * hs;
            T sr = T(1), si = T(0);
            int at = 0;   // R_at^at is (sr, si)
            for (int m = warp; m < p; m += 8) {
                for (; at < m; ++at) {
                    const T f = hcoef<T>(c_hf, c_hff, at + 1);
                    const T nr = f * (x * sr - y * si), ni = f * (x * si + y * sr);
                    sr = nr;
                    si = ni;
                }
                T r1 = sr, i1 = si, r0 = T(0), i0 = T(0);
                h[kidx_re(m, m)] = sr;
                if (m > 0) h[kidx_im(m, m)] = si;
                for (int n = m + 1; n < p; ++n) {
                    const int q = n * (n + 1) / 2 + m;
                    const T az = hcoef<T>(c_ha, c_haf, q) * z, br = hcoef<T>(c_hb, c_hbf, q) * r2;
                    const T cr = az * r1 - br * r0, ci = az * i1 - br * i0;
                    h[kidx_re(n, m)] = cr;
                    if (m > 0) h[kidx_im(n, m)] = ci;
                    r0 = r1;
                    i0 = i1;
                    r1 = cr;
                    i1 = ci;
                }
            }
        }
        __syncthreads();
        if ((int)threadIdx.x < P2)
            for (int j = 0; j < cnt; ++j) {
                const T h = H[j * hs + threadIdx.x];
#pragma unroll
                for (int c = 0; c < CT; ++c) acc[c] += h * rw[j * CT + c];
            }
    }
    __syncthreads();
    if ((int)threadIdx.x < P2)
#pragma unroll
        for (int c = 0; c < CT; ++c)
            if (c < C) W[c * P2 + threadIdx.x] = acc[c];
    __syncthreads();
    const T sc = T(-1) / (T(b) * T(b));
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        int n = (int)sqrtf((float)k + 0.5f);
        const int ro = k - n * n, m = (ro + 1) / 2;
        const bool im = ro > 0 && (ro % 2 == 0);
        const T A = sqrt(T((n - m) * (n + m))), al = sqrt(T((n + m) * (n + m - 1))), bu = sqrt(T((n - m) * (n - m - 1)));
        const T f = m == 0 ? T(1) : T(2);
        // moments of R_{n-1}^{m-1} (l), R_{n-1}^m (c), R_{n-1}^{m+1} (u)
        auto get = [&](const T *w, int mm, T &re, T &imv) {
            re = imv = T(0);
            const bool neg = mm < 0;   // R^{-1} = -conj(R^1)
            if (neg) mm = 1;
            if (mm > n - 1) return;
            re = w[kidx_re(n - 1, mm)];
            if (mm > 0) imv = w[kidx_im(n - 1, mm)];
            if (neg) re = -re;
        };
        for (int bb = 0; bb < B; ++bb) {
            T v = T(0);
            if (n > 0) {
                const T *w = W + (size_t)bb * ncomp * P2;
                T cr, ci;
                get(w + (ncomp == 3 ? 2 * P2 : 0), m, cr, ci);
                v = A * (im ? ci : cr);
                if (ncomp == 3) {
                    T lr, li, ur, ui;
                    get(w, m - 1, lr, li);
                    get(w, m + 1, ur, ui);
                    v += T(0.5) * (im ? -al * li + bu * ui : -al * lr + bu * ur);
                    get(w + P2, m - 1, lr, li);
                    get(w + P2, m + 1, ur, ui);
                    v += T(0.5) * (im ? -(al * lr + bu * ur) : al * li + bu * ui);   // -i (s_r + i s_i)
                }
            }
            le[(t * B + bb) * ldk + k] = sc * f * v;
        }
    }
}

gf_status upload_harmonic_coefs(int device) {
    static std::mutex mu;
    static unsigned long long done = 0;
    std::lock_guard<std::mutex> lk(mu);
    if (device >= 0 && device < 64 && ((done >> device) & 1ull)) return GF_OK;
    constexpr int NT = kMaxP * (kMaxP + 1) / 2;
    double ha[NT] = {}, hb[NT] = {}, hf[kMaxP] = {};
    float haf[NT], hbf[NT], hff[kMaxP];
    for (int n = 1; n < kMaxP; ++n) {
        for (int m = 0; m < n; ++m) {
            const double inv = 1.0 / std::sqrt((double)((n + m) * (n - m)));
            ha[n * (n + 1) / 2 + m] = (2 * n - 1) * inv;
            hb[n * (n + 1) / 2 + m] = n - 1 > m ? std::sqrt((double)((n - 1 + m) * (n - 1 - m))) * inv : 0.0;
        }
        hf[n] = -std::sqrt((2.0 * n - 1.0) / (2.0 * n));
    }
    for (int t = 0; t < NT; ++t) {
        haf[t] = (float)ha[t];
        hbf[t] = (float)hb[t];
    }
    for (int n = 0; n < kMaxP; ++n) hff[n] = (float)hf[n];
    GF_CUDA(cudaMemcpyToSymbol(c_ha, ha, sizeof(ha)));
    GF_CUDA(cudaMemcpyToSymbol(c_hb, hb, sizeof(hb)));
    GF_CUDA(cudaMemcpyToSymbol(c_hf, hf, sizeof(hf)));
    GF_CUDA(cudaMemcpyToSymbol(c_haf, haf, sizeof(haf)));
    GF_CUDA(cudaMemcpyToSymbol(c_hbf, hbf, sizeof(hbf)));
    GF_CUDA(cudaMemcpyToSymbol(c_hff, hff, sizeof(hff)));
    if (device >= 0 && device < 64) done |= 1ull << device;
    return GF_OK;
}

template <class T, int CT>
gf_status launch_l2p_adj(gf_plan_s *plan, const double *r, int ncomp, int B, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &leaf = F->lev[F->L];
    const int P2 = F->p * F->p;
    const size_t h = std::max<size_t>(((32 * (P2 | 1) + 3) & ~3), (size_t)ncomp * B * P2);
    const size_t shm = sizeof(T) * (std::max<size_t>(h, ((32 * (P2 | 1) + 3) & ~3) + 32 * CT));
    GF_TRY((ensure_smem(l2p_adj<T, CT>, shm)));
    l2p_adj<T, CT><<<(unsigned)leaf.nt, 256, shm, st>>>(
        F->leaf_beg, F->perm, sizeof(T) == 8 ? (const T *)F->tloc_d : (const T *)F->tloc_f, r, ncomp, plan->M, B, F->p,
        F->K, F->KS, F->b, (T *)leaf.le);
    GF_KERNEL_DONE();
    return GF_OK;
}

// ---------------------------------------------------------------- folded P^T
// Column c of the transposed P2M: a box's dual multipole expansion times the
// transposed operator of the all-positive octant, class by class
// (Z_chi[v] = sum over the components k of class chi of P[v][k] x[k]), then the
// inverse of the fold over the eight mirrored voxels,
//   out[v mirrored to o] = sum_chi s_o(chi) Z_chi[v].
// NV = 64: boxes of level L - 1 (octants of 4^3 voxels), stored into the
// gradient; NV = 8: leaves (2^3), added to it.  Thread (v, group) holds four
// columns.  FP32: the sums are compensated (the product's and the sum's
// rounding errors are kept beside them), so they carry what an FP64
// accumulation of the FP32 products did; two columns form a packed pair.
// Bound by FP32 issue (ten packed instructions a product), next
// to writing the gradient.  128^3, p = 12, 16 models: with the M2M^T to the leaves
// and the near field below, 34.1 -> 0.76 ms; from the boxes of level L - 1 416 us,
// the slab leaves 127 us, the near field 215 us.
struct P2MTArgs {
    const void *me;                 // dual expansions
    const void *tab;                // [off[8]][NV], class order, zero where perm is -1
    const int *perm;                // [off[8]] component of each place, or -1
    int off[9];                     // classes, multiples of four
    int ldk, B;
    uint32_t ncol, first;           // columns; first box
    int32_t blo[3], bn[3];          // block of the boxes
    int32_t gn[3], voff[3];
    int64_t nvox;
    double scale;
    ScalePair sp;
    int pair_ok;                    // scale through sp (FP32)
    double *grad;
};

constexpr int kTCols = 4;

__device__ __forceinline__ void two_sum2(uint64_t a, uint64_t b, uint64_t &s, uint64_t &e) {
    s = add2(a, b);
    const uint64_t bp = sub2(s, a);
    e = add2(sub2(a, sub2(s, bp)), sub2(b, bp));
}

template <class T, int NV>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 1) p2m_transpose(P2MTArgs a) {
    extern __shared__ __align__(16) unsigned char shraw[];
    constexpr int PB = 128 / NV * kTCols, XP = PB + 4;   // columns; row pitch (spreads the staging over the banks)
    T *xs = reinterpret_cast<T *>(shraw);                // [off[8]][XP], class order
    constexpr int E = NV == 64 ? 4 : 2;     // octant edge
    const int tid = threadIdx.x;
    const uint32_t col0 = blockIdx.x * PB;
    const T *me = reinterpret_cast<const T *>(a.me) + (int64_t)a.first * a.B * a.ldk;
    const int rows = a.off[8];
    for (int e = tid; e < rows * PB; e += 128) {
        const int pos = e % rows, c = e / rows;
        const uint32_t col = min(col0 + c, a.ncol - 1);
        const int k = a.perm[pos];
        xs[pos * XP + c] = k >= 0 ? __ldg(me + (int64_t)col * a.ldk + k) : T(0);
    }
    __syncthreads();
    const int v = tid % NV, cg = tid / NV;
    const T *t = reinterpret_cast<const T *>(a.tab) + v;
    const T *x = xs + cg * kTCols;
    double out[kTCols][8];
    if constexpr (sizeof(T) == 4) {
        uint64_t zh[2][8], zl[2][8];
        float tn[4];   // the next four operator entries, in flight
#pragma unroll
        for (int q = 0; q < 4; ++q) tn[q] = __ldg(t + q * NV);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            uint64_t s[2] = {0, 0}, c[2] = {0, 0};
#pragma unroll 1
            for (int pos = a.off[e]; pos < a.off[e + 1]; pos += 4) {
                float tv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) tv[q] = tn[q];
                if (pos + 4 < rows)
#pragma unroll
                    for (int q = 0; q < 4; ++q) tn[q] = __ldg(t + (pos + 4 + q) * NV);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint64_t t2 = pk2(tv[q], tv[q]), tm = pk2(-tv[q], -tv[q]);
                    const ulonglong2 x4 = *reinterpret_cast<const ulonglong2 *>(x + (pos + q) * XP);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const uint64_t xv = u ? x4.y : x4.x, pr = mul2(t2, xv);
                        const uint64_t ep = fma2(tm, xv, pr);   // minus the product's rounding error
                        uint64_t ns, es;
                        two_sum2(s[u], pr, ns, es);
                        s[u] = ns;
                        c[u] = add2(c[u], sub2(es, ep));
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                zh[u][e] = s[u];
                zl[u][e] = c[u];
            }
        }
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
#pragma unroll
            for (int o = 0; o < 8; ++o)
                if (!((o >> ax) & 1)) {
                    const int h = o | (1 << ax);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const uint64_t p0 = zh[u][o], p1 = zh[u][h], q0 = zl[u][o], q1 = zl[u][h];
                        uint64_t sp, ep, sm, em;
                        two_sum2(p0, p1, sp, ep);
                        two_sum2(p0, sub2(0, p1), sm, em);
                        zh[u][h] = sp;   // positive side: a0 + a1
                        zl[u][h] = add2(ep, add2(q0, q1));
                        zh[u][o] = sm;   // negative side: a0 - a1
                        zl[u][o] = add2(em, sub2(q0, q1));
                    }
                }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                float h0, h1, l0, l1;
                up2(zh[u][o], h0, h1);
                up2(zl[u][o], l0, l1);
                out[2 * u][o] = a.pair_ok ? scaled_pair(h0, l0, a.sp) : pair_to_f64(h0, l0) * a.scale;
                out[2 * u + 1][o] = a.pair_ok ? scaled_pair(h1, l1, a.sp) : pair_to_f64(h1, l1) * a.scale;
            }
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            double s[kTCols] = {};
#pragma unroll 2
            for (int pos = a.off[e]; pos < a.off[e + 1]; ++pos) {
                const double tv = __ldg(t + pos * NV);
#pragma unroll
                for (int c = 0; c < kTCols; ++c) s[c] = fma(tv, (double)x[pos * XP + c], s[c]);
            }
#pragma unroll
            for (int c = 0; c < kTCols; ++c) out[c][e] = s[c] * a.scale;
        }
#pragma unroll
        for (int c = 0; c < kTCols; ++c)
#pragma unroll
            for (int ax = 0; ax < 3; ++ax)
#pragma unroll
                for (int o = 0; o < 8; ++o)
                    if (!((o >> ax) & 1)) {
                        const double p0 = out[c][o], p1 = out[c][o | (1 << ax)];
                        out[c][o | (1 << ax)] = p0 + p1;
                        out[c][o] = p0 - p1;
                    }
    }
    const int vx = v % E, vy = (v / E) % E, vz = v / (E * E);
#pragma unroll
    for (int c = 0; c < kTCols; ++c) {
        const uint32_t col = col0 + cg * kTCols + c;
        if (col >= a.ncol) break;
        const uint32_t rel = col / (uint32_t)a.B, bb = col - rel * a.B, box = a.first + rel;
        const uint32_t byz = box / (uint32_t)a.bn[0], bz = byz / (uint32_t)a.bn[1];
        const int i0 = 2 * E * (a.blo[0] + (int)(box - byz * a.bn[0])) - a.voff[0],
                  j0 = 2 * E * (a.blo[1] + (int)(byz - bz * a.bn[1])) - a.voff[1], k0 = 2 * E * (a.blo[2] + (int)bz) - a.voff[2];
        double *g = a.grad + (int64_t)bb * a.nvox;
        int64_t at[8];
        double old[8];
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const int i = i0 + ((o & 1) ? E + vx : E - 1 - vx), j = j0 + ((o & 2) ? E + vy : E - 1 - vy),
                      k = k0 + ((o & 4) ? E + vz : E - 1 - vz);
            const bool in = i >= 0 && j >= 0 && k >= 0 && i < a.gn[0] && j < a.gn[1] && k < a.gn[2];
            at[o] = in ? ((int64_t)k * a.gn[1] + j) * a.gn[0] + i : -1;
            old[o] = NV == 8 && in ? g[at[o]] : 0.0;   // all reads in flight before the first write
        }
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (at[o] >= 0) g[at[o]] = NV == 8 ? old[o] + out[c][o] : out[c][o];
    }
}

// ---------------------------------------------------------------- N^T beside the folded P^T
// One warp per source leaf of 4^3 voxels (two per lane) and chunk of BT batch
// members: for every observer of the neighbouring observer leaves the kernel
// vector sum_q w_q d / |d|^3 of both voxels is made once and multiplied by the
// chunk's weights (NC components each); sums over one observer leaf are merged
// with TwoSum and added to the gradient.  Leaves without an observer leaf
// beside them are left at once.  Bound by the weighting (BT fused multiply-adds
// a pair and component) and reading the weights.
struct NearTArgs {
    const int32_t *leaf_beg, *perm;
    const void *tloc;
    const double *r;
    int64_t M;
    int B, nq;
    const int32_t *imap;       // level L window map
    int32_t mlo[3], mn[3];
    int32_t blo[3], bn[3];     // leaf source block
    uint32_t first, nleaf;     // leaves of the slabs
    const QuadRule *qr;
    int32_t gn[3], voff[3];
    int64_t nvox;
    double scale, eps2;
    double *grad;
};

constexpr int kNearTWarps = 4;

template <class T, int NC, int BT>
__global__ void __launch_bounds__(kNearTWarps * 32) near_transpose(NearTArgs a) {
    constexpr int W = NC * BT, RS = 4 + ((W + 3) & ~3);   // staged observer: position, weights
    __shared__ __align__(16) T stage[kNearTWarps][32 * RS];
    __shared__ T node[kMaxQuad][4];   // node offsets from the voxel's lower corner, weights
    for (int q = threadIdx.x; q < a.nq; q += blockDim.x) {
        for (int d = 0; d < 3; ++d) node[q][d] = (T)(0.5 + 0.5 * a.qr->xi[q][d]);
        node[q][3] = (T)a.qr->wn[q];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t e = blockIdx.x * kNearTWarps + warp;
    if (e >= a.nleaf) return;
    const uint32_t leaf = a.first + e, lyz = leaf / (uint32_t)a.bn[0], lz = lyz / (uint32_t)a.bn[1];
    const int S[3] = {a.blo[0] + (int)(leaf - lyz * a.bn[0]), a.blo[1] + (int)(lyz - lz * a.bn[1]), a.blo[2] + (int)lz};
    const int b0 = blockIdx.y * BT;
    // the neighbouring observer leaves (lane nb of the 27)
    int tl = -1;
    if (lane < 27) {
        const int wx = S[0] + lane % 3 - 1 - a.mlo[0], wy = S[1] + (lane / 3) % 3 - 1 - a.mlo[1],
                  wz = S[2] + lane / 9 - 1 - a.mlo[2];
        if (wx >= 0 && wy >= 0 && wz >= 0 && wx < a.mn[0] && wy < a.mn[1] && wz < a.mn[2])
            tl = a.imap[((int64_t)wz * a.mn[1] + wy) * a.mn[0] + wx];
    }
    unsigned todo = __ballot_sync(0xffffffffu, tl >= 0);
    if (!todo) return;
    T *os = stage[warp];
    const T *tloc = reinterpret_cast<const T *>(a.tloc);
    const T eps2 = (T)a.eps2;
    const T vx = T(lane & 3) - T(2), vy = T((lane >> 2) & 3) - T(2), vz0 = T(lane >> 4) - T(2), vz1 = vz0 + T(2);
    T hi[2][BT], lo[2][BT];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < BT; ++c) hi[u][c] = lo[u][c] = T(0);
    while (todo) {
        const int nb = __ffs(todo) - 1;
        todo &= todo - 1;
        const int t = __shfl_sync(0xffffffffu, tl, nb);
        const T ox = T(4 * (nb % 3 - 1)), oy = T(4 * ((nb / 3) % 3 - 1)), oz = T(4 * (nb / 9 - 1));
        const int j0 = a.leaf_beg[t], j1 = a.leaf_beg[t + 1];
        T part[2][BT];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int c = 0; c < BT; ++c) part[u][c] = T(0);
        for (int c0 = j0; c0 < j1; c0 += 32) {
            const int cnt = min(32, j1 - c0);
            __syncwarp();
            if (lane < cnt) {
                const int64_t jj = c0 + lane;
                T *o = os + lane * RS;
                o[0] = tloc[3 * jj] + ox;
                o[1] = tloc[3 * jj + 1] + oy;
                o[2] = tloc[3 * jj + 2] + oz;
                const int64_t cj = a.perm[jj];
#pragma unroll
                for (int c = 0; c < BT; ++c)
#pragma unroll
                    for (int d = 0; d < NC; ++d)
                        o[4 + c * NC + d] = b0 + c < a.B ? (T)a.r[((int64_t)(b0 + c) * a.M + cj) * NC + d] : T(0);
            }
            __syncwarp();
            // the kernel vector of one node
            auto pair = [&](T ddx, T ddy, T ddz, T wq, T (&k)[3]) {
                const T r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                T k3;
                if constexpr (sizeof(T) == 4) {
                    // the reciprocal square root, refined by one Newton step
                    const float y = rsqrt_ftz(r2);
                    const float ri = fmaf(0.5f * y, fmaf(-r2 * y, y, 1.f), y);
                    k3 = r2 > eps2 ? wq * ri * ri * ri : 0.f;
                } else {
                    k3 = __double_as_longlong(r2) > __double_as_longlong(eps2) ? inv_r3(r2, wq) : 0.0;
                }
                if (NC == 3) {
                    k[0] += k3 * ddx;
                    k[1] += k3 * ddy;
                }
                k[2] += k3 * ddz;
            };
            auto weigh = [&](const T *o, const T (&k)[2][3]) {
#pragma unroll
                for (int c = 0; c < BT; ++c)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (NC == 3) {
                            part[u][c] += k[u][0] * o[4 + 3 * c];
                            part[u][c] += k[u][1] * o[5 + 3 * c];
                            part[u][c] += k[u][2] * o[6 + 3 * c];
                        } else {
                            part[u][c] += k[u][2] * o[4 + c];
                        }
                    }
            };
            if (a.nq == 1) {
                const T bx = vx + node[0][0], by = vy + node[0][1], bz0 = vz0 + node[0][2], bz1 = vz1 + node[0][2],
                        wq = node[0][3];
                for (int s = 0; s < cnt; ++s) {
                    const T *o = os + s * RS;
                    T k[2][3] = {};
                    pair(o[0] - bx, o[1] - by, o[2] - bz0, wq, k[0]);
                    pair(o[0] - bx, o[1] - by, o[2] - bz1, wq, k[1]);
                    weigh(o, k);
                }
            } else {
                for (int s = 0; s < cnt; ++s) {
                    const T *o = os + s * RS;
                    T k[2][3] = {};
                    for (int q = 0; q < a.nq; ++q) {
                        const T dx = o[0] - (vx + node[q][0]), dy = o[1] - (vy + node[q][1]), wq = node[q][3];
                        pair(dx, dy, o[2] - (vz0 + node[q][2]), wq, k[0]);
                        pair(dx, dy, o[2] - (vz1 + node[q][2]), wq, k[1]);
                    }
                    weigh(o, k);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int c = 0; c < BT; ++c) two_sum(hi[u][c], lo[u][c], part[u][c]);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = 4 * S[0] + (lane & 3) - a.voff[0], j = 4 * S[1] + ((lane >> 2) & 3) - a.voff[1],
                  k = 4 * S[2] + (lane >> 4) + 2 * u - a.voff[2];
        if (i < 0 || j < 0 || k < 0 || i >= a.gn[0] || j >= a.gn[1] || k >= a.gn[2]) continue;
#pragma unroll
        for (int c = 0; c < BT; ++c)
            if (b0 + c < a.B)
                a.grad[(int64_t)(b0 + c) * a.nvox + ((int64_t)k * a.gn[1] + j) * a.gn[0] + i] +=
                    ((double)hi[u][c] + (double)lo[u][c]) * a.scale;
    }
}

// ---------------------------------------------------------------- N^T, P^T
// One warp per source leaf.  Each lane owns up to two voxels of the leaf;
// the observers of every neighbouring observer leaf are staged in shared
// memory (offset from this leaf's centre and the weights) and each lane
// accumulates, for its voxels' quadrature nodes, sum_j r_j . d / |d|^3 with
// d the observer minus the node.  The dual multipole expansion is then
// expanded back over the voxels with the P2M matrix.  Per-leaf partial sums
// are merged with TwoSum; the result is scaled by G h and scattered to the
// caller's grid order.
constexpr int kAdjWarps = 4;
constexpr int kAdjChunk = 32;
constexpr int kAdjMaxB = 16;

template <class T>
__device__ __forceinline__ void two_sum_a(T &hi, T &lo, T x) {
    const T s = hi + x;
    const T bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
}

struct AdjArgs {
    const int32_t *leaf_beg, *perm;
    const void *tloc;
    const double *r;
    int ncomp;
    int64_t M;
    int B, K, ldk, b, nq, p;
    const int32_t *imap;       // level L window map
    int64_t mlo[3], mn[3];
    int64_t blo[3], bn[3];     // leaf source block
    const void *me;            // dual ME at the leaves
    const void *P;             // [b^3][K]
    const QuadRule *qr;
    int64_t gn[3];             // grid voxels
    int64_t voff[3];
    double scale, eps2;
    double *grad;
};

template <class T>
__global__ void __launch_bounds__(kAdjWarps * 32)
adj_eval(AdjArgs a) {
    extern __shared__ unsigned char shraw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int B = a.B;
    // per-warp slice: observers [kAdjChunk][3 + 3 B]
    const int ostride = 3 + 3 * B;
    T *os = reinterpret_cast<T *>(shraw) + (size_t)warp * kAdjChunk * ostride;
    const T *tloc = reinterpret_cast<const T *>(a.tloc);
    const T *me = reinterpret_cast<const T *>(a.me);
    const T *P = reinterpret_cast<const T *>(a.P);
    const int b = a.b, b3 = b * b * b;
    const int64_t nleaf = a.bn[0] * a.bn[1] * a.bn[2];
    const T half_b = T(0.5) * T(b);
    const T eps2 = (T)a.eps2;
    for (int64_t sl = (int64_t)blockIdx.x * kAdjWarps + warp; sl < nleaf; sl += (int64_t)gridDim.x * kAdjWarps) {
        const int64_t lx = sl % a.bn[0], ly = (sl / a.bn[0]) % a.bn[1], lz = sl / (a.bn[0] * a.bn[1]);
        const int64_t Sx = a.blo[0] + lx, Sy = a.blo[1] + ly, Sz = a.blo[2] + lz;
        for (int v0 = 0; v0 < b3; v0 += 64) {
            int vv[2];
            vv[0] = v0 + lane;
            vv[1] = v0 + lane + 32;
            T hi[2][kAdjMaxB], lo[2][kAdjMaxB];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int bb = 0; bb < kAdjMaxB; ++bb) hi[u][bb] = lo[u][bb] = T(0);
            for (int nb = 0; nb < 27; ++nb) {
                const int dx = nb % 3 - 1, dy = (nb / 3) % 3 - 1, dz = nb / 9 - 1;
                const int64_t wx = Sx + dx - a.mlo[0], wy = Sy + dy - a.mlo[1], wz = Sz + dz - a.mlo[2];
                if (wx < 0 || wy < 0 || wz < 0 || wx >= a.mn[0] || wy >= a.mn[1] || wz >= a.mn[2]) continue;
                const int32_t t = a.imap[(wz * a.mn[1] + wy) * a.mn[0] + wx];
                if (t < 0) continue;
                const int j0 = a.leaf_beg[t], j1 = a.leaf_beg[t + 1];
                T part[2][kAdjMaxB];
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int bb = 0; bb < kAdjMaxB; ++bb) part[u][bb] = T(0);
                for (int c0 = j0; c0 < j1; c0 += kAdjChunk) {
                    const int cnt = min(kAdjChunk, j1 - c0);
                    __syncwarp();
                    if (lane < cnt) {
                        const int64_t jj = c0 + lane;
                        T *o = os + lane * ostride;
                        o[0] = tloc[3 * jj + 0] + T(dx * b);
                        o[1] = tloc[3 * jj + 1] + T(dy * b);
                        o[2] = tloc[3 * jj + 2] + T(dz * b);
                        const int64_t cj = a.perm[jj];
                        for (int bb = 0; bb < B; ++bb) {
                            if (a.ncomp == 3) {
                                o[3 + 3 * bb + 0] = (T)a.r[((int64_t)bb * a.M + cj) * 3 + 0];
                                o[3 + 3 * bb + 1] = (T)a.r[((int64_t)bb * a.M + cj) * 3 + 1];
                                o[3 + 3 * bb + 2] = (T)a.r[((int64_t)bb * a.M + cj) * 3 + 2];
                            } else {
                                o[3 + 3 * bb + 0] = T(0);
                                o[3 + 3 * bb + 1] = T(0);
                                o[3 + 3 * bb + 2] = (T)a.r[(int64_t)bb * a.M + cj];
                            }
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int v = vv[u];
                        if (v >= b3) continue;
                        const int vx = v % b, vy = (v / b) % b, vz = v / (b * b);
                        for (int q = 0; q < a.nq; ++q) {
                            const T sx = T(vx) + (T)(0.5 + 0.5 * a.qr->xi[q][0]) - half_b;
                            const T sy = T(vy) + (T)(0.5 + 0.5 * a.qr->xi[q][1]) - half_b;
                            const T sz = T(vz) + (T)(0.5 + 0.5 * a.qr->xi[q][2]) - half_b;
                            const T wq = (T)a.qr->wn[q];
                            for (int s = 0; s < cnt; ++s) {
                                const T *o = os + s * ostride;
                                const T ddx = o[0] - sx, ddy = o[1] - sy, ddz = o[2] - sz;
                                const T r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                                T ri = T(0);
                                if (r2 > eps2) ri = T(1) / sqrt(r2);
                                const T k3 = wq * ri * ri * ri;
#pragma unroll
                                for (int bb = 0; bb < kAdjMaxB; ++bb)
                                    if (bb < B)
                                        part[u][bb] += k3 * (o[3 + 3 * bb] * ddx + o[4 + 3 * bb] * ddy +
                                                             o[5 + 3 * bb] * ddz);
                            }
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int bb = 0; bb < kAdjMaxB; ++bb)
                        if (bb < B) two_sum_a(hi[u][bb], lo[u][bb], part[u][bb]);
            }
            // far part and scatter
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int v = vv[u];
                if (v >= b3) continue;
                const int64_t gi = Sx * b + v % b - a.voff[0], gj = Sy * b + (v / b) % b - a.voff[1],
                              gk = Sz * b + v / (b * b) - a.voff[2];
                const bool in = gi >= 0 && gj >= 0 && gk >= 0 && gi < a.gn[0] && gj < a.gn[1] && gk < a.gn[2];
                for (int bb = 0; bb < B && bb < kAdjMaxB; ++bb) {
                    const T *mer = me + (sl * B + bb) * a.ldk;
                    double far = 0.0;
                    for (int k = 0; k < a.K; ++k) far += (double)P[(size_t)v * a.K + k] * (double)mer[k];
                    if (in) {
                        const double val = ((double)hi[u][bb] + (double)lo[u][bb] + far) * a.scale;
                        a.grad[(int64_t)bb * a.gn[0] * a.gn[1] * a.gn[2] + (gk * a.gn[1] + gj) * a.gn[0] + gi] = val;
                    }
                }
            }
        }
    }
}

}  // namespace

gf_status fmm_adjoint_prepare(gf_plan_s *plan, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    DeviceArena &A = plan->arena;
    GF_TRY(upload_harmonic_coefs(plan->device));
    for (int l = 2; l <= F->L; ++l) {
        FmmLevel &lv = F->lev[l];
        int64_t n = 1;
        for (int d = 0; d < 3; ++d) {
            F->mlo[l][d] = lv.slo[d] - 3;
            F->mn[l][d] = lv.sn[d] + 6;
            n *= F->mn[l][d];
        }
        GF_TRY(A.alloc_n(&F->imap[l], n));
        GF_CUDA(cudaMemsetAsync(F->imap[l], 0xff, sizeof(int32_t) * n, st));
        if (lv.nt > 0) {
            fill_imap<<<ceil_div(lv.nt, 256), 256, 0, st>>>(lv.tkey, lv.nt, F->mlo[l][0], F->mlo[l][1], F->mlo[l][2],
                                                            F->mn[l][0], F->mn[l][1], F->mn[l][2], F->imap[l]);
            GF_KERNEL_DONE();
        }
        if (l < F->L) {
            GF_TRY(A.alloc_n(&F->child[l], std::max<int64_t>(lv.nt, 1) * 8));
            GF_CUDA(cudaMemsetAsync(F->child[l], 0xff, sizeof(int32_t) * std::max<int64_t>(lv.nt, 1) * 8, st));
            const FmmLevel &ch = F->lev[l + 1];
            if (ch.nt > 0) {
                fill_child<<<ceil_div(ch.nt, 256), 256, 0, st>>>(ch.tkey, ch.tparent, ch.nt, F->child[l]);
                GF_KERNEL_DONE();
            }
        }
        // source boxes per parity class, in the z-slabs that the M2L^T writes
        F->scls_off[l][0] = 0;
        const int64_t nz = std::max<int64_t>(0, lv.m2l_z1 - lv.m2l_z0 + 1);
        for (int c = 0; c < 8; ++c) {
            int64_t cnt = 1;
            for (int d = 0; d < 3; ++d) {
                const int64_t par = (c >> d) & 1, lo = lv.slo[d] + (d == 2 ? lv.m2l_z0 : 0), n = d == 2 ? nz : lv.sn[d];
                const int64_t i0 = (par - (lo & 1) + 2) & 1;
                cnt *= n > i0 ? (n - i0 + 1) / 2 : 0;
            }
            F->scls_off[l][c + 1] = F->scls_off[l][c] + cnt;
        }
    }
    return GF_OK;
}

namespace {

template <class T, int NV>
gf_status launch_p2m_transpose(gf_plan_s *plan, P2MTArgs a, int level, int64_t first, int64_t count, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    if (count <= 0) return GF_OK;
    const FmmLevel &lv = F->lev[level];
    a.me = lv.me;
    a.tab = NV == 64 ? (sizeof(T) == 8 ? (const void *)F->p2m_upt_d : (const void *)F->p2m_upt_f)
                     : (sizeof(T) == 8 ? (const void *)F->p2m_leaft_d : (const void *)F->p2m_leaft_f);
    for (int d = 0; d < 3; ++d) {
        a.blo[d] = (int32_t)lv.slo[d];
        a.bn[d] = (int32_t)lv.sn[d];
    }
    a.first = (uint32_t)first;
    a.ncol = (uint32_t)(count * a.B);
    constexpr int PB = 128 / NV * kTCols;
    const size_t shm = sizeof(T) * (size_t)a.off[8] * (PB + 4);
    GF_TRY((ensure_smem(p2m_transpose<T, NV>, shm)));
    p2m_transpose<T, NV><<<ceil_div((int64_t)a.ncol, PB), 128, shm, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

// P^T and N^T of 4^3-voxel leaves under a mirror-symmetric rule: from the
// boxes of level L - 1 (up) into every voxel, then the slabs of leaves that
// hold their own dual expansions (every leaf when !up) and the near field.
template <class T>
gf_status fold_eval(gf_plan_s *plan, const double *r, int ncomp, int B, double *grad, bool up, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const FmmLevel &leaf = F->lev[F->L];
    P2MTArgs a;
    memset(&a, 0, sizeof(a));
    a.perm = F->tab->cls_perm;
    for (int c = 0; c <= 8; ++c) a.off[c] = F->tab->cls_off[c];
    a.ldk = F->KS;
    a.B = B;
    a.nvox = plan->nvox;
    a.scale = plan->G * F->h;
    a.pair_ok = scale_pair(a.scale, a.sp) ? 1 : 0;
    a.grad = grad;
    for (int d = 0; d < 3; ++d) {
        a.gn[d] = (int32_t)plan->grid.n[d];
        a.voff[d] = (int32_t)F->voff[d];
    }
    if (up)
        GF_TRY((launch_p2m_transpose<T, 64>(plan, a, F->L - 1, 0, F->lev[F->L - 1].ns, st)));
    else
        GF_CUDA(cudaMemsetAsync(grad, 0, sizeof(double) * (size_t)B * plan->nvox, st));
    const int64_t slab = leaf.sn[0] * leaf.sn[1];
    const int64_t z0 = leaf.m2l_z0, nz = std::max<int64_t>(0, leaf.m2l_z1 - leaf.m2l_z0 + 1);
    if (up)
        GF_TRY((launch_p2m_transpose<T, 8>(plan, a, F->L, z0 * slab, nz * slab, st)));
    else
        GF_TRY((launch_p2m_transpose<T, 8>(plan, a, F->L, 0, leaf.ns, st)));
    if (nz == 0) return GF_OK;
    NearTArgs n;
    memset(&n, 0, sizeof(n));
    n.leaf_beg = F->leaf_beg;
    n.perm = F->perm;
    n.tloc = sizeof(T) == 8 ? (const void *)F->tloc_d : (const void *)F->tloc_f;
    n.r = r;
    n.M = plan->M;
    n.B = B;
    n.nq = F->nq;
    n.imap = F->imap[F->L];
    for (int d = 0; d < 3; ++d) {
        n.mlo[d] = (int32_t)F->mlo[F->L][d];
        n.mn[d] = (int32_t)F->mn[F->L][d];
        n.blo[d] = (int32_t)leaf.slo[d];
        n.bn[d] = (int32_t)leaf.sn[d];
        n.gn[d] = a.gn[d];
        n.voff[d] = a.voff[d];
    }
    n.first = (uint32_t)(z0 * slab);
    n.nleaf = (uint32_t)(nz * slab);
    n.qr = quad_device(plan);
    n.nvox = plan->nvox;
    n.scale = a.scale;
    n.eps2 = sizeof(T) == 8 ? 1e-18 : 1e-12;
    n.grad = grad;
    const unsigned gx = ceil_div(n.nleaf, kNearTWarps);
#define GF_NEAR_T(NC, BT) near_transpose<T, NC, BT><<<dim3(gx, ceil_div(B, BT)), kNearTWarps * 32, 0, st>>>(n)
    if (ncomp == 1) {
        if (B == 1)
            GF_NEAR_T(1, 1);
        else if (B <= 4)
            GF_NEAR_T(1, 4);
        else
            GF_NEAR_T(1, 16);
    } else if (B == 1) {
        GF_NEAR_T(3, 1);
    } else {
        GF_NEAR_T(3, 4);
    }
#undef GF_NEAR_T
    GF_KERNEL_DONE();
    return GF_OK;
}

template <class T>
gf_status run_adjoint(gf_plan_s *plan, const double *r, int ncomp, int B, double *grad, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    const int K = F->K, L = F->L;
    const FmmLevel &leaf = F->lev[L];
    // E^T: dual local expansions of the observer leaves
    if (leaf.nt > 0) {
        const int C = ncomp * B;
        if (C <= 4)
            GF_TRY((launch_l2p_adj<T, 4>(plan, r, ncomp, B, st)));
        else if (C <= 16)
            GF_TRY((launch_l2p_adj<T, 16>(plan, r, ncomp, B, st)));
        else
            GF_TRY((launch_l2p_adj<T, 48>(plan, r, ncomp, B, st)));
    }
    // L^T: children to parents (the transpose of the top FP64 translation
    // stays in FP64 in mixed precision)
    for (int l = L - 1; l >= 2; --l) {
        if (sizeof(T) == 4 && l <= 2)
            GF_TRY((translate_run<T, double>(plan, l, 3, B, st)));
        else
            GF_TRY((translate_run<T, T>(plan, l, 3, B, st)));
    }
    // M2L^T at every level, into the z-slabs that an interaction list reaches
    // (the others' dual multipole expansions are zero)
    for (int l = 2; l <= L; ++l) {
        const FmmLevel &lv = F->lev[l];
        const int64_t row = (int64_t)B * F->KS * sizeof(T), slab = lv.sn[0] * lv.sn[1] * row;
        const int64_t z0 = lv.m2l_z1 >= lv.m2l_z0 ? lv.m2l_z0 : lv.sn[2],
                      z1 = lv.m2l_z1 >= lv.m2l_z0 ? lv.m2l_z1 + 1 : lv.sn[2];
        char *me = (char *)lv.me;
        if (z0 > 0) GF_CUDA(cudaMemsetAsync(me, 0, z0 * slab, st));
        if (z1 < lv.sn[2]) GF_CUDA(cudaMemsetAsync(me + z1 * slab, 0, (lv.sn[2] - z1) * slab, st));
    }
    GF_TRY(m2l_run<T>(plan, B, true, st));
    // M2M^T: parents to children, top down (to the leaves unless the folded P^T
    // takes level L - 1 to the voxels)
    const bool fold = p2m_fold_ok(plan) && leaf.ns * B <= 0x7fffffff;
    const bool up = fold && L - 1 > 2;
    for (int l = 3; l <= (up ? L - 1 : L); ++l) {
        if (sizeof(T) == 4 && l - 1 <= 2)
            GF_TRY((translate_run<T, double>(plan, l, 2, B, st)));
        else
            GF_TRY((translate_run<T, T>(plan, l, 2, B, st)));
    }
    if (fold) return fold_eval<T>(plan, r, ncomp, B, grad, up, st);
    // P^T and N^T, scaled by G h, scattered to grid order
    AdjArgs a;
    a.leaf_beg = F->leaf_beg;
    a.perm = F->perm;
    a.tloc = sizeof(T) == 8 ? (const void *)F->tloc_d : (const void *)F->tloc_f;
    a.r = r;
    a.ncomp = ncomp;
    a.M = plan->M;
    a.B = B;
    a.K = K;
    a.ldk = F->KS;
    a.b = F->b;
    a.nq = F->nq;
    a.p = F->p;
    a.imap = F->imap[L];
    for (int d = 0; d < 3; ++d) {
        a.mlo[d] = F->mlo[L][d];
        a.mn[d] = F->mn[L][d];
        a.blo[d] = leaf.slo[d];
        a.bn[d] = leaf.sn[d];
        a.gn[d] = plan->grid.n[d];
        a.voff[d] = F->voff[d];
    }
    a.me = leaf.me;
    a.P = sizeof(T) == 8 ? (const void *)F->p2m_d : (const void *)F->p2m_f;
    a.qr = quad_device(plan);
    a.scale = plan->G * F->h;
    a.eps2 = sizeof(T) == 8 ? 1e-18 : 1e-12;
    a.grad = grad;
    const int64_t nleaf = leaf.ns;
    const size_t shm = sizeof(T) * kAdjWarps * kAdjChunk * (3 + 3 * B);
    GF_TRY(ensure_smem(adj_eval<T>, shm));
    const unsigned grid = (unsigned)std::min<int64_t>((nleaf + kAdjWarps - 1) / kAdjWarps, 152 * 32);
    adj_eval<T><<<grid, kAdjWarps * 32, shm, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

}  // namespace

gf_status fmm_adjoint(gf_plan_s *plan, const double *r, int ncomp, int B, double *grad, cudaStream_t st) {
    if (B > kAdjMaxB) {
        set_error("the FMM adjoint takes at most %d batch members per call", kAdjMaxB);
        return GF_ERR_UNSUPPORTED;
    }
    if (plan->M == 0) {
        GF_CUDA(cudaMemsetAsync(grad, 0, sizeof(double) * B * plan->nvox, st));
        return GF_OK;
    }
    FmmPlan *F = plan->fmm;
    if (!F->adj_ready) {   // adjoint-only structures, built once per plan
        GF_TRY(fmm_adjoint_prepare(plan, plan->arena.stream));
        GF_TRY(m2l_tc_prepare_adj(plan));
        GF_CUDA(cudaStreamSynchronize(plan->arena.stream));
        F->adj_ready = true;
    }
    if (plan->fmm->mixed) return run_adjoint<float>(plan, r, ncomp, B, grad, st);
    return run_adjoint<double>(plan, r, ncomp, B, grad, st);
}

}  // namespace gf
