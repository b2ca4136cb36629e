// gf_m2l.cu -- M2L over the interaction list, as a batched dense contraction:
// on the tensor cores in mixed precision (tiles of 128 columns of one parity
// class, offset by offset), on the SIMT cores otherwise (columns folded by
// mirror symmetry).  Sources outside the source block contribute zeros.  Each
// output is written once, so the result is deterministic.
#include <cuda_fp16.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "gf_fold.cuh"
#include "gf_m2l.cuh"

namespace gf {

__constant__ signed char c_il[8][189][3];

gf_status m2l_upload_offsets(const signed char h_il[8][189][3]) {
    GF_CUDA(cudaMemcpyToSymbol(c_il, h_il, sizeof(signed char) * 8 * 189 * 3));
    return GF_OK;
}

namespace {

// Byte offset of FP16 element (row, k), k < 32, in a [rows][32] tile stored
// K-major with the 64-byte swizzle: 8-row atoms of 512 bytes, the 16-byte
// chunk index (8 halves) XOR-ed with bits 1-2 of the row inside the atom.
__host__ __device__ __forceinline__ uint32_t swz64h(int row, int k) {
    return (uint32_t)((row >> 3) * 512 + (row & 7) * 64 + ((((k >> 3) ^ (row >> 1)) & 3) << 4) + (k & 7) * 2);
}

// Column scales of an M2L operator set (one block per output component n <
// Npad): s_n = 2^(14 - ceil(log2 max |T_o[n][k]|)), the maximum over the
// used offset slots and every input k.  cs[n] = s_n, cs[Npad + n] = 1 / s_n
// (1 for empty columns and n >= K).
__global__ void m2l_colscale(const double *__restrict__ tab, int K, int Npad, float *__restrict__ cs) {
    __shared__ double red[256];
    const int n = blockIdx.x;
    double mx = 0.0;
    if (n < K)
        for (int e = threadIdx.x; e < 343 * K; e += blockDim.x) {
            const int off = e / K, kin = e - off * K;
            const int dx = off % 7 - 3, dy = (off / 7) % 7 - 3, dz = off / 49 - 3;
            if (max(abs(dx), max(abs(dy), abs(dz))) < 2) continue;
            mx = fmax(mx, fabs(tab[(size_t)off * K * K + (size_t)kin * K + n]));
        }
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        int sh = 0;
        if (red[0] > 0.0) {
            int e;
            const double f = frexp(red[0], &e);   // red = f 2^e, f in [0.5, 1)
            sh = 14 - (f == 0.5 ? e - 1 : e);
        }
        cs[n] = ldexpf(1.f, sh);
        cs[Npad + n] = ldexpf(1.f, -sh);
    }
}

// FP16 operator images of the tensor-core M2L: img[off][c][part][Npad][32],
// part 0 = FP16(T s), part 1 = FP16(T s - part 0), T = T_off[k_out][k_in]
// for the 32 inputs of chunk c, s = the column scale of k_out.
__global__ void build_h16_images(const double *__restrict__ tab, int K, int Npad, int nck,
                                 const float *__restrict__ cs, __half *__restrict__ img) {
    const int off = blockIdx.x;
    const int dx = off % 7 - 3, dy = (off / 7) % 7 - 3, dz = off / 49 - 3;
    const bool used = max(abs(dx), max(abs(dy), abs(dz))) >= 2;
    const size_t tile = (size_t)Npad * 32;
    for (int c = 0; c < nck; ++c) {
        __half *hi = img + ((size_t)off * nck + c) * 2 * tile;
        __half *lo = hi + tile;
        for (int e = threadIdx.x; e < Npad * 32; e += blockDim.x) {
            const int n = e / 32, kk = e % 32, kin = 32 * c + kk;
            const double v = (used && n < K && kin < K) ? tab[(size_t)off * K * K + (size_t)kin * K + n] * cs[n] : 0.0;
            const float f = (float)v;
            const __half h = __float2half_rn(f);
            const uint32_t o = swz64h(n, kk) / 2;
            hi[o] = h;
            lo[o] = __float2half_rn(f - __half2float(h));
        }
    }
}

}  // namespace

gf_status m2l_prepare_tables(Tables *T, cudaStream_t st) {
    const int npad = (T->K + 15) & ~15;
    if (npad > 256) return GF_OK;  // beyond one MMA's N: SIMT only
    T->tc_npad = npad;
    T->tc_nck_h = (T->K + 31) / 32;
    const size_t n = (size_t)343 * T->tc_nck_h * 2 * npad * 32;
    for (int adj = 0; adj < 2; ++adj) {
        const double *tab = adj ? T->am2l_d : T->m2l_d;
        void *&img = adj ? T->am2l_tc : T->m2l_tc;
        float *&cs = adj ? T->am2l_cs : T->m2l_cs;
        GF_CUDA(cudaMalloc(&cs, 2 * npad * sizeof(float)));
        m2l_colscale<<<npad, 256, 0, st>>>(tab, T->K, npad, cs);
        GF_KERNEL_DONE();
        GF_CUDA(cudaMalloc(&img, n * sizeof(__half)));
        build_h16_images<<<343, 256, 0, st>>>(tab, T->K, npad, T->tc_nck_h, cs, (__half *)img);
        GF_KERNEL_DONE();
    }
    return GF_OK;
}

namespace {

__device__ __forceinline__ int64_t dm(uint64_t k, int s) {
    int64_t c = 0;
    for (int bit = 0; bit < 21; ++bit) c |= (int64_t)((k >> (3 * bit + s)) & 1) << bit;
    return c;
}

// Boxes of a dense block [lo, lo + n) whose coordinates have the parities of
// class `cls` (bit a = parity on axis a): per-axis first offset and count.
__host__ __device__ __forceinline__ void class_lattice(int cls, const int64_t *lo, const int64_t *n, int64_t *i0,
                                                       int64_t *cnt) {
    for (int a = 0; a < 3; ++a) {
        const int64_t par = (cls >> a) & 1;
        i0[a] = (par - (lo[a] & 1) + 2) & 1;
        cnt[a] = n[a] > i0[a] ? (n[a] - i0[a] + 1) / 2 : 0;
    }
}

// j-th box of class `cls` in a dense block: coordinates relative to lo.
__device__ __forceinline__ void class_box(int cls, const int64_t *lo, const int64_t *n, int64_t j, int64_t &x,
                                          int64_t &y, int64_t &z) {
    int64_t i0[3], c[3];
    class_lattice(cls, lo, n, i0, c);
    x = i0[0] + 2 * (j % c[0]);
    y = i0[1] + 2 * ((j / c[0]) % c[1]);
    z = i0[2] + 2 * (j / (c[0] * c[1]));
}

// ---------------------------------------------------------------- SIMT
// The M2L on the SIMT cores (FP64 plans; GF_FLAG_M2L_SIMT; degrees beyond one
// MMA's width), folded by mirror symmetry: the up to eight offsets
// (+-a, +-b, +-c) of a box's list have operators that are signed copies of
// T_(a, b, c), so their sources are folded (an 8-point Walsh-Hadamard transform)
// and take one K x K product: 56 products for the 189 offsets of an interior
// box, 28 for the 63 of a box above its sources.  The FP64 pipe (two
// instructions a clock and SM) bounds it, so everything else -- gathering,
// table reads, index work -- only has to stay out of its way.  One launch
// takes every level (the longest lists, the upper levels, first); a block owns
// P columns (box, batch member), any parity classes mixed, and runs the 56
// magnitudes in turn; thread (i, group) sums component i of a 16-byte group of
// columns.  128^3 voxels, p = 14, 256^2 stations, FP64: the M2L 275 -> 10.8 ms
// (each level a launch of 8..64 blocks before, one after another; the FP64 pipe
// is now 95% busy on an active SM).
struct FoldLevel {
    const void *in;          // forward: ME_l; adjoint: LE_l duals
    void *out;               // forward: LE_l; adjoint: ME_l duals
    const uint64_t *tkey;    // forward: observer boxes
    const int32_t *imap;     // adjoint: observer box of a place, or -1
    int32_t blo[3], bn[3];   // source block
    int32_t mlo[3], mn[3];   // adjoint: extent of the map
    uint32_t ncol, blk0;     // columns; first block of the level
};

struct FoldM2LArgs {
    FoldLevel lv[kMaxLevels + 1];
    int lmin, lmax;
    int K, ldk, B, adj;
    const void *tab;             // [343][K][K], input component major
    uint32_t part_lo, part_hi;   // source partition (forward)
};

template <class T, int P>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 512 : 640, sizeof(T) == 8 ? 2 : 1)
m2l_fold(const __grid_constant__ FoldM2LArgs a) {
    constexpr int G = Lay<T, P>::G, NG = Lay<T, P>::NG;
    constexpr int Q = sizeof(T) == 8 ? 2 : 4;   // staged inputs per thread (FP64: two blocks' registers fit an SM)
    extern __shared__ __align__(16) unsigned char shraw[];
    T *xs = reinterpret_cast<T *>(shraw);   // folded inputs (Lay)
    __shared__ int64_t crow[P * 8];
    __shared__ int ccoord[P][3], cmember[P];
    const int K = a.K, tid = threadIdx.x, nthr = blockDim.x;
    int l = a.lmin;
    while (l < a.lmax && blockIdx.x >= a.lv[l + 1].blk0) ++l;
    const FoldLevel &L = a.lv[l];
    const uint32_t col0 = (blockIdx.x - L.blk0) * P;
    if (tid < P) {   // the columns' boxes, relative to the source block
        const uint32_t col = min(col0 + tid, L.ncol - 1), box = col / (uint32_t)a.B;
        cmember[tid] = (int)(col - box * a.B);
        if (!a.adj) {
            const uint64_t key = L.tkey[box];
            for (int d = 0; d < 3; ++d) ccoord[tid][d] = (int)dm(key, d) - L.blo[d];
        } else {
            const uint32_t yz = box / (uint32_t)L.bn[0], z = yz / (uint32_t)L.bn[1];
            ccoord[tid][0] = (int)(box - yz * L.bn[0]);
            ccoord[tid][1] = (int)(yz - z * L.bn[1]);
            ccoord[tid][2] = (int)z;
        }
    }
    const bool on = tid < K * NG;
    const int grp = on ? tid / K : 0, i = on ? tid - grp * K : 0, cls = parity_of(i);
    const T *in = reinterpret_cast<const T *>(L.in);
    Acc<T, G> acc;
    acc.zero();
    for (int mag = 0; mag < 64; ++mag) {
        const int ma[3] = {mag & 3, (mag >> 2) & 3, mag >> 4};
        if (max(ma[0], max(ma[1], ma[2])) < 2) continue;
        __syncthreads();   // the previous magnitude's inputs have been used
        int any = 0;
        if (tid < 8 * P) {
            // source at (s_x a, s_y b, s_z c), s = - where the bit of o is clear
            const int c = tid >> 3, o = tid & 7;
            int64_t row = -1;
            int s[3];
            bool ok = col0 + c < L.ncol;
            for (int d = 0; d < 3; ++d) {
                const int off = ((o >> d) & 1) ? ma[d] : -ma[d];
                const int t = ccoord[c][d], par = (t + L.blo[d]) & 1;
                // the list reaches [-2, 3] from an even place, [-3, 2] from an odd
                // one; a zero component is counted once
                ok = ok && off >= -2 - par && off <= 3 - par && (ma[d] != 0 || ((o >> d) & 1));
                s[d] = t + off;
            }
            if (ok && !a.adj) {
                ok = s[0] >= 0 && s[1] >= 0 && s[2] >= 0 && s[0] < L.bn[0] && s[1] < L.bn[1] && s[2] < L.bn[2] &&
                     in_source_part(s[0] + L.blo[0], s[1] + L.blo[1], s[2] + L.blo[2], l - 2, a.part_lo, a.part_hi);
                if (ok) row = ((((int64_t)s[2] * L.bn[1] + s[1]) * L.bn[0] + s[0]) * a.B + cmember[c]) * a.ldk;
            } else if (ok) {
                const int w[3] = {s[0] + L.blo[0] - L.mlo[0], s[1] + L.blo[1] - L.mlo[1], s[2] + L.blo[2] - L.mlo[2]};
                if (w[0] >= 0 && w[1] >= 0 && w[2] >= 0 && w[0] < L.mn[0] && w[1] < L.mn[1] && w[2] < L.mn[2]) {
                    const int32_t m = L.imap[((int64_t)w[2] * L.mn[1] + w[1]) * L.mn[0] + w[0]];
                    if (m >= 0) row = ((int64_t)m * a.B + cmember[c]) * a.ldk;
                }
            }
            crow[tid] = row;
            any = row >= 0 ? 1 << o : 0;
        }
        const int sides = tid < 32 * ((8 * P + 31) / 32) ? __reduce_or_sync(0xffffffffu, any) : 0;
        const int has = __syncthreads_or(sides) ? 1 : 0;
        if (!has) continue;
        // Q inputs of one column per thread; a mirror pair with one side
        // missing throughout the column needs no additions
        for (int e = tid; e < (((K + 3) & ~3) / Q) * P; e += nthr) {
            const int c = e % P, j0 = Q * (e / P);
            T v[Q][8];
            int have = 0;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const int64_t row = crow[c * 8 + o];
                have |= (row >= 0) << o;
                if constexpr (Q == 4) {
                    T w[4];
                    load4<T, T>(in, row, j0, K, w);
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q][o] = w[q];
                } else {
#pragma unroll
                    for (int q = 0; q < Q; ++q) v[q][o] = row >= 0 && j0 + q < K ? __ldg(in + row + j0 + q) : T(0);
                }
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int hi_set = d == 0 ? 0xaa : d == 1 ? 0xcc : 0xf0;
                const bool lo_any = have & ~hi_set & 0xff, hi_any = have & hi_set;
#pragma unroll
                for (int o = 0; o < 8; ++o)
                    if (!((o >> d) & 1)) {
                        const int h = o | (1 << d);
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            const T lo = v[q][o], hi = v[q][h];
                            if (lo_any && hi_any) {
                                v[q][o] = hi + lo;
                                v[q][h] = hi - lo;
                            } else if (hi_any) {
                                v[q][o] = hi;
                            } else {
                                v[q][h] = -lo;
                            }
                        }
                    }
                have |= (have & hi_set) >> (1 << d) | (have & ~hi_set & 0xff) << (1 << d);
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int sw = parity_of(j0 + q) ^ (((j0 + q) >> 2) & 7);
#pragma unroll
                for (int d = 0; d < 8; ++d) xs[Lay<T, P>::at(j0 + q, d ^ sw, c)] = v[q][d];
            }
        }
        __syncthreads();
        const T *t = reinterpret_cast<const T *>(a.tab) + (size_t)((ma[2] + 3) * 49 + (ma[1] + 3) * 7 + ma[0] + 3) * K * K + i;
#pragma unroll 2
        for (int g = 0; 4 * g < K; ++g) {
            T tv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) tv[q] = 4 * g + q < K ? __ldg(t + (size_t)(4 * g + q) * K) : T(0);
            const T *x = xs + ((size_t)(4 * g * NG + grp) * 8 + (cls ^ (g & 7) ^ (grp & 7))) * G;
#pragma unroll
            for (int q = 0; q < 4; ++q) acc.add(0, tv[q], x + q * 8 * P);
        }
    }
    if (!on) return;
    T *out = reinterpret_cast<T *>(L.out);
#pragma unroll
    for (int c = 0; c < G; ++c) {
        const uint32_t col = col0 + grp * G + c;
        if (col < L.ncol) out[(int64_t)col * a.ldk + i] = acc.get(c);
    }
}

// ---------------------------------------------------------------- tcgen05
// Tensor-core M2L (mixed precision, and FP64 plans that ask for it).  A CTA
// owns 128 target columns -- (box, batch member) pairs of one parity class of
// one level -- and, offset by offset, computes
// D_o[col][k_out] = sum_k_in ME[t + o][k_in] T_o[k_out][k_in] on the tensor
// cores from FP16 parts, A_hi B_hi + A_hi B_lo + A_lo B_hi (K = 16 per MMA),
// with FP32 accumulation.  Both operands are scaled by powers of two so that
// every part that matters is a normal FP16 number: the inputs of a level by
// 2^sh (largest |input| into (2^14, 2^15]), each output column of the operator
// images by its own factor; the write-back divides both out exactly.  The
// inputs are split once per level by a small kernel before the M2L.  Inputs
// come in chunks of 32, two to a stage, through a ring of shared-memory stages
// (64-byte swizzle), filled by warp-specialised producers:
//   warps 0-3   A producers: 16-byte asynchronous copies straight into the
//               stage (eight lanes per row's 128 contiguous bytes), which is
//               signalled once they have landed;
//   warp 4      one thread issues the MMAs of a stage and commits them to the
//               stage's "empty" barrier (and, after an offset's last chunk,
//               to the bank's "full" barrier);
//   warp 5      one thread bulk-copies the pre-split, pre-swizzled operator
//               image of each stage;
//   warps 6-13  promoters: after each offset they read the finished bank of
//               tensor memory and add it into FP32 registers (two banks
//               alternate, so the tensor cores never accumulate more than one
//               offset: their FP32 accumulation rounds differently from
//               IEEE and long chains over zero-mean data lose digits).
// Offsets whose source boxes are all missing are skipped by every role (a
// per-tile list built first).  Every wait is bounded and watches an abort
// flag; a wait that gives up sets status[1], and the CTA then drains its
// copies and MMAs (bounded) and frees its tensor memory.

struct TcLevel {
    float *le;            // output rows (LE_l or adjoint ME_l duals)
    const int32_t *order;
    const uint64_t *tkey;
    int64_t blo[3], bn[3];
    int64_t cls_off[9];
    int adj;
    int64_t slab0;        // adjoint: boxes of the source block before [blo, bn)
    const int32_t *imap;
    int64_t mlo[3], mn[3];
    const uint32_t *amax;        // largest |input| of the level (float bits)
    const unsigned char *split;  // the level's inputs split into scaled FP16 parts
    int shift;                   // level - 2 (source partition test)
};

struct TcArgs {
    const TcLevel *lv;          // device array indexed by level
    int lmin, nent;             // entries e = (level - lmin) * 8 + class
    int tile_begin[kMaxLevels * 8 + 1];
    int K, ldk, B, Npad, nck, nst;
    int le_f64;                 // the output rows are FP64 (an FP64 plan's local expansions)
    const unsigned char *img;   // operator images, one [hi|lo] tile pair per (slot, chunk)
    const float *cs;            // column scales of the image ([Npad] scale, [Npad] inverse)
    int *status;
    long wait_tries;            // bound of every barrier wait (kWaitTries)
    uint32_t part_lo, part_hi;  // forward: source partition (in_source_part)
    // forward with msplit = 2: each tile's active offsets are shared by two
    // CTAs (blockIdx 2 t and 2 t + 1); each writes its partial rows to mpart
    // (slot = blockIdx, [128][Npad]) and counts itself in mcnt ([tile][8]
    // promoter warps, zero at launch); the second to arrive adds the other's
    // rows to its own and writes the tile.
    int msplit;
    float *mpart;
    int *mcnt;
    int test_stall;             // testing aid: the MMA issuer first waits on a barrier that
                                // nothing completes, so the bounded-wait failure path runs
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a K-major operand with the 64-byte
// swizzle (8-row atoms of 512 bytes).
__device__ __forceinline__ uint64_t umma_desc64(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;             // leading byte offset (unused, swizzled K-major)
    d |= (uint64_t)(512 >> 4) << 32;    // stride byte offset: one 8-row atom
    d |= (uint64_t)1 << 46;             // descriptor version
    d |= (uint64_t)4 << 61;             // 64-byte swizzle
    return d;
}

__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    // D = FP32, A = B = FP16 (format 0), both K-major
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Power-of-two scale sig = 2^sh that brings the largest |input| m of an
// M2L level into (2^14, 2^15] (the top of the FP16 range, far from its
// subnormals), from the bits of m: ceil(log2 m) = E + (mantissa != 0) for
// m = 1.mantissa * 2^E.  sh is clamped to [-126, 126]; m = 0 gives 1.
__device__ __forceinline__ void input_scale(uint32_t mbits, float &sig, float &inv) {
    int sh = 0;
    if (mbits != 0u) {
        const int eb = (int)(mbits >> 23);   // biased exponent (0: subnormal)
        const int cl = (eb == 0 ? -126 : eb - 127) + ((mbits & 0x7FFFFFu) != 0u ? 1 : 0);
        sh = min(126, max(-126, 15 - cl));
    }
    sig = __int_as_float((127 + sh) << 23);
    inv = __int_as_float((127 - sh) << 23);
}

// Input chunk that an offset processes at step j of its nck steps: the
// highest chunk first (see the MMA issue order).
__host__ __device__ __forceinline__ int chunk_of(int nck, int j) { return nck - 1 - j; }

constexpr long kWaitTries = 1l << 24;
constexpr long kTestWaitTries = 1l << 12;   // wait bound under GF_FLAG_TEST_WAIT_TIMEOUT

__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(addr), "r"(parity)
                 : "memory");
    return ok != 0;
}

// Bounded wait on phase `parity` of an mbarrier that also gives up when
// another role has set the abort flag; a timeout sets the flag.
__device__ __forceinline__ bool mbar_wait_ab(uint32_t addr, uint32_t parity, volatile int *abort_flag,
                                             long tries) {
    for (long it = 0; it < tries; ++it) {
        if (mbar_try(addr, parity)) return true;
        if ((it & 255) == 255 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

// Bounded wait that ignores the abort flag (used to drain in-flight work).
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, long tries) {
    for (long it = 0; it < tries; ++it)
        if (mbar_try(addr, parity)) return true;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t addr) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void commit_to(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// Read 8 accumulator columns starting at address ta (this warp's 32 lanes).
__device__ __forceinline__ void tmem_ld8(uint32_t ta, float *v) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ta));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

constexpr int kTcWarps = 14;
constexpr int kTcThreads = kTcWarps * 32;
constexpr int kTcMaxStages = 8;
constexpr uint32_t kTcCols = 512;           // two banks of 256 columns
constexpr uint32_t kTcA = 2u * 8192u;       // A hi + lo: 128 rows x 64 bytes each

constexpr int kTcChunks = 2;                // 32-input chunks per pipeline stage (12 MMAs per barrier wait)

__host__ __device__ constexpr uint32_t tc_stage_bytes(int Npad) { return kTcA + 2u * (uint32_t)Npad * 64u; }
constexpr size_t kTcSmemBudget = 227 * 1024 - 2048;
inline int tc_stages(int Npad) {
    const int n = (int)(kTcSmemBudget / ((size_t)kTcChunks * tc_stage_bytes(Npad)));
    return n > kTcMaxStages ? kTcMaxStages : n;
}
size_t tc_smem_bytes(int Npad) { return (size_t)tc_stages(Npad) * kTcChunks * tc_stage_bytes(Npad) + 1024; }

// 16-byte asynchronous global -> shared copy; nbytes = 0 fills zeros.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t nbytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(nbytes) : "memory");
}

// NS >= Npad / 2: FP32 sums held per promoter thread.
template <int NS>
__global__ void __launch_bounds__(kTcThreads, 1)
m2l_tc(TcArgs a) {
    extern __shared__ unsigned char dsm[];
    unsigned char *base = dsm + ((1024 - (smem_u32(dsm) & 1023)) & 1023);
    // afull: the stage's A operand has landed (128 producer arrivals); bfull:
    // its operator image has landed (the copy's own transaction count, so the
    // copying thread can always wait for its copies, whatever the producers do)
    __shared__ __align__(8) uint64_t afull[kTcMaxStages], bfull[kTcMaxStages], empty[kTcMaxStages];
    __shared__ __align__(8) uint64_t stall_bar;
    __shared__ __align__(8) uint64_t bank_full[2], bank_empty[2];
    __shared__ uint32_t tslot;
    __shared__ int abort_flag;
    __shared__ uint32_t omask[6];   // M2L: offsets with at least one source box in this tile
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int B = a.B, Npad = a.Npad, nck = a.nck, NST = a.nst;
    const int nsum = Npad / 2;
    const uint32_t b_bytes = 2u * (uint32_t)Npad * 64u;
    constexpr int S = kTcChunks;
    const uint32_t stage_bytes = S * tc_stage_bytes(Npad);   // [A: S x (hi, lo)][B: S x (hi, lo)]
    volatile int *abortp = &abort_flag;
    const int nbox = 128 / B;
    constexpr int noff = 189;
    const int msplit = max(1, a.msplit);
    const int utile = (int)blockIdx.x / msplit, uhalf = (int)blockIdx.x - utile * msplit;   // tile, share
    struct Ctx {
        const TcLevel *L;
        int cls, tile;
        int64_t cbeg, ccnt;
    };
    // (level, class, tile within the class) of tile t
    auto ctx_of = [&](int t) -> Ctx {
        int e = 0;
        while (e + 1 < a.nent && a.tile_begin[e + 1] <= t) ++e;
        Ctx c;
        c.L = &a.lv[a.lmin + e / 8];
        c.cls = e % 8;
        c.tile = t - a.tile_begin[e];
        c.cbeg = c.L->cls_off[c.cls];
        c.ccnt = c.L->cls_off[c.cls + 1] - c.cbeg;
        return c;
    };

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)),
                     "r"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            // 128 producer threads; the operator copy's expect-tx arrival
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&afull[i])), "r"(128));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bfull[i])), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty[i])), "r"(1));
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bank_full[i])), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bank_empty[i])), "r"(8));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&stall_bar)), "r"(1));
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (tid < 6) omask[tid] = 0;

    // producer role: column `row` of the tile
    const int row = tid & 127;
    const int slot = row / B, bb = row - slot * B;
    const Ctx pc = ctx_of(utile);
    int64_t tbox = -1, tc0 = 0, tc1 = 0, tc2 = 0;
    int64_t qbn0 = 0, qbn1 = 0, qbn2 = 0;   // the level's source block extent, kept in registers
    int qadj = 0;
    auto set_target = [&]() {
        tbox = -1;
        tc0 = tc1 = tc2 = 0;
        const TcLevel &L = *pc.L;
        qbn0 = L.bn[0];
        qbn1 = L.bn[1];
        qbn2 = L.bn[2];
        qadj = L.adj;
        const int64_t sidx = (int64_t)pc.tile * nbox + slot;
        if (warp >= 4 || slot >= nbox || sidx >= pc.ccnt) return;
        if (!L.adj) {
            tbox = L.order[pc.cbeg + sidx];
            const uint64_t key = L.tkey[tbox];
            tc0 = dm(key, 0) - L.blo[0];
            tc1 = dm(key, 1) - L.blo[1];
            tc2 = dm(key, 2) - L.blo[2];
        } else {
            class_box(pc.cls, L.blo, L.bn, sidx, tc0, tc1, tc2);
            tbox = (tc2 * L.bn[1] + tc1) * L.bn[0] + tc0;
        }
    };
    set_target();
    // input row of this column at offset oi of the current tile (-1: none)
    auto src_row = [&](int oi) -> int64_t {
        if (tbox < 0) return -1;
        const TcLevel &L = *pc.L;
        const int cls = pc.cls;
        const int64_t sx = tc0 + c_il[cls][oi][0], sy = tc1 + c_il[cls][oi][1], sz = tc2 + c_il[cls][oi][2];
        if (!qadj) {
            if (sx >= 0 && sy >= 0 && sz >= 0 && sx < qbn0 && sy < qbn1 && sz < qbn2 &&
                in_source_part(sx + L.blo[0], sy + L.blo[1], sz + L.blo[2], L.shift, a.part_lo, a.part_hi))
                return (((sz * qbn1 + sy) * qbn0 + sx) * B + bb) * a.ldk;
            return -1;
        }
        const int64_t wx = sx + L.blo[0] - L.mlo[0], wy = sy + L.blo[1] - L.mlo[1], wz = sz + L.blo[2] - L.mlo[2];
        if (wx >= 0 && wy >= 0 && wz >= 0 && wx < L.mn[0] && wy < L.mn[1] && wz < L.mn[2]) {
            const int32_t m = L.imap[(wz * L.mn[1] + wy) * L.mn[0] + wx];
            if (m >= 0) return ((int64_t)m * B + bb) * a.ldk;
        }
        return -1;
    };
    __syncthreads();
    if (warp < 4) {
        for (int w = 0; w * 32 < noff; ++w) {
            uint32_t bits = 0;
            for (int b = 0; b < 32 && 32 * w + b < noff; ++b)
                if (src_row(32 * w + b) >= 0) bits |= 1u << b;
            bits = __reduce_or_sync(0xffffffffu, bits);
            if (lane == 0 && bits) atomicOr(&omask[w], bits);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (msplit > 1) {
        // keep this CTA's share of the tile's active offsets: ranks
        // [uhalf tot / msplit, (uhalf + 1) tot / msplit) in offset order
        if (tid == 0) {
            int tot = 0;
            for (int w = 0; w < 6; ++w) tot += __popc(omask[w]);
            const int lo = uhalf * tot / msplit, hi = (uhalf + 1) * tot / msplit;
            int rank = 0;
            for (int w = 0; w < 6; ++w) {
                uint32_t m = omask[w], keep = 0;
                while (m) {
                    const int b = __ffs(m) - 1;
                    m &= m - 1;
                    if (rank >= lo && rank < hi) keep |= 1u << b;
                    ++rank;
                }
                omask[w] = keep;
            }
        }
        __syncthreads();
    }
    const uint32_t tmem = tslot;
    int G = 0;   // offsets run by this CTA
    for (int w = 0; w < 6; ++w) G += __popc(omask[w]);
    const int nsp = (nck + S - 1) / S;   // stages per offset
    const int iters = G * nsp;       // stages run by this CTA
    // the next offset to run after oi within a tile (noff when none is left)
    auto next_off = [&](int oi) -> int {
        for (++oi; oi < noff; ++oi)
            if (omask[oi >> 5] & (1u << (oi & 31))) return oi;
        return noff;
    };

    if (warp < 4) {
        // ---------------- A producers
        int qo = next_off(-1), qc = 0;
        int64_t qs = qo < noff ? src_row(qo) : -1;
        auto take = [&](int &c_out, int64_t &s_out) {   // next chunk in sequence
            c_out = qc;
            s_out = qs;
            if (++qc == nck) {
                qc = 0;
                qo = next_off(qo);
                qs = qo < noff ? src_row(qo) : -1;
            }
        };
        // FP16 inputs, scaled and split in advance: once a stage is free,
        // each thread copies its row's 64-byte high and low pieces of the
        // stage's chunks straight into it (16-byte asynchronous copies to
        // the swizzled positions; a missing source copies zeros), waits for
        // them and signals the stage.  The copies overlap the MMAs of the
        // previous stage.
        const unsigned char *spl = pc.L->split;   // every tile of a launch reads the same levels
        int s = 0;
        uint32_t ph = 0;
        for (int it = 0; it < iters; ++it) {
            if (it >= NST && !mbar_wait_ab(smem_u32(&empty[s]), ph ^ 1, abortp, a.wait_tries)) break;
            unsigned char *stage = base + (size_t)s * stage_bytes;
            int c0 = 0, nc = S;
#pragma unroll
            for (int q = 0; q < S; ++q) {
                if (q > 0 && c0 + q >= nck) break;   // the offset's last stage may hold fewer chunks
                int cc;
                int64_t sr;
                take(cc, sr);
                if (q == 0) {
                    c0 = cc;
                    nc = min(S, nck - c0);
                }
                // chunks run from the highest inputs down (chunk_of), and the
                // stage keeps its chunks in ascending order
                const int pc = chunk_of(nck, cc);
                // the warp's 32 rows in 8 passes of 4: eight lanes copy one
                // row's 128 contiguous bytes (pieces 0-3 high, 4-7 low)
                const uint32_t sub = smem_u32(stage + (nc - 1 - q) * kTcA);
                const int k = lane & 7;
                const uint32_t kpart = k < 4 ? 0u : 8192u;
                const int kk = 8 * (k & 3);
#pragma unroll
                for (int pp = 0; pp < 8; ++pp) {
                    const int rl = 4 * pp + (lane >> 3);
                    const int64_t srp = __shfl_sync(0xffffffffu, (long long)sr, rl);
                    const int r = (row & ~31) + rl;
                    const unsigned char *src = srp >= 0 ? spl + (size_t)srp * 4 + (size_t)pc * 128 + 16 * k : spl;
                    cp_async16(sub + kpart + swz64h(r, kk), src, srp >= 0 ? 16u : 0u);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(smem_u32(&afull[s]));
            if (++s == NST) {
                s = 0;
                ph ^= 1;
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");   // no copy outlives the loop (abort)
    } else if (warp == 4) {
        // ---------------- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_f16(128, Npad);
            int s = 0, c0 = 0, g = 0;
            uint32_t ph = 0;
            int last = -1;
            // testing aid: a wait that nothing completes runs out, sets the abort
            // flag, and every role stops, drains and reports through status[1]
            const bool stalled = a.test_stall && !mbar_wait_ab(smem_u32(&stall_bar), 0, abortp, a.wait_tries);
            for (int it = 0; it < (stalled ? 0 : iters); ++it) {
                if (!mbar_wait_ab(smem_u32(&afull[s]), ph, abortp, a.wait_tries)) break;
                if (!mbar_wait_ab(smem_u32(&bfull[s]), ph, abortp, a.wait_tries)) break;
                if (c0 == 0 && g >= 2 &&
                    !mbar_wait_ab(smem_u32(&bank_empty[g & 1]), ((g - 2) >> 1) & 1, abortp, a.wait_tries))
                    break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const unsigned char *stage = base + (size_t)s * stage_bytes;
                const uint32_t d = tmem + (uint32_t)(g & 1) * 256u;
                const int nc = min(S, nck - c0);
                // Inputs in descending order: the stage's chunks from the last
                // slot down, each chunk's k-steps from the last down, and in each
                // k-step the two small cross products before the main one.  The
                // accumulator adds of the tensor cores truncate, so every add made
                // once the sum has its full size costs up to an ulp of it, all of
                // the same sign; leading with the small high-order terms leaves
                // only the last few adds at full size.
                for (int q = 0; q < nc; ++q) {
                    const int sl = nc - 1 - q;
                    const int c = chunk_of(nck, c0 + nc - 1) + sl;   // the input chunk in slot sl
                    const uint32_t sa = smem_u32(stage + sl * kTcA);
                    const uint32_t sb = smem_u32(stage + S * kTcA + sl * b_bytes);
                    // k-steps of 32 bytes (16 inputs) holding inputs
                    const int nks = min(2, (a.K - 32 * c + 15) / 16);
                    for (int ks = nks - 1; ks >= 0; --ks) {
                        const uint32_t ko = ks * 32;
                        const uint64_t ah = umma_desc64(sa + ko), al = umma_desc64(sa + 8192 + ko);
                        const uint64_t bh = umma_desc64(sb + ko), bl = umma_desc64(sb + (uint32_t)Npad * 64 + ko);
                        const uint32_t acc = (c0 > 0 || q > 0 || ks < nks - 1) ? 1u : 0u;
                        mma_f16(d, ah, bl, idesc, acc);
                        mma_f16(d, al, bh, idesc, 1u);
                        mma_f16(d, ah, bh, idesc, 1u);
                    }
                }
                commit_to(&empty[s]);
                last = it;
                c0 += S;
                if (c0 >= nck) {
                    commit_to(&bank_full[g & 1]);
                    c0 = 0;
                    ++g;
                }
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
            // drain: the last commit covers every MMA issued
            if (last >= 0) mbar_wait(smem_u32(&empty[last % NST]), (uint32_t)((last / NST) & 1), a.wait_tries);
        }
    } else if (warp == 5) {
        // ---------------- operator images
        if (lane == 0) {
            int s = 0, c0 = 0;
            int oi = next_off(-1);
            const int bcls = pc.cls;
            uint32_t ph = 0;
            int last = -1;
            for (int it = 0; it < iters; ++it) {
                if (it >= NST && !mbar_wait_ab(smem_u32(&empty[s]), ph ^ 1, abortp, a.wait_tries)) break;
                const int dx = c_il[bcls][oi][0], dy = c_il[bcls][oi][1], dz = c_il[bcls][oi][2];
                const int slot_off = (dz + 3) * 49 + (dy + 3) * 7 + (dx + 3);
                unsigned char *stage = base + (size_t)s * stage_bytes;
                // the stage's chunks of the operator image are contiguous
                // (ascending, the lowest being that of the stage's last chunk)
                const int ncs = min(S, nck - c0);
                const uint32_t nbytes = (uint32_t)ncs * b_bytes;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&bfull[s])),
                             "r"(nbytes));
                const unsigned char *srcimg = a.img + ((size_t)slot_off * nck + chunk_of(nck, c0 + ncs - 1)) * b_bytes;
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        smem_u32(stage + S * kTcA)),
                    "l"(srcimg), "r"(nbytes), "r"(smem_u32(&bfull[s]))
                    : "memory");
                last = it;
                c0 += S;
                if (c0 >= nck) {
                    c0 = 0;
                    oi = next_off(oi);
                }
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
            // drain: every copy issued must have landed before the CTA exits;
            // the last NST stages may still have copies in flight (earlier ones
            // were consumed by MMAs before their stage was reused), and each
            // stage's copy completes its own barrier
            for (int j = last - NST + 1 > 0 ? last - NST + 1 : 0; j <= last; ++j)
                mbar_wait(smem_u32(&bfull[j % NST]), (uint32_t)((j / NST) & 1), a.wait_tries);
        }
    }
    // ---------------- promoters (warps 6-13) and the write-back of each tile
    const int pw = warp - 6;
    const int pq = warp & 3, ph_half = pw >> 2;   // TMEM lane quarter, column half
    bool ok = true;
    if (pw >= 0) {
        float acc[NS];
#pragma unroll
        for (int q = 0; q < NS; ++q) acc[q] = 0.f;
        for (int g = 0; g < G; ++g) {
            bool w_ok = mbar_wait_ab(smem_u32(&bank_full[g & 1]), (g >> 1) & 1, abortp, a.wait_tries);
            w_ok = __all_sync(0xffffffffu, w_ok);   // tcgen05.ld is warp-collective
            if (!w_ok) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t tb =
                tmem + ((uint32_t)(pq * 32) << 16) + (uint32_t)(g & 1) * 256u + (uint32_t)(ph_half * nsum);
#pragma unroll
            for (int j0 = 0; j0 < NS; j0 += 8) {
                if (j0 < nsum) {
                    float t[8];
                    tmem_ld8(tb + j0, t);
#pragma unroll
                    for (int q = 0; q < 8; ++q) acc[j0 + q] += t[q];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bank_empty[g & 1]));
        }
        if (*abortp) ok = false;
        if (ok) {
            // write this tile's rows
            const TcLevel &L = *pc.L;
            const int r = pq * 32 + lane;
            const int oslot = r / B, obb = r - oslot * B;
            const int64_t os = (int64_t)pc.tile * nbox + oslot;
            bool write = true;
            {
                // undo the column scales of the image and the input scale
                float sig, sig_inv;
                input_scale(*L.amax, sig, sig_inv);
                const float4 *ci = reinterpret_cast<const float4 *>(a.cs + Npad + ph_half * nsum);
#pragma unroll
                for (int q = 0; q < NS; q += 4)
                    if (q < nsum) {
                        const float4 c4 = __ldg(ci + q / 4);
                        acc[q] = acc[q] * c4.x * sig_inv;
                        acc[q + 1] = acc[q + 1] * c4.y * sig_inv;
                        acc[q + 2] = acc[q + 2] * c4.z * sig_inv;
                        acc[q + 3] = acc[q + 3] * c4.w * sig_inv;
                    }
            }
            if (msplit > 1) {
                // this warp's slice of the tile (32 rows, half the columns):
                // partial rows out, then the second CTA to arrive adds the
                // other's rows (a + b = b + a, so the sum does not depend on
                // which CTA is second) and writes the tile
                float4 *mine =
                    reinterpret_cast<float4 *>(a.mpart + ((size_t)blockIdx.x * 128 + r) * Npad + ph_half * nsum);
#pragma unroll
                for (int q = 0; q < NS; q += 4)
                    if (q < nsum) mine[q / 4] = make_float4(acc[q], acc[q + 1], acc[q + 2], acc[q + 3]);
                __threadfence();
                __syncwarp();
                int second = 0;
                if (lane == 0) second = atomicAdd(a.mcnt + (size_t)utile * 8 + pw, 1) == msplit - 1;
                second = __shfl_sync(0xffffffffu, second, 0);
                write = second != 0;
                if (write) {
                    __threadfence();
                    const float4 *other = reinterpret_cast<const float4 *>(
                        a.mpart + ((size_t)(utile * msplit + (1 - uhalf)) * 128 + r) * Npad + ph_half * nsum);
#pragma unroll
                    for (int q = 0; q < NS; q += 4)
                        if (q < nsum) {
                            const float4 o4 = __ldcg(other + q / 4);
                            acc[q] += o4.x;
                            acc[q + 1] += o4.y;
                            acc[q + 2] += o4.z;
                            acc[q + 3] += o4.w;
                        }
                }
            }
            if (write && oslot < nbox && os < pc.ccnt) {
                int64_t obox;
                if (!L.adj) {
                    obox = L.order[pc.cbeg + os];
                } else {
                    int64_t ox, oy, oz;
                    class_box(pc.cls, L.blo, L.bn, os, ox, oy, oz);
                    obox = L.slab0 + (oz * L.bn[1] + oy) * L.bn[0] + ox;
                }
                // 16-byte stores of the whole half row: columns from K up to
                // Npad hold zeros (the operator images are zero there) and stay
                // inside the row's padding (Npad <= ldk)
                float4 *dst = reinterpret_cast<float4 *>(L.le + (obox * B + obb) * a.ldk + ph_half * nsum);
                if (a.le_f64) {
                    // an FP64 plan's local expansions: rows of ldk >= Npad doubles
                    double *dd = reinterpret_cast<double *>(L.le) + (obox * B + obb) * a.ldk + ph_half * nsum;
#pragma unroll
                    for (int q = 0; q < NS; q += 4)
                        if (q < nsum) {
                            dd[q] = (double)acc[q];
                            dd[q + 1] = (double)acc[q + 1];
                            dd[q + 2] = (double)acc[q + 2];
                            dd[q + 3] = (double)acc[q + 3];
                        }
                } else {
#pragma unroll
                    for (int q = 0; q < NS; q += 4)
                        if (q < nsum) dst[q / 4] = make_float4(acc[q], acc[q + 1], acc[q + 2], acc[q + 3]);
                }
            }
        }
    }
    const bool failed = __syncthreads_or(!ok || abort_flag);
    if (failed && tid == 0) atomicOr(a.status + 1, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols));
}

}  // namespace

// Bytes of the split FP16 inputs of levels 2..l-1 (the start of level l in
// the split buffer), for the plan's largest batch.
static size_t split_offset(const FmmPlan *F, int adj, int l) {
    size_t off = 0;
    for (int k = 2; k < l; ++k) off += (size_t)(adj ? F->lev[k].nt : F->lev[k].ns) * F->B * F->KS * sizeof(float);
    return off;
}

gf_status m2l_tc_prepare_adj(gf_plan_s *plan) {
    FmmPlan *F = plan->fmm;
    if (!F->mixed || !F->tab->m2l_tc) return GF_OK;
    GF_TRY(plan->arena.alloc((void **)&F->tc_split_adj, std::max<size_t>(16, split_offset(F, 1, F->L + 1))));
    for (int adj = 1; adj < 2; ++adj) {
        std::vector<TcLevel> h(F->L + 1);
        memset(h.data(), 0, h.size() * sizeof(TcLevel));
        for (int l = 2; l <= F->L; ++l) {
            const FmmLevel &lv = F->lev[l];
            TcLevel &t = h[l];
            t.le = (float *)(adj ? lv.me : lv.le);
            t.order = lv.m2l_order;
            t.tkey = lv.tkey;
            t.adj = adj;
            t.imap = F->imap[l];
            for (int d = 0; d < 3; ++d) {
                t.blo[d] = lv.slo[d];
                t.bn[d] = lv.sn[d];
                t.mlo[d] = F->mlo[l][d];
                t.mn[d] = F->mn[l][d];
            }
            if (adj) {   // output: the z-slabs an interaction list reaches
                t.blo[2] += lv.m2l_z0;
                t.bn[2] = std::max<int64_t>(0, lv.m2l_z1 - lv.m2l_z0 + 1);
                t.slab0 = lv.m2l_z0 * lv.sn[0] * lv.sn[1];
            }
            for (int c = 0; c <= 8; ++c) t.cls_off[c] = adj ? F->scls_off[l][c] : lv.cls_off[c];
            t.amax = F->tc_amax + (adj ? kMaxLevels + 1 : 0) + l;
            t.split = (adj ? F->tc_split_adj : F->tc_split) + split_offset(F, adj, l);
            t.shift = l - 2;
        }
        std::vector<unsigned char> &hb = adj ? F->tc_levels_adj_host : F->tc_levels_host;
        void *&dev = adj ? F->tc_levels_adj : F->tc_levels;
        hb.assign(reinterpret_cast<unsigned char *>(h.data()), reinterpret_cast<unsigned char *>(h.data() + h.size()));
        GF_TRY(plan->arena.alloc(&dev, hb.size()));
        GF_TRY(upload_small(dev, hb.data(), hb.size(), plan->arena.stream));
    }
    return GF_OK;
}

gf_status m2l_tc_prepare(gf_plan_s *plan) {
    FmmPlan *F = plan->fmm;
    if (!(F->mixed || F->m2l_tc64) || !F->tab->m2l_tc) return GF_OK;
    GF_TRY(plan->arena.alloc((void **)&F->tc_amax, 2 * (kMaxLevels + 1) * sizeof(uint32_t)));
    GF_TRY(plan->arena.alloc((void **)&F->tc_split, std::max<size_t>(16, split_offset(F, 0, F->L + 1))));
    {
        // partial rows of the forward M2L's tiles when two CTAs share each
        // (tiles counted for the plan's largest batch: the most tiles)
        const int nbox = 128 / std::max(1, std::min(F->B, 128));
        int64_t tiles = 0;
        for (int l = 2; l <= F->L; ++l)
            for (int c = 0; c < 8; ++c) {
                const int64_t cnt = F->lev[l].nt > 0 ? F->lev[l].cls_off[c + 1] - F->lev[l].cls_off[c] : 0;
                tiles += (cnt + nbox - 1) / nbox;
            }
        if (tiles > 0 && 2 * tiles <= (int64_t)sm_count()) {
            GF_TRY(plan->arena.alloc((void **)&F->m2l_part, (size_t)tiles * 2 * 128 * F->tab->tc_npad * sizeof(float)));
            GF_TRY(plan->arena.alloc((void **)&F->m2l_cnt, (size_t)tiles * 8 * sizeof(int)));
            F->m2l_part_tiles = (int)tiles;
        }
    }
    for (int adj = 0; adj < 1; ++adj) {
        std::vector<TcLevel> h(F->L + 1);
        memset(h.data(), 0, h.size() * sizeof(TcLevel));
        for (int l = 2; l <= F->L; ++l) {
            const FmmLevel &lv = F->lev[l];
            TcLevel &t = h[l];
            t.le = (float *)(adj ? lv.me : lv.le);
            t.order = lv.m2l_order;
            t.tkey = lv.tkey;
            t.adj = adj;
            t.imap = F->imap[l];
            for (int d = 0; d < 3; ++d) {
                t.blo[d] = lv.slo[d];
                t.bn[d] = lv.sn[d];
                t.mlo[d] = F->mlo[l][d];
                t.mn[d] = F->mn[l][d];
            }
            if (adj) {   // output: the z-slabs an interaction list reaches
                t.blo[2] += lv.m2l_z0;
                t.bn[2] = std::max<int64_t>(0, lv.m2l_z1 - lv.m2l_z0 + 1);
                t.slab0 = lv.m2l_z0 * lv.sn[0] * lv.sn[1];
            }
            for (int c = 0; c <= 8; ++c) t.cls_off[c] = adj ? F->scls_off[l][c] : lv.cls_off[c];
            t.amax = F->tc_amax + (adj ? kMaxLevels + 1 : 0) + l;
            t.split = (adj ? F->tc_split_adj : F->tc_split) + split_offset(F, adj, l);
            t.shift = l - 2;
        }
        std::vector<unsigned char> &hb = adj ? F->tc_levels_adj_host : F->tc_levels_host;
        void *&dev = adj ? F->tc_levels_adj : F->tc_levels;
        hb.assign(reinterpret_cast<unsigned char *>(h.data()), reinterpret_cast<unsigned char *>(h.data() + h.size()));
        GF_TRY(plan->arena.alloc(&dev, hb.size()));
        GF_TRY(upload_small(dev, hb.data(), hb.size(), plan->arena.stream));
    }
    return GF_OK;
}

namespace {

// Largest |x| over the first kin components of every row of each level's
// M2L input (forward: ME_l; adjoint: the LE_l duals), as the bits of a
// non-negative float, combined with atomicMax (out[] zeroed before).
struct AmaxArgs {
    const float4 *in[kMaxLevels + 1];   // FP32 rows, or (f64) FP64 rows read through in64
    const double *in64[kMaxLevels + 1];
    int64_t rows[kMaxLevels + 1];
    uint32_t *out;
    int lmin, ld4, kin;
    int f64;                            // inputs are FP64 rows of 4 ld4 doubles
};

__global__ void __launch_bounds__(256) input_absmax(AmaxArgs a) {
    const int l = a.lmin + (int)blockIdx.y;
    if (a.f64) {
        // FP64 rows: element by element
        const double *p = a.in64[l];
        const int ld = 4 * a.ld4;
        const int64_t n = a.rows[l] * ld;
        float m = 0.f;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
            if ((int)(i % ld) < a.kin) m = fmaxf(m, fabsf((float)__ldg(p + i)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(a.out + l, __float_as_uint(m));
        return;
    }
    const float4 *p = a.in[l];
    const int64_t n = a.rows[l] * a.ld4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    float m = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            v[u] = i + u * stride < n ? __ldg(p + i + u * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = (int)((i + u * stride) % a.ld4) * 4;
            if (c < a.kin) m = fmaxf(m, fabsf(v[u].x));
            if (c + 1 < a.kin) m = fmaxf(m, fabsf(v[u].y));
            if (c + 2 < a.kin) m = fmaxf(m, fabsf(v[u].z));
            if (c + 3 < a.kin) m = fmaxf(m, fabsf(v[u].w));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(a.out + l, __float_as_uint(m));
}

// Split every M2L input row into the FP16 operand parts the tensor-core
// M2L copies: x s = hi + lo + O(2^-22 |x s|), s = the level's input scale;
// per row and 32-wide chunk, 64 bytes of hi then 64 bytes of lo (inputs
// beyond kin are zero).
struct SplitArgs {
    unsigned char *out[kMaxLevels + 1];
};

__global__ void __launch_bounds__(256) input_split(AmaxArgs a, SplitArgs o, int nck) {
    const int l = a.lmin + (int)blockIdx.y;
    float sig, sig_inv;
    input_scale(a.out[l], sig, sig_inv);
    const int64_t items = a.rows[l] * nck;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / nck;
        const int c = (int)(i - r * nck);
        float4 v[8];
        if (a.f64) {
            // FP64 rows (4 ld4 doubles): 32 inputs rounded to FP32 (the parts carry 22 bits)
            const double2 *s2 = reinterpret_cast<const double2 *>(a.in64[l] + r * 4 * a.ld4 + 32 * c);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const double2 d0 = __ldg(s2 + 2 * q), d1 = __ldg(s2 + 2 * q + 1);
                v[q] = make_float4((float)d0.x, (float)d0.y, (float)d1.x, (float)d1.y);
            }
        } else {
            const float4 *src = a.in[l] + r * a.ld4 + 8 * c;
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __ldg(src + q);
        }
        uint4 *dst = reinterpret_cast<uint4 *>(o.out[l] + (size_t)i * 128);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float x8[8] = {v[2 * q].x,     v[2 * q].y,     v[2 * q].z,     v[2 * q].w,
                                 v[2 * q + 1].x, v[2 * q + 1].y, v[2 * q + 1].z, v[2 * q + 1].w};
            uint32_t h[4], lo[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int kin = 32 * c + 8 * q + 2 * j;
                const float x0 = kin < a.kin ? x8[2 * j] * sig : 0.f;
                const float x1 = kin + 1 < a.kin ? x8[2 * j + 1] * sig : 0.f;
                const __half2 hh = __floats2half2_rn(x0, x1);
                const float2 hf = __half22float2(hh);
                const __half2 ll = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
                memcpy(&h[j], &hh, 4);
                memcpy(&lo[j], &ll, 4);
            }
            dst[q] = make_uint4(h[0], h[1], h[2], h[3]);
            dst[4 + q] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
}

gf_status tc_launch(TcArgs &a, int tiles, cudaStream_t st) {
    if (tiles == 0) return GF_OK;
    const int grid = tiles * std::max(1, a.msplit);
    const size_t shm = tc_smem_bytes(a.Npad);
    a.nst = tc_stages(a.Npad);
    const int nsum = a.Npad / 2;
#define GF_TC_LAUNCH(NS)                                        \
    do {                                                        \
        GF_TRY((ensure_smem(m2l_tc<NS>, shm)));                 \
        m2l_tc<NS><<<grid, kTcThreads, shm, st>>>(a);           \
    } while (0)
    if (nsum <= 32)
        GF_TC_LAUNCH(32);
    else if (nsum <= 64)
        GF_TC_LAUNCH(64);
    else if (nsum <= 96)
        GF_TC_LAUNCH(96);
    else
        GF_TC_LAUNCH(128);
#undef GF_TC_LAUNCH
    GF_KERNEL_DONE();
    return GF_OK;
}

gf_status m2l_run_tc(gf_plan_s *plan, int B, bool adj, cudaStream_t st, cudaEvent_t fork) {
    FmmPlan *F = plan->fmm;
    const Tables *T = F->tab;
    TcArgs a;
    memset(&a, 0, sizeof(a));
    a.K = F->K;
    a.ldk = F->KS;
    a.B = B;
    a.Npad = T->tc_npad;
    a.nck = T->tc_nck_h;
    a.status = plan->d_status;
    a.wait_tries = kWaitTries;
    a.msplit = 1;
    a.lv = reinterpret_cast<const TcLevel *>(adj ? F->tc_levels_adj : F->tc_levels);
    a.lmin = 2;
    a.img = (const unsigned char *)(adj ? T->am2l_tc : T->m2l_tc);
    a.cs = adj ? T->am2l_cs : T->m2l_cs;
    a.le_f64 = F->m2l_tc64 ? 1 : 0;
    a.part_lo = adj ? 0u : plan->part_lo;
    a.part_hi = adj ? 64u : plan->part_hi;
    if (plan->opt.reserved0 & GF_FLAG_TEST_WAIT_TIMEOUT) {
        a.test_stall = 1;
        a.wait_tries = kTestWaitTries;
    }
    if (F->L < 2) return GF_OK;
    // the largest |input| of every level, for the FP16 input scales
    {
        AmaxArgs m;
        memset(&m, 0, sizeof(m));
        m.out = F->tc_amax + (adj ? kMaxLevels + 1 : 0);
        m.lmin = 2;
        m.ld4 = F->KS / 4;
        m.kin = F->K;
        m.f64 = F->m2l_tc64 ? 1 : 0;
        int64_t most = 0;
        // forward: only the z-slabs of each level's source block that an
        // interaction list reaches (rows run x fastest, then y, then z)
        int64_t row0[kMaxLevels + 1] = {};
        for (int l = 2; l <= F->L; ++l) {
            const FmmLevel &lv = F->lev[l];
            int64_t r0 = 0, nr = (adj ? lv.nt : lv.ns) * B;
            if (!adj) {
                const int64_t slab = lv.sn[0] * lv.sn[1] * B;
                r0 = lv.m2l_z1 >= lv.m2l_z0 ? lv.m2l_z0 * slab : 0;
                nr = lv.m2l_z1 >= lv.m2l_z0 ? (lv.m2l_z1 - lv.m2l_z0 + 1) * slab : 0;
            }
            row0[l] = r0;
            m.in[l] = (const float4 *)(adj ? lv.le : lv.me) + r0 * m.ld4;
            m.in64[l] = (const double *)(adj ? lv.le : lv.me) + r0 * 4 * m.ld4;
            m.rows[l] = nr;
            most = std::max(most, m.rows[l] * m.ld4);
        }
        const int gx = (int)std::min<int64_t>(8 * 152, std::max<int64_t>(1, (most + 1023) / 1024));
        if (adj || !F->amax_fused) {   // else the kernels that wrote the expansions took it
            GF_CUDA(cudaMemsetAsync(m.out, 0, (kMaxLevels + 1) * sizeof(uint32_t), st));
            input_absmax<<<dim3(gx, F->L - 1), 256, 0, st>>>(m);
            GF_KERNEL_DONE();
        }
        SplitArgs o;
        memset(&o, 0, sizeof(o));
        for (int l = 2; l <= F->L; ++l)
            o.out[l] = (adj ? F->tc_split_adj : F->tc_split) + split_offset(F, adj, l) + (size_t)row0[l] * F->KS * 4;
        input_split<<<dim3(gx, F->L - 1), 256, 0, st>>>(m, o, T->tc_nck_h);
        GF_KERNEL_DONE();
    }
    if (!adj) stage_mark(plan, 4, st);
    const int nbox = 128 / B;
    int tiles = 0, e = 0;
    for (int l = 2; l <= F->L; ++l)
        for (int c = 0; c < 8; ++c, ++e) {
            a.tile_begin[e] = tiles;
            const int64_t *off = adj ? F->scls_off[l] : F->lev[l].cls_off;
            const int64_t cnt = (adj || F->lev[l].nt > 0) ? off[c + 1] - off[c] : 0;
            tiles += (int)((cnt + nbox - 1) / nbox);
        }
    a.tile_begin[e] = tiles;
    a.nent = e;
    // when two CTAs per tile still fit the SMs at once, every tile's offsets
    // are shared by two: each chain of offsets is half as long (and each
    // FP32 sum of offsets half as deep)
    if (!adj && F->m2l_part && tiles <= F->m2l_part_tiles && 2 * tiles <= sm_count()) {
        a.msplit = 2;
        a.mpart = F->m2l_part;
        a.mcnt = F->m2l_cnt;
        GF_CUDA(cudaMemsetAsync(F->m2l_cnt, 0, (size_t)tiles * 8 * sizeof(int), st));
    }
    if (fork) GF_CUDA(cudaEventRecord(fork, st));
    return tc_launch(a, tiles, st);
}

}  // namespace

template <class T, int P>
gf_status launch_m2l_fold(FoldM2LArgs &a, cudaStream_t st) {
    uint64_t blocks = 0;
    for (int l = a.lmin; l <= a.lmax; ++l) {
        a.lv[l].blk0 = (uint32_t)blocks;
        blocks += (a.lv[l].ncol + (uint64_t)P - 1) / P;
    }
    if (blocks == 0) return GF_OK;
    const size_t shm = sizeof(T) * (size_t)((a.K + 3) & ~3) * 8 * P;
    GF_TRY((ensure_smem(m2l_fold<T, P>, shm)));
    const int threads = (a.K * Lay<T, P>::NG + 31) & ~31;
    m2l_fold<T, P><<<(unsigned)blocks, threads, shm, st>>>(a);
    GF_KERNEL_DONE();
    return GF_OK;
}

// Every level of the M2L (adj: of its transpose) on the SIMT cores.
template <class T>
gf_status m2l_run_fold(gf_plan_s *plan, int B, bool adj, cudaStream_t st) {
    FmmPlan *F = plan->fmm;
    if (B > 32) {
        set_error("M2L supports at most 32 batch members");
        return GF_ERR_UNSUPPORTED;
    }
    FoldM2LArgs a;
    memset(&a, 0, sizeof(a));
    int64_t total = 0;
    for (int l = 2; l <= F->L; ++l) {
        const FmmLevel &lv = F->lev[l];
        FoldLevel &t = a.lv[l];
        t.in = adj ? lv.le : lv.me;
        t.out = adj ? lv.me : lv.le;
        t.tkey = lv.tkey;
        t.imap = F->imap[l];
        for (int d = 0; d < 3; ++d) {
            t.blo[d] = (int32_t)lv.slo[d];
            t.bn[d] = (int32_t)lv.sn[d];
            t.mlo[d] = (int32_t)F->mlo[l][d];
            t.mn[d] = (int32_t)F->mn[l][d];
        }
        int64_t ncol = lv.nt * B;
        if (adj) {   // the z-slabs an interaction list reaches
            const int64_t slab = lv.sn[0] * lv.sn[1];
            t.blo[2] += (int32_t)lv.m2l_z0;
            t.bn[2] = (int32_t)std::max<int64_t>(0, lv.m2l_z1 - lv.m2l_z0 + 1);
            t.out = (T *)lv.me + lv.m2l_z0 * slab * B * F->KS;
            ncol = t.bn[2] * slab * B;
        }
        t.ncol = (uint32_t)ncol;
        total += ncol;
    }
    if (total > (int64_t)0x7fffffff) {
        set_error("too many expansions for one launch (%lld)", (long long)total);
        return GF_ERR_UNSUPPORTED;
    }
    a.lmin = 2;
    a.lmax = F->L;
    a.K = F->K;
    a.ldk = F->KS;
    a.B = B;
    a.adj = adj ? 1 : 0;
    a.part_lo = adj ? 0u : plan->part_lo;
    a.part_hi = adj ? 64u : plan->part_hi;
    const Tables *Tb = F->tab;
    a.tab = sizeof(T) == 8 ? (const void *)(adj ? Tb->am2l_d : Tb->m2l_d) : (const void *)(adj ? Tb->am2l_f : Tb->m2l_f);
    // columns per block: more share a table element, fewer fill the SMs evenly
    const int64_t sms = sm_count();
    if constexpr (sizeof(T) == 8) {
        if (total >= 8 * sms && F->K <= 256) return launch_m2l_fold<T, 4>(a, st);   // at most 512 threads
        if (total >= sms) return launch_m2l_fold<T, 2>(a, st);
        return launch_m2l_fold<T, 1>(a, st);
    } else {
        if (total >= 16 * sms) return launch_m2l_fold<T, 8>(a, st);
        return launch_m2l_fold<T, 2>(a, st);
    }
}

template <class T>
gf_status m2l_run(gf_plan_s *plan, int B, bool adj, cudaStream_t st, cudaEvent_t fork) {
    FmmPlan *F = plan->fmm;
    const bool tc = (sizeof(T) == 4 || (F->m2l_tc64 && !adj)) && F->tab->m2l_tc && (adj ? F->tc_levels_adj : F->tc_levels) &&
                    !(plan->opt.reserved0 & GF_FLAG_M2L_SIMT) && B <= 128 &&
                    tc_stages(F->tab->tc_npad) >= 2;
    if (tc) return m2l_run_tc(plan, B, adj, st, fork);
    if (!adj) stage_mark(plan, 4, st);   // no input split on this path
    if (fork) GF_CUDA(cudaEventRecord(fork, st));
    return m2l_run_fold<T>(plan, B, adj, st);
}

template gf_status m2l_run<float>(gf_plan_s *, int, bool, cudaStream_t, cudaEvent_t);
template gf_status m2l_run<double>(gf_plan_s *, int, bool, cudaStream_t, cudaEvent_t);

}  // namespace gf
