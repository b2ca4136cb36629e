// gf_m2l.cu -- M2L over the interaction list, as a batched dense contraction:
// on the tensor cores (tiles of 128 columns of one parity class, offset by
// offset) from FP16 parts in mixed precision and from BF16 digits in FP64, or on
// the SIMT cores (columns folded by mirror symmetry): small FP64 plans, the FP64
// transpose, and where a plan asks for it.  Sources outside the source block
// contribute zeros.  Every sum is made in an order that the plan fixes, so the
// result is deterministic.
#include <cuda_fp16.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "gf_fold.cuh"
#include "gf_m2l.cuh"

namespace gf {

// Interaction-list offsets of each parity class, dx | dy | dz << 0 | 8 | 16
// as signed bytes.
__constant__ int c_il[8][189];
// Per class, axis and displacement d = -3 .. 3 along it: the offsets with that
// displacement, as bits of six words.
__constant__ uint32_t c_axis[8][3][7][6];

gf_status m2l_upload_offsets(const signed char h_il[8][189][3]) {
    int packed[8][189];
    static uint32_t axis[8][3][7][6];
    memset(axis, 0, sizeof(axis));
    for (int c = 0; c < 8; ++c)
        for (int i = 0; i < 189; ++i)
            for (int d = 0; d < 3; ++d) axis[c][d][h_il[c][i][d] + 3][i >> 5] |= 1u << (i & 31);
    GF_CUDA(cudaMemcpyToSymbol(c_axis, axis, sizeof(axis)));
    for (int c = 0; c < 8; ++c)
        for (int i = 0; i < 189; ++i)
            packed[c][i] = (uint8_t)h_il[c][i][0] | (uint8_t)h_il[c][i][1] << 8 | (uint8_t)h_il[c][i][2] << 16;
    GF_CUDA(cudaMemcpyToSymbol(c_il, packed, sizeof(packed)));
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

// Every third bit of a Morton key from bit s on, gathered.
__device__ __forceinline__ int64_t dm(uint64_t k, int s) {
    uint64_t x = (k >> s) & 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x001f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x001f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x00000000001fffffull;
    return (int64_t)x;
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
        // (a strided loop: the block of a small degree has fewer threads than entries)
        for (int e = tid; e < 8 * P; e += nthr) {
            // source at (s_x a, s_y b, s_z c), s = - where the bit of o is clear
            const int c = e >> 3, o = e & 7;
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
            crow[e] = row;
            any |= row >= 0;
        }
        if (!__syncthreads_or(any)) continue;
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
// come in chunks of 32, one to a stage.  Two pipelines take the units of the CTA in
// turn, each with a ring of shared-memory stages (64-byte swizzle), a tensor-memory
// bank and warps of its own:
//   warps 0-1, 2-3  A producers: 16-byte asynchronous copies straight into the
//               stage (eight lanes per row's 128 contiguous bytes); each
//               thread's arrival on the stage's barrier is made by its copies
//               as they land, so the producers run as far ahead as there are
//               free stages;
//   warps 4, 14 one thread issues the MMAs of a stage and commits them to the
//               stage's "empty" barrier (and, after an offset's last chunk,
//               to the bank's "full" barrier);
//   warps 5, 15 one thread bulk-copies the pre-split, pre-swizzled operator
//               image of each stage;
//   warps 6-13  promoters, of both: after each offset they read the finished bank
//               of tensor memory and add it into FP32 registers (the tensor
//               cores never accumulate more than one offset: their FP32
//               accumulation rounds differently from IEEE and long chains over
//               zero-mean data lose digits).
// Offsets whose source boxes are all missing are skipped by every role: the
// active offsets of every tile are found beforehand (tile_mask) as bit masks
// and counts.  Work is dealt out in units of one (tile, active offset): with up
// to kStreamTiles tiles the launch has at most one CTA per SM, and CTA c of G
// takes the units [c T / G, (c + 1) T / G) of the T in tile order, whatever tiles
// they fall in, so that no SM waits for the longest tile (the upper levels' lists
// are twice as long as a surface's leaf lists, and a few tiles more than SMs
// made a second wave).  The partial rows of a tile cut by that are summed in CTA
// order by a second launch (m2l_join), spread over the chip: one CTA's last
// arrival summing them took longer than the tile's units when a tile was shared
// by twenty CTAs.  With more tiles a CTA takes one whole tile.
// What bounds it: serial latencies.  169 components are 33 MMAs of 128 x 176 x 16
// an offset, 2,900 cycles of the tensor cores; an issuing thread waits out most of
// each MMA and spends as long again on barriers, fences and commits, and a stage's
// refill (wake-up, 16 copies a thread, L2) takes longer than another stage's MMAs.
// One pipeline took 5,800 cycles an offset; two, each hiding the other's, 5,000.
// Measured against one CTA, or two, per tile and producers that waited for their
// copies: the 8 tiles of a 32^3 grid under a plane of stations 260 -> 33 us + 6 us to
// join; the 156 of a 464^3 grid (K = 121) 327 -> 127 + 14; 16 grids of 128^3 846 -> 397; a 2^25-point
// set 1,050 -> 522; 128^3 with observers throughout 1,236 -> 1,011.  (A gather by TMA
// of the rows took 20 cycles a row, three times as long in all.)
// Every wait is bounded and watches an abort
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
    const unsigned char *split;  // the level's inputs split into scaled FP16 parts (FP64 slices: BF16 digits)
    const double *rscale;        // FP64 slices: the rows' scales
    int64_t src0;                // FP64 slices: first box of the source block that has split rows
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
    int ntiles;
    const uint32_t *tmask;      // [ntiles][8]: 189 offset bits, [6]: how many
    int stream;                 // units dealt out over the grid (else one tile per CTA)
    int min_units;              // a CTA takes no fewer units than this (stream)
    float *mpart;               // [gridDim][Npad / 4][prow] float4: partial rows of CTA c's first tile, when
                                // an earlier CTA starts it
    int prow;                   // rows of a tile that may hold a target, at most
    int4 *mcut;                 // [gridDim + 1] (stream): CTA c's first tile, the units before it and up to its
                                // end, G; [gridDim].x: T
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

constexpr int kTcWarps = 16;
constexpr int kTcThreads = kTcWarps * 32;
constexpr int kTcMaxStages = 4;             // of each of the two pipelines
constexpr uint32_t kTcCols = 512;           // two banks of 256 columns
constexpr uint32_t kTcA = 2u * 8192u;       // A hi + lo: 128 rows x 64 bytes each

__host__ __device__ constexpr uint32_t tc_stage_bytes(int Npad) { return kTcA + 2u * (uint32_t)Npad * 64u; }
constexpr int kScanItems = 3;               // tiles per thread of the unit scan
constexpr int kStreamTiles = kTcThreads * kScanItems;
constexpr size_t kTcSmemBudget = 227 * 1024 - 2048 - 4 * (kStreamTiles + 1);
inline int tc_stages(int Npad) {
    const int n = (int)(kTcSmemBudget / (size_t)tc_stage_bytes(Npad)) / 2;   // per pipeline
    return n > kTcMaxStages ? kTcMaxStages : n;
}
size_t tc_smem_bytes(int Npad) { return 2 * (size_t)tc_stages(Npad) * tc_stage_bytes(Npad) + 1024; }

// 16-byte asynchronous global -> shared copy; nbytes = 0 fills zeros.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t nbytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(nbytes) : "memory");
}

struct TcTile {
    const TcLevel *L;
    int cls, tile;        // tile within the class
    int64_t cbeg, ccnt;   // the class's targets
};

// (level, class, tile within the class) of tile t
__device__ __forceinline__ TcTile tile_of(const TcArgs &a, int t) {
    int e = 0, hi = a.nent;   // tile_begin[e] <= t < tile_begin[hi]
    while (hi - e > 1) {
        const int mid = (e + hi) >> 1;
        if (a.tile_begin[mid] <= t)
            e = mid;
        else
            hi = mid;
    }
    TcTile c;
    c.L = &a.lv[a.lmin + e / 8];
    c.cls = e % 8;
    c.tile = t - a.tile_begin[e];
    c.cbeg = c.L->cls_off[c.cls];
    c.ccnt = c.L->cls_off[c.cls + 1] - c.cbeg;
    return c;
}

// What locates the source rows of a target box at an offset, in registers:
// its position in the window of boxes that have rows (forward: the level's
// source block; adjoint: the target boxes' bounding box, through imap).
struct TcTarget {
    int x, y, z, n0, n1, n2;
    const int32_t *imap;
};

// Target of a tile's slot (a position no offset can reach if there is none).
__device__ __forceinline__ TcTarget target_of(const TcTile &t, int nbox, int slot) {
    const TcLevel &L = *t.L;
    TcTarget q;
    q.imap = L.imap;
    q.x = q.y = q.z = -1000;
    if (!L.adj) {
        q.imap = nullptr;
        q.n0 = (int)L.bn[0];
        q.n1 = (int)L.bn[1];
        q.n2 = (int)L.bn[2];
    } else {
        q.n0 = (int)L.mn[0];
        q.n1 = (int)L.mn[1];
        q.n2 = (int)L.mn[2];
    }
    const int64_t sidx = (int64_t)t.tile * nbox + slot;
    if (slot >= nbox || sidx >= t.ccnt) return q;
    if (!L.adj) {
        const uint64_t key = L.tkey[L.order[t.cbeg + sidx]];
        q.x = (int)(dm(key, 0) - L.blo[0]);
        q.y = (int)(dm(key, 1) - L.blo[1]);
        q.z = (int)(dm(key, 2) - L.blo[2]);
    } else {
        int64_t c0, c1, c2;
        class_box(t.cls, L.blo, L.bn, sidx, c0, c1, c2);
        q.x = (int)(c0 + L.blo[0] - L.mlo[0]);
        q.y = (int)(c1 + L.blo[1] - L.mlo[1]);
        q.z = (int)(c2 + L.blo[2] - L.mlo[2]);
    }
    return q;
}

// Index of the source box's rows at list offset oi of class cls (-1: none).
__device__ __forceinline__ int64_t source_of(const TcArgs &a, const TcLevel *L, const TcTarget &q, int cls, int oi) {
    const int o = c_il[cls][oi];
    const int sx = q.x + (signed char)o, sy = q.y + (signed char)(o >> 8), sz = q.z + (signed char)(o >> 16);
    if ((unsigned)sx >= (unsigned)q.n0 || (unsigned)sy >= (unsigned)q.n1 || (unsigned)sz >= (unsigned)q.n2) return -1;
    const int64_t i = ((int64_t)sz * q.n1 + sy) * q.n0 + sx;
    if (q.imap) return q.imap[i];
    if ((a.part_lo != 0 || a.part_hi < 64) &&
        !in_source_part(sx + L->blo[0], sy + L->blo[1], sz + L->blo[2], L->shift, a.part_lo, a.part_hi))
        return -1;
    return i;
}

// The active offsets of tile t (256 threads of one block): bit masks and their
// count, at least one (a tile without sources runs one offset of zeros).
__device__ __forceinline__ void tile_mask(const TcArgs &a, int t, uint32_t *tmask) {
    __shared__ uint32_t words[6];
    const TcTile tile = tile_of(a, t);
    const int row = threadIdx.x & 127, half = threadIdx.x >> 7;   // offset words 3 half .. 3 half + 2
    // the batch members of a box share its offsets
    const bool on = row % a.B == 0;
    const TcTarget q = target_of(tile, 128 / a.B, row / a.B);
    __syncthreads();
    if (threadIdx.x < 6) words[threadIdx.x] = 0;
    __syncthreads();
    // where every source inside the window counts: the offsets that stay inside it on
    // every axis, from the axes' own masks (63 constants a thread in place of 96
    // tests of an offset: the launch that ends with this 12.1 -> 4.9 us at 32^3)
    const bool whole = !q.imap && a.part_lo == 0 && a.part_hi >= 64;
    for (int w = 3 * half; w < 3 * half + 3; ++w) {
        uint32_t bits = 0;
        if (on && whole) {
            uint32_t in[3] = {0, 0, 0};
#pragma unroll
            for (int d = 0; d < 7; ++d) {
                if ((unsigned)(q.x + d - 3) < (unsigned)q.n0) in[0] |= c_axis[tile.cls][0][d][w];
                if ((unsigned)(q.y + d - 3) < (unsigned)q.n1) in[1] |= c_axis[tile.cls][1][d][w];
                if ((unsigned)(q.z + d - 3) < (unsigned)q.n2) in[2] |= c_axis[tile.cls][2][d][w];
            }
            bits = in[0] & in[1] & in[2];
        } else if (on)
            for (int b = 0; b < 32 && 32 * w + b < 189; ++b)
                if (source_of(a, tile.L, q, tile.cls, 32 * w + b) >= 0) bits |= 1u << b;
        bits = __reduce_or_sync(0xffffffffu, bits);
        if ((threadIdx.x & 31) == 0 && bits) atomicOr(&words[w], bits);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int n = 0;
        for (int w = 0; w < 6; ++w) n += __popc(words[w]);
        if (n == 0) words[0] = n = 1;
        for (int w = 0; w < 6; ++w) tmask[8 * (size_t)t + w] = words[w];
        tmask[8 * (size_t)t + 6] = (uint32_t)n;
    }
}

// The active offsets of a tile in order, from the one of rank `skip` on.
struct OffsetIter {
    const uint32_t *m;
    int w;
    uint32_t bits;
    __device__ __forceinline__ void open(const uint32_t *tmask, int t, int skip) {
        m = tmask + 8 * (size_t)t;
        w = 0;
        bits = __ldg(m);
        while (skip > 0) {
            const int n = __popc(bits);
            if (n <= skip) {
                skip -= n;
                bits = __ldg(m + ++w);
            } else {
                for (; skip > 0; --skip) bits &= bits - 1;
            }
        }
    }
    __device__ __forceinline__ int next() {
        while (!bits) bits = __ldg(m + ++w);
        const int b = __ffs(bits) - 1;
        bits &= bits - 1;
        return 32 * w + b;
    }
};

// Output row of row r of a tile (-1: none).
__device__ __forceinline__ int64_t out_row(const TcArgs &a, const TcTile &t, int nbox, int r) {
    const TcLevel &L = *t.L;
    const int slot = r / a.B, bb = r - slot * a.B;
    const int64_t sidx = (int64_t)t.tile * nbox + slot;
    if (slot >= nbox || sidx >= t.ccnt) return -1;
    if (!L.adj) return (int64_t)L.order[t.cbeg + sidx] * a.B + bb;
    int64_t x, y, z;
    class_box(t.cls, L.blo, L.bn, sidx, x, y, z);
    return (L.slab0 + (z * L.bn[1] + y) * L.bn[0] + x) * a.B + bb;
}

// Store four columns of an output row; columns from K up to Npad hold zeros
// (the operator images are zero there) and stay inside the row's padding
// (Npad <= ldk).
__device__ __forceinline__ void store4(const TcArgs &a, const TcLevel &L, int64_t row, int col, float4 v) {
    if (a.le_f64) {
        double2 *d = reinterpret_cast<double2 *>(reinterpret_cast<double *>(L.le) + row * a.ldk + col);
        d[0] = make_double2(v.x, v.y);
        d[1] = make_double2(v.z, v.w);
    } else {
        *reinterpret_cast<float4 *>(L.le + row * a.ldk + col) = v;
    }
}

__device__ __forceinline__ float4 read4(const TcArgs &a, const TcLevel &L, int64_t row, int col) {
    if (!a.le_f64) return *reinterpret_cast<const float4 *>(L.le + row * a.ldk + col);
    const double2 *d = reinterpret_cast<const double2 *>(reinterpret_cast<const double *>(L.le) + row * a.ldk + col);
    return make_float4((float)d[0].x, (float)d[0].y, (float)d[1].x, (float)d[1].y);   // FP32 values
}

// Tiles cut between CTAs: the first CTA's sums, in the output rows, plus the other
// CTAs' partial rows in CTA order.  Blocks (c - 1, .) look at the boundary before
// CTA c and, when it is the first one inside its tile, finish the tile's rows, the
// columns split over blockIdx.y.
// A chain of dependent loads with little behind it: kJoin partial rows are on their way
// before the first CTA's sum is asked for, and the blocks are small, to start beside
// those of the near field.  44^3 voxels under 256^2 stations, p = 8: 111.0 us a forward
// (that sum first, a column at a time, blocks of 512), now 108.6; 45 x 182 x 28, p = 13:
// 242.7, 237.4; 179^3, p = 10: 250.9, 246.4; 49^3 under 98^2 with their volume too,
// p = 12: 334.1, 324.3.
constexpr int kJoin = 4;
__global__ void __launch_bounds__(256) m2l_join(const __grid_constant__ TcArgs a) {
    const int c = (int)blockIdx.x + 1;
    const int4 cut = a.mcut[c];
    const uint32_t G = (uint32_t)cut.w, T = a.mcut[gridDim.x + 1].x;
    if (c >= (int)G) return;
    const uint32_t p0 = (uint32_t)cut.y, p1 = (uint32_t)cut.z;
    if ((uint32_t)((uint64_t)c * T / G) == p0) return;
    // CTAs holding the tile's first and last unit
    const int cf = (int)((((uint64_t)p0 + 1) * G - 1) / T), cl = (int)(((uint64_t)p1 * G - 1) / T);
    if (c != cf + 1) return;
    const int r = threadIdx.x & 127;
    const TcTile tile = tile_of(a, cut.x);
    const int64_t row = out_row(a, tile, 128 / a.B, r);
    if (row < 0) return;
    const size_t slot = (size_t)(a.Npad / 4) * a.prow;
    const float4 *p = reinterpret_cast<const float4 *>(a.mpart) + r;
    for (int q = 2 * (int)blockIdx.y + (threadIdx.x >> 7); q < a.Npad / 4; q += 2 * (int)gridDim.y) {
        float4 s;
        for (int e = cf + 1; e <= cl; e += kJoin) {
            float4 v[kJoin];
#pragma unroll
            for (int i = 0; i < kJoin; ++i)
                if (e + i <= cl) v[i] = __ldg(p + (e + i) * slot + (size_t)q * a.prow);
            if (e == cf + 1) s = read4(a, *tile.L, row, 4 * q);
#pragma unroll
            for (int i = 0; i < kJoin; ++i)
                if (e + i <= cl) {
                    s.x += v[i].x;
                    s.y += v[i].y;
                    s.z += v[i].z;
                    s.w += v[i].w;
                }
        }
        store4(a, *tile.L, row, 4 * q, s);
    }
}

// NS >= Npad / 2: FP32 sums held per promoter thread.
template <int NS>
__global__ void __launch_bounds__(kTcThreads, 1)
m2l_tc(const __grid_constant__ TcArgs a) {
    extern __shared__ unsigned char dsm[];
    unsigned char *base = dsm + ((1024 - (smem_u32(dsm) & 1023)) & 1023);
    // Of each pipeline: afull: the stage's A operand has landed (64 producer
    // arrivals); bfull: its operator image has landed (the copy's own transaction
    // count, so the copying thread can always wait for its copies, whatever the
    // producers do)
    __shared__ __align__(8) uint64_t afull_[2][kTcMaxStages], bfull_[2][kTcMaxStages], empty_[2][kTcMaxStages];
    __shared__ __align__(8) uint64_t stall_bar;
    __shared__ __align__(8) uint64_t bank_full[2], bank_empty[2];
    __shared__ uint32_t tslot;
    __shared__ int abort_flag;
    __shared__ uint32_t pref[kStreamTiles + 1];   // stream: units before each tile
    __shared__ uint32_t wtot[kTcWarps];
    __shared__ int first_tile;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int B = a.B, Npad = a.Npad, nck = a.nck, NST = a.nst;
    const int nsum = Npad / 2;
    const uint32_t b_bytes = 2u * (uint32_t)Npad * 64u;
    const uint32_t stage_bytes = tc_stage_bytes(Npad);   // [A: hi, lo][B: hi, lo]
    volatile int *abortp = &abort_flag;
    const int nbox = 128 / B;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)),
                     "r"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < 2 * kTcMaxStages; ++i) {
            // 64 producer threads; the operator copy's expect-tx arrival
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&afull_[0][0] + i)), "r"(64));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bfull_[0][0] + i)), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty_[0][0] + i)), "r"(1));
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bank_full[i])), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bank_empty[i])), "r"(8));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&stall_bar)), "r"(1));
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    // this CTA's units [u0, u1), in tile order from tile t0 on; P(t) = units
    // before tile t
    uint32_t G = 1, T = 0;
    uint32_t u0 = 0, u1 = 0;
    if (a.stream) {
        uint32_t n[kScanItems], sum = 0;
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) {
            const int t = tid * kScanItems + q;
            n[q] = t < a.ntiles ? __ldg(a.tmask + 8 * (size_t)t + 6) : 0;
            sum += n[q];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < kTcWarps; ++w) {
            if (w < warp) before += wtot[w];
            T += wtot[w];
        }
        uint32_t run = before + incl - sum;
        G = min(gridDim.x, max(1u, T / (uint32_t)a.min_units));
        if (blockIdx.x < G) {
            u0 = (uint32_t)((uint64_t)blockIdx.x * T / G);
            u1 = (uint32_t)((uint64_t)(blockIdx.x + 1) * T / G);
        }
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) {
            const int t = tid * kScanItems + q;
            if (t <= a.ntiles) pref[t] = run;
            if (t < a.ntiles && u0 >= run && u0 < run + n[q]) first_tile = t;
            run += n[q];
        }
        if (tid == 0) pref[a.ntiles] = T;
    } else {
        if (tid == 0) first_tile = (int)blockIdx.x;
        u1 = __ldg(a.tmask + 8 * (size_t)blockIdx.x + 6);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    const int units = (int)(u1 - u0);
    const int t0 = units > 0 ? first_tile : 0;
    if (a.stream && tid == 0) {   // for m2l_join
        a.mcut[blockIdx.x] = make_int4(t0, (int)pref[t0], (int)pref[t0 + 1], (int)G);
        if (blockIdx.x == 0) a.mcut[gridDim.x] = make_int4((int)T, 0, 0, 0);
    }
    // rank of the first unit taken of tile t, and how many are taken
    auto seg_lo = [&](int t) -> int { return a.stream && pref[t] < u0 ? (int)(u0 - pref[t]) : 0; };
    auto seg_n = [&](int t) -> int {
        return a.stream ? (int)(min(u1, pref[t + 1]) - max(u0, pref[t])) : units;
    };

    // This role's pipeline: units pipe, pipe + 2, ... of the CTA's, in stages of its
    // own ring.
    const int pipe = warp < 4 ? warp >> 1 : warp >= 14 ? 1 : 0;
    unsigned char *ring = base + (size_t)pipe * NST * stage_bytes;
    uint64_t *afull = afull_[pipe], *bfull = bfull_[pipe], *empty = empty_[pipe];
    // The units in order: tile, and offset within its class's list.
    struct Walk {
        int t, left, oi;
        OffsetIter it;
    };
    auto step = [&](Walk &w) {
        if (w.left == 0) {
            ++w.t;
            w.left = seg_n(w.t);
            w.it.open(a.tmask, w.t, seg_lo(w.t));
        }
        --w.left;
        w.oi = w.it.next();
    };
    Walk walk;
    walk.t = t0 - 1;
    walk.left = 0;

    if (warp < 4) {
        // ---------------- A producers: FP16 inputs, scaled and split in advance;
        // a warp does rows [64 half, 64 half + 64) of its pipeline's stages
        const int half = warp & 1;
        const int k = lane & 7;                       // 16-byte piece of a row's chunk: 0-3 high, 4-7 low
        const uint32_t kpart = k < 4 ? 0u : 8192u;
        const int rl0 = lane >> 3;
        int opened = -1, cls = 0;
        const TcLevel *L = nullptr;
        const unsigned char *split = nullptr;
        TcTarget q[2];
        const unsigned char *ahead[2] = {nullptr, nullptr};   // split parts of this lane's two rows at the next unit
        auto locate = [&]() {
            if (walk.t != opened) {
                opened = walk.t;
                const TcTile tile = tile_of(a, walk.t);
                L = tile.L;
                cls = tile.cls;
                split = L->split;
#pragma unroll
                for (int e = 0; e < 2; ++e) q[e] = target_of(tile, nbox, (64 * half + 32 * e + lane) / B);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t src = source_of(a, L, q[e], cls, walk.oi);
                ahead[e] = src >= 0 ? split + (src * B + (64 * half + 32 * e + lane) % B) * a.ldk * 4 : nullptr;
            }
        };
        int s = 0, n_done = 0;
        uint32_t ph = 0;
        bool stop = false;
        if (pipe < units) {
            if (pipe) step(walk);
            step(walk);
            locate();
        }
        for (int u = pipe; u < units && !stop; u += 2) {
            // the warp's 64 rows in 16 passes of 4, eight lanes per row: each
            // lane's piece of its sixteen rows
            const unsigned char *rp[16];
            uint32_t have = 0;
#pragma unroll
            for (int pp = 0; pp < 16; ++pp) {
                const unsigned char *o = (const unsigned char *)__shfl_sync(
                    0xffffffffu, (unsigned long long)ahead[pp >> 3], 4 * (pp & 7) + rl0);
                rp[pp] = (o ? o : split) + 16 * k;
                have |= (uint32_t)(o != nullptr) << pp;
            }
            if (u + 2 < units) {   // located a unit early, off the pipeline's path
                step(walk);
                step(walk);
                locate();
            }
            for (int j = 0; j < nck; ++j) {
                if (n_done >= NST && !mbar_wait_ab(smem_u32(&empty[s]), ph ^ 1, abortp, a.wait_tries)) {
                    stop = true;
                    break;
                }
                const uint32_t sub = smem_u32(ring) + (uint32_t)s * stage_bytes + kpart;
                const int ck = chunk_of(nck, j);
#pragma unroll
                for (int pp = 0; pp < 16; ++pp)
                    cp_async16(sub + swz64h(64 * half + 4 * pp + rl0, 8 * (k & 3)), rp[pp] + 128 * ck,
                               (have >> pp) & 1u ? 16u : 0u);
                // the thread's arrival, made when its copies have landed
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&afull[s])) : "memory");
                ++n_done;
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");   // no copy outlives the loop
    } else if (warp == 4 || warp == 14) {
        // ---------------- MMA issuers
        const uint32_t idesc = idesc_f16(128, Npad);
        const uint64_t desc0 = umma_desc64(smem_u32(ring));   // addresses: lowest bits, in units of 16 bytes
        const uint32_t d = tmem + (uint32_t)pipe * 256u;
        int s = 0, last = -1;
        uint32_t ph = 0;
        // testing aid: a wait that nothing completes runs out, sets the abort
        // flag, and every role stops, drains and reports through status[1]
        bool stop = pipe == 0 && a.test_stall && !mbar_wait_ab(smem_u32(&stall_bar), 0, abortp, a.wait_tries);
        stop = __any_sync(0xffffffffu, stop);
        // Inputs in descending order: chunk by chunk from the last, each chunk's
        // k-steps of 16 inputs from the last down, and in each k-step the two
        // small cross products before the main one.  The accumulator adds of the
        // tensor cores truncate, so every add made once the sum has its full size
        // costs up to an ulp of it, all of the same sign; leading with the small
        // high-order terms leaves only the last few adds at full size.
        for (int g = pipe; g < units && !stop; g += 2)
            for (int j = 0; j < nck; ++j) {
                // lanes 0, 1: the stage's operands; 2: the bank, read out by the
                // promoters of two units before
                uint32_t bar = 0, par = ph;
                if (lane < 2) {
                    bar = smem_u32(lane ? &bfull[s] : &afull[s]);
                } else if (lane == 2 && j == 0 && g >= 2) {
                    bar = smem_u32(&bank_empty[pipe]);
                    par = ((g - 2) >> 1) & 1;
                }
                bool done = bar == 0;
                long tries = 0;
                for (; tries < a.wait_tries; ++tries) {
                    if (!done) done = mbar_try(bar, par);
                    if (__all_sync(0xffffffffu, done)) break;
                    if ((tries & 255) == 255 && __any_sync(0xffffffffu, *abortp != 0)) tries = a.wait_tries;
                }
                if (tries >= a.wait_tries) {
                    *abortp = 1;
                    stop = true;
                    break;
                }
                __syncwarp();
                if (lane == 0) {
                    // the producers' copies are generic-proxy writes; the MMAs read
                    // shared memory through the async proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint64_t ah = desc0 + (uint32_t)s * (stage_bytes >> 4), al = ah + (8192 >> 4);
                    const uint64_t bh = ah + (kTcA >> 4), bl = bh + Npad * 4;
                    uint32_t acc = j > 0 ? 1u : 0u;
                    if (a.K > 32 * chunk_of(nck, j) + 16) {   // else one k-step holds inputs
                        mma_f16(d, ah + 2, bl + 2, idesc, acc);
                        mma_f16(d, al + 2, bh + 2, idesc, 1u);
                        mma_f16(d, ah + 2, bh + 2, idesc, 1u);
                        acc = 1u;
                    }
                    mma_f16(d, ah, bl, idesc, acc);
                    mma_f16(d, al, bh, idesc, 1u);
                    mma_f16(d, ah, bh, idesc, 1u);
                    commit_to(&empty[s]);
                    if (j + 1 == nck) commit_to(&bank_full[pipe]);
                }
                ++last;
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
        // drain: the last commit covers every MMA issued
        if (last >= 0) mbar_wait(smem_u32(&empty[last % NST]), (uint32_t)((last / NST) & 1), a.wait_tries);
    } else if (warp == 5 || warp == 15) {
        // ---------------- operator images
        if (lane == 0) {
            int s = 0, n_done = 0, opened = -1, cls = 0;
            uint32_t ph = 0;
            bool stop = false;
            for (int u = pipe; u < units && !stop; u += 2) {
                if (u > 0) step(walk);
                step(walk);
                if (walk.t != opened) {
                    opened = walk.t;
                    cls = tile_of(a, walk.t).cls;
                }
                const int o = c_il[cls][walk.oi];
                const int dx = (signed char)o, dy = (signed char)(o >> 8), dz = (signed char)(o >> 16);
                const unsigned char *img = a.img + (size_t)((dz + 3) * 49 + (dy + 3) * 7 + (dx + 3)) * nck * b_bytes;
                for (int j = 0; j < nck; ++j) {
                    if (n_done >= NST && !mbar_wait_ab(smem_u32(&empty[s]), ph ^ 1, abortp, a.wait_tries)) {
                        stop = true;
                        break;
                    }
                    const uint32_t stage = smem_u32(ring) + (uint32_t)s * stage_bytes;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&bfull[s])),
                                 "r"(b_bytes));
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            stage + kTcA),
                        "l"(img + (size_t)chunk_of(nck, j) * b_bytes), "r"(b_bytes), "r"(smem_u32(&bfull[s]))
                        : "memory");
                    ++n_done;
                    if (++s == NST) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            // drain: every copy issued must have landed before the CTA exits;
            // the last NST stages may still have copies in flight (earlier ones
            // were consumed by MMAs before their stage was reused), and each
            // stage's copy completes its own barrier
            for (int j = max(0, n_done - NST); j < n_done; ++j)
                mbar_wait(smem_u32(&bfull[j % NST]), (uint32_t)((j / NST) & 1), a.wait_tries);
        }
    }
    // ---------------- promoters (warps 6-13) and the write-back of each tile
    const int pw = warp - 6;
    const int pq = warp & 3, ph_half = pw >> 2;   // TMEM lane quarter, column half
    bool ok = true;
    if (pw >= 0 && pw < 8) {
        float acc[NS];
        int g = 0;   // units promoted so far (bank g & 1)
        for (int t = t0; g < units; ++t) {
            const int n = seg_n(t);
#pragma unroll
            for (int q = 0; q < NS; ++q) acc[q] = 0.f;
            for (int e = 0; e < n; ++e, ++g) {
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
                        float v[8];
                        tmem_ld8(tb + j0, v);
#pragma unroll
                        for (int q = 0; q < 8; ++q) acc[j0 + q] += v[q];
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bank_empty[g & 1]));
            }
            if (*abortp) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const TcTile tile = tile_of(a, t);
            const TcLevel &L = *tile.L;
            const int r = pq * 32 + lane;
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
            if (a.stream && pref[t] < u0) {
                // the rest of an earlier CTA's tile: partial rows, added by m2l_join
                const int q4 = nsum / 4;
                float4 *mine = reinterpret_cast<float4 *>(a.mpart) +
                               ((size_t)blockIdx.x * (Npad / 4) + ph_half * q4) * a.prow + r;
#pragma unroll
                for (int q = 0; q < NS; q += 4)
                    if (q < nsum && r < a.prow)
                        mine[(q / 4) * a.prow] = make_float4(acc[q], acc[q + 1], acc[q + 2], acc[q + 3]);
                continue;
            }
            const int64_t row = out_row(a, tile, nbox, r);
            if (row >= 0) {
#pragma unroll
                for (int q = 0; q < NS; q += 4)
                    if (q < nsum)
                        store4(a, L, row, ph_half * nsum + q, make_float4(acc[q], acc[q + 1], acc[q + 2], acc[q + 3]));
            }
        }
    }
    const bool failed = __syncthreads_or(!ok || abort_flag);
    if (failed && tid == 0) atomicOr(a.status + 1, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols));
}

// ------------------------------------------------ FP64 from BF16 digits
// The FP64 M2L on the tensor cores (GB300's FP64 pipe runs at 1/64 of its FP32
// rate; its tensor cores add 8-bit integers' products exactly).  Every input row
// is scaled by a power of two of its own and every operator column by one of its
// own, and both are written as kSl = 7 digits in base 256, -128..128, exact in
// BF16 (56 bits); powers of two per input component, taken from the operators,
// balance the orders first.  Digit products of equal weight, i + j = d <= 6, add
// up in one FP32 accumulator: d + 1 products of at most 2^14 for each of up to 289
// inputs.  That is at most 2^24, so exact whatever the digits, for d <= 3 up to
// p = 15 and for d <= 2 at p = 16.  A later sum passes 2^24 only if nearly all its
// products agree in sign and are of the largest size (of random digits it is
// some 2^18), and then loses units of its own weight, 2^-24 (p = 16, d = 3) or
// 2^-32 and less of the first digits'.  (The splitting into exactly multipliable
// slices is Ozaki, Ogita, Oishi and Rump's, 2012.)  What is left out, d >= 7, and the
// last place of the digits are some 2^-54 of a row's largest term, as much as FP64
// rounds away in one of its additions; a component far below its row's largest has
// fewer than 53 bits.
//
// The pipeline is m2l_tc's: tiles of 128 targets, units of one (tile, column
// group, offset) dealt out over the grid, chunks of 16 inputs in a ring of stages
// (32-byte rows, 32-byte swizzle), seven accumulators of up to 64 columns in
// tensor memory.  After an offset the promoters turn the seven sums into one
// 64-bit integer, exactly, and add it to FP64 sums with the source row's scale.
// The batch members go one after the other, tiles of 128 boxes of one member:
// where a tile is cut decides how its sum associates, and a member's result is
// the same alone and in a batch.
// Bound by shared-memory and L2 operand traffic and by the promoters, which the
// tensor cores wait for (no second bank fits).  128^3 with 1,360 targets at p = 14:
// 1,710 us, where the SIMT M2L takes 10.8 ms; the fields differ by 2e-16.
constexpr int kSl = 7;
constexpr int kOzWarps = 14, kOzThreads = 32 * kOzWarps, kOzScanItems = 4, kOzMaxStages = 8;
constexpr int kOzStreamTiles = kOzThreads * kOzScanItems;
constexpr int kOzCols = 64;                              // columns of a group, at most
constexpr uint32_t kOzA = kSl * 128u * 32u;              // A slices of a stage
__host__ __device__ constexpr uint32_t oz_stage_bytes(int ng) { return kOzA + (uint32_t)kSl * ng * 32u; }
inline int oz_stages(int ng) {
    const int n = (int)((227 * 1024 - 2048 - 4 * (kOzStreamTiles + 1)) / oz_stage_bytes(ng));
    return n > kOzMaxStages ? kOzMaxStages : n;
}
inline int oz_groups(int K) { return (K + kOzCols - 1) / kOzCols; }
inline int oz_group_cols(int K) { return ((K + oz_groups(K) - 1) / oz_groups(K) + 15) & ~15; }
inline int oz_chunks(int K) { return (K + 15) / 16; }
constexpr int kOzRowChunk = 256;                         // bytes of a row's chunk: 7 slices of 16 digits, padded

struct OzArgs {
    TcArgs t;                   // ntiles: of 128 targets; the launch's are (tile, group) pairs
    int ngrp, ng, nck;          // column groups, columns of a group, chunks of 16 inputs
    int nb, bb;                 // batch members of the rows, and the one this launch does (t.B = 1)
    const unsigned char *img;   // [343][ngrp][nck][kSl][ng rows of 32 bytes, swizzled]
    const double *cinv;         // [ngrp ng] inverse column scales
    double *part;               // [gridDim][ng][t.prow] partial rows
};

// Byte offset of 16-byte half h of row r in a slice (8-row atoms of 256 bytes).
__host__ __device__ __forceinline__ uint32_t swz32(int r, int h) {
    return (uint32_t)r * 32u + (uint32_t)((h ^ ((r >> 2) & 1)) << 4);
}

__device__ __forceinline__ uint64_t umma_desc32(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;             // leading byte offset (unused, swizzled K-major)
    d |= (uint64_t)(256 >> 4) << 32;    // stride byte offset: one 8-row atom
    d |= (uint64_t)1 << 46;             // descriptor version
    d |= (uint64_t)6 << 61;             // 32-byte swizzle
    return d;
}

// D = FP32, A = B = BF16 (format 1), both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Digits of v, |v| <= 2^55, as BF16: v = sum_i d_i 256^(6 - i), those of -v the
// negatives of v's.
__device__ __forceinline__ void bf16_digits(long long v, uint16_t d[kSl]) {
    const uint16_t sign = v < 0 ? 0x8000u : 0u;
    v = v < 0 ? -v : v;
#pragma unroll
    for (int i = kSl - 1; i >= 0; --i) {
        const int q = i > 0 ? (int)(signed char)(v & 255) : (int)v;
        v = (v - q) >> 8;
        d[i] = (uint16_t)(__float_as_uint((float)q) >> 16) ^ (q ? sign : 0u);   // |q| <= 128: 8 bits
    }
}

// The integer v as FP64, truncated to 53 bits, without the FP64 pipe
__device__ __forceinline__ double i64_to_f64(long long v) {
    const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)m);
    const unsigned long long n = m << (lz & 63);   // leading one at bit 63
    const unsigned hi = (v < 0 ? 0x80000000u : 0u) + ((unsigned)(63 - lz + 1022) << 20) + (unsigned)(n >> 43);
    return m ? __hiloint2double((int)hi, (int)(unsigned)(n >> 11)) : 0.0;
}

__global__ void __launch_bounds__(kOzThreads, 1) m2l_oz(const __grid_constant__ OzArgs o) {
    extern __shared__ unsigned char dsm[];
    unsigned char *base = dsm + ((1024 - (smem_u32(dsm) & 1023)) & 1023);
    __shared__ __align__(8) uint64_t afull[kOzMaxStages], bfull[kOzMaxStages], empty[kOzMaxStages];
    __shared__ __align__(8) uint64_t bank_full, bank_empty;
    __shared__ uint32_t tslot;
    __shared__ int abort_flag;
    __shared__ uint32_t pref[kOzStreamTiles + 1];   // stream: units before each (tile, group)
    __shared__ uint32_t wtot[kOzWarps];
    __shared__ int first_tile;
    const TcArgs &a = o.t;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nck = o.nck, NST = a.nst, NG = o.ng, ngrp = o.ngrp;
    const int ntg = a.ntiles * ngrp;
    const uint32_t stage_bytes = oz_stage_bytes(NG), b_bytes = (uint32_t)kSl * NG * 32u;
    volatile int *abortp = &abort_flag;
    constexpr int nbox = 128;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)),
                     "r"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&afull[i])), "r"(128));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bfull[i])), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty[i])), "r"(1));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bank_full)), "r"(1));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bank_empty)), "r"(8));
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    // this CTA's units [u0, u1), as in m2l_tc with (tile, group) pairs for tiles
    uint32_t G = 1, T = 0, u0 = 0, u1 = 0;
    if (a.stream) {
        uint32_t n[kOzScanItems], sum = 0;
#pragma unroll
        for (int q = 0; q < kOzScanItems; ++q) {
            const int t = tid * kOzScanItems + q;
            n[q] = t < ntg ? __ldg(a.tmask + 8 * (size_t)(t / ngrp) + 6) : 0;
            sum += n[q];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int q = 1; q < 32; q <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, q);
            if (lane >= q) incl += v;
        }
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < kOzWarps; ++w) {
            if (w < warp) before += wtot[w];
            T += wtot[w];
        }
        uint32_t run = before + incl - sum;
        G = min(gridDim.x, max(1u, T / (uint32_t)a.min_units));
        if (blockIdx.x < G) {
            u0 = (uint32_t)((uint64_t)blockIdx.x * T / G);
            u1 = (uint32_t)((uint64_t)(blockIdx.x + 1) * T / G);
        }
#pragma unroll
        for (int q = 0; q < kOzScanItems; ++q) {
            const int t = tid * kOzScanItems + q;
            if (t <= ntg) pref[t] = run;
            if (t < ntg && u0 >= run && u0 < run + n[q]) first_tile = t;
            run += n[q];
        }
        if (tid == 0) pref[ntg] = T;
    } else {
        if (tid == 0) first_tile = (int)blockIdx.x;
        u1 = __ldg(a.tmask + 8 * (size_t)((int)blockIdx.x / ngrp) + 6);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    const int units = (int)(u1 - u0);
    const int t0 = units > 0 ? first_tile : 0;
    if (a.stream && tid == 0) {   // for m2l_oz_join
        a.mcut[blockIdx.x] = make_int4(t0, (int)pref[t0], (int)pref[t0 + 1], (int)G);
        if (blockIdx.x == 0) a.mcut[gridDim.x] = make_int4((int)T, 0, 0, 0);
    }
    auto seg_lo = [&](int t) -> int { return a.stream && pref[t] < u0 ? (int)(u0 - pref[t]) : 0; };
    auto seg_n = [&](int t) -> int {
        return a.stream ? (int)(min(u1, pref[t + 1]) - max(u0, pref[t])) : units;
    };
    // the source box's row index of row `row` of the tile, unit by unit (-1: none)
    struct Rows {
        int t, left, cls, slot;
        const TcLevel *L;
        TcTarget q;
        OffsetIter it;
    };
    auto next_row = [&](Rows &w) -> int64_t {
        if (w.left == 0) {
            ++w.t;
            w.left = seg_n(w.t);
            w.it.open(a.tmask, w.t / ngrp, seg_lo(w.t));
            const TcTile tile = tile_of(a, w.t / ngrp);
            w.L = tile.L;
            w.cls = tile.cls;
            w.q = target_of(tile, nbox, w.slot);
        }
        --w.left;
        const int64_t src = source_of(a, w.L, w.q, w.cls, w.it.next());
        return src >= 0 ? (src - w.L->src0) * o.nb + o.bb : -1;
    };

    bool ok = true;
    if (warp < 4) {
        // ---------------- A producers: 16 lanes per row's 14 pieces of 16 bytes
        Rows w{};
        w.t = t0 - 1;
        w.slot = tid;
        const int piece = lane & 15;
        const int64_t ldb = (int64_t)nck * kOzRowChunk;
        int s = 0, n_done = 0;
        uint32_t ph = 0;
        bool stop = false;
        const unsigned char *ahead = nullptr;
        auto locate = [&]() {
            const int64_t r = next_row(w);
            ahead = r >= 0 ? w.L->split + r * ldb : nullptr;
        };
        if (units > 0) locate();
        const unsigned char *any = units > 0 ? w.L->split : nullptr;   // a valid address for rows without a source
        for (int u = 0; u < units && !stop; ++u) {
            const unsigned char *src = ahead;
            if (u + 1 < units) locate();
            const unsigned char *rp[16];
            uint32_t have = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const unsigned char *q =
                    (const unsigned char *)__shfl_sync(0xffffffffu, (unsigned long long)src, 2 * i + (lane >> 4));
                rp[i] = (q ? q : any) + 16 * piece;
                have |= (uint32_t)(q != nullptr) << i;
            }
            for (int j = 0; j < nck; ++j) {
                if (n_done >= NST && !mbar_wait_ab(smem_u32(&empty[s]), ph ^ 1, abortp, a.wait_tries)) {
                    stop = true;
                    break;
                }
                if (piece < 2 * kSl) {
                    const uint32_t sub = smem_u32(base) + (uint32_t)s * stage_bytes + (uint32_t)(piece >> 1) * 4096u;
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        cp_async16(sub + swz32(warp * 32 + 2 * i + (lane >> 4), piece & 1), rp[i] + j * kOzRowChunk,
                                   (have >> i) & 1u ? 16u : 0u);
                }
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&afull[s])) : "memory");
                ++n_done;
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");   // no copy outlives the loop
    } else if (warp == 4) {
        // ---------------- MMA issuer
        const uint32_t idesc = idesc_bf16(128, NG);
        const uint64_t desc0 = umma_desc32(smem_u32(base));
        int s = 0, last = -1, it = 0;
        uint32_t ph = 0;
        bool stop = false;
        for (int g = 0; g < units && !stop; ++g) {
            for (int j = 0; j < nck && !stop; ++j) {
                // lanes 0, 1: the stage's operands; 2: the bank, read out after the unit before
                uint32_t bar = 0, par = ph;
                if (lane < 2) {
                    bar = smem_u32(lane ? &bfull[s] : &afull[s]);
                } else if (lane == 2 && j == 0 && g >= 1) {
                    bar = smem_u32(&bank_empty);
                    par = (g - 1) & 1;
                }
                bool done = bar == 0;
                long tries = 0;
                for (; tries < a.wait_tries; ++tries) {
                    if (!done) done = mbar_try(bar, par);
                    if (__all_sync(0xffffffffu, done)) break;
                    if ((tries & 255) == 255 && __any_sync(0xffffffffu, *abortp != 0)) tries = a.wait_tries;
                }
                if (tries >= a.wait_tries) {
                    *abortp = 1;
                    stop = true;
                    break;
                }
                __syncwarp();
                if (lane == 0) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint64_t ad = desc0 + (uint32_t)s * (stage_bytes >> 4), bd = ad + (kOzA >> 4);
#pragma unroll
                    for (int i = 0; i < kSl; ++i)
#pragma unroll
                        for (int e = 0; e < kSl - i; ++e)
                            mma_f16(tmem + (uint32_t)((i + e) * NG), ad + i * (4096 >> 4), bd + (uint32_t)(e * NG * 2), idesc,
                                    j > 0 || i > 0 ? 1u : 0u);
                    commit_to(&empty[s]);
                    if (j + 1 == nck) commit_to(&bank_full);
                }
                last = it++;
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
        }
        if (last >= 0) mbar_wait(smem_u32(&empty[last % NST]), (uint32_t)((last / NST) & 1), a.wait_tries);
    } else if (warp == 5) {
        // ---------------- operator images
        if (lane == 0) {
            int t = t0 - 1, left = 0, cls = 0;
            OffsetIter it;
            int s = 0, n_done = 0, last = -1;
            uint32_t ph = 0;
            bool stop = false;
            for (int u = 0; u < units && !stop; ++u) {
                if (left == 0) {
                    ++t;
                    left = seg_n(t);
                    it.open(a.tmask, t / ngrp, seg_lo(t));
                    cls = tile_of(a, t / ngrp).cls;
                }
                --left;
                const int q = c_il[cls][it.next()];
                const int dx = (signed char)q, dy = (signed char)(q >> 8), dz = (signed char)(q >> 16);
                const unsigned char *img =
                    o.img + ((size_t)((dz + 3) * 49 + (dy + 3) * 7 + (dx + 3)) * ngrp + t % ngrp) * nck * b_bytes;
                for (int j = 0; j < nck; ++j) {
                    if (n_done >= NST && !mbar_wait_ab(smem_u32(&empty[s]), ph ^ 1, abortp, a.wait_tries)) {
                        stop = true;
                        break;
                    }
                    const uint32_t stage = smem_u32(base) + (uint32_t)s * stage_bytes;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&bfull[s])),
                                 "r"(b_bytes));
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            stage + kOzA),
                        "l"(img + (size_t)j * b_bytes), "r"(b_bytes), "r"(smem_u32(&bfull[s]))
                        : "memory");
                    last = n_done++;
                    if (++s == NST) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            // drain, as in m2l_tc
            for (int j = last - NST + 1 > 0 ? last - NST + 1 : 0; j <= last; ++j)
                mbar_wait(smem_u32(&bfull[j % NST]), (uint32_t)((j / NST) & 1), a.wait_tries);
        }
    } else {
        // ---------------- promoters: a row and half the columns per thread
        constexpr int NH = kOzCols / 2;
        const int pw = warp - 6, pq = warp & 3, half = pw >> 2, nh = NG / 2;
        const int r = pq * 32 + lane;
        Rows w{};
        w.t = t0 - 1;
        w.slot = r;
        double acc[NH];
        int64_t ahead = units > 0 ? next_row(w) : -1;
        double scale = ahead >= 0 ? __ldg(w.L->rscale + ahead) : 0.0;
        int g = 0;
        for (int t = t0; g < units; ++t) {
            const int n = seg_n(t);
#pragma unroll
            for (int q = 0; q < NH; ++q) acc[q] = 0.0;
            for (int e = 0; e < n; ++e, ++g) {
                const double sc = scale;
                if (g + 1 < units) {   // the next unit's scale, on its way meanwhile
                    ahead = next_row(w);
                    scale = ahead >= 0 ? __ldg(w.L->rscale + ahead) : 0.0;
                }
                bool w_ok = mbar_wait_ab(smem_u32(&bank_full), g & 1, abortp, a.wait_tries);
                w_ok = __all_sync(0xffffffffu, w_ok);   // tcgen05.ld is warp-collective
                if (!w_ok) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t tb = tmem + ((uint32_t)(pq * 32) << 16) + (uint32_t)(half * nh);
#pragma unroll
                for (int c0 = 0; c0 < NH; c0 += 4) {
                    if (c0 < nh) {
                        uint32_t d[kSl][4];
#pragma unroll
                        for (int i = 0; i < kSl; ++i)
                            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                         : "=r"(d[i][0]), "=r"(d[i][1]), "=r"(d[i][2]), "=r"(d[i][3])
                                         : "r"(tb + (uint32_t)(i * NG + c0)));
                        // (the registers pass through the wait: nothing reads them before it)
                        asm volatile("tcgen05.wait::ld.sync.aligned;"
                                     : "+r"(d[0][0]), "+r"(d[0][1]), "+r"(d[0][2]), "+r"(d[0][3]), "+r"(d[1][0]),
                                       "+r"(d[1][1]), "+r"(d[1][2]), "+r"(d[1][3]), "+r"(d[2][0]), "+r"(d[2][1]),
                                       "+r"(d[2][2]), "+r"(d[2][3]), "+r"(d[3][0]), "+r"(d[3][1]));
                        asm volatile("" : "+r"(d[3][2]), "+r"(d[3][3]), "+r"(d[4][0]), "+r"(d[4][1]), "+r"(d[4][2]),
                                          "+r"(d[4][3]), "+r"(d[5][0]), "+r"(d[5][1]), "+r"(d[5][2]), "+r"(d[5][3]),
                                          "+r"(d[6][0]), "+r"(d[6][1]), "+r"(d[6][2]), "+r"(d[6][3]));
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            int v[kSl];
#pragma unroll
                            for (int i = 0; i < kSl; ++i) v[i] = __float2int_rn(__uint_as_float(d[i][c]));
                            // in units of 256^-5 of the first digits' products; |d_0| <= 289 2^14 and so on:
                            // below 2^63
                            long long x = (long long)(v[0] * 256 + v[1]) * 65536 + (long long)v[2] * 256 + v[3];
                            x = x * 65536 + (long long)v[4] * 256 + v[5] + v[6] / 256;
                            acc[c0 + c] = fma(i64_to_f64(x), sc, acc[c0 + c]);
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bank_empty));
            }
            if (*abortp) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const int col0 = (t % ngrp) * NG + half * nh;
            if (a.stream && pref[t] < u0) {
                // the rest of an earlier CTA's tile: partial rows, added by m2l_oz_join
                double *mine = o.part + ((size_t)blockIdx.x * NG + half * nh) * a.prow + r;
#pragma unroll
                for (int q = 0; q < NH; ++q)
                    if (q < nh && r < a.prow) mine[q * a.prow] = acc[q];
                continue;
            }
            const TcTile tile = tile_of(a, t / ngrp);
            const int64_t row = out_row(a, tile, nbox, r);
            if (row >= 0) {
                double *dst = reinterpret_cast<double *>(tile.L->le) + (row * o.nb + o.bb) * a.ldk + col0;
#pragma unroll
                for (int q = 0; q < NH; ++q)
                    if (q < nh && col0 + q < a.K) dst[q] = acc[q] * __ldg(o.cinv + col0 + q);
            }
        }
    }
    const bool failed = __syncthreads_or(!ok || abort_flag);
    if (failed && tid == 0) atomicOr(a.status + 1, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols));
}

// The cut (tile, group)s' partial rows, added in CTA order (see m2l_join; the
// column scales are powers of two, so it does not matter when they are applied).
// 128^3 voxels 3,889 -> 3,884 us a forward, 83^3 1,272 -> 1,267, of the loads' order
// and of 8 blocks to a boundary in place of 2.
__global__ void __launch_bounds__(512) m2l_oz_join(const __grid_constant__ OzArgs o) {
    constexpr int kRows = 8;   // partial rows on their way
    const TcArgs &a = o.t;
    const int c = (int)blockIdx.x + 1;
    const int4 cut = a.mcut[c];
    const uint32_t G = (uint32_t)cut.w, T = a.mcut[gridDim.x + 1].x;
    if (c >= (int)G) return;
    const uint32_t p0 = (uint32_t)cut.y, p1 = (uint32_t)cut.z;
    if ((uint32_t)((uint64_t)c * T / G) == p0) return;
    const int cf = (int)((((uint64_t)p0 + 1) * G - 1) / T), cl = (int)(((uint64_t)p1 * G - 1) / T);
    if (c != cf + 1) return;
    const int r = threadIdx.x & 127;
    const TcTile tile = tile_of(a, cut.x / o.ngrp);
    const int64_t row = out_row(a, tile, 128, r);
    if (row < 0) return;
    const int col0 = (cut.x % o.ngrp) * o.ng;
    double *dst = reinterpret_cast<double *>(tile.L->le) + (row * o.nb + o.bb) * a.ldk + col0;
    const double *p = o.part + r;
    const size_t slot = (size_t)o.ng * a.prow;
    for (int q = 4 * (int)blockIdx.y + (threadIdx.x >> 7); q < o.ng && col0 + q < a.K; q += 4 * (int)gridDim.y) {
        double s = 0.0, scale = 0.0;
        for (int e = cf + 1; e <= cl; e += kRows) {
            double v[kRows];
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (e + i <= cl) v[i] = __ldg(p + (e + i) * slot + (size_t)q * a.prow);
            if (e == cf + 1) {
                scale = __ldg(o.cinv + col0 + q);
                s = dst[q];
            }
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (e + i <= cl) s = fma(v[i], scale, s);
        }
        dst[q] = s;
    }
}

// Power-of-two exponents of the operator set: se[k] per input component, ce[n]
// per output column, |T_o[n][k]| 2^(-se[k] - ce[n]) <= 1 over all offsets, each
// reached within a factor of two or so.  One block; two sweeps.
__global__ void __launch_bounds__(1024) oz_exponents(const double *__restrict__ cmax, int K, int *__restrict__ se,
                                                     int *__restrict__ ce) {
    __shared__ int c1[(kMaxP + 1) * (kMaxP + 1)], s1[(kMaxP + 1) * (kMaxP + 1)];
    auto expo = [](double v) { return v > 0.0 ? ilogb(v) + 1 : -2000; };   // v < 2^expo
    for (int n = threadIdx.x; n < K; n += blockDim.x) {
        int e = -2000;
        for (int k = 0; k < K; ++k) e = max(e, expo(cmax[(size_t)k * K + n]));
        c1[n] = e;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        int e = -2000;
        for (int n = 0; n < K; ++n)
            if (c1[n] > -2000) e = max(e, expo(cmax[(size_t)k * K + n]) - c1[n]);
        s1[k] = e > -1000 ? e : 0;
        se[k] = s1[k];
    }
    __syncthreads();
    for (int n = threadIdx.x; n < K; n += blockDim.x) {
        int e = -2000;
        for (int k = 0; k < K; ++k) e = max(e, expo(cmax[(size_t)k * K + n]) - s1[k]);
        ce[n] = e > -1000 ? e : 0;
    }
}

// Largest |T_o[n][k]| over the offsets, per (k, n).
__global__ void oz_absmax(const double *__restrict__ tab, int KK, double *__restrict__ cmax) {
    const int e = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (e >= KK) return;
    double m = 0.0;
    for (int off = 0; off < 343; ++off) {
        const int dx = off % 7 - 3, dy = (off / 7) % 7 - 3, dz = off / 49 - 3;
        if (max(abs(dx), max(abs(dy), abs(dz))) >= 2) m = fmax(m, fabs(tab[(size_t)off * KK + e]));
    }
    cmax[e] = m;
}

__global__ void oz_images(const double *__restrict__ tab, int K, int ngrp, int ng, int nck, const int *__restrict__ se,
                          const int *__restrict__ ce, double *__restrict__ cinv, unsigned char *__restrict__ img) {
    const int off = blockIdx.x, grp = blockIdx.y;
    const int dx = off % 7 - 3, dy = (off / 7) % 7 - 3, dz = off / 49 - 3;
    const bool used = max(abs(dx), max(abs(dy), abs(dz))) >= 2;
    const size_t tile = (size_t)kSl * ng * 32;
    unsigned char *dst = img + ((size_t)off * ngrp + grp) * nck * tile;
    for (int e = threadIdx.x; e < nck * ng * 16; e += blockDim.x) {
        const int kk = e % 16, n = e / 16 % ng, ck = e / (16 * ng), k = 16 * ck + kk, col = grp * ng + n;
        long long v = 0;
        if (used && k < K && col < K)
            v = llrint(ldexp(tab[(size_t)off * K * K + (size_t)k * K + col], 55 - se[k] - ce[col]));
        uint16_t d[kSl];
        bf16_digits(v, d);
#pragma unroll
        for (int i = 0; i < kSl; ++i)
            *reinterpret_cast<uint16_t *>(dst + ck * tile + (size_t)i * ng * 32 + swz32(n, kk >> 3) + (kk & 7) * 2) = d[i];
    }
    if (off == 0)
        for (int n = threadIdx.x; n < ng; n += blockDim.x)
            cinv[grp * ng + n] = grp * ng + n < K ? ldexp(1.0, ce[grp * ng + n]) : 0.0;
}

// The inputs' rows as digits, and the rows' scales: one warp per row; the last
// row of blocks finds the tiles' active offsets.
struct OzSplitArgs {
    const double *in[kMaxLevels + 1];
    unsigned char *out[kMaxLevels + 1];
    double *rscale[kMaxLevels + 1];
    int64_t rows[kMaxLevels + 1];
    const int *se;
    int lmin, ldk, K, nck;
};

__global__ void __launch_bounds__(256)
oz_split(const __grid_constant__ OzSplitArgs o, const __grid_constant__ TcArgs tc, uint32_t *tmask) {
    if (blockIdx.y == gridDim.y - 1) {
        for (int t = (int)blockIdx.x; t < tc.ntiles; t += (int)gridDim.x) tile_mask(tc, t, tmask);
        return;
    }
    const int l = o.lmin + (int)blockIdx.y, lane = threadIdx.x & 31;
    constexpr int NV = ((kMaxP + 1) * (kMaxP + 1) + 31) / 32;
    int sk[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) sk[q] = lane + 32 * q < o.K ? __ldg(o.se + lane + 32 * q) : 0;
    for (int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r < o.rows[l]; r += (int64_t)gridDim.x * 8) {
        const double *src = o.in[l] + r * o.ldk;
        double x[NV];
        int em = 0;   // largest biased exponent of x 2^se, 0x7ff + ... for infinities and NaN
        bool bad = false;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int k = lane + 32 * q;
            x[q] = k < o.K ? __ldg(src + k) : 0.0;
            const int e = (int)((__double_as_longlong(x[q]) >> 52) & 0x7ff);
            bad |= e == 0x7ff;
            if (e > 0) em = max(em, e + sk[q]);
        }
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, q));
        bad = __any_sync(0xffffffffu, bad);
        const int E = em - 1022;   // |x 2^se| < 2^E
        if (lane == 0) o.rscale[l][r] = bad ? __longlong_as_double(0x7ff8000000000000ll) : em > 0 ? ldexp(1.0, E - 54) : 0.0;
        unsigned char *dst = o.out[l] + r * (int64_t)o.nck * kOzRowChunk;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int k = lane + 32 * q;
            if (k >= 16 * o.nck) continue;
            // one bit more, rounded off
            long long v = bad || em <= 0 ? 0 : to_fix(x[q], 56 - E + sk[q]);
            v = (v + (v >= 0 ? 1 : -1)) / 2;
            uint16_t d[kSl];
            bf16_digits(v, d);
#pragma unroll
            for (int i = 0; i < kSl; ++i)
                *reinterpret_cast<uint16_t *>(dst + (k >> 4) * kOzRowChunk + i * 32 + (k & 15) * 2) = d[i];
        }
    }
}

}  // namespace

// Bytes of the split FP16 inputs of levels 2..l-1 (the start of level l in
// the split buffer), for the plan's largest batch.
static size_t split_offset(const FmmPlan *F, int adj, int l) {
    size_t off = 0;
    for (int k = 2; k < l; ++k) off += (size_t)(adj ? F->lev[k].nt : F->lev[k].ns) * F->B * F->KS * sizeof(float);
    return off;
}

float *tc_split_rows(const FmmPlan *F, int level) {
    return reinterpret_cast<float *>(F->tc_split + split_offset(F, 0, level));
}

// Tiles of the M2L (adj: of its transpose) for batches of B.
static int64_t tc_tiles(const FmmPlan *F, bool adj, int B, int *tile_begin) {
    const int nbox = 128 / B;
    int64_t tiles = 0;
    int e = 0;
    for (int l = 2; l <= F->L; ++l)
        for (int c = 0; c < 8; ++c, ++e) {
            if (tile_begin) tile_begin[e] = (int)tiles;
            const int64_t *off = adj ? F->scls_off[l] : F->lev[l].cls_off;
            const int64_t cnt = (adj || F->lev[l].nt > 0) ? off[c + 1] - off[c] : 0;
            tiles += (cnt + nbox - 1) / nbox;
        }
    if (tile_begin) tile_begin[e] = (int)tiles;
    return tiles;
}

// Rows of a tile that may hold a target, at most, for batches of B.
static int tc_tile_rows(const FmmPlan *F, bool adj, int B) {
    const int64_t nbox = 128 / B;
    int64_t most = 1;
    for (int l = 2; l <= F->L; ++l)
        for (int c = 0; c < 8; ++c) {
            const int64_t *off = adj ? F->scls_off[l] : F->lev[l].cls_off;
            if (adj || F->lev[l].nt > 0) most = std::max(most, std::min(nbox, off[c + 1] - off[c]));
        }
    return (int)(most * B);
}

// CTAs of a launch that deals out units: one per SM, no more than could have
// kMinUnits each, and no more than the partial rows held serve; 0: whole tiles
// (too many of them, or rows for fewer CTAs than tiles).
constexpr int kMinUnits = 6;
static int64_t tc_stream_ctas(int64_t tiles, int64_t rows, int prow) {
    if (tiles > kStreamTiles) return 0;
    const int64_t c = std::max<int64_t>(1, std::min<int64_t>(sm_count(), tiles * 189 / kMinUnits));
    return std::min(c, rows / prow) >= std::min<int64_t>(tiles, sm_count()) ? std::min(c, rows / prow) : 0;
}

size_t m2l_tc_bytes(int p, bool fp64) {
    const int npad = ((p + 1) * (p + 1) + 15) & ~15;
    const size_t cuts = (size_t)(sm_count() + 1) * sizeof(int4) + 4096;
    if (fp64) return (size_t)sm_count() * 128 * kOzCols * sizeof(double) + cuts;
    return npad > 256 ? 0 : (size_t)sm_count() * 128 * npad * sizeof(float) + cuts;
}

// Bytes that the plan can still allocate within the size it was announced with
// (gf_plan_bytes): what is left of the open chunk, or a chunk of its own
// (alloc_exact).  Point plans, and FP64 plans with the M2L on FP16 parts, have no
// announced size.
static size_t announced_room(const gf_plan_s *plan) {
    if (plan->fmm->points || plan->fmm->m2l_tc64) return SIZE_MAX;
    const DeviceArena &A = plan->arena;
    const size_t all = fmm_bytes_estimate(&plan->grid, plan->quad.nq, plan->M, &plan->opt, plan->tight);
    return all > A.bytes ? std::max(A.left, all - A.bytes) : A.left;
}

// Scratch of n bytes, `room` at most: of its own size in a small plan, whose chunks
// would multiply what it holds; from a chunk in a plan of 64 MB or more, because a
// piece of another size splits a chunk that the pool holds for the next plan
// (creating one took 200 us longer).
static gf_status take_scratch(gf_plan_s *plan, void **p, size_t n, size_t room) {
    DeviceArena &A = plan->arena;
    return A.next >= ((size_t)32 << 20) && A.next >= n && room >= A.next ? A.alloc(p, n) : A.alloc_exact(p, n);
}

// Masks of the tiles and the partial rows of cut tiles, for every batch up to the
// plan's largest (which has the most tiles).  Only rows that hold targets are kept:
// a 32^3 grid under a plane of stations has 16 to a tile, 1.7 MB for 152 CTAs, where
// two whole tiles to a CTA took 27 MB.  The forward's rows serve the adjoint too when
// they suffice.  A plan without room for them takes whole tiles.
static gf_status m2l_tc_workspaces(gf_plan_s *plan, bool adj) {
    FmmPlan *F = plan->fmm;
    if (F->B > 128) return GF_OK;
    const int64_t tiles = tc_tiles(F, adj, F->B, nullptr);
    if (tiles == 0) return GF_OK;
    GF_TRY(plan->arena.alloc((void **)&F->m2l_mask[adj], (size_t)tiles * 8 * sizeof(uint32_t)));
    int64_t rows = 0, ctas = 0;
    for (int B = 1; B <= F->B; ++B) {
        const int64_t c = tc_stream_ctas(tc_tiles(F, adj, B, nullptr), INT64_MAX, 1);
        rows = std::max(rows, c * tc_tile_rows(F, adj, B));
        ctas = std::max(ctas, c);
    }
    const size_t row = F->tab->tc_npad * sizeof(float), cut = (size_t)(sm_count() + 1) * sizeof(int4) + 512;
    size_t room = SIZE_MAX;
    if (plan->tight) {
        room = adj ? 0 : announced_room(plan);
        rows = room > cut ? std::min<int64_t>(rows, (int64_t)std::min<size_t>((room - cut) / row, INT64_MAX)) : 0;
    }
    if (rows == 0 || (rows <= F->m2l_part_rows && ctas <= F->m2l_part_ctas)) return GF_OK;
    rows = std::max(rows, F->m2l_part_rows);
    ctas = std::max<int64_t>(ctas, F->m2l_part_ctas);
    unsigned char *mem = nullptr;
    if (take_scratch(plan, (void **)&mem, rows * row + cut, room) != GF_OK) return GF_OK;
    F->m2l_part = (float *)mem;
    F->m2l_cut = (int4 *)(mem + ((rows * row + 255) & ~(size_t)255));
    F->m2l_part_rows = rows;
    F->m2l_part_ctas = (int)ctas;
    return GF_OK;
}

// The level table of the forward (or its transpose) on the device.
static gf_status m2l_tc_levels(gf_plan_s *plan, bool adj) {
    FmmPlan *F = plan->fmm;
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
    return upload_small(dev, hb.data(), hb.size(), plan->arena.stream);
}

gf_status m2l_tc_prepare_adj(gf_plan_s *plan) {
    FmmPlan *F = plan->fmm;
    if (!F->mixed || !F->tab->m2l_tc) return GF_OK;
    GF_TRY(plan->arena.alloc((void **)&F->tc_split_adj, std::max<size_t>(16, split_offset(F, 1, F->L + 1))));
    GF_TRY(m2l_tc_workspaces(plan, true));
    return m2l_tc_levels(plan, true);
}

gf_status m2l_tc_prepare(gf_plan_s *plan) {
    FmmPlan *F = plan->fmm;
    if (!(F->mixed || F->m2l_tc64) || !F->tab->m2l_tc) return GF_OK;
    GF_TRY(plan->arena.alloc((void **)&F->tc_amax, 2 * (kMaxLevels + 1) * sizeof(uint32_t)));
    GF_TRY(plan->arena.alloc((void **)&F->tc_split, std::max<size_t>(16, split_offset(F, 0, F->L + 1))));
    GF_TRY(m2l_tc_workspaces(plan, false));
    return m2l_tc_levels(plan, false);
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

// The last row of blocks finds the active offsets of the tiles (tile_mask)
// beside the split.
__global__ void __launch_bounds__(256)
input_split(const __grid_constant__ AmaxArgs a, const __grid_constant__ SplitArgs o, int nck,
            const __grid_constant__ TcArgs tc, uint32_t *tmask) {
    if (blockIdx.y == gridDim.y - 1) {
        for (int t = (int)blockIdx.x; t < tc.ntiles; t += (int)gridDim.x) tile_mask(tc, t, tmask);
        return;
    }
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

gf_status tc_launch(TcArgs &a, int grid, cudaStream_t st) {
    if (a.ntiles == 0) return GF_OK;
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
    a.nent = 8 * (F->L - 1);
    a.ntiles = (int)tc_tiles(F, adj, B, a.tile_begin);
    a.tmask = F->m2l_mask[adj];
    a.mcut = F->m2l_cut;
    a.mpart = F->m2l_part;
    a.min_units = kMinUnits;
    a.prow = tc_tile_rows(F, adj, B);
    const int64_t ctas = std::min<int64_t>(F->m2l_part_ctas, tc_stream_ctas(a.ntiles, F->m2l_part_rows, a.prow));
    a.stream = ctas > 0;
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
        const int gs = std::max(gx, std::min(a.ntiles, 8 * 152));
        input_split<<<dim3(gs, F->L), 256, 0, st>>>(m, o, T->tc_nck_h, a, F->m2l_mask[adj]);
        GF_KERNEL_DONE();
    }
    if (!adj) stage_mark(plan, 4, st);
    if (fork) GF_CUDA(cudaEventRecord(fork, st));
    GF_TRY(tc_launch(a, a.stream ? (int)ctas : a.ntiles, st));
    if (a.stream && ctas > 1) {
        m2l_join<<<dim3((unsigned)ctas - 1, 8), 256, 0, st>>>(a);
        GF_KERNEL_DONE();
    }
    return GF_OK;
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

// ---------------------------------------------------------------- FP64 on the tensor cores
namespace {

std::mutex g_oz_mu;

// The digit images of an operator set, built with the first plan that uses
// them and kept as long as the tables they come from.
gf_status oz_tables(const Tables *T, cudaStream_t st, const OzTables **out) {
    std::lock_guard<std::mutex> lk(g_oz_mu);
    OzTables &z = *T->oz;
    if (!z.img) {
        const int K = T->K, ngrp = oz_groups(K), ng = oz_group_cols(K), nck = oz_chunks(K);
        double *cmax = nullptr;
        int *e = nullptr;
        unsigned char *img = nullptr;
        const size_t nimg = (size_t)343 * ngrp * nck * kSl * ng * 32;
        cudaError_t err = cudaMalloc(&cmax, ((size_t)K * K + (size_t)ngrp * ng) * sizeof(double));
        if (err == cudaSuccess) err = cudaMalloc(&e, 2 * (size_t)K * sizeof(int));
        if (err == cudaSuccess) err = cudaMalloc(&img, nimg);
        if (err == cudaSuccess) {
            double *cinv = cmax + (size_t)K * K;
            oz_absmax<<<ceil_div(K * K, 256), 256, 0, st>>>(T->m2l_d, K * K, cmax);
            oz_exponents<<<1, 1024, 0, st>>>(cmax, K, e, e + K);
            oz_images<<<dim3(343, ngrp), 256, 0, st>>>(T->m2l_d, K, ngrp, ng, nck, e, e + K, cinv, img);
            err = cudaGetLastError();
            if (err == cudaSuccess) err = cudaStreamSynchronize(st);
            if (err == cudaSuccess) {
                z.cinv = cinv;
                z.se = e;
                z.img = img;
            }
        }
        if (!z.img) {
            cudaFree(cmax);
            cudaFree(e);
            cudaFree(img);
            cudaGetLastError();
            *out = nullptr;   // no room: the SIMT M2L serves the plan
            if (err == cudaErrorMemoryAllocation) return GF_OK;
            set_error("cannot make the digit M2L's operators: %s", cudaGetErrorString(err));
            return GF_ERR_CUDA;
        }
    }
    *out = &z;
    return GF_OK;
}

// Rows of a level's split inputs: the z-slabs its M2L reads.
int64_t oz_rows(const FmmLevel &lv) {
    return lv.m2l_z1 >= lv.m2l_z0 ? (lv.m2l_z1 - lv.m2l_z0 + 1) * lv.sn[0] * lv.sn[1] : 0;
}

}  // namespace

// FP64 plans: the digit M2L's workspaces, when it is the faster one and they
// fit what the plan's size was announced as (gf_plan_bytes; point plans have no
// announced size).
gf_status m2l_oz_prepare(gf_plan_s *plan) {
    FmmPlan *F = plan->fmm;
    F->oz = nullptr;
    if (F->mixed || F->m2l_tc64 || F->L < 2 || F->B > 32 || (plan->opt.reserved0 & GF_FLAG_M2L_SIMT)) return GF_OK;
    const int K = F->K, ngrp = oz_groups(K), ng = oz_group_cols(K), nck = oz_chunks(K);
    const int64_t tiles = tc_tiles(F, false, 1, nullptr);
    if (tiles == 0 || tiles * ngrp > 0x7fffffff) return GF_OK;
    int64_t cols = 0, rows = 0;
    for (int l = 2; l <= F->L; ++l) {
        cols += F->lev[l].nt * F->B;
        rows += oz_rows(F->lev[l]) * F->B;
    }
    // Microseconds, from measurements at p = 4 to 16: a (tile, group, offset) unit
    // here, some 130 offsets to a tile padded to 128 targets, against a wave of the
    // SIMT M2L, which takes as many targets to a block as it would.  16^3 to 48^3
    // grids under a plane of observers (20 to 189 targets) stay there: 48^3 at
    // p = 12 1,109 us against 1,173 for the whole forward; from 64^3 on (340 targets)
    // the digits win: 2,256 against 1,271 us, 128^3 12.6 against 6.9 ms at p = 14.
    const double oz_us = F->B * (tiles * 130.0 * ngrp / sm_count() + 2.0) * (1.2 * nck + 8.0);
    const int64_t sms = sm_count(), P = cols >= 8 * sms && K <= 256 ? 4 : cols >= sms ? 2 : 1;
    const double fold_us = 0.8e-4 * K * K * (double)((cols + sms * P - 1) / (sms * P) * (sms * P));
    if (oz_us > 0.85 * fold_us) return GF_OK;
    const int64_t ctas = std::min<int64_t>(sm_count(), tiles * ngrp * 189);
    const size_t row_bytes = (size_t)nck * kOzRowChunk;
    const size_t part_bytes = (size_t)ctas * ng * tc_tile_rows(F, false, 1) * sizeof(double);
    const size_t inputs = (size_t)rows * (row_bytes + sizeof(double)) + (size_t)tiles * 8 * sizeof(uint32_t) +
                          (F->L + 1) * sizeof(TcLevel) + (size_t)(ctas + 1) * sizeof(int4) + 4096;
    const size_t room = announced_room(plan);
    if (inputs > room) return GF_OK;
    const bool stream = tiles * ngrp <= kOzStreamTiles && inputs + part_bytes <= room;
    // whole tiles in place of few dealt-out ones: the longest lists, rounds of blocks
    if (!stream && tiles * ngrp <= kOzStreamTiles &&
        F->B * ((tiles * ngrp + sms - 1) / sms * 189.0 + 2.0) * (1.2 * nck + 8.0) > 0.85 * fold_us)
        return GF_OK;
    const size_t need = inputs + (stream ? part_bytes : 0);
    const OzTables *z = nullptr;
    GF_TRY(oz_tables(F->tab, plan->arena.stream, &z));
    if (!z) return GF_OK;
    unsigned char *mem = nullptr;
    if (take_scratch(plan, (void **)&mem, need, room) != GF_OK) {   // no room: the SIMT M2L serves the plan
        cudaGetLastError();
        return GF_OK;
    }
    auto take = [&](size_t n) {
        unsigned char *p = mem;
        mem += (n + 255) & ~(size_t)255;
        return p;
    };
    F->oz_split = take((size_t)rows * row_bytes);
    F->oz_rscale = (double *)take((size_t)rows * sizeof(double));
    F->m2l_mask[0] = (uint32_t *)take((size_t)tiles * 8 * sizeof(uint32_t));
    F->oz_part = stream ? (double *)take(part_bytes) : nullptr;
    F->m2l_cut = stream ? (int4 *)take((size_t)(ctas + 1) * sizeof(int4)) : nullptr;
    std::vector<TcLevel> h(F->L + 1);
    memset(h.data(), 0, h.size() * sizeof(TcLevel));
    int64_t r0 = 0;
    for (int l = 2; l <= F->L; ++l) {
        const FmmLevel &lv = F->lev[l];
        TcLevel &t = h[l];
        t.le = (float *)lv.le;
        t.order = lv.m2l_order;
        t.tkey = lv.tkey;
        for (int d = 0; d < 3; ++d) {
            t.blo[d] = lv.slo[d];
            t.bn[d] = lv.sn[d];
        }
        for (int c = 0; c <= 8; ++c) t.cls_off[c] = lv.cls_off[c];
        t.shift = l - 2;
        t.split = F->oz_split + r0 * row_bytes;
        t.rscale = F->oz_rscale + r0;
        t.src0 = oz_rows(lv) > 0 ? lv.m2l_z0 * lv.sn[0] * lv.sn[1] : 0;
        F->oz_row0[l] = r0;
        r0 += oz_rows(lv) * F->B;
    }
    F->oz_levels = take(h.size() * sizeof(TcLevel));
    GF_TRY(upload_small(F->oz_levels, h.data(), h.size() * sizeof(TcLevel), plan->arena.stream));
    F->oz = z;
    return GF_OK;
}

static gf_status m2l_run_oz(gf_plan_s *plan, int B, cudaStream_t st, cudaEvent_t fork) {
    FmmPlan *F = plan->fmm;
    const OzTables *z = F->oz;
    OzArgs o;
    memset(&o, 0, sizeof(o));
    TcArgs &a = o.t;
    a.K = F->K;
    a.ldk = F->KS;
    a.B = 1;
    a.status = plan->d_status;
    a.wait_tries = kWaitTries;
    a.lv = reinterpret_cast<const TcLevel *>(F->oz_levels);
    a.lmin = 2;
    a.part_lo = plan->part_lo;
    a.part_hi = plan->part_hi;
    a.nent = 8 * (F->L - 1);
    a.ntiles = (int)tc_tiles(F, false, 1, a.tile_begin);
    a.tmask = F->m2l_mask[0];
    a.mcut = F->m2l_cut;
    a.prow = tc_tile_rows(F, false, 1);
    a.min_units = 1;
    o.nb = B;
    o.ngrp = oz_groups(F->K);
    o.ng = oz_group_cols(F->K);
    o.nck = oz_chunks(F->K);
    o.img = z->img;
    o.cinv = z->cinv;
    o.part = F->oz_part;
    a.nst = oz_stages(o.ng);
    const int64_t ntg = (int64_t)a.ntiles * o.ngrp;
    a.stream = ntg <= kOzStreamTiles && o.part;
    OzSplitArgs p;
    memset(&p, 0, sizeof(p));
    p.se = z->se;
    p.lmin = 2;
    p.ldk = F->KS;
    p.K = F->K;
    p.nck = o.nck;
    int64_t most = 1;
    for (int l = 2; l <= F->L; ++l) {
        const FmmLevel &lv = F->lev[l];
        p.rows[l] = oz_rows(lv) * B;
        p.in[l] = (const double *)lv.me + (p.rows[l] > 0 ? lv.m2l_z0 * lv.sn[0] * lv.sn[1] : 0) * B * F->KS;
        p.out[l] = F->oz_split + F->oz_row0[l] * o.nck * kOzRowChunk;
        p.rscale[l] = F->oz_rscale + F->oz_row0[l];
        most = std::max(most, p.rows[l]);
    }
    const int gx = (int)std::min<int64_t>(8 * 152, std::max<int64_t>((most + 7) / 8, std::min(a.ntiles, 8 * 152)));
    oz_split<<<dim3(gx, F->L), 256, 0, st>>>(p, a, F->m2l_mask[0]);
    GF_KERNEL_DONE();
    stage_mark(plan, 4, st);
    if (fork) GF_CUDA(cudaEventRecord(fork, st));
    if (a.ntiles == 0) return GF_OK;
    const size_t shm = (size_t)a.nst * oz_stage_bytes(o.ng) + 1024;
    GF_TRY(ensure_smem(m2l_oz, shm));
    const int64_t grid = a.stream ? std::min<int64_t>(sm_count(), ntg * 189) : ntg;
    for (o.bb = 0; o.bb < B; ++o.bb) {
        m2l_oz<<<(unsigned)grid, kOzThreads, shm, st>>>(o);
        GF_KERNEL_DONE();
        if (a.stream && grid > 1) {
            m2l_oz_join<<<dim3((unsigned)grid - 1, 8), 512, 0, st>>>(o);
            GF_KERNEL_DONE();
        }
    }
    return GF_OK;
}

// Whether the M2L runs from FP16 parts on the tensor cores.
static bool m2l_on_f16(const gf_plan_s *plan, int B, bool adj) {
    const FmmPlan *F = plan->fmm;
    return (F->mixed || (F->m2l_tc64 && !adj)) && F->tab->m2l_tc && (adj ? F->tc_levels_adj : F->tc_levels) &&
           !(plan->opt.reserved0 & GF_FLAG_M2L_SIMT) && B <= 128 && tc_stages(F->tab->tc_npad) >= 2;
}

bool m2l_fills_sms(const gf_plan_s *plan, int B) { return m2l_on_f16(plan, B, false) || plan->fmm->oz; }

template <class T>
gf_status m2l_run(gf_plan_s *plan, int B, bool adj, cudaStream_t st, cudaEvent_t fork) {
    FmmPlan *F = plan->fmm;
    if (m2l_on_f16(plan, B, adj)) return m2l_run_tc(plan, B, adj, st, fork);
    if (sizeof(T) == 8 && !adj && F->oz) return m2l_run_oz(plan, B, st, fork);
    if (!adj) stage_mark(plan, 4, st);   // no input split on this path
    if (fork) GF_CUDA(cudaEventRecord(fork, st));
    return m2l_run_fold<T>(plan, B, adj, st);
}

template gf_status m2l_run<float>(gf_plan_s *, int, bool, cudaStream_t, cudaEvent_t);
template gf_status m2l_run<double>(gf_plan_s *, int, bool, cudaStream_t, cudaEvent_t);

}  // namespace gf
