// gf_prim.cu -- exclusive scan, stable LSD radix sort and a bounding-box
// reduction, written for the octree build.
#include <float.h>
#include <string.h>

#include <algorithm>

#include "gf_prim.cuh"

namespace gf {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;   // 1024

// Sort tiles: 256 threads of 8 keys, or of 16 from kBigSort keys on (longer runs
// to write; fewer keys would leave SMs idle).  512 threads of 16: the scatter of
// 2^25 keys 164 us in place of 151.
constexpr int64_t kBigSort = 4 << 20;
constexpr int kRadix = 256;
constexpr int kSmallTile = 256 * 8, kBigTile = 256 * 16;

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Exclusive scan of one 1024-element tile per block; block totals to sums.
__global__ void __launch_bounds__(kScanThreads)
scan_tiles(const int64_t *__restrict__ in, int64_t *__restrict__ out, int64_t n,
           int64_t *__restrict__ sums) {
    __shared__ int64_t warp_tot[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t loc = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0;
        loc += v[i];
    }
    const int64_t incl = warp_incl_scan(loc);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < kScanThreads / 32 ? warp_tot[lane] : 0;
        const int64_t wi = warp_incl_scan(w);
        if (lane < kScanThreads / 32) warp_tot[lane] = wi - w;
        if (lane == kScanThreads / 32 - 1) sums[blockIdx.x] = wi;
    }
    __syncthreads();
    int64_t run = warp_tot[warp] + incl - loc;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
}

__global__ void add_tile_offsets(int64_t *__restrict__ out, int64_t n, const int64_t *__restrict__ offs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += offs[i / kScanTile];
}

__global__ void write_total(int64_t *__restrict__ out, int64_t n, const int64_t *__restrict__ offs,
                            const int64_t *__restrict__ sums, int64_t nb) {
    out[n] = offs[nb - 1] + sums[nb - 1];
}

// Whole scan in one block (n <= kSmallScan).  Warp w owns a run of
// consecutive rows of 32 items; a first sweep sums the run (independent
// loads), one block-wide scan of the run totals gives every run its offset,
// and a second sweep scans the run row by row (the reads of four rows ahead of
// the row in hand).  Latency is all there is to it: rows a warp reads at once
// instead of a run per thread, 32,768 items 59 -> 17 us.  Also the total into out[n] when asked.  (`in` may
// alias `out`: the second sweep reads each item before writing it.)
constexpr int kSmallThreads = 1024;
constexpr int kSmallRows = 32;   // per warp
constexpr int64_t kSmallScan = (int64_t)kSmallRows * kSmallThreads;

__global__ void __launch_bounds__(kSmallThreads)
scan_small(const int64_t *in, int64_t *out, int64_t n, int write_tot) {
    __shared__ int64_t warp_tot[kSmallThreads / 32 + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = (int)((n + kSmallThreads - 1) / kSmallThreads);
    const int64_t b0 = (int64_t)warp * rows * 32 + lane;
    int64_t loc = 0;
#pragma unroll 8
    for (int i = 0; i < rows; ++i)
        if (b0 + 32 * i < n) loc += in[b0 + 32 * i];
    const int64_t incl = warp_incl_scan(loc);
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int64_t w = warp_tot[lane];
        const int64_t wi = warp_incl_scan(w);
        warp_tot[lane] = wi - w;
        if (lane == 31) warp_tot[32] = wi;
    }
    __syncthreads();
    int64_t run = warp_tot[warp];
    for (int i = 0; i < rows; i += 4) {
        int64_t v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = i + q < rows && b0 + 32 * (i + q) < n ? in[b0 + 32 * (i + q)] : 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t s = warp_incl_scan(v[q]);
            if (i + q < rows && b0 + 32 * (i + q) < n) out[b0 + 32 * (i + q)] = run + s - v[q];
            run += __shfl_sync(0xffffffffu, s, 31);
        }
    }
    if (threadIdx.x == 0 && write_tot) out[n] = warp_tot[32];
}

gf_status scan_rec(const int64_t *in, int64_t *out, int64_t n, int64_t *scratch, cudaStream_t st,
                   bool write_tot) {
    if (n <= 0) {
        if (write_tot) GF_CUDA(cudaMemsetAsync(out, 0, sizeof(int64_t), st));
        return GF_OK;
    }
    if (n <= kSmallScan) {
        scan_small<<<1, kSmallThreads, 0, st>>>(in, out, n, write_tot ? 1 : 0);
        GF_KERNEL_DONE();
        return GF_OK;
    }
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    int64_t *sums = scratch;            // [nb]
    int64_t *offs = scratch + nb;       // [nb + 1]
    scan_tiles<<<(unsigned)nb, kScanThreads, 0, st>>>(in, out, n, sums);
    GF_KERNEL_DONE();
    GF_TRY(scan_rec(sums, offs, nb, scratch + 2 * nb + 1, st, false));
    add_tile_offsets<<<ceil_div(n, 256), 256, 0, st>>>(out, n, offs);
    GF_KERNEL_DONE();
    if (write_tot) {
        write_total<<<1, 1, 0, st>>>(out, n, offs, sums, nb);
        GF_KERNEL_DONE();
    }
    return GF_OK;
}

// -------------------------------------------------------------- radix sort
// Counts of a pass: hist[digit][block] (rows of ld entries, a multiple of 4).  All
// of a thread's keys are read before the first is counted: 2^25 keys 67 -> 30 us
// (20 us to read them); four tiles to a block, a quarter of the writes, took 78.
template <class K, int T, int R>
__global__ void __launch_bounds__(T)
radix_hist(const K *__restrict__ keys, int64_t n, int shift, int64_t ld, uint32_t *__restrict__ hist) {
    __shared__ uint32_t cnt[kRadix];
    const int64_t base = (int64_t)blockIdx.x * (T * R) + threadIdx.x;
    K k[R];
#pragma unroll
    for (int r = 0; r < R; ++r) k[r] = base + r * T < n ? keys[base + r * T] : 0;
    cnt[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (base + r * T < n) atomicAdd(&cnt[(k[r] >> shift) & 0xff], 1u);
    __syncthreads();
    hist[(int64_t)threadIdx.x * ld + blockIdx.x] = cnt[threadIdx.x];
}

// Exclusive scan of each digit's row in place, its total to tot[digit]: one block
// a digit, 1,024 counts at a time; the scatter adds the digits' own scan.  All SMs
// take part: for 262,144 keys 2.5 us where one block over all the digits' 32,768
// counts took 24; for 2^25, 8 where tiles, their sums and a sweep to add them took 23.
__global__ void __launch_bounds__(256)
radix_rows(uint32_t *__restrict__ hist, int64_t nb, int64_t ld, uint32_t *__restrict__ tot) {
    __shared__ uint32_t wsum[2][8];
    uint32_t *row = hist + (int64_t)blockIdx.x * ld;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t run = 0;
    int buf = 0;
    for (int64_t b = 0; b < nb; b += 1024, buf ^= 1) {
        const int64_t i = b + 4 * threadIdx.x;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (i < nb) {
            v = *reinterpret_cast<const uint4 *>(row + i);
            if (i + 1 >= nb) v.y = 0;
            if (i + 2 >= nb) v.z = 0;
            if (i + 3 >= nb) v.w = 0;
        }
        const uint32_t four = v.x + v.y + v.z + v.w;
        uint32_t incl = four;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[buf][warp] = incl;
        __syncthreads();
        uint32_t before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const uint32_t t = wsum[buf][w];
            if (w < warp) before += t;
            all += t;
        }
        if (i < nb) {
            uint4 o;
            o.x = run + before + incl - four;
            o.y = o.x + v.x;
            o.z = o.y + v.y;
            o.w = o.z + v.z;
            *reinterpret_cast<uint4 *>(row + i) = o;
        }
        run += all;
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = run;
}

// Stable scatter.  Each warp ranks its own run of 32 R consecutive keys, row by
// row, against its own digit counts (warp-level synchronisation only); one
// block-wide step turns the warps' counts into offsets, and the keys go out
// from registers.  Equal digits keep their relative order.  vals == nullptr:
// the values are the indices.  Bound by the scattered writes (a tile's keys of a
// digit are a run, 16 on average in the large tiles); ranking a block's row at a
// time, five block barriers to 256 keys, it was bound by those: 200 us a pass over
// 2^25 (64-bit) keys, now 124 for 32-bit ones.
template <class K, int T, int R>
__global__ void __launch_bounds__(T)
radix_scatter(const K *__restrict__ keys, const int32_t *__restrict__ vals, int64_t n, int shift, int64_t ld,
              const uint32_t *__restrict__ offs, const uint32_t *__restrict__ tot, K *__restrict__ keys_out,
              int32_t *__restrict__ vals_out) {
    constexpr int kWarps = T / 32;
    __shared__ uint32_t wcnt[kWarps][kRadix];
    __shared__ uint32_t dsum[kRadix / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = (int64_t)blockIdx.x * (T * R) + warp * (32 * R) + lane;
    const unsigned lt_mask = (1u << lane) - 1u;
    K k[R];
    int32_t v[R];
    uint32_t rank[R];
#pragma unroll
    for (int r = 0; r < R; ++r) k[r] = base + 32 * r < n ? keys[base + 32 * r] : 0;
    // thread d: where digit d's keys of this block begin
    const uint32_t mine = tot[threadIdx.x], start = offs[(int64_t)threadIdx.x * ld + blockIdx.x];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = vals && base + 32 * r < n ? vals[base + 32 * r] : (int32_t)(base + 32 * r);
    for (int d = lane; d < kRadix; d += 32) wcnt[warp][d] = 0;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const bool valid = base + 32 * r < n;
        const int d = valid ? (int)((k[r] >> shift) & 0xff) : kRadix;   // invalid -> sentinel
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t old = valid ? wcnt[warp][d] : 0;
        rank[r] = old + __popc(peers & lt_mask);
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) wcnt[warp][d] = old + __popc(peers);
        __syncwarp();
    }
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) dsum[warp] = incl;
    __syncthreads();
    {   // digit threadIdx.x: its keys of the warps before, from its own start
        uint32_t acc = start + incl - mine;
#pragma unroll
        for (int w = 0; w < kRadix / 32; ++w)
            if (w < warp) acc += dsum[w];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = acc;
            acc += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (base + 32 * r < n) {
            const uint32_t pos = wcnt[warp][(k[r] >> shift) & 0xff] + rank[r];
            keys_out[pos] = k[r];
            vals_out[pos] = v[r];
        }
}

template <class K, int T, int R>
gf_status radix_pass(const K *keys, const int32_t *vals, int64_t n, int shift, uint32_t *hist, K *keys_out,
                     int32_t *vals_out, cudaStream_t st) {
    static_assert(T == kRadix, "a thread to a digit");
    const int64_t nb = (n + T * R - 1) / (T * R), ld = (nb + 3) / 4 * 4;
    uint32_t *tot = hist + ld * kRadix;
    radix_hist<K, T, R><<<(unsigned)nb, T, 0, st>>>(keys, n, shift, ld, hist);
    GF_KERNEL_DONE();
    radix_rows<<<kRadix, 256, 0, st>>>(hist, nb, ld, tot);
    GF_KERNEL_DONE();
    radix_scatter<K, T, R><<<(unsigned)nb, T, 0, st>>>(keys, vals, n, shift, ld, hist, tot, keys_out, vals_out);
    GF_KERNEL_DONE();
    return GF_OK;
}

// -------------------------------------------------------------- bbox
// Bounding box on the integer units: a double's bits map to an unsigned key
// with the same order (negative values: all bits flipped; others: the sign
// bit set), so min/max are integer operations (FP64 is slow on this GPU)
// and the blocks combine with 64-bit atomics.
__device__ __forceinline__ unsigned long long order_key(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__global__ void __launch_bounds__(256)
bbox_keys(const double *__restrict__ p, int64_t n, unsigned long long *__restrict__ out) {
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const unsigned long long k = order_key(p[3 * i + a]);
            mn[a] = k < mn[a] ? k : mn[a];
            mx[a] = k > mx[a] ? k : mx[a];
        }
    }
    // one atomic of each kind to a block: the atomics of all warps, on six
    // addresses, took most of the 21 us of 262,144 points (now 5)
    __shared__ unsigned long long red[6][8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, mn[a], o), y = __shfl_xor_sync(0xffffffffu, mx[a], o);
            mn[a] = x < mn[a] ? x : mn[a];
            mx[a] = y > mx[a] ? y : mx[a];
        }
        if (lane == 0) {
            red[a][warp] = mn[a];
            red[3 + a][warp] = mx[a];
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        unsigned long long m = red[threadIdx.x][0];
        for (int w = 1; w < 8; ++w) {
            const unsigned long long x = red[threadIdx.x][w];
            m = threadIdx.x < 3 ? (x < m ? x : m) : (x > m ? x : m);
        }
        if (threadIdx.x < 3)
            atomicMin(out + threadIdx.x, m);
        else
            atomicMax(out + threadIdx.x, m);
    }
}

// keys back to doubles
__global__ void bbox_decode(const unsigned long long *__restrict__ k, double *__restrict__ out) {
    if (threadIdx.x < 6) {
        const unsigned long long u = k[threadIdx.x];
        out[threadIdx.x] = __longlong_as_double((long long)((u >> 63) ? (u & 0x7fffffffffffffffull) : ~u));
    }
}

__global__ void bbox_init(unsigned long long *__restrict__ k) {
    if (threadIdx.x < 6) k[threadIdx.x] = threadIdx.x < 3 ? ~0ull : 0ull;
}

}  // namespace

size_t scan_scratch_bytes(int64_t n) {
    size_t tot = 0;
    int64_t m = n;
    do {
        const int64_t nb = (m + kScanTile - 1) / kScanTile;
        tot += (size_t)(2 * nb + 1);
        m = nb;
    } while (m > 1);
    return (tot + 16) * sizeof(int64_t);
}

size_t sort_scratch_bytes(int64_t n) {
    const int64_t tile = n >= kBigSort ? kBigTile : kSmallTile;
    const int64_t ld = ((n + tile - 1) / tile + 3) / 4 * 4;
    return (size_t)(ld + 1) * kRadix * sizeof(uint32_t);
}

gf_status exclusive_scan_i64(const int64_t *in, int64_t *out, int64_t n, void *scratch, cudaStream_t st) {
    return scan_rec(in, out, n, reinterpret_cast<int64_t *>(scratch), st, true);
}

static int sort_passes(int bits) { return std::max(1, (bits + 7) / 8); }

template <class K>
K *radix_sort_input(K *keys, K *keys_alt, int bits) {
    return sort_passes(bits) % 2 ? keys_alt : keys;
}

template <class K>
gf_status radix_sort(K *keys, int32_t *vals, K *keys_alt, int32_t *vals_alt, int64_t n, int bits, void *scratch,
                     cudaStream_t st) {
    if (n <= 0) return GF_OK;
    uint32_t *hist = reinterpret_cast<uint32_t *>(scratch);
    const int passes = sort_passes(bits);
    // odd: from keys_alt; each pass crosses over, the last one into keys
    K *ka = passes % 2 ? keys_alt : keys, *kb = passes % 2 ? keys : keys_alt;
    int32_t *va = passes % 2 ? vals_alt : vals, *vb = passes % 2 ? vals : vals_alt;
    for (int ps = 0; ps < passes; ++ps) {
        const int32_t *vin = ps ? va : nullptr;
        if (n >= kBigSort)
            GF_TRY((radix_pass<K, 256, 16>(ka, vin, n, 8 * ps, hist, kb, vb, st)));
        else
            GF_TRY((radix_pass<K, 256, 8>(ka, vin, n, 8 * ps, hist, kb, vb, st)));
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    return GF_OK;
}
template uint32_t *radix_sort_input(uint32_t *, uint32_t *, int);
template uint64_t *radix_sort_input(uint64_t *, uint64_t *, int);
template gf_status radix_sort(uint32_t *, int32_t *, uint32_t *, int32_t *, int64_t, int, void *, cudaStream_t);
template gf_status radix_sort(uint64_t *, int32_t *, uint64_t *, int32_t *, int64_t, int, void *, cudaStream_t);

// Small host arrays travel to the device as kernel arguments (pieces of
// kUploadWords words), not as host-to-device copies: a plan build then
// never queues behind a large copy the caller has in flight on another
// stream, and the host memory may be reused as soon as the call returns.
namespace {
constexpr int kUploadWords = 960;
struct UploadPiece {
    uint32_t w[kUploadWords];
};
__global__ void upload_piece(UploadPiece pc, int nw, uint32_t *__restrict__ dst) {
    for (int i = threadIdx.x; i < nw; i += blockDim.x) dst[i] = pc.w[i];
}
}  // namespace

gf_status upload_small(void *dst, const void *src, size_t nbytes, cudaStream_t st) {
    if (nbytes % 4 != 0 || ((uintptr_t)dst & 3) != 0) {
        set_error("upload_small: %zu bytes to %p (whole aligned words only)", nbytes, dst);
        return GF_ERR_INVALID_ARG;
    }
    const size_t nw = nbytes / 4;
    const unsigned char *s8 = static_cast<const unsigned char *>(src);
    uint32_t *d = static_cast<uint32_t *>(dst);
    for (size_t w0 = 0; w0 < nw; w0 += kUploadWords) {
        UploadPiece pc;
        const int n = (int)std::min<size_t>(kUploadWords, nw - w0);
        memcpy(pc.w, s8 + 4 * w0, 4 * (size_t)n);
        upload_piece<<<1, 256, 0, st>>>(pc, n, d + w0);
        GF_KERNEL_DONE();
    }
    return GF_OK;
}

gf_status bbox3(const double *pts, int64_t n, double *out, cudaStream_t st) {
    // out must have room for 12 doubles: the integer keys follow the result
    if (n <= 0) return GF_OK;
    unsigned long long *k = reinterpret_cast<unsigned long long *>(out + 6);
    bbox_init<<<1, 32, 0, st>>>(k);
    GF_KERNEL_DONE();
    const int nb = (int)std::min<int64_t>(4 * 152, (n + 255) / 256);
    bbox_keys<<<nb, 256, 0, st>>>(pts, n, k);
    GF_KERNEL_DONE();
    bbox_decode<<<1, 32, 0, st>>>(k, out);
    GF_KERNEL_DONE();
    return GF_OK;
}

}  // namespace gf
