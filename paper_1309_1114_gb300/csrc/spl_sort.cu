// spl_sort.cu -- depth ordering of the tile lists for the general absorption
// form (Eq. 1 with E_p != A_p), where the particles a ray crosses must be
// taken in depth order (the sort step of Sec. 4 with a depth key).
//
// A stable least-significant-digit radix sort of 64-bit keys, digits of up to 8 bits:
// per pass, every block of kSortTile keys counts its digits (hist[digit][block]),
// one exclusive scan over the digit-major table gives every (digit, block) its
// output base, and every block scatters its keys in their original order.
// Stability inside a block: each warp owns a contiguous run of keys taken 32
// at a time; lanes holding the same digit are ranked by ballots over the digit's bits
// (a match of the lanes' digits bound the scatter: 10M depth keys 87 us a pass, 70 so),
// the warp keeps a running count per digit, and the warps' per-digit counts are
// prefixed in shared memory.
//
// Depth order of a frame: the particles are sorted by their depth key (equal depths stay
// in index order), and the tile lists are then written in that order
// (spl_raster.cu: depth_entries_kernel) and sorted, stably, by tile alone.
#include "spl_geom.cuh"

namespace spl {

constexpr int kSortThreads = 256;
// keys per thread: 8 keep the scatter at 48 registers and 5 CTAs per SM
// without spills (four passes over 10M keys and five over 30M: 3.77 ms; 16 keys, 99
// registers and 2 CTAs per SM: 4.64; 4 keys at 6 or 8 CTAs per SM: 4.12 and 3.84)
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;            // keys per block

__device__ __forceinline__ unsigned digit_of(unsigned long long k, int shift, unsigned mask) {
    return (unsigned)(k >> shift) & mask;
}

// hist[d * nblocks + b] = keys of block b with digit d.
__global__ void __launch_bounds__(kSortThreads) radix_hist_kernel(const unsigned long long *keys,
                                                                  int64_t n, int shift, unsigned mask,
                                                                  int *hist, int nblocks) {
    __shared__ int cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t b0 = (int64_t)blockIdx.x * kSortTile + threadIdx.x;
    unsigned long long key[kSortItems];            // every load before the first count
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) key[r] = b0 + r * kSortThreads < n ? keys[b0 + r * kSortThreads] : 0ull;
#pragma unroll
    for (int r = 0; r < kSortItems; ++r)
        if (b0 + r * kSortThreads < n) atomicAdd(&cnt[digit_of(key[r], shift, mask)], 1);
    __syncthreads();
    if (threadIdx.x <= mask) hist[threadIdx.x * nblocks + blockIdx.x] = cnt[threadIdx.x];
}

// Stable scatter of block b's keys to base[d * nblocks + b] + rank; the last pass
// writes the keys' low halves, the ids, to ids + *first.
template <bool LAST>
__global__ void __launch_bounds__(kSortThreads, 5) radix_scatter_kernel(const unsigned long long *in,
                                                                     unsigned long long *out,
                                                                     unsigned *ids, const long long *first,
                                                                     int64_t n, int shift, unsigned mask,
                                                                     const int *base, int nblocks) {
    constexpr int NW = kSortThreads / 32;
    __shared__ int wcnt[NW][256];      // per warp and digit: count, then offset
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int d = lane; d <= (int)mask; d += 32) wcnt[warp][d] = 0;
    __syncwarp();
    // warp w owns keys [b0 + w * 32 * kSortItems, ... + 32 * kSortItems), in
    // rounds of 32 consecutive keys
    const int64_t w0 = (int64_t)blockIdx.x * kSortTile + (int64_t)warp * 32 * kSortItems;
    unsigned long long key[kSortItems];
    int rnk[kSortItems];
    // all of the warp's keys are loaded before the ranking rounds, whose warp
    // barriers would otherwise serialise the loads' latencies
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t i = w0 + r * 32 + lane;
        key[r] = i < n ? in[i] : 0ull;
    }
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t i = w0 + r * 32 + lane;
        const bool valid = i < n;
        const int d = valid ? (int)digit_of(key[r], shift, mask) : -1;
        // the lanes with this lane's digit, a ballot per bit
        unsigned m = __ballot_sync(0xffffffffu, valid);
        for (unsigned bit = 1; bit <= mask; bit <<= 1) {
            const unsigned v = __ballot_sync(0xffffffffu, d & bit);
            m &= d & bit ? v : ~v;
        }
        int before = 0;
        if (valid) before = wcnt[warp][d];
        rnk[r] = before + __popc(m & lt);
        __syncwarp();
        if (valid && lane == __ffs(m) - 1) wcnt[warp][d] = before + __popc(m);
        __syncwarp();
    }
    __syncthreads();
    // per digit: offsets of the warps inside the block, plus the block's base
    if (threadIdx.x <= mask) {
        const int d = threadIdx.x;     // kSortThreads == 256 digits at most
        int run = base[d * nblocks + blockIdx.x];
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int c = wcnt[w][d];
            wcnt[w][d] = run;
            run += c;
        }
    }
    __syncthreads();
    if (LAST && first) ids += *first;
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t i = w0 + r * 32 + lane;
        if (i >= n) continue;
        const int to = wcnt[warp][digit_of(key[r], shift, mask)] + rnk[r];
        if (LAST)
            ids[to] = (unsigned)key[r];
        else
            out[to] = key[r];
    }
}

int radix_blocks(int64_t n) { return (int)((n + kSortTile - 1) / kSortTile); }

// Exclusive scan of m ints for the digit table: blocks of kScanChunk values
// are reduced, the block sums scanned by one CTA (scan_kernel), and every
// block then scans its values from its base.  out[m] = total.
constexpr int kScanThreads = 1024, kScanPer = 8, kScanChunk = kScanThreads * kScanPer;

__device__ __forceinline__ int block_exclusive(int v, int *wsum, int &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int w = wsum[lane];
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += u;
        }
        wsum[lane] = wi - w;
        if (lane == 31) wsum[32] = wi;
    }
    __syncthreads();
    total = wsum[32];
    const int r = wsum[warp] + incl - v;
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const int *in, int m, int *part) {
    __shared__ int wsum[33];
    const int base = blockIdx.x * kScanChunk + threadIdx.x * kScanPer;
    int v = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k)
        if (base + k < m) v += in[base + k];
    int total;
    block_exclusive(v, wsum, total);
    if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(const int *in, int m,
                                                                  const int *pbase, int nparts,
                                                                  int *out) {
    __shared__ int wsum[33];
    const int base = blockIdx.x * kScanChunk + threadIdx.x * kScanPer;
    int v[kScanPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        v[k] = base + k < m ? in[base + k] : 0;
        sum += v[k];
    }
    int total;
    int run = pbase[blockIdx.x] + block_exclusive(sum, wsum, total);
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (base + k < m) out[base + k] = run;
        run += v[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) out[m] = pbase[nparts];
}

static int scan_parts(int m) { return (m + kScanChunk - 1) / kScanChunk; }

// Ints of radix scratch for n keys: digit counts, scanned bases, block sums.
int64_t radix_scratch_ints(int64_t n) {
    const int64_t nb = radix_blocks(n > 0 ? n : 1);
    const int64_t parts = scan_parts((int)(256 * nb));
    return 512 * nb + 2 + 2 * (parts + 1);
}

// part: 2 (m / kScanChunk + 2) ints.  A small table in one launch: the three of a large
// one are most of a small sort's time (21k particles: the sort 0.24 ms, 0.13 so).
constexpr int kFewDigits = 16384;
void launch_wide_scan(int m, const int *in, int *out, int *part, cudaStream_t s) {
    if (m <= kFewDigits) {
        launch_scan(m, in, out, s);
        return;
    }
    const int np = scan_parts(m);
    int *pbase = part + np + 1;
    scan_reduce_kernel<<<np, kScanThreads, 0, s>>>(in, m, part);
    ++g_launches;
    launch_scan(np, part, pbase, s);
    scan_apply_kernel<<<np, kScanThreads, 0, s>>>(in, m, pbase, np, out);
    ++g_launches;
}

// Sorts keys[0, n) by their bits [shift, shift + bits), in passes of at most eight of
// them, and writes the low halves of the sorted keys to ids + *first (first null: ids); tmp
// holds n keys (keys and tmp are both overwritten); hist holds radix_scratch_ints(n) ints.
static void radix_sort_ids(unsigned long long *keys, unsigned long long *tmp, int64_t n, int shift,
                           int bits, unsigned *ids, const long long *first, int *hist, cudaStream_t s) {
    const int passes = bits > 8 ? (bits + 7) / 8 : 1, per = bits > passes ? (bits + passes - 1) / passes : 1;
    const unsigned mask = (1u << per) - 1u;
    const int nb = radix_blocks(n);
    const int m = (int)(mask + 1u) * nb;
    int *cnt = hist, *bases = hist + m + 1, *part = bases + m + 1;
    for (int p = 0; p < passes; ++p, shift += per) {
        radix_hist_kernel<<<nb, kSortThreads, 0, s>>>(keys, n, shift, mask, cnt, nb);
        ++g_launches;
        launch_wide_scan(m, cnt, bases, part, s);
        if (p == passes - 1)
            radix_scatter_kernel<true><<<nb, kSortThreads, 0, s>>>(keys, nullptr, ids, first, n, shift,
                                                                   mask, bases, nb);
        else
            radix_scatter_kernel<false><<<nb, kSortThreads, 0, s>>>(keys, tmp, nullptr, nullptr, n, shift,
                                                                    mask, bases, nb);
        ++g_launches;
        unsigned long long *t = keys;
        keys = tmp;
        tmp = t;
    }
}

// ---------------------------------------------------------------------------
// Depth order of a frame.
// ---------------------------------------------------------------------------

// Particle keys: (float bits of the depth key) << 32 | index; the depth key is
// positive for every active particle (z_c > z_near > 0), so its bits order as
// the value.  Inactive or non-absorbing records go last.
__global__ void depth_keys_kernel(const float2 *rec2, int64_t n, unsigned long long *keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float2 q = rec2[i];                  // (A, depth key); A = 0 where inactive
        const unsigned hi = q.x > 0.f ? __float_as_uint(q.y) : 0xFFFFFFFFu;
        keys[i] = ((unsigned long long)hi << 32) | (unsigned long long)(unsigned)i;
    }
}

static int bits_for(unsigned long long v) {
    int b = 0;
    while (b < 64 && (v >> b) != 0ull) ++b;
    return b;
}

// The tile lists of one view, all its entries in the medium list slots off[0 .. ntiles]
// (device offsets into entries; the host passes their total, off[ntiles] - off[0], known
// after the binning synchronisation), front to back in every tile.  The particles are
// sorted by depth, their (tile, particle) keys written in that order, and the keys sorted
// by tile, stably: lists filled in any order and sorted by (tile, depth rank) took five
// passes over the entries where this takes two, and three kernels to make and undo the
// ranks (clustered 10M / 1024^2 from the counts to the sorted lists: 2.98 -> 1.20 ms; with
// 16-pixel tiles, 79M entries: 6.29 -> 1.81 ms).
// pkeys/ptmp: n particle keys each; ekeys/etmp: total entry keys each; by_depth: n ids;
// hist: radix_scratch_ints(max(n, total)) ints.
void launch_depth_order(const Views &vs, const Rec *recs, const float2 *rec2, unsigned *entries,
                        const long long *off, int ntiles, long long total, unsigned long long *pkeys,
                        unsigned long long *ptmp, unsigned long long *ekeys, unsigned long long *etmp,
                        unsigned *by_depth, int *hist, DevStats *st, int sms, cudaStream_t s) {
    const int64_t n = vs.n;
    if (n <= 0 || total <= 0) return;
    depth_keys_kernel<<<sms * 8, 256, 0, s>>>(rec2, n, pkeys);
    ++g_launches;
    // the keys start in index order and every pass is stable, so sorting by
    // the depth bits alone leaves equal depths in index order: the index bits
    // need no passes of their own
    radix_sort_ids(pkeys, ptmp, n, 32, 32, by_depth, nullptr, hist, s);
    launch_depth_entries(vs, recs, by_depth, ekeys, total, hist, st, s);
    radix_sort_ids(ekeys, etmp, total, 32, bits_for((unsigned long long)(ntiles - 1)), entries, off, hist, s);
}

}  // namespace spl
