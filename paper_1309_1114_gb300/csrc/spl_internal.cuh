// spl_internal.cuh -- shared declarations of the GB300 Splotch renderer.
//
// Data layout in HBM (one frame):
//   particles   SoA: x, y, z (FP32) and h, I, s (FP32 or binary16), owned by the
//               context, read once per frame by the rasteriser.
//   records     one 32-byte Rec per particle id (and view):
//                 r0 = { packed (xi, yi) as two int16, xf, yf, kq }
//                 r1 = { r^2 (negative when inactive), e_R, e_G, e_B }
//               where x_s = xi + xf with xf in [0, 1) (the integer part keeps
//               the sub-pixel position exact to ~1e-7 px in FP32) and
//               kq = log2(e) / sigma_s^2, so exp(-d^2/sigma^2) = 2^(-kq d^2).
//   counts      int32 [NLIST][n_tiles]: entries per (list, tile), then an
//               exclusive scan into offsets [NLIST * n_tiles + 1].
//   entries     uint32 particle ids, grouped by list, then by tile.
//   image       caller-owned H x W x 3 FP32.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace spl {

// Lists a particle can be binned into (Sec. 4 classes by screen radius).
enum : int { L_POINT = 0, L_SMALL = 1, L_MEDIUM = 2, L_LARGE = 3, NLIST = 4 };
enum : int { CLS_INACTIVE = -2, CLS_POINT = 0, CLS_SMALL = 1, CLS_MEDIUM = 2, CLS_LARGE = 3 };

// Device-side error bits (reported as SPL_EDEVICE).
enum : unsigned { ERR_LIST_OVERFLOW = 1u, ERR_INDEX = 2u };

constexpr int kMaxPalette = 1024;
constexpr int kTileThreads = 256;        // 8 warps per tile CTA

// Per-frame constants (camera in double-float: hi + lo pairs of FP32).
struct FrameConst {
    float2 Rxy_hi[3], Rxy_lo[3];   // columns of the rows (right, up')
    float2 Exy_hi, Exy_lo;         // those rows times the eye
    float2 f2_hi, f2_lo;           // focal length, (f, -f): y_s grows downwards
    float2 half;                   // (width / 2, height / 2)
    float Rz_hi[3], Rz_lo[3];      // row fwd
    float Ez_hi, Ez_lo;
    float fhi;                     // focal length rounded to float
    float z_near;
    float sig_fac;             // sigma_per_h / s_box
    float chi;
    float r_sml2, r_small2, r_large2;   // squared class radii
    float s_min, s_inv;        // colour-scalar normalisation
    float brightness;
    int npal;
    int width, height;
    int tile, ntx, nty, ntiles;
    int tile_shift;            // log2(tile)
    // place of this view in a batch of views
    int view;                  // index in the batch
    int tile_base;             // first global tile: global tile = tile_base + local tile
    int slot_base;             // first list slot: slot = slot_base + list * ntiles + tile
    int absorb;                // general absorption (Eq. 1, E != A): one depth-sorted list per tile
    float absorption;          // A = absorption * brightness * I
    int log_flags;             // 1: log10 of I, 2: log10 of s before normalisation
    long long rec_base;        // first record: record = rec_base + particle id
};

// Kernels launched by this host thread: every launch site adds one, and a
// render reports the difference across its own launches.
extern thread_local long long g_launches;

// A batch of views rendered together: one particle set, nviews cameras.
// Per-view constants live in device memory; the tile side is common.
constexpr int kMaxViews = 64;
struct Views {
    const FrameConst *fcs;     // device, nviews entries
    int nviews;
    int total_tiles;           // sum over views of ntiles
    int tile;                  // common tile side
    int64_t n;                 // particles
};

// Device status block (one per context).
// Everything before `err` is cleared at the start of every frame; `err`
// accumulates until the host reads and clears it.
struct DevStats {
    unsigned long long n_active, n_point, n_small, n_medium, n_large;
    unsigned int n_large_ids;  // large records appended this frame
    int totals[NLIST];         // entries per list, summed over views
    long long slot_total;      // all entries (written by the slot scan)
    int item_totals[2];        // work items of the tile pass and of the large pass
    int item_counter[3];       // dynamic work-item counters of the two passes and the covering pass
    unsigned int err;          // ERR_* bits
};

// A work item of the persistent tile / large passes: a tile (global index
// over the batch) and a range of one of its lists, or every list of a tile
// light enough to be done by one CTA, which then stores its pixels instead of
// adding them (its range is the tile's medium list).  lv packs the view (high
// bits), whether the item is its tile's only large item (kSole), and the list
// (low 7 bits, kAllLists for "every list").
struct WorkItem {
    int tile, lv;
    long long start, end;
};
constexpr int kAllLists = 0x7F, kSole = 0x80;
__host__ __device__ inline int item_view(const WorkItem &w) { return w.lv >> 8; }
__host__ __device__ inline bool item_sole(const WorkItem &w) { return (w.lv & kSole) != 0; }
__host__ __device__ inline int item_list(const WorkItem &w) {
    return (w.lv & kAllLists) == kAllLists ? -1 : (w.lv & kAllLists);
}

// Largest list segment one work item takes (per list), so that a crowded
// tile (a halo core holding 1e5-1e6 particles) is spread over many CTAs.
constexpr int kSegPoint = 8192, kSegSmall = 2048, kSegMedium = 1024, kSegLarge = 512;
// A frame with less than two such segments for each CTA of the persistent passes
// leaves most of them idle (200k particles on 256^2: 64 tiles, one item each, tile
// pass 0.064 ms).  There the segments shrink with the frame's entries, down to
// 1/8 of the above: two batches of the tile pass (0.047 ms; 1/4 and 1/16 within 5 %).
constexpr int kSegShrink = 8;
struct Segs {
    int len[NLIST];
};

// Binning CTAs: each takes kChunk consecutive particles and aggregates their
// list slots in a shared-memory hash table of kHash slots, which the scatter
// reuses (one table per CTA and view).
constexpr int kHashBits = 11;
constexpr int kHash = 1 << kHashBits;
constexpr int kChunk = 2048;
// Sets that give the SMs less than kFewChunks CTAs of that size go through half chunks
// with half tables, and those that give them less than kQuarter through quarters: a CTA takes
// its chunk 256 particles at a time, so that a longer chunk is a longer chain (200k
// particles: raster 0.032 -> 0.022, lists 0.043 -> 0.029 ms in quarters; 1.3M clustered: 0.107 ->
// 0.079, 0.163 -> 0.098 in halves), but every table adds each of its slots to the global counts
// (10M: raster 0.369 ms, 0.588 in quarters; the two meet near 3M).  1.3M in quarters and
// halves: clustered frame 1.084 and 1.097 ms, uniform 0.781 and 0.676; 1.7M clustered 0.338 and 0.312.
struct BinShape {
    int chunk, hash_bits;
};
constexpr int kFewChunks = 10, kQuarter = 3;
__host__ __device__ inline BinShape bin_shape(int64_t n, int sms) {
    if (n < (int64_t)sms * kQuarter * kChunk) return BinShape{kChunk / 4, kHashBits - 2};
    return n < (int64_t)sms * kFewChunks * kChunk ? BinShape{kChunk / 2, kHashBits - 1}
                                                  : BinShape{kChunk, kHashBits};
}
__host__ __device__ constexpr int64_t ctab_entries(int64_t n, int nviews) {
    return ((n + kChunk - 1) / kChunk > 0 ? (n + kChunk - 1) / kChunk : 1) *
           (nviews > 0 ? nviews : 1) * kHash;
}

// One rasterised particle: r0 = (packed pixel xi, yi; sub-pixel xf, yf;
// 1 / (sigma^2 ln 2)), r1 = (r^2; e_R, e_G, e_B).  The two halves sit in one
// 32-byte record, so that a gather through a tile list reads one sector.
struct Rec {
    float4 r0, r1;
};
static_assert(sizeof(Rec) == 32, "32-byte records");

struct RasterArgs {
    int64_t n;
    const float *x, *y, *z;
    const void *h, *I, *s;
    const float *pal;          // npal * 3
    const float *cr, *cg, *cb; // optional per-particle colour components (replace the palette)
    float h_log2_min;          // ATTR 3: h = 2^(h_log2_min + code / 4096)
    Rec *recs;                 // nviews * n records
    float2 *rec2;              // absorption mode: (A, depth key) per record, else null
    int *counts;               // list slots of all views: entries counted through the CTA tables
    int *ovf;                  // list slots: entries placed through the cursors (see BinArgs)
    int2 *ctab;                // per (CTA, view): the CTA hash table, (slot, offset in the slot)
    unsigned *large_ids;       // record indices, capacity nviews * n
    DevStats *st;
    BinShape shape;
};

// A list slot's range [offsets[k], offsets[k+1]) holds first the entries
// whose place the rasteriser's CTA tables fixed (counts[k] of them: CTA b's
// share starts at offsets[k] + its table's offset), then the entries placed
// one warp group at a time through cursor[k] = offsets[k] + counts[k]: those
// of keys that found no room in a CTA table, and the large list (ovf[k]).
struct BinArgs {
    const Rec *recs;
    const unsigned *large_ids;
    long long *cursor;         // list slots, starts at offsets + counts
    int *full;                 // per tile: large entries that cover it, placed from the list's end
    int *counts;
    int *ovf;
    const long long *offsets;
    const int2 *ctab;
    unsigned *entries;         // record indices
    int64_t entries_cap;
    DevStats *st;
    BinShape shape;
};

struct TileArgs {
    const Rec *recs;
    const long long *offsets;  // list slots of all views, + 1 (64-bit list positions)
    const unsigned *entries;
    long long entries_cap;     // a replayed graph's lists may end beyond it (then flagged)
    const WorkItem *items;
    int items_cap;
    float *const *images;      // device array: one image per view
    DevStats *st;
    const int *order;          // optional: processing order of each pass's items
    long long *item_cycles;    // optional: SM clock cycles spent on each item
    int accumulate;            // add into the images instead of storing (streamed chunks)
    const int *full;           // per tile: entries at the end of its large list that cover it
    int cover;                 // large pass: those go through the covering pass
    const float2 *rec2;        // absorption mode: per record (A, depth key)
    float4 *partial;           // absorption mode: (C, T) per pixel of every split item
    float *front;              // absorption mode, optional: per segment, how much it lets through
};

// Tile-cost network 32 -> 64 (ReLU) -> 1; parameter vector layout
// W1[64][32] row-major, b1[64], w2[64], b2.
constexpr int kFeat = 32, kHid = 64;
constexpr int kNParam = kHid * kFeat + 2 * kHid + 1;

// Launchers (stream-ordered, no synchronisation).  Every count the kernels
// need after binning (entries, work items) is read from device memory, so
// the whole sequence can be captured in a CUDA graph.
void launch_raster(const Views &v, RasterArgs a, int attr, int sms, cudaStream_t s);
void launch_count_large(const Views &v, const BinArgs &a, int sms, cudaStream_t s);

// The start of a frame: zeroes the slot counts and the frame's statistics; a single
// view's constants and image (fcs not null) are written from the arguments.
struct SetupArgs {
    FrameConst fc;
    float *image;
    FrameConst *fcs;           // device, or null: copied by the caller
    float **images;
    int *counts, *ovf, *full;  // full: a quarter as many
    int slots;
    DevStats *st;
};
void launch_setup(const SetupArgs &a, int sms, cudaStream_t s);

// Slot counts and ovf to list offsets, cursors, item offsets ([tile-pass items | large
// items]) and the totals in st.  sms > 0: segments shrink on small frames (see
// kSegShrink); 0: full segments.  part: slot_parts(total_tiles) values of scratch.
struct SlotArgs {
    const int *counts, *ovf;
    long long *offsets, *cursor, *part;
    int *item_counts, *item_offsets;
    DevStats *st;
};
void launch_slots(const Views &v, const SlotArgs &a, int sms, cudaStream_t s);
size_t slot_parts(int tiles);

// Exclusive scan of in[0..m) into out[0..m] (out[m] = total).
void launch_scan(int m, const int *in, int *out, cudaStream_t s);
void launch_wide_scan(int m, const int *in, int *out, int *part, cudaStream_t s);

// The tile lists, the work items and (zero) the cleared images.  The caller fills the
// first five fields of l.
struct ListArgs {
    const int *item_offsets;
    WorkItem *items;
    int items_cap, seg_sms;
    float *const *images;
    int large_blocks, item_blocks, zero_blocks;
    bool scatter = true;          // fill the lists of points, small and medium particles
};
void launch_lists(const Views &v, BinArgs a, ListArgs l, bool zero, int sms, cudaStream_t s);
void launch_tile_pass(const Views &v, const TileArgs &a, int sms, cudaStream_t s);
// The covering pass starts twice as many items as the large pass alone; it pays where a
// tile's large list is long (687k heavy-tailed particles, 20 large entries per tile:
// large pass 0.072 ms without it, 0.096 with; 100M, 1227 per tile: 4.96 and 3.44 ms).
inline bool cover_pays(long long large_entries, int tiles, int tile) {
    return tile > 16 && large_entries >= 64LL * tiles;
}
void launch_large_pass(const Views &v, const TileArgs &a, int sms, cudaStream_t s);
// The absorption mode's segments in the order of their depth, and what lies in front of
// each; worth it once more segments than are worked on at a time follow others (3542
// segments of 290 tiles: absorb and composition 1.40 ms without it, 0.70 with; 640 of 85: 0.154 and
// 0.156).
inline bool front_pays(int items, int tiles, int sms) { return items >= tiles + 3 * sms; }
// the cost whose bucket in the order of the items is b (up to 255)
__host__ __device__ inline float bucket_cost(int b) { return 25.f - ((float)(b < 255 ? b : 255) + 0.5f) / 12.8f; }
void launch_segment_order(const TileArgs &a, const int *item_offsets, int tile, float *cost, cudaStream_t s);
// Absorption mode: the depth-ordered pass and the composition of split tiles.
void launch_absorb_pass(const Views &v, const TileArgs &a, const int *item_offsets, int sms,
                        cudaStream_t s);
int radix_blocks(int64_t n);
int64_t radix_scratch_ints(int64_t n);
void launch_depth_order(const Views &vs, const Rec *recs, const float2 *rec2, unsigned *entries,
                        const long long *off, int ntiles, long long total, unsigned long long *pkeys,
                        unsigned long long *ptmp, unsigned long long *ekeys, unsigned long long *etmp,
                        unsigned *by_depth, int *hist, DevStats *st, int sms, cudaStream_t s);
void launch_depth_entries(const Views &vs, const Rec *recs, const unsigned *by_depth,
                          unsigned long long *keys, long long total, int *counts, DevStats *st,
                          cudaStream_t s);
void launch_epilogue_ea(float *image, int64_t nvals, int sms, cudaStream_t s);
// FP32 attributes h, I, s into storage layout `store` (SPL_ATTR_* value).
void launch_encode_attrs(const float *h, const float *I, const float *s, int64_t n, int store,
                         float h_log2_min, void *ho, void *Io, void *so, int sms, cudaStream_t st);
// cursor[k] = offsets[k] + counts[k] for the m list slots, full = 0 (re-arms the scatter).
void launch_slot_cursor(int m, const int *counts, const long long *offsets, long long *cursor,
                        int *full, cudaStream_t s);
// Apply the E=A map to every view's image (the image pointers are read from
// device memory, so a graph can replay them).
void launch_epilogue_views(const Views &v, float *const *images, int sms, cudaStream_t s);
void launch_count_work(const FrameConst &fc, const Rec *recs, int64_t n,
                       unsigned long long *work, int sms, cudaStream_t s);

// Scheduling of the work items (spl_sched.cu): per-item features, predicted
// cost (network or count heuristic), and a longest-first order per pass.
void launch_item_entries(const Views &v, const TileArgs &a, int *n_entries, int sms,
                         cudaStream_t s);
void launch_item_features(const Views &v, const TileArgs &a, float area_scale, int max_sample,
                          float *feat, int *n_entries, int sms, cudaStream_t s);
void launch_item_cost(const float *feat, const int *n_entries, const float *theta,
                      const float *heur, int items_cap, const DevStats *st, float *cost,
                      cudaStream_t s);
void launch_order_items(const float *cost, int items_cap, DevStats *st, int *hist, int *order,
                        cudaStream_t s);

// Network kernels (spl_mlp.cu); B samples, features row-major [B][32].
void launch_mlp_forward(const float *theta, const float *x, int64_t B, float *y, cudaStream_t s);
void launch_mlp_loss_grad(const float *theta, const float *x, const float *t, int64_t B,
                          float *work, float *grad, float *loss, cudaStream_t s);
void launch_mlp_adam(float *theta, const float *grad, float *m, float *v, int64_t np, int64_t step,
                     float lr, float b1, float b2, float eps, cudaStream_t s);
// One CTA's partial gradient and loss, and the CTAs of a gradient pass.
constexpr int kGradRow = kNParam + 3, kGradBlocks = 152;
size_t mlp_work_floats();
// logc[k] = log(cycles[k]) (cycles clamped to >= 1).
void launch_log_cycles(const long long *cycles, int64_t n, float *logc, cudaStream_t s);

// View of a global tile index (binary search over the views' tile bases).
__device__ __forceinline__ int view_of_tile(const FrameConst *fcs, int nviews, int g) {
    int lo = 0, hi = nviews - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (fcs[mid].tile_base <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace spl
