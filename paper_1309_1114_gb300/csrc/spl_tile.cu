// spl_tile.cu -- the rendering passes (Sec. 4.1-4.3 and Eq. 2).
//
// Work is cut into items: a T x T tile of the image (the tiling of Eq. 8)
// together with its lists, or -- for a crowded tile, the load imbalance of
// the Remarks of Sec. 4 -- a bounded segment of one of its lists.  Persistent
// CTAs take items from a device counter.  A tile that is one item is written
// by exactly one CTA with plain stores; the segments of a crowded tile add
// their partial tiles into the (zeroed) image with one atomic add per pixel
// and channel, instead of one per contribution (the write races of
// Sec. 3.2.2 / Fig. 3).
//
// Inside an item a warp owns 16 x 8 pixels (two 8 x 8 blocks, see Quad), each lane a few
// of them, and keeps its pixels' three channels in registers.  Then:
//   - point particles (r <= r_sml, Sec. 4.1) add their emission to one pixel
//     of a shared-memory copy of the tile; lanes of a warp that hit the same
//     pixel are summed with warp shuffles first;
//   - small particles (r_sml < r <= r_small, a few pixels wide): one thread
//     per particle walks the particle's pixel box, into shared memory;
//   - medium and large particles are taken in batches (the chunks of n_p
//     particles of Sec. 4.2): the CTA first tabulates, per particle, the
//     column weights w_x(i) = exp(-dx^2/sigma^2) and the row terms
//     e * w_y(j) (Eq. 2 is separable: exp(-(dx^2+dy^2)/sigma^2) = w_x w_y),
//     then every warp whose blocks the particle reaches adds
//     e * w_y * w_x into its registers: three FMAs per pixel, plus a clip
//     test folded into one saturating add on the FMA pipe (see below); two
//     rows go through one packed FP32x2 instruction (the row table is laid
//     out in row pairs);
//   - finally each thread adds the shared-memory part to its registers and
//     writes its pixels once.
// The large pass (r > r_large, Sec. 4.3) runs after the tile pass with the
// same scheme over segments of the tiles' large lists and adds its partial
// tiles into the image; tiles that lie wholly inside a disc go through the
// covering pass.
//
// Clip (Eq. 2: zero beyond chi*sigma).  With B = 2^20 / r^2 the tables hold
// dx^2 * B per column and (r^2 - dy^2) * B + 1 per row; the clip factor is
// m = saturate((r^2 - dy^2) B + 1 - dx^2 B), which is exactly 1 inside the
// disc and exactly 0 outside it, except for pixels whose distance lies within
// r * (1 + 5e-7) -- inside the band where FP32 and FP64 may legitimately
// disagree on an inclusive clip test anyway.
#include "spl_tile.cuh"

namespace spl {

// One small particle (a few pixels wide) into the shared tile, by one thread:
// the pixel box inside the tile, the clip test and the weight of Eq. 2 per
// pixel, and one shared-memory add per channel.  A tiny splat costs a few
// pixels of work here instead of a batch-table share and a band visit.
template <int W>
__device__ __forceinline__ void thread_small(const FrameConst &fc, float4 r0, float4 r1, int x0,
                                             int y0, float (*sacc)[W][W]) {
    PixBox b;
    if (!splat_box(fc, r0, r1.x, b)) return;
    const int i0 = max(b.i0, x0), i1 = min(b.i1, x0 + W - 1);
    const int j0 = max(b.j0, y0), j1 = min(b.j1, y0 + W - 1);
    const int xi = unpack_xi(r0.x), yi = unpack_yi(r0.x);
    const float xh = 0.5f - r0.y, yh = 0.5f - r0.z;
    const float kq = r0.w, r2 = r1.x;
    for (int j = j0; j <= j1; ++j) {
        const float dy = (float)(j - yi) + yh;
        const float rem = r2 - dy * dy;
        for (int i = i0; i <= i1; ++i) {
            const float dx = (float)(i - xi) + xh;
            const float dx2 = dx * dx;
            if (dx2 <= rem) {
                const float w = ex2_neg(kq * (dx2 + dy * dy));
                atomicAdd(&sacc[0][j - y0][i - x0], r1.y * w);
                atomicAdd(&sacc[1][j - y0][i - x0], r1.z * w);
                atomicAdd(&sacc[2][j - y0][i - x0], r1.w * w);
            }
        }
    }
}

// Points of one warp, one record (r0, r1) per valid lane: lanes that hit the
// same pixel are summed inside the warp first (match + shuffles), then one lane adds.
// The points belong to the T-pixel tile at (tx0, ty0); those in the W-pixel part of it
// at (x0, y0) are added.
template <int T, int W>
__device__ __forceinline__ void warp_points(const TileArgs &a, bool valid, float4 r0, float4 r1,
                                            int tx0, int ty0, int x0, int y0, float (*sacc)[W][W],
                                            int lane) {
    int key = -1;
    float er = 0.f, eg = 0.f, eb = 0.f;
    int i = 0, j = 0;
    if (valid) {
        i = unpack_xi(r0.x) - x0;
        j = unpack_yi(r0.x) - y0;
        if ((unsigned)i < (unsigned)W && (unsigned)j < (unsigned)W) {
            key = j * W + i;
            er = r1.y; eg = r1.z; eb = r1.w;
        } else if ((unsigned)(i + x0 - tx0) >= (unsigned)T || (unsigned)(j + y0 - ty0) >= (unsigned)T) {
            atomicOr(&a.st->err, ERR_INDEX);      // outside its tile, not just this part of it
        }
    }
    const unsigned m = __match_any_sync(0xffffffffu, key);
    if (__any_sync(0xffffffffu, key >= 0 && __popc(m) > 1)) {
        float sr = 0.f, sg = 0.f, sb = 0.f;
        for (int q = 0; q < 32; ++q) {
            const float vr = __shfl_sync(0xffffffffu, er, q);
            const float vg = __shfl_sync(0xffffffffu, eg, q);
            const float vb = __shfl_sync(0xffffffffu, eb, q);
            if ((m >> q) & 1u) { sr += vr; sg += vg; sb += vb; }
        }
        er = sr; eg = sg; eb = sb;
    }
    if (key >= 0 && lane == __ffs(m) - 1) {
        atomicAdd(&sacc[0][j][i], er);
        atomicAdd(&sacc[1][j][i], eg);
        atomicAdd(&sacc[2][j][i], eb);
    }
}

// ---------------------------------------------------------------------------
// Quarter-warp splatting over 8 x 8 blocks.  A warp owns two adjacent 8 x 8
// blocks of the tile; two of its quarter-warps take two particles of the left
// block's list at a time, the other two two of the right block's, a lane holding
// 4 x 2 pixels of its block.  The two quarters of a block are added at the end of
// the item.
//
// What bounds it: the shared-memory data pipe (76 % of its peak on the clustered
// 10M / 1024^2 frame; issue slots 63 %, FMA pipe 58 %).  One particle per warp step
// over a 16 x 8 band, a lane 2 x 2 pixels, took 8 wavefronts per 128 pixels at 54 %
// covered pixels: 28.7 shared-load wavefronts and 128 instructions per list entry, the pipe at 81 %.
// 8 x 8 blocks are covered to 65 %, and a lane's eight pixels share its four 16-byte loads
// (12 wavefronts per 256 pixels): 20.5 wavefronts and 102 instructions.  Tile pass of that
// frame 4.58 -> 3.84 ms.  Also measured there: a lane 4 x 4 pixels of a 16 x 8 band
// (fewest wavefronts, but 48 accumulators leave 16 warps per SM: 4.65), the same with
// producer warps and an mbarrier ring (4.50), 3 CTAs per SM (4.55), the clip as
// compare and select on the ALU pipe for half or all of the columns (3.87, 4.12).
// ---------------------------------------------------------------------------
//
// W is the side of the pixels a CTA works on: 32 for 32-pixel tiles (8 warps, 16 blocks);
// a 64-pixel tile is four such parts, each its own piece of work over the same list
// (particles that miss the part are not tabulated), added to the image by atomics; 16 for 16-pixel tiles, whose two
// pairs of blocks are shared by four warps each, a warp taking 16 of a batch's 64
// particles.  A lane per pixel over 16 x 2 bands (16), and 64 x 8 bands with 128
// registers (64), took 7.98 and 8.69 ms on the clustered 10M / 1024^2 frame; these
// take 4.39 and 5.95.
template <int W>
struct Quad {
    static constexpr int P = 64;                   // particles per batch
    // one particle's tables: W / 2 column pairs (w_a, w_b, dx_a^2 B, dx_b^2 B), W / 2 row
    // pairs (e_R w_a, e_R w_b, e_G w_a, e_G w_b), W / 2 row pairs (e_B w_a, e_B w_b, rem_a,
    // rem_b); the 16 bytes of padding and the slot order put neighbouring particles in
    // different banks
    static constexpr int ROWA = 8 * W, ROWB = 16 * W, BYTES = 24 * W + 16;
    __device__ static __forceinline__ unsigned slot(int p) {
        return (unsigned)((p & ~7) | ((p & 1) << 2) | ((p >> 1) & 3));
    }
    static constexpr int BL = W / 8;               // blocks along a side
    static constexpr int BANDS = BL * BL / 2;      // pairs of blocks, one per warp
    static constexpr int G = 8 / BANDS;            // warps per pair
    static constexpr int kNone = P * BYTES;        // tables of a particle that adds nothing
    static constexpr int kStage = kNone + BYTES;   // two batches of records
    static constexpr int kMask = kStage + 2 * P * 32;   // per block: the particles that reach it
    static constexpr int kLists = kMask + 16 * 8;
    static constexpr int LIST = 72;                // a block's particles (slots), padded
    static constexpr int kSmem = kLists + 16 * LIST;
    // the shared tile of the points and small particles, then (G > 1) the warps' partial
    // sums, reuse the tables
    static constexpr int kPart = 12 * W * W;
    static_assert(kPart + (G > 1 ? G * 12 * W * W : 0) <= kNone, "the tables hold both");
    static_assert(W == 16 || 12 * 64 * 64 <= kNone, "the tables hold a 64-pixel tile");
};

// Tabulate particle (r0, r1) into the block tab: thread q of its four fills
// column pairs and row pairs q, q + 4, ....  Pixel offsets are exact
// integers plus the sub-pixel part; two columns (rows) go through one packed
// FP32x2 instruction.  B only needs to be the same on both sides of the clip
// test, so a fast reciprocal serves.
template <int W>
__device__ __forceinline__ void quad_tabulate(float4 r0, float4 r1, int x0, int y0, unsigned tab,
                                              int q) {
    const float B = __fdividef(1048576.f, r1.x);
    const f32x2 nkq = pack2(-r0.w, -r0.w), B2 = pack2(B, B);
    const float xf = (float)(x0 - unpack_xi(r0.x) + 2 * q), yf = (float)(y0 - unpack_yi(r0.x) + 2 * q);
    const f32x2 x2 = pack2(xf, xf + 1.f), y2 = pack2(yf, yf + 1.f);
    const f32x2 xh = pack2(0.5f - r0.y, 0.5f - r0.y), yh = pack2(0.5f - r0.z, 0.5f - r0.z);
    const unsigned at = tab + 16 * q;
#pragma unroll
    for (int u = 0; u < W / 8; ++u) {
        const f32x2 d = add2(add2(x2, pack2(8.f * u, 8.f * u)), xh);
        const f32x2 d2 = mul2(d, d);
        float ta, tb, wa, wb;
        unpack2(mul2(d2, nkq), ta, tb);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
        sts2x2(at + 64 * u, pack2(wa, wb), mul2(d2, B2));
    }
    const f32x2 er = pack2(r1.y, r1.y), eg = pack2(r1.z, r1.z), eb = pack2(r1.w, r1.w);
    const f32x2 rr = pack2(r1.x, r1.x), one = pack2(1.f, 1.f), mone = pack2(-1.f, -1.f);
#pragma unroll
    for (int u = 0; u < W / 8; ++u) {
        const f32x2 d = add2(add2(y2, pack2(8.f * u, 8.f * u)), yh);
        const f32x2 d2 = mul2(d, d);
        float ta, tb, wa, wb;
        unpack2(mul2(d2, nkq), ta, tb);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
        const f32x2 w = pack2(wa, wb);
        sts2x2(at + Quad<W>::ROWA + 64 * u, mul2(er, w), mul2(eg, w));
        sts2x2(at + Quad<W>::ROWB + 64 * u, mul2(eb, w), fma2v(fma2v(d2, mone, rr), B2, one));
    }
}

// The n_ent list entries at ent into this lane's pixels: v[k][y][c] = channel c of row
// (2 rg + y), column (4 cg + 2 (quarter & 1) + k) of the lane's block.  FILTER: some of the
// list's particles miss these pixels altogether.
template <int W, bool FILTER>
__device__ __forceinline__ void quad_list(const TileArgs &a, const unsigned *ent, int n_ent, int x0, int y0,
                                          unsigned smem, float (&v)[2][2][3]) {
    using Q = Quad<W>;
    constexpr int P = Q::P, BL = Q::BL;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int band = warp % Q::BANDS, group = warp / Q::BANDS;
    const int brow = band / (BL / 2), bcol = band % (BL / 2) * 2;     // left block of the pair
    const unsigned lt = (1u << lane) - 1u;
    const int quarter = lane >> 3, side = quarter >> 1, cg = lane & 1, rg = (lane >> 1) & 3;
    const unsigned col_at = smem + (unsigned)((bcol + side) * 8 + 4 * cg) * 8u;
    const unsigned row_at = smem + Q::ROWA + (unsigned)(brow * 4 + rg) * 16u;
    const unsigned stage = smem + Q::kStage;
    const unsigned lists = smem + Q::kLists + (unsigned)(2 * warp) * Q::LIST;
    f32x2 acc[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k][0] = acc[k][1] = acc[k][2] = 0ull;
    // thread 2p + h copies half h of staged particle p; the id of the batch
    // after the next is fetched ahead
    const int sp = tid >> 1;
    const unsigned half = (unsigned)(tid & 1);
    const unsigned stage_at = stage + half * (P * 16) + (unsigned)sp * 16u;
    unsigned id = 0;
    if (sp < P && sp < n_ent) {
        cp_async16(stage_at, reinterpret_cast<const char *>(a.recs + ent[sp]) + half * 16);
        if (P + sp < n_ent) id = ent[P + sp];
    }
    unsigned buf = 0;
#pragma unroll 1
    for (int base = 0; base < n_ent; base += P) {
        const unsigned st = stage + buf * (P * 32);
        cp_async_wait();
        __syncthreads();
        if (sp < P && base + P + sp < n_ent) {
            cp_async16(stage_at + (buf ^ 1u) * (P * 32),
                       reinterpret_cast<const char *>(a.recs + id) + half * 16);
            if (base + 2 * P + sp < n_ent) id = ent[base + 2 * P + sp];
        }
        {
            const int p = tid >> 2, q = tid & 3;
            bool valid = base + p < n_ent;
            const float4 r0 = lds4(st + p * 16), r1 = lds4(st + P * 16 + p * 16);
            // does the disc (with a margin) reach the rectangles of pixel centres of
            // the blocks in row q of blocks?  A superset of the blocks that hold a
            // covered pixel: a block visited in vain adds clipped zeros.  Lane b <
            // BL^2 gathers the eight bits of block b.
            const float r = r1.x * rsqrtf(r1.x) + 1e-3f;      // approximate: far inside the margin
            const float ax = (float)(x0 - unpack_xi(r0.x)) + (0.5f - r0.y);
            const float ay = (float)(y0 + 8 * q - unpack_yi(r0.x)) + (0.5f - r0.z);
            const float ny = fmaxf(ay, fminf(0.f, ay + 7.f)), room = r * r - ny * ny;
            unsigned bits = 0, any = 0;
#pragma unroll
            for (int u = 0; u < BL; ++u) {
                const float nx = fmaxf(ax + (float)(8 * u), fminf(0.f, ax + (float)(8 * u + 7)));
                const unsigned h = __ballot_sync(0xffffffffu, valid && q < BL && nx * nx <= room);
                if ((lane & (BL - 1)) == u) bits = h;
                any |= h;
            }
            if (lane < BL * BL) {
                const unsigned m = every_fourth(bits >> (lane / BL));
                asm volatile("st.shared.u8 [%0], %1;" ::"r"(smem + Q::kMask + 8 * lane + warp), "r"(m) : "memory");
            }
            if (FILTER) valid = (any >> (lane & ~3)) & 0xfu;
            if (valid) quad_tabulate<W>(r0, r1, x0, y0, smem + Q::slot(p) * Q::BYTES, q);
        }
        __syncthreads();
        // the lists of this warp's blocks (of its share of the batch), padded to whole steps
        const unsigned masks = smem + Q::kMask + 8u * (unsigned)(brow * BL + bcol);
        uint4 m;
        if (Q::G == 1) {
            m = ldsu4(masks);
        } else {
            static_assert(Q::G == 1 || Q::G == 4, "sixteen particles per warp");
            m.x = lds_u16(masks + 2 * group);
            m.z = lds_u16(masks + 8 + 2 * group);
            m.y = m.w = 0u;
        }
        const int first = group * (P / Q::G) + lane;
        const int na = __popc(m.x), nl = na + __popc(m.y), nb = __popc(m.z), nr = nb + __popc(m.w);
        const int n = nl > nr ? nl : nr;
        const unsigned sa = Q::slot(first), sb = sa + 32;
        if (nl + lane < n + 2) sts_u8(lists + nl + lane, P);
        if (nr + lane < n + 2) sts_u8(lists + Q::LIST + nr + lane, P);
        if (Q::G == 1) {
            if (nl + 32 + lane < n + 2) sts_u8(lists + nl + 32 + lane, P);
            if (nr + 32 + lane < n + 2) sts_u8(lists + Q::LIST + nr + 32 + lane, P);
            if ((m.y >> lane) & 1u) sts_u8(lists + na + __popc(m.y & lt), sb);
            if ((m.w >> lane) & 1u) sts_u8(lists + Q::LIST + nb + __popc(m.w & lt), sb);
        }
        if ((m.x >> lane) & 1u) sts_u8(lists + __popc(m.x & lt), sa);
        if ((m.z >> lane) & 1u) sts_u8(lists + Q::LIST + __popc(m.z & lt), sa);
        __syncwarp();
        unsigned at = lists + (unsigned)side * Q::LIST + (unsigned)(quarter & 1);
        unsigned off = lds_u8(at);
#pragma unroll 1
        for (int i = 0; i < n; i += 2) {
            const unsigned ca = col_at + off * Q::BYTES, ra = row_at + off * Q::BYTES;
            at += 2;
            off = lds_u8(at);
            const float4 c0 = lds4(ca), c1 = lds4(ca + 16);
            f32x2 er, eg, eb, rem;
            lds2x2(ra, er, eg);
            lds2x2(ra + (Q::ROWB - Q::ROWA), eb, rem);
            const float wx[4] = {c0.x, c0.y, c1.x, c1.y}, dxb[4] = {c0.z, c0.w, c1.z, c1.w};
            float rem_a, rem_b;
            unpack2(rem, rem_a, rem_b);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const f32x2 clip = pack2(__saturatef(rem_a - dxb[k]), __saturatef(rem_b - dxb[k]));
                const f32x2 w = mul2(clip, pack2(wx[k], wx[k]));
                fma2(acc[k][0], er, w);
                fma2(acc[k][1], eg, w);
                fma2(acc[k][2], eb, w);
            }
        }
        buf ^= 1u;
    }
    // add the two quarters of a block: each keeps two of the four columns
    const bool odd = quarter & 1;
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float a0, a1, b0, b1;
            unpack2(acc[k][c], a0, a1);
            unpack2(acc[k + 2][c], b0, b1);
            v[k][0][c] = (odd ? b0 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : b0, 8);
            v[k][1][c] = (odd ? b1 : a1) + __shfl_xor_sync(0xffffffffu, odd ? a1 : b1, 8);
        }
}

// Write one pixel's channel: stored (only item of its tile) or added atomically.
__device__ __forceinline__ void put_value(float *dst, float v, bool store) {
    if (store)
        *dst = v;
    else if (v != 0.f)
        atomicAdd(dst, v);
}

// Points and small particles of an item into the shared tile: thread t of n
// takes every n-th small particle, warp w of the n / 32 every (n / 32)-th run
// of 32 points (Sec. 4.1).
template <int T, int W>
__device__ __forceinline__ void shared_lists(const FrameConst &fc, const TileArgs &a, long long lb0,
                                             long long le0, long long lb1, long long le1, int tx0,
                                             int ty0, int x0, int y0,
                                             float (*sacc)[W][W], int t, int n) {
    const int lane = t & 31;
#pragma unroll 1
    for (long long base = lb0 + (t & ~31); base < le0; base += n) {
        float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
        const bool valid = base + lane < le0;
        if (valid) {
            const Rec rc = a.recs[a.entries[base + lane]];
            r0 = rc.r0;
            r1 = rc.r1;
        }
        warp_points<T, W>(a, valid, r0, r1, tx0, ty0, x0, y0, sacc, lane);
    }
#pragma unroll 1
    for (long long k = lb1 + t; k < le1; k += n) {
        const Rec rc = a.recs[a.entries[k]];
        thread_small<W>(fc, rc.r0, rc.r1, x0, y0, sacc);
    }
}

// The entries of a large item that cover its whole tile: the last ones of the tile's
// list, from the first result to the second.  They go through the covering pass, unless
// they are too few to be worth a start there.
constexpr int kFewFull = 64;
__device__ __forceinline__ long long item_full_start(const TileArgs &a, const FrameConst &fc,
                                                     const WorkItem &w) {
    const int slot = fc.slot_base + L_LARGE * fc.ntiles + w.tile - fc.tile_base;
    const long long from = max(w.start, a.offsets[slot + 1] - a.full[w.tile]);
    return w.end - from < kFewFull ? w.end : from;
}

// Persistent pass over the work items of every view of the batch: the tile
// pass takes items [0, item_totals[0]), the large pass the next
// item_totals[1] (both counts read from device memory).
constexpr int kItemCtas = 4;      // per SM: 64 registers, 56 KB of shared memory at W = 32

// Points and small particles of an item of a 64-pixel tile, over the whole tile: each of its
// four parts going through these lists cost more than it shared (7.9M points and
// small particles on 195 x 89: tile pass 0.394 ms, 0.299 so).
__device__ __forceinline__ void whole_tile_lists(const Views &vs, const TileArgs &a, const WorkItem &w,
                                                 const FrameConst &fc, int tx0, int ty0,
                                                 float (*sacc)[64][64]) {
    const int list = item_list(w), tid = threadIdx.x;
    const long long cap = a.entries_cap;
    long long lb0 = 0, le0 = 0, lb1 = 0, le1 = 0;
    if (list < 0) {
        const long long *o = a.offsets + fc.slot_base + w.tile - fc.tile_base;
        lb0 = min(o[L_POINT * fc.ntiles], cap); le0 = min(o[L_POINT * fc.ntiles + 1], cap);
        lb1 = min(o[L_SMALL * fc.ntiles], cap); le1 = min(o[L_SMALL * fc.ntiles + 1], cap);
    } else if (list == L_POINT) {
        lb0 = min(w.start, cap); le0 = min(w.end, cap);
    } else if (list == L_SMALL) {
        lb1 = min(w.start, cap); le1 = min(w.end, cap);
    }
    if (le0 <= lb0 && le1 <= lb1) return;
    for (int k = tid; k < 3 * 64 * 64; k += kTileThreads) (&sacc[0][0][0])[k] = 0.f;
    __syncthreads();
    shared_lists<64, 64>(fc, a, lb0, le0, lb1, le1, tx0, ty0, tx0, ty0, sacc, tid, kTileThreads);
    __syncthreads();
    float *image = a.images[item_view(w)];
    for (int k = tid; k < 3 * 64 * 64; k += kTileThreads) {
        const int row = k / 192, x3 = k % 192;
        if (ty0 + row < fc.height && tx0 + x3 / 3 < fc.width)
            put_value(image + (int64_t)3 * fc.width * (ty0 + row) + 3 * tx0 + x3, sacc[x3 % 3][row][x3 / 3],
                      false);
    }
}

// The cycles of an item, when they are recorded (zeroed by the caller; the parts of a tile
// add up).
__device__ __forceinline__ void finish(const TileArgs &a, int idx, long long t_start) {
    if (!a.item_cycles) return;
    __syncthreads();
    if (threadIdx.x == 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(&a.item_cycles[idx]),
                  (unsigned long long)(clock64() - t_start));
}

template <int T, bool LARGE>
__global__ void __launch_bounds__(kTileThreads, kItemCtas) item_kernel(Views vs, TileArgs a) {
    // a 64-pixel tile: four parts for its medium (large) particles, and in the tile pass a
    // fifth for its points and small particles, over the whole tile
    constexpr int W = T == 16 ? 16 : 32, SIDE = T / W;
    constexpr int SUB = SIDE * SIDE + (T == 64 && !LARGE ? 1 : 0);
    using Q = Quad<W>;
    extern __shared__ float4 smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int *counter = &a.st->item_counter[LARGE ? 1 : 0];
    const int item0 = LARGE ? a.st->item_totals[0] : 0;
    const int n_work = min(a.st->item_totals[LARGE ? 1 : 0], a.items_cap - item0) * SUB;
    if (tid < Q::BYTES / 16) smem_raw[Q::kNone / 16 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    float (*sacc)[W][W] = reinterpret_cast<float (*)[W][W]>(smem_raw);   // after the tables
    __shared__ int s_item[2];
    __shared__ long long s_range[4];       // of an item with every list: its points, its small particles
    __shared__ FrameConst sfc;
    // The item after this one is taken while this one is worked on, an item of a
    // light tile carries its medium range, and the view's constants are read only
    // when the view changes: a light tile's time is the chain of loads before its
    // first batch.
    int cur_view = -1, next = 0;
    if (tid == 0) s_item[0] = atomicAdd(counter, 1);
    for (int turn = 0;; turn ^= 1) {
        __syncthreads();
        const int it = s_item[turn];
        if (it >= n_work) break;
        if (tid == 0) next = atomicAdd(counter, 1);
        const int idx = item0 + (a.order ? a.order[item0 + it / SUB] : it / SUB), sub = it % SUB;
        const WorkItem w = a.items[idx];
        const int view = item_view(w), list = item_list(w);
        const long long t_start = clock64();
        if (view != cur_view) {
            const int words = (int)(sizeof(FrameConst) / sizeof(int));
            if (tid < words)
                reinterpret_cast<int *>(&sfc)[tid] =
                    reinterpret_cast<const int *>(vs.fcs + view)[tid];
            __syncthreads();
            cur_view = view;
        }
        const FrameConst &fc = sfc;
        const int tile = w.tile - fc.tile_base;
        const int tx0 = (tile % fc.ntx) * T, ty0 = (tile / fc.ntx) * T;
        const int x0 = tx0 + sub % SIDE * W, y0 = ty0 + sub / SIDE * W;
        // (a part of a tile may lie outside the image)
        const long long cap = SUB == 1 || (x0 < fc.width && y0 < fc.height) ? a.entries_cap : 0;
        if constexpr (T == 64 && !LARGE) {
            if (sub == SIDE * SIDE) {
                whole_tile_lists(vs, a, w, fc, tx0, ty0, reinterpret_cast<float (*)[64][64]>(smem_raw));
                finish(a, idx, t_start);
                if (tid == 0) s_item[turn ^ 1] = next;
                continue;
            }
        }
        if (list < 0 && tid < 4)
            s_range[tid] = a.offsets[fc.slot_base + (tid < 2 ? L_POINT : L_SMALL) * fc.ntiles + tile + (tid & 1)];
        // medium (tile pass) or large (large pass) particles into registers; never past
        // the entries written
        const bool mine = list < 0 || list >= L_MEDIUM;
        const long long lb2 = min(w.start, cap);
        const long long last = LARGE && T > 16 && a.cover ? item_full_start(a, fc, w) : w.end;
        const int n2 = mine ? (int)(min(last, cap) - lb2) : 0;
        float quad[2][2][3];
        quad_list<W, (SIDE > 1)>(a, a.entries + lb2, n2, x0, y0,
                                (unsigned)__cvta_generic_to_shared(smem_raw), quad);

        // points and small particles go through the shared tile, which reuses
        // the table space (the tables are dead once every warp is past here)
        long long lb0 = 0, le0 = 0, lb1 = 0, le1 = 0;
        if (SIDE > 1) {
            // (see whole_tile_lists)
        } else if (list < 0) {
            if (n2 <= 0) __syncthreads();   // s_range (the batches' barriers otherwise)
            lb0 = min(s_range[0], cap); le0 = min(s_range[1], cap);
            lb1 = min(s_range[2], cap); le1 = min(s_range[3], cap);
        } else if (list == L_POINT) {
            lb0 = min(w.start, cap); le0 = min(w.end, cap);
        } else if (list == L_SMALL) {
            lb1 = min(w.start, cap); le1 = min(w.end, cap);
        }
        const bool shared_tile = le0 > lb0 || le1 > lb1;
        if (shared_tile) {
            __syncthreads();
            for (int k = tid; k < 3 * W * W; k += kTileThreads) (&sacc[0][0][0])[k] = 0.f;
            __syncthreads();
            shared_lists<T, W>(fc, a, lb0, le0, lb1, le1, tx0, ty0, x0, y0, sacc, tid, kTileThreads);
            __syncthreads();
        }
        // write: shared part + registers; plain stores where no other item of the
        // pass writes the tile: the large pass adds to what the tile pass left (687k
        // heavy-tailed particles on 3633 x 1145, one large item per tile: 0.112 ms with
        // atomic adds, 0.072 with plain ones)
        const bool store = LARGE ? item_sole(w) : list < 0 && SIDE == 1;
        const int onto = LARGE ? 1 : a.accumulate;
        float *image = a.images[view];
        const int64_t pitch = (int64_t)3 * fc.width;
        const int band = warp % Q::BANDS, quarter = lane >> 3;
        const int row = band / (Q::BL / 2) * 8 + ((lane >> 1) & 3) * 2;
        const int cx = band % (Q::BL / 2) * 16 + (quarter >> 1) * 8 + (lane & 1) * 4 + (quarter & 1) * 2;
        if constexpr (Q::G == 1) {
            float *dst = image + pitch * (y0 + row) + 3 * (x0 + cx);
            bool in[2][2];
#pragma unroll
            for (int y = 0; y < 2; ++y)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    in[y][k] = y0 + row + y < fc.height && x0 + cx + k < fc.width;
                    if (!shared_tile) continue;
#pragma unroll
                    for (int c = 0; c < 3; ++c) quad[k][y][c] += sacc[c][row + y][cx + k];
                }
            if (store && onto) {     // every load before the first store
                float old[2][2][3];
#pragma unroll
                for (int u = 0; u < 12; ++u) {
                    const int y = u / 6, k = u / 3 % 2, c = u % 3;
                    old[y][k][c] = in[y][k] ? dst[pitch * y + 3 * k + c] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 12; ++u) quad[u / 3 % 2][u / 6][u % 3] += old[u / 6][u / 3 % 2][u % 3];
            }
#pragma unroll
            for (int u = 0; u < 12; ++u) {
                const int y = u / 6, k = u / 3 % 2, c = u % 3;
                if (in[y][k]) put_value(dst + pitch * y + 3 * k + c, quad[k][y][c], store);
            }
        } else {
            // the warps' partial sums through shared memory, then one pixel per thread
            float (*part)[3][W][W] = reinterpret_cast<float (*)[3][W][W]>(
                reinterpret_cast<char *>(smem_raw) + Q::kPart);
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 12; ++u) {
                const int y = u / 6, k = u / 3 % 2, c = u % 3;
                part[warp / Q::BANDS][c][row + y][cx + k] = quad[k][y][c];
            }
            __syncthreads();
            static_assert(Q::G == 1 || W * W == kTileThreads, "one pixel per thread");
            const int px = tid % W, py = tid / W;
            if (x0 + px < fc.width && y0 + py < fc.height) {
                float *dst = image + pitch * (y0 + py) + 3 * (x0 + px);
                float v[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    v[c] = shared_tile ? sacc[c][py][px] : 0.f;
#pragma unroll
                    for (int g = 0; g < Q::G; ++g) v[c] += part[g][c][py][px];
                }
                if (store && onto) {
                    const float o0 = dst[0], o1 = dst[1], o2 = dst[2];
                    v[0] += o0; v[1] += o1; v[2] += o2;
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) put_value(dst + c, v[c], store);
            }
        }
        finish(a, idx, t_start);
        if (tid == 0) s_item[turn ^ 1] = next;
    }
}

// ---------------------------------------------------------------------------
// The covering pass: large particles over tiles that lie wholly inside their discs (most
// tiles of a particle much wider than a tile).  No clip, and every pixel is covered, so
// that a lane can hold 4 x 4 pixels and a warp half the tile: per particle a warp loads four
// column weights and four rows' terms (10 wavefronts per 512 pixels, where the blocks of
// the tile pass take 26) and adds 48 products per lane.  The two warps of a tile are
// repeated four times over the particles.  16 warps per SM leave it bound by latency
// (FMA pipe 40 %, 50 cycles per entry and SM where the tile pass took 78).  Large pass of
// the 100M heavy-tailed frame 4.96 -> 3.44 ms, of 1M particles in six orbit views 6.89 ->
// 5.33 ms.
// ---------------------------------------------------------------------------
struct Cover {
    static constexpr int P = 64;
    // one particle's tables: 32 column weights, 16 row pairs (e_R w_a, e_R w_b, e_G w_a,
    // e_G w_b), 16 row pairs (e_B w_a, e_B w_b); padding and slot order as in Quad
    static constexpr int ROWA = 128, ROWB = 384, BYTES = 544;
    __device__ static __forceinline__ unsigned slot(int p) {
        return (unsigned)((p & ~3) | ((p & 1) << 1) | ((p >> 1) & 1));
    }
    static constexpr int kStage = P * BYTES;
    static constexpr int kSmem = kStage + 2 * P * 32;
    static constexpr int kTile = 3 * 32 * 32;      // floats; two tiles reuse the tables
    static_assert(2 * 4 * kTile <= kStage, "the tables hold two tiles");
};
constexpr int kCoverCtas = 2, kCoverUnroll = 2;   // 128 registers (3 CTAs at 80 spill: 7 % longer)

template <int T>
__global__ void __launch_bounds__(kTileThreads, kCoverCtas) cover_kernel(Views vs, TileArgs a) {
    constexpr int W = 32, SIDE = T / W, SUB = SIDE * SIDE, P = Cover::P;
    extern __shared__ float4 smem_raw[];
    __shared__ int s_item[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned smem = (unsigned)__cvta_generic_to_shared(smem_raw);
    float *tiles = reinterpret_cast<float *>(smem_raw);
    int *counter = &a.st->item_counter[2];
    const int item0 = a.st->item_totals[0];
    const int n_work = min(a.st->item_totals[1], a.items_cap - item0) * SUB;
    // this lane's pixels: columns 4 cg .. 4 cg + 3, row pairs rg and rg + 1
    const int cg = lane & 7, rg = (warp & 1) * 8 + (lane >> 3) * 2, group = warp >> 1;
    const unsigned at0 = smem + Cover::slot(group) * Cover::BYTES;
    const unsigned col_at = at0 + 16u * cg, row_at = at0 + Cover::ROWA + 16u * rg;
    const unsigned blue_at = at0 + Cover::ROWB + 8u * rg;
    const int sp = tid >> 1;
    const unsigned half = (unsigned)(tid & 1);
    const unsigned stage = smem + Cover::kStage, stage_at = stage + half * (P * 16) + (unsigned)sp * 16u;
    // where there are few items most have nothing for this pass: eight at a time, one
    // lane each
    const int step = n_work < 8 * (int)gridDim.x ? 8 : 1;
    __shared__ unsigned s_some;
    int next = 0;
    unsigned some = 0;                     // items of the current step still to be done
    if (tid == 0) s_item[0] = atomicAdd(counter, step);
    for (int turn = 0, it0 = 0;;) {
        __syncthreads();
        if (!some) {
            it0 = s_item[turn];
            if (it0 >= n_work) break;
            turn ^= 1;
            if (tid == 0) next = atomicAdd(counter, step);
            if (warp == 0) {
                bool has = lane < step && it0 + lane < n_work;
                if (has) {
                    const WorkItem w = a.items[item0 + (it0 + lane) / SUB];
                    has = item_full_start(a, vs.fcs[item_view(w)], w) < w.end;
                }
                const unsigned m = __ballot_sync(0xffffffffu, has);
                if (lane == 0) {
                    s_some = m;
                    s_item[turn] = next;
                }
            }
            __syncthreads();
            some = s_some;
            if (!some) continue;
        }
        const int it = it0 + __ffs(some) - 1;
        some &= some - 1u;
        const int idx = item0 + it / SUB, sub = it % SUB;
        const WorkItem w = a.items[idx];
        const FrameConst &fc = vs.fcs[item_view(w)];
        const int tile = w.tile - fc.tile_base;
        const int x0 = (tile % fc.ntx) * T + sub % SIDE * W, y0 = (tile / fc.ntx) * T + sub / SIDE * W;
        const long long lb = item_full_start(a, fc, w);
        int n = (int)(min(w.end, a.entries_cap) - lb);
        if (x0 >= fc.width || y0 >= fc.height) n = 0;
        if (n > 0) {
            const long long t_start = clock64();
            const unsigned *ent = a.entries + lb;
            f32x2 acc[2][4][3];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[m][k][0] = acc[m][k][1] = acc[m][k][2] = 0ull;
            unsigned id = 0;
            if (sp < P && sp < n) {
                cp_async16(stage_at, reinterpret_cast<const char *>(a.recs + ent[sp]) + half * 16);
                if (P + sp < n) id = ent[P + sp];
            }
            unsigned buf = 0;
#pragma unroll 1
            for (int base = 0; base < n; base += P) {
                const int cnt = n - base < P ? n - base : P;
                const unsigned st = stage + buf * (P * 32);
                cp_async_wait();
                __syncthreads();
                if (sp < P && base + P + sp < n) {
                    cp_async16(stage_at + (buf ^ 1u) * (P * 32),
                               reinterpret_cast<const char *>(a.recs + id) + half * 16);
                    if (base + 2 * P + sp < n) id = ent[base + 2 * P + sp];
                }
                const int p = tid >> 2, q = tid & 3;
                if (p < cnt) {
                    // thread q of a particle's four: pairs q, q + 4, q + 8, q + 12 of columns and rows
                    const float4 r0 = lds4(st + p * 16), r1 = lds4(st + P * 16 + p * 16);
                    const f32x2 nkq = pack2(-r0.w, -r0.w);
                    const float xf = (float)(x0 - unpack_xi(r0.x) + 2 * q);
                    const float yf = (float)(y0 - unpack_yi(r0.x) + 2 * q);
                    const f32x2 xh = pack2(0.5f - r0.y, 0.5f - r0.y), yh = pack2(0.5f - r0.z, 0.5f - r0.z);
                    const f32x2 er = pack2(r1.y, r1.y), eg = pack2(r1.z, r1.z), eb = pack2(r1.w, r1.w);
                    const unsigned tab = smem + Cover::slot(p) * Cover::BYTES;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const f32x2 dx = add2(pack2(xf + 8.f * u, xf + 8.f * u + 1.f), xh);
                        const f32x2 dy = add2(pack2(yf + 8.f * u, yf + 8.f * u + 1.f), yh);
                        float ta, tb, wa, wb;
                        unpack2(mul2(mul2(dx, dx), nkq), ta, tb);
                        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
                        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
                        sts2(tab + 8 * q + 32 * u, pack2(wa, wb));
                        unpack2(mul2(mul2(dy, dy), nkq), ta, tb);
                        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
                        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
                        const f32x2 wy = pack2(wa, wb);
                        sts2x2(tab + Cover::ROWA + 16 * q + 64 * u, mul2(er, wy), mul2(eg, wy));
                        sts2(tab + Cover::ROWB + 8 * q + 32 * u, mul2(eb, wy));
                    }
                }
                __syncthreads();
                unsigned off = 0;
#pragma unroll kCoverUnroll
                for (int i = group; i < cnt; i += 4, off += 4 * Cover::BYTES) {
                    const float4 c = lds4(col_at + off);
                    f32x2 er0, eg0, er1, eg1, eb0, eb1;
                    lds2x2(row_at + off, er0, eg0);
                    lds2x2(row_at + off + 16, er1, eg1);
                    lds2x2(blue_at + off, eb0, eb1);
                    const float wx[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const f32x2 wk = pack2(wx[k], wx[k]);
                        fma2(acc[0][k][0], er0, wk);
                        fma2(acc[0][k][1], eg0, wk);
                        fma2(acc[0][k][2], eb0, wk);
                        fma2(acc[1][k][0], er1, wk);
                        fma2(acc[1][k][1], eg1, wk);
                        fma2(acc[1][k][2], eb1, wk);
                    }
                }
                buf ^= 1u;
            }
            // the four groups' sums: 2 and 3 through shared memory to 0 and 1, then 1 to 0,
            // whose sum every thread writes
            auto exchange = [&](float *t, bool put) {
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float *d = t + (c * W + 2 * (rg + m)) * W + 4 * cg + k;
                            float lo, hi;
                            unpack2(acc[m][k][c], lo, hi);
                            if (put) {
                                d[0] = lo;
                                d[W] = hi;
                            } else {
                                acc[m][k][c] = pack2(lo + d[0], hi + d[W]);
                            }
                        }
            };
            __syncthreads();
            if (group >= 2) exchange(tiles + (group - 2) * Cover::kTile, true);
            __syncthreads();
            if (group < 2) exchange(tiles + group * Cover::kTile, false);
            if (group == 1) exchange(tiles + Cover::kTile, true);
            __syncthreads();
            if (group == 0) {
                exchange(tiles + Cover::kTile, false);
                exchange(tiles, true);
            }
            __syncthreads();
            const bool sole = item_sole(w);
            float *image = a.images[item_view(w)];
            // 12 values per thread, every load before the first store
            constexpr int PER = Cover::kTile / kTileThreads;
            float v[PER];
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int k = tid + u * kTileThreads, row = k / (3 * W), x3 = k % (3 * W);
                v[u] = tiles[(x3 % 3 * W + row) * W + x3 / 3];
                if (sole && y0 + row < fc.height && x0 + x3 / 3 < fc.width)
                    v[u] += image[(int64_t)3 * fc.width * (y0 + row) + 3 * x0 + x3];
            }
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int k = tid + u * kTileThreads, row = k / (3 * W), x3 = k % (3 * W);
                if (y0 + row < fc.height && x0 + x3 / 3 < fc.width)
                    put_value(image + (int64_t)3 * fc.width * (y0 + row) + 3 * x0 + x3, v[u], sole);
            }
            finish(a, idx, t_start);
        }
    }
}

template <int T>
static void launch_cover_t(const Views &vs, const TileArgs &a, int sms, cudaStream_t s) {
    cudaFuncSetAttribute(cover_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cover::kSmem);
    cover_kernel<T><<<sms * kCoverCtas, kTileThreads, Cover::kSmem, s>>>(vs, a);
    ++g_launches;
}

template <int T, bool LARGE>
static void launch_items_t(const Views &vs, const TileArgs &a, int sms, cudaStream_t s) {
    constexpr size_t bytes = Quad<(T == 16 ? 16 : 32)>::kSmem;
    cudaFuncSetAttribute(item_kernel<T, LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)bytes);
    item_kernel<T, LARGE><<<sms * kItemCtas, kTileThreads, bytes, s>>>(vs, a);
    ++g_launches;
}

template <bool LARGE>
static void launch_items(const Views &vs, const TileArgs &a, int sms, cudaStream_t s) {
    if (vs.tile == 16)
        launch_items_t<16, LARGE>(vs, a, sms, s);
    else if (vs.tile == 64)
        launch_items_t<64, LARGE>(vs, a, sms, s);
    else
        launch_items_t<32, LARGE>(vs, a, sms, s);
}

void launch_tile_pass(const Views &vs, const TileArgs &a, int sms, cudaStream_t s) {
    launch_items<false>(vs, a, sms, s);
}

void launch_large_pass(const Views &vs, const TileArgs &a, int sms, cudaStream_t s) {
    launch_items<true>(vs, a, sms, s);
    if (!a.cover) return;
    if (vs.tile == 32)
        launch_cover_t<32>(vs, a, sms, s);
    else if (vs.tile == 64)
        launch_cover_t<64>(vs, a, sms, s);
}

// E_p = A_p solution of Eq. 1 applied to the additive sum: I = 1 - exp(-S).
__global__ void epilogue_ea_kernel(float *img, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        img[i] = -expm1f(-img[i]);
}

void launch_epilogue_ea(float *image, int64_t nvals, int sms, cudaStream_t s) {
    if (nvals <= 0) return;
    int64_t blocks = (nvals + 255) / 256;
    blocks = blocks < (int64_t)sms * 4 ? blocks : (int64_t)sms * 4;
    epilogue_ea_kernel<<<(unsigned)blocks, 256, 0, s>>>(image, nvals);
    ++g_launches;
}

// Grid-stride over every pixel value of every view (blockIdx.y = view).
__global__ void views_ea_kernel(Views vs, float *const *images) {
    const int v = blockIdx.y;
    const FrameConst &fc = vs.fcs[v];
    float *img = images[v];
    const int64_t n = (int64_t)3 * fc.width * fc.height;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        img[i] = -expm1f(-img[i]);
}

void launch_epilogue_views(const Views &vs, float *const *images, int sms, cudaStream_t s) {
    views_ea_kernel<<<dim3(sms * 2, vs.nviews), 256, 0, s>>>(vs, images);
    ++g_launches;
}

}  // namespace spl
