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
// Inside an item a warp owns a band of the tile (two 8 x 8 blocks for T = 32, see
// Quad; 16 x 2 pixels for T = 16, 64 x 8 for T = 64), each lane a few pixels of it
// (T = 16: one pixel; T = 64: two columns 32 apart, eight rows), and keeps its
// pixels' three channels in registers.  Then:
//   - point particles (r <= r_sml, Sec. 4.1) add their emission to one pixel
//     of a shared-memory copy of the tile; lanes of a warp that hit the same
//     pixel are summed with warp shuffles first;
//   - small particles (r_sml < r <= r_small, a few pixels wide): one thread
//     per particle walks the particle's pixel box, into shared memory;
//   - medium and large particles are taken in batches (the chunks of n_p
//     particles of Sec. 4.2): the CTA first tabulates, per particle, the
//     column weights w_x(i) = exp(-dx^2/sigma^2) and the row terms
//     e * w_y(j) (Eq. 2 is separable: exp(-(dx^2+dy^2)/sigma^2) = w_x w_y),
//     then every warp whose band the particle reaches adds
//     e * w_y * w_x into its registers: three FMAs per pixel, plus a clip
//     test folded into one saturating add on the FMA pipe (see below);
//     where a lane holds an even number of rows, two rows go through one
//     packed FP32x2 instruction (the row table is laid out in row pairs);
//   - finally each thread adds the shared-memory part to its registers and
//     writes its pixels once.
// The large pass (r > r_large, Sec. 4.3) runs after the tile pass with the
// same scheme over segments of the tiles' large lists and adds its partial
// tiles into the image.
//
// Clip (Eq. 2: zero beyond chi*sigma).  With B = 2^20 / r^2 the tables hold
// dx^2 * B per column and (r^2 - dy^2) * B + 1 per row; the clip factor is
// m = saturate((r^2 - dy^2) B + 1 - dx^2 B), which is exactly 1 inside the
// disc and exactly 0 outside it, except for pixels whose distance lies within
// r * (1 + 5e-7) -- inside the band where FP32 and FP64 may legitimately
// disagree on an inclusive clip test anyway.
#include "spl_tile.cuh"

namespace spl {

// The registers of one thread's pixels: RPL rows x CPL columns x RGB, held
// as row pairs when the rows are processed two at a time.
template <int T, bool PAIRED = Shape<T>::PAIRED>
struct Acc {
    using S = Shape<T>;
    float v[S::RPL][S::CPL][3];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int q = 0; q < S::RPL; ++q)
#pragma unroll
            for (int k = 0; k < S::CPL; ++k) v[q][k][0] = v[q][k][1] = v[q][k][2] = 0.f;
    }
    __device__ __forceinline__ float get(int q, int k, int c) const { return v[q][k][c]; }
};
template <int T>
struct Acc<T, true> {
    using S = Shape<T>;
    f32x2 v[S::RPL / 2][S::CPL][3];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int q = 0; q < S::RPL / 2; ++q)
#pragma unroll
            for (int k = 0; k < S::CPL; ++k) v[q][k][0] = v[q][k][1] = v[q][k][2] = 0ull;
    }
    __device__ __forceinline__ float get(int q, int k, int c) const {
        float lo, hi;
        unpack2(v[q >> 1][k][c], lo, hi);
        return (q & 1) ? hi : lo;
    }
};

// One small particle (a few pixels wide) into the shared tile, by one thread:
// the pixel box inside the tile, the clip test and the weight of Eq. 2 per
// pixel, and one shared-memory add per channel.  A tiny splat costs a few
// pixels of work here instead of a batch-table share and a band visit.
template <int T>
__device__ __forceinline__ void thread_small(const FrameConst &fc, float4 r0, float4 r1, int x0,
                                             int y0, float (*sacc)[T][T]) {
    PixBox b;
    if (!splat_box(fc, r0, r1.x, b)) return;
    const int i0 = max(b.i0, x0), i1 = min(b.i1, x0 + T - 1);
    const int j0 = max(b.j0, y0), j1 = min(b.j1, y0 + T - 1);
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
template <int T>
__device__ __forceinline__ void warp_points(const TileArgs &a, bool valid, float4 r0, float4 r1,
                                            int x0, int y0, float (*sacc)[T][T], int lane) {
    int key = -1;
    float er = 0.f, eg = 0.f, eb = 0.f;
    int i = 0, j = 0;
    if (valid) {
        i = unpack_xi(r0.x) - x0;
        j = unpack_yi(r0.x) - y0;
        if ((unsigned)i < (unsigned)T && (unsigned)j < (unsigned)T) {
            key = j * T + i;
            er = r1.y; eg = r1.z; eb = r1.w;
        } else {
            atomicOr(&a.st->err, ERR_INDEX);
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

// Tabulate the separable factors of a batch of cnt <= 32 staged particles:
// swx[p][c] = (w_x, dx^2 B) for tile column c; for tile row j the row terms
// e_R w_y, e_G w_y, e_B w_y and (r^2 - dy^2) B + 1.  Rows are stored one
// float4 per row, or -- when the rows go two at a time -- per row pair
// (2m, 2m+1) in two tables, srow[p][m] = (e_R w_y, same for row 2m+1, e_G w_y,
// e_G w_y') in the first half of the row space and (e_B w_y, e_B w_y', rem,
// rem') in the second, so that every packed operand is one aligned half of a
// 16-byte load and the eight threads of a particle store consecutive entries.  Thread (p, q) = (tid / 8,
// tid % 8) fills columns q, q + 8, q + 16, ... (and the same rows, or row
// pairs q, q + 8, ...) of particle p.  It also decides for row band q whether
// the disc reaches it (bit p of band_mask[q]).  B only needs to be the same
// on both sides of the clip test, so a fast reciprocal serves.
template <int T>
__device__ __forceinline__ void tabulate(const float4 *st0, const float4 *st1, int cnt, int x0,
                                         int y0, float2 (*swx)[Shape<T>::WXS], float4 (*srow)[T],
                                         unsigned *band_mask, int tid) {
    using S = Shape<T>;
    const int p = tid >> 3, q = tid & 7;
    // every lane runs to the end (the band bits are combined by a ballot); the
    // entries of particles p >= cnt are written but never read (no band bit)
    const bool valid = p < cnt;
    const float4 r0 = st0[valid ? p : 0], r1 = st1[valid ? p : 0];
    const float kq = r0.w, r2 = r1.x;
    const float B = __fdividef(1048576.f, r2);
    const int xi = unpack_xi(r0.x), yi = unpack_yi(r0.x);
    const float xh = 0.5f - r0.y, yh = 0.5f - r0.z;
    // the disc's radius for the band test (conservative by 1e-3 px)
    const float r = r2 * rsqrtf(r2) + 1e-3f;   // approximate: far inside the margin
    // offsets of this thread's first column and row from the particle centre;
    // the others follow by adding small integers (exact in FP32)
    const float dxq = ((float)(x0 - xi) + xh) + (float)q;
#pragma unroll
    for (int u = 0; u < S::PER; ++u) {
        const int k = q + 8 * u;
        const float dx = dxq + (float)(8 * u);
        const float dx2 = dx * dx;
        swx[p][k] = make_float2(ex2_neg(kq * dx2), dx2 * B);
    }
    if constexpr (S::PAIRED) {
        const float dyq = ((float)(y0 - yi) + yh) + (float)(2 * q);
#pragma unroll
        for (int u = 0; u < S::PER / 2; ++u) {
            const int m = q + 8 * u;
            const float dya = dyq + (float)(16 * u), dyb = dya + 1.f;
            const float a2 = dya * dya, b2 = dyb * dyb;
            const float wa = ex2_neg(kq * a2), wb = ex2_neg(kq * b2);
            float4 *rowA = reinterpret_cast<float4 *>(srow), *rowB = rowA + S::P * (T / 2);
            rowA[p * (T / 2) + m] = make_float4(r1.y * wa, r1.y * wb, r1.z * wa, r1.z * wb);
            rowB[p * (T / 2) + m] =
                make_float4(r1.w * wa, r1.w * wb, fmaf(r2 - a2, B, 1.f), fmaf(r2 - b2, B, 1.f));
        }
    } else {
#pragma unroll
        for (int u = 0; u < S::PER; ++u) {
            const int k = q + 8 * u;
            const float dy = (float)(y0 + k - yi) + yh;
            const float dy2 = dy * dy;
            const float wy = ex2_neg(kq * dy2);
            srow[p][k] = make_float4(r1.y * wy, r1.z * wy, r1.w * wy, fmaf(r2 - dy2, B, 1.f));
        }
    }
    // row band q: columns [bx BW, bx BW + BW), rows [by BH, by BH + BH); the
    // disc (with a margin) must reach the rectangle of the band's pixel
    // centres.  A superset of the bands that hold a covered pixel: a band
    // visited in vain adds clipped zeros.
    const int bx0 = (q % S::NBX) * S::BW, by0 = (q / S::NBX) * S::BH;
    const float ax = (float)(x0 + bx0 - xi) + xh, ay = (float)(y0 + by0 - yi) + yh;
    const float nx = fmaxf(ax, fminf(0.f, ax + (float)(S::BW - 1)));
    const float ny = fmaxf(ay, fminf(0.f, ay + (float)(S::BH - 1)));
    const bool hit = valid && nx * nx + ny * ny <= r * r;
    // lane 8j + q holds particle 4w + j of warp w and band q: lane q < 8 gathers
    // its band's four bits and sets them with one atomic
    const unsigned hb = __ballot_sync(0xffffffffu, hit);
    const int lane = tid & 31;
    if (lane < 8) {
        const unsigned nib = ((hb >> lane) & 1u) | (((hb >> (lane + 8)) & 1u) << 1) |
                             (((hb >> (lane + 16)) & 1u) << 2) | (((hb >> (lane + 24)) & 1u) << 3);
        if (nib) atomicOr(&band_mask[lane], nib << (4 * (tid >> 5)));
    }
}

// Add tabulated particle p into the registers of this thread's pixels.  The
// clip factor is exactly 1 inside the disc and 0 outside (see the top).
template <int T>
__device__ __forceinline__ void band_splat(const float2 *wxp, const float4 *rowp, int col, int row0,
                                           Acc<T, false> &acc) {
    using S = Shape<T>;
    float wx[S::CPL], dxb[S::CPL];
#pragma unroll
    for (int k = 0; k < S::CPL; ++k) {
        const float2 v = wxp[col + S::CSTEP * k];
        wx[k] = v.x;
        dxb[k] = v.y;
    }
#pragma unroll
    for (int q = 0; q < S::RPL; ++q) {
        const float4 rv = rowp[row0 + q];
#pragma unroll
        for (int k = 0; k < S::CPL; ++k) {
            const float wk = wx[k] * __saturatef(rv.w - dxb[k]);
            acc.v[q][k][0] = fmaf(rv.x, wk, acc.v[q][k][0]);
            acc.v[q][k][1] = fmaf(rv.y, wk, acc.v[q][k][1]);
            acc.v[q][k][2] = fmaf(rv.z, wk, acc.v[q][k][2]);
        }
    }
}

// The same two rows at a time: per row pair two 16-byte loads, and per
// column two scalar clips, one packed multiply and three packed FMAs (R, G, B
// of both rows).
// rowp points at the particle's first-half row-pair table (see tabulate).
template <int T>
__device__ __forceinline__ void band_splat(const float2 *wxp, const float4 *rowp, int col, int row0,
                                           Acc<T, true> &acc) {
    using S = Shape<T>;
    float dxb[S::CPL];
    f32x2 ww[S::CPL];
#pragma unroll
    for (int k = 0; k < S::CPL; ++k) {
        const float2 v = wxp[col + S::CSTEP * k];
        ww[k] = pack2(v.x, v.x);
        dxb[k] = v.y;
    }
    const ulonglong2 *ra_ = reinterpret_cast<const ulonglong2 *>(rowp) + row0 / 2;
    const ulonglong2 *rb_ = ra_ + S::P * (T / 2);
#pragma unroll
    for (int m = 0; m < S::RPL / 2; ++m) {
        const ulonglong2 a = ra_[m], b = rb_[m];
        float ra, rb;
        unpack2(b.y, ra, rb);
#pragma unroll
        for (int k = 0; k < S::CPL; ++k) {
            const f32x2 w = mul2(pack2(__saturatef(ra - dxb[k]), __saturatef(rb - dxb[k])), ww[k]);
            fma2(acc.v[m][k][0], a.x, w);
            fma2(acc.v[m][k][1], a.y, w);
            fma2(acc.v[m][k][2], b.x, w);
        }
    }
}

// ---------------------------------------------------------------------------
// T = 32: quarter-warp splatting over 8 x 8 blocks.  A warp owns two adjacent 8 x 8
// blocks of the tile; two of its quarter-warps take two particles of the left
// block's list at a time, the other two two of the right block's, a lane holding
// 4 x 2 pixels of its block.  The two quarters of a block are added at the end of
// the item.
//
// What bounds it: the shared-memory data pipe (77 % of its peak on the clustered
// 10M / 1024^2 frame; issue slots 65 %, FMA pipe 55 %).  One particle per warp step
// over a 16 x 8 band, a lane 2 x 2 pixels, took 8 wavefronts per 128 pixels at 54 %
// covered pixels: 34.6 wavefronts and 124 instructions per list entry, the pipe at 82 %.
// 8 x 8 blocks are covered to 65 %, and a lane's eight pixels share its four 16-byte loads
// (12 wavefronts per 256 pixels): 28.5 wavefronts and 108 instructions.  Tile pass of that
// frame 4.58 -> 3.84 ms.  Also measured there: a lane 4 x 4 pixels of a 16 x 8 band
// (fewest wavefronts, but 48 accumulators leave 16 warps per SM: 4.65), the same with
// producer warps and an mbarrier ring (4.50), 3 CTAs per SM (4.55), the clip as
// compare and select on the ALU pipe for half or all of the columns (3.87, 4.12).
// ---------------------------------------------------------------------------
struct Quad {
    static constexpr int T = 32, P = 64;           // tile side, particles per batch
    // one particle's tables: 16 column pairs (w_a, w_b, dx_a^2 B, dx_b^2 B), 16 row pairs
    // (e_R w_a, e_R w_b, e_G w_a, e_G w_b), 16 row pairs (e_B w_a, e_B w_b, rem_a, rem_b);
    // the 16 bytes of padding and the slot order put neighbouring particles in
    // different banks
    static constexpr int ROWA = 256, ROWB = 512, BYTES = 784;
    __device__ static __forceinline__ unsigned slot(int p) {
        return (unsigned)((p & ~7) | ((p & 1) << 2) | ((p >> 1) & 3));
    }
    static constexpr int kNone = P * BYTES;        // tables of a particle that adds nothing
    static constexpr int kStage = kNone + BYTES;   // two batches of records
    static constexpr int kMask = kStage + 2 * P * 32;   // per block: the particles that reach it
    static constexpr int kLists = kMask + 16 * 8;
    static constexpr int LIST = 72;                // a block's particles (slots), padded
    static constexpr int kSmem = kLists + 16 * LIST;
};

__device__ __forceinline__ float4 lds4(unsigned a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void lds2x2(unsigned a, f32x2 &u, f32x2 &v) {
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(u), "=l"(v) : "r"(a));
}
__device__ __forceinline__ uint4 ldsu4(unsigned a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts2x2(unsigned a, f32x2 u, f32x2 v) {
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(a), "l"(u), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned lds_u8(unsigned a) {
    unsigned v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u8(unsigned a, unsigned v) {
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// Tabulate particle (r0, r1) into the block tab: thread q of its four fills
// column pairs and row pairs q, q + 4, q + 8, q + 12.  Pixel offsets are exact
// integers plus the sub-pixel part; two columns (rows) go through one packed
// FP32x2 instruction.  B only needs to be the same on both sides of the clip
// test, so a fast reciprocal serves.
__device__ __forceinline__ void quad_tabulate(float4 r0, float4 r1, int x0, int y0, unsigned tab,
                                              int q) {
    const float B = __fdividef(1048576.f, r1.x);
    const f32x2 nkq = pack2(-r0.w, -r0.w), B2 = pack2(B, B);
    const float xf = (float)(x0 - unpack_xi(r0.x) + 2 * q), yf = (float)(y0 - unpack_yi(r0.x) + 2 * q);
    const f32x2 x2 = pack2(xf, xf + 1.f), y2 = pack2(yf, yf + 1.f);
    const f32x2 xh = pack2(0.5f - r0.y, 0.5f - r0.y), yh = pack2(0.5f - r0.z, 0.5f - r0.z);
    const unsigned at = tab + 16 * q;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
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
    for (int u = 0; u < 4; ++u) {
        const f32x2 d = add2(add2(y2, pack2(8.f * u, 8.f * u)), yh);
        const f32x2 d2 = mul2(d, d);
        float ta, tb, wa, wb;
        unpack2(mul2(d2, nkq), ta, tb);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
        const f32x2 w = pack2(wa, wb);
        sts2x2(at + Quad::ROWA + 64 * u, mul2(er, w), mul2(eg, w));
        sts2x2(at + Quad::ROWB + 64 * u, mul2(eb, w), fma2v(fma2v(d2, mone, rr), B2, one));
    }
}

// Bits 0, 4, ..., 28 of v gathered into the low byte.
__device__ __forceinline__ unsigned every_fourth(unsigned v) {
    v &= 0x11111111u;
    v = (v | (v >> 3)) & 0x03030303u;
    v = (v | (v >> 6)) & 0x000f000fu;
    return (v | (v >> 12)) & 0xffu;
}

// The list [lb, le) into this lane's pixels: v[k][y][c] = channel c of row
// (2 rg + y), column (4 cg + 2 (quarter & 1) + k) of the lane's block.
__device__ __forceinline__ void quad_list(const TileArgs &a, long long lb, long long le, int x0, int y0,
                                          unsigned smem, float (&v)[2][2][3]) {
    constexpr int P = Quad::P;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int quarter = lane >> 3, side = quarter >> 1, cg = lane & 1, rg = (lane >> 1) & 3;
    const unsigned col_at = smem + (unsigned)((warp & 1) * 16 + side * 8 + 4 * cg) * 8u;
    const unsigned row_at = smem + Quad::ROWA + (unsigned)((warp >> 1) * 4 + rg) * 16u;
    const unsigned stage = smem + Quad::kStage;
    const unsigned lists = smem + Quad::kLists + (unsigned)(2 * warp) * Quad::LIST;
    f32x2 acc[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k][0] = acc[k][1] = acc[k][2] = 0ull;
    // thread 2p + h copies half h of staged particle p; the id of the batch
    // after the next is fetched ahead
    const int sp = tid >> 1;
    const unsigned half = (unsigned)(tid & 1);
    const unsigned stage_at = stage + half * (P * 16) + (unsigned)sp * 16u;
    unsigned id = 0;
    if (sp < P && lb + sp < le) {
        id = a.entries[lb + sp];
        cp_async16(stage_at, reinterpret_cast<const char *>(a.recs + id) + half * 16);
        if (lb + P + sp < le) id = a.entries[lb + P + sp];
    }
    unsigned buf = 0;
#pragma unroll 1
    for (long long base = lb; base < le; base += P) {
        const int cnt = (int)(le - base < P ? le - base : P);
        const unsigned st = stage + buf * (P * 32);
        cp_async_wait();
        __syncthreads();
        if (sp < P && base + P + sp < le) {
            cp_async16(stage_at + (buf ^ 1u) * (P * 32),
                       reinterpret_cast<const char *>(a.recs + id) + half * 16);
            if (base + 2 * P + sp < le) id = a.entries[base + 2 * P + sp];
        }
        {
            const int p = tid >> 2, q = tid & 3;
            const bool valid = p < cnt;
            const float4 r0 = lds4(st + p * 16), r1 = lds4(st + P * 16 + p * 16);
            // does the disc (with a margin) reach the rectangles of pixel centres of
            // the blocks in row q of blocks?  A superset of the blocks that hold a
            // covered pixel: a block visited in vain adds clipped zeros.  Lane b < 16
            // gathers the eight bits of block b.
            const float r = r1.x * rsqrtf(r1.x) + 1e-3f;      // approximate: far inside the margin
            const float ax = (float)(x0 - unpack_xi(r0.x)) + (0.5f - r0.y);
            const float ay = (float)(y0 + 8 * q - unpack_yi(r0.x)) + (0.5f - r0.z);
            const float ny = fmaxf(ay, fminf(0.f, ay + 7.f)), room = r * r - ny * ny;
            unsigned bits = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float nx = fmaxf(ax + (float)(8 * u), fminf(0.f, ax + (float)(8 * u + 7)));
                const unsigned h = __ballot_sync(0xffffffffu, valid && nx * nx <= room);
                if ((lane & 3) == u) bits = h;
            }
            if (lane < 16) {
                const unsigned m = every_fourth(bits >> (lane >> 2));
                asm volatile("st.shared.u8 [%0], %1;" ::"r"(smem + Quad::kMask + 8 * lane + warp), "r"(m) : "memory");
            }
            if (valid) quad_tabulate(r0, r1, x0, y0, smem + Quad::slot(p) * Quad::BYTES, q);
        }
        __syncthreads();
        // the lists of this warp's blocks, padded to whole steps
        const uint4 m = ldsu4(smem + Quad::kMask + 16 * warp);
        const int na = __popc(m.x), nl = na + __popc(m.y), nb = __popc(m.z), nr = nb + __popc(m.w);
        const int n = nl > nr ? nl : nr;
        const unsigned sa = Quad::slot(lane), sb = sa + 32;
        if (nl + lane < n + 2) sts_u8(lists + nl + lane, P);
        if (nr + lane < n + 2) sts_u8(lists + Quad::LIST + nr + lane, P);
        if (nl + 32 + lane < n + 2) sts_u8(lists + nl + 32 + lane, P);
        if (nr + 32 + lane < n + 2) sts_u8(lists + Quad::LIST + nr + 32 + lane, P);
        if ((m.x >> lane) & 1u) sts_u8(lists + __popc(m.x & lt), sa);
        if ((m.y >> lane) & 1u) sts_u8(lists + na + __popc(m.y & lt), sb);
        if ((m.z >> lane) & 1u) sts_u8(lists + Quad::LIST + __popc(m.z & lt), sa);
        if ((m.w >> lane) & 1u) sts_u8(lists + Quad::LIST + nb + __popc(m.w & lt), sb);
        __syncwarp();
        unsigned at = lists + (unsigned)side * Quad::LIST + (unsigned)(quarter & 1);
        unsigned off = lds_u8(at);
#pragma unroll 1
        for (int i = 0; i < n; i += 2) {
            const unsigned ca = col_at + off * Quad::BYTES, ra = row_at + off * Quad::BYTES;
            at += 2;
            off = lds_u8(at);
            const float4 c0 = lds4(ca), c1 = lds4(ca + 16);
            f32x2 er, eg, eb, rem;
            lds2x2(ra, er, eg);
            lds2x2(ra + (Quad::ROWB - Quad::ROWA), eb, rem);
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

// Write one pixel's channel: stored (only item of its tile; added to the
// previous chunks' sum when accumulating) or added atomically.
__device__ __forceinline__ void put_value(float *dst, float v, bool store, int accumulate) {
    if (store)
        *dst = accumulate ? *dst + v : v;
    else if (v != 0.f)
        atomicAdd(dst, v);
}

// Points and small particles of an item into the shared tile: thread t of n
// takes every n-th small particle, warp w of the n / 32 every (n / 32)-th run
// of 32 points (Sec. 4.1).
template <int T>
__device__ __forceinline__ void shared_lists(const FrameConst &fc, const TileArgs &a, long long lb0,
                                             long long le0, long long lb1, long long le1, int x0, int y0,
                                             float (*sacc)[T][T], int t, int n) {
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
        warp_points<T>(a, valid, r0, r1, x0, y0, sacc, lane);
    }
#pragma unroll 1
    for (long long k = lb1 + t; k < le1; k += n) {
        const Rec rc = a.recs[a.entries[k]];
        thread_small<T>(fc, rc.r0, rc.r1, x0, y0, sacc);
    }
}

// Dynamic shared memory of one CTA (bytes), T = 16 and 64: the batch tables
// srow and swx, then the staged records st0, st1.  The shared tile sacc of the
// point and small passes (3 T^2 floats) reuses the table space: those passes
// run after the medium list, when the tables are no longer read.
template <int T>
__host__ __device__ constexpr size_t table_bytes() {
    using S = Shape<T>;
    return sizeof(float4) * S::P * T + sizeof(float2) * S::P * S::WXS;
}
static_assert(table_bytes<16>() >= sizeof(float) * 3 * 16 * 16, "shared tile fits the tables");
static_assert(table_bytes<64>() >= sizeof(float) * 3 * 64 * 64, "shared tile fits the tables");
template <int T>
__host__ __device__ constexpr size_t smem_bytes() {
    return T == Quad::T ? (size_t)Quad::kSmem : table_bytes<T>() + sizeof(float4) * 4 * Shape<T>::P;
}

template <int T>
constexpr int min_ctas() { return T == 64 ? 2 : 4; }

// Persistent pass over the work items of every view of the batch: the tile
// pass takes items [0, item_totals[0]), the large pass the next
// item_totals[1] (both counts read from device memory).
template <int T, bool LARGE>
__global__ void __launch_bounds__(kTileThreads, min_ctas<T>()) item_kernel(Views vs, TileArgs a) {
    extern __shared__ float4 smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int *counter = &a.st->item_counter[LARGE ? 1 : 0];
    const int item0 = LARGE ? a.st->item_totals[0] : 0;
    const int n_items = min(a.st->item_totals[LARGE ? 1 : 0], a.items_cap - item0);
    constexpr bool QUAD = T == Quad::T;
    if constexpr (QUAD) {
        if (tid < Quad::BYTES / 16) smem_raw[Quad::kNone / 16 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    using S = Shape<T>;
    constexpr int NW = kTileThreads / 32;
    float4 (*srow)[T] = reinterpret_cast<float4 (*)[T]>(smem_raw);
    float2 (*swx)[S::WXS] = reinterpret_cast<float2 (*)[S::WXS]>(smem_raw + S::P * T);
    float (*sacc)[T][T] = reinterpret_cast<float (*)[T][T]>(smem_raw);   // after the tables
    float4 *st0 = reinterpret_cast<float4 *>(reinterpret_cast<char *>(smem_raw) + table_bytes<T>());
    float4 *st1 = st0 + 2 * S::P;
    __shared__ unsigned band_mask[2][NW];
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
        if (it >= n_items) break;
        if (tid == 0) next = atomicAdd(counter, 1);
        const int idx = item0 + (a.order ? a.order[item0 + it] : it);
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
        const int x0 = (tile % fc.ntx) * T, y0 = (tile / fc.ntx) * T;
        if (list < 0 && tid < 4)
            s_range[tid] = a.offsets[fc.slot_base + (tid < 2 ? L_POINT : L_SMALL) * fc.ntiles + tile + (tid & 1)];
        const bool mine = list < 0 || list >= L_MEDIUM;   // medium (tile pass) or large (large pass)
        const long long cap = a.entries_cap;              // never past the entries written
        const long long lb2 = mine ? min(w.start, cap) : 0, le2 = mine ? min(w.end, cap) : 0;
        const int col = (warp % S::NBX) * S::BW + (lane % S::LW) * S::CMUL;
        const int row0 = (warp / S::NBX) * S::BH + (lane / S::LW) * S::RPL;
        Acc<T> acc;
        float quad[2][2][3];
        if constexpr (QUAD) {
            quad_list(a, lb2, le2, x0, y0, (unsigned)__cvta_generic_to_shared(smem_raw), quad);
        } else {
            acc.zero();
            // medium (or large) particles: tabulate a batch, then every row band
            // adds it.  Records are staged in two alternating buffers (with two
            // band-mask sets): the next batch is stored while the bands of this one
            // are added, and the batch after it is fetched into registers.
            float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0;
            if (lb2 < le2) {
                if (lb2 + tid < le2 && tid < S::P) {
                    const unsigned id = a.entries[lb2 + tid];
                    const Rec rc = a.recs[id];
                    st0[tid] = rc.r0;
                    st1[tid] = rc.r1;
                }
                if (tid < NW) band_mask[0][tid] = 0u;
                if (lb2 + S::P + tid < le2 && tid < S::P) {
                    const unsigned id = a.entries[lb2 + S::P + tid];
                    const Rec rc = a.recs[id];
                    n0 = rc.r0;
                    n1 = rc.r1;
                }
                __syncthreads();
            }
            int buf = 0;
#pragma unroll 1
            for (long long base = lb2; base < le2; base += S::P) {
                const int cnt = (int)(le2 - base < S::P ? le2 - base : S::P);
                tabulate<T>(st0 + buf * S::P, st1 + buf * S::P, cnt, x0, y0, swx, srow, band_mask[buf],
                            tid);
                __syncthreads();
                // stage the next batch (its buffer and masks were last used a batch ago)
                if (tid < S::P) {
                    if (base + S::P + tid < le2) {
                        st0[(buf ^ 1) * S::P + tid] = n0;
                        st1[(buf ^ 1) * S::P + tid] = n1;
                    }
                    if (base + 2 * S::P + tid < le2) {
                        const unsigned id = a.entries[base + 2 * S::P + tid];
                        const Rec rc = a.recs[id];
                        n0 = rc.r0;
                        n1 = rc.r1;
                    }
                }
                if (tid < NW) band_mask[buf ^ 1][tid] = 0u;
                // this warp's row band: only the particles that reach it
                unsigned mask = band_mask[buf][warp];
                while (mask) {
                    const int p = __ffs(mask) - 1;
                    mask &= mask - 1u;
                    band_splat<T>(swx[p], S::PAIRED ? srow[0] + p * (T / 2) : srow[p], col, row0, acc);
                }
                __syncthreads();
                buf ^= 1;
            }
        }

        // points and small particles go through the shared tile, which reuses
        // the table space (the tables are dead once every warp is past here)
        long long lb0 = 0, le0 = 0, lb1 = 0, le1 = 0;
        if (list < 0) {
            if (lb2 >= le2) __syncthreads();   // s_range (the batches' barriers otherwise)
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
            for (int k = tid; k < 3 * T * T; k += kTileThreads) (&sacc[0][0][0])[k] = 0.f;
            __syncthreads();
            shared_lists<T>(fc, a, lb0, le0, lb1, le1, x0, y0, sacc, tid, kTileThreads);
            __syncthreads();
        }
        // write: shared part + registers
        // plain stores where no other item of the pass writes the tile: the large
        // pass adds to what the tile pass left (687k heavy-tailed particles on 3633 x
        // 1145, one large item per tile: 0.112 ms with atomic adds, 0.072 with plain ones)
        const bool store = LARGE ? item_sole(w) : list < 0;
        const int onto = LARGE ? 1 : a.accumulate;
        float *image = a.images[view];
        if constexpr (QUAD) {
            const int quarter = lane >> 3;
            const int row = (warp >> 1) * 8 + ((lane >> 1) & 3) * 2;
            const int cx = (warp & 1) * 16 + (quarter >> 1) * 8 + (lane & 1) * 4 + (quarter & 1) * 2;
            float *dst = image + 3 * ((int64_t)(y0 + row) * fc.width + x0 + cx);
            const int64_t pitch = (int64_t)3 * fc.width;
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
                if (in[y][k]) put_value(dst + pitch * y + 3 * k + c, quad[k][y][c], store, 0);
            }
        } else {
#pragma unroll
            for (int q = 0; q < S::RPL; ++q) {
                const int row = row0 + q;
#pragma unroll
                for (int k = 0; k < S::CPL; ++k) {
                    const int cx = col + S::CSTEP * k;
                    if (y0 + row >= fc.height || x0 + cx >= fc.width) continue;
                    float *dst = image + 3 * ((int64_t)(y0 + row) * fc.width + x0 + cx);
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        put_value(dst + c, (shared_tile ? sacc[c][row][cx] : 0.f) + acc.get(q, k, c),
                                  store, onto);
                }
            }
        }
        if (a.item_cycles) {
            __syncthreads();
            if (tid == 0) a.item_cycles[idx] = clock64() - t_start;
        }
        if (tid == 0) s_item[turn ^ 1] = next;
    }
}

template <int T, bool LARGE>
static void launch_items_t(const Views &vs, const TileArgs &a, int sms, cudaStream_t s) {
    constexpr size_t bytes = smem_bytes<T>();
    cudaFuncSetAttribute(item_kernel<T, LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)bytes);
    item_kernel<T, LARGE><<<sms * min_ctas<T>(), kTileThreads, bytes, s>>>(vs, a);
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
