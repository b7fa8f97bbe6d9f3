// spl_absorb.cu -- the general absorption pass (Eq. 1 with E_p != A_p):
// front-to-back compositing over depth-sorted tile lists, and the composition
// of the partials of split tiles.
#include "spl_tile.cuh"

namespace spl {

// ---------------------------------------------------------------------------
// General absorption (Eq. 1 with E_p != A_p).  Across particle p a ray's
// intensity becomes I exp(-tau) + S (1 - exp(-tau)) with tau = A_p w_p and the
// source term S = E_p / A_p; for the particles of a pixel taken front to back
// this is the same as keeping the transmittance T of the particles in front
// and adding T S (1 - exp(-tau)), then T *= exp(-tau) (the ray starts with
// zero intensity behind the last particle).  Every tile's list holds all its
// particles (points included) sorted front to back by (depth, index); a work
// item runs its range in that order with (T, C) per pixel in registers.  A
// tile that is one item stores C; the segments of a crowded tile store their
// (C, T) partials, and absorb_combine_kernel composes them in segment order:
// C = C_1 + T_1 C_2 + T_1 T_2 C_3 ..., which is the same recurrence.
// ---------------------------------------------------------------------------

// Quarter-warps over 8 x 8 blocks, as in the additive pass (spl_tile.cu: blocks, bands,
// parts of a tile), except that a pixel's particles must be taken in order.  The item's
// list is cut into RANGES contiguous ranges; a batch holds 64 / RANGES particles of
// each, and a quarter-warp takes its block's particles of its own range one after
// the other: the two quarters of a block (and the four warps that share a pair of blocks at
// W = 16) work on different ranges, whose (C, T) are composed at the end.
//
// What bounds it: issue and latency -- 14 packed operations per pixel pair and step beside the
// loads, and each pixel's T is a chain.  One particle per warp step over a 16 x 8 band, a
// lane 2 x 2 pixels, records fetched between two barriers, took 9.48 ms on the
// clustered 10M / 1024^2 frame (covered to 54 %; 8 x 8 blocks to 65 %); this takes
// 8.13 ms (1.24 since hidden segments are left out, below).
template <int W>
struct Absorb {
    static constexpr int P = 64;                   // particles per batch
    // one particle's tables: W / 2 column pairs (w_a, w_b, dx_a^2 B, dx_b^2 B), W / 2 row
    // pairs (A w_a, A w_b, rem_a, rem_b), then (E / A per channel, each value twice; A).  A point:
    // 1 in its column and 0 elsewhere, A in its row, and no clip (0 and 2).  The odd
    // number of 16-byte words puts neighbouring particles in different banks.
    static constexpr int ROWS = 8 * W, SRC = 16 * W, BYTES = 16 * W + 48;
    static constexpr int BL = W / 8, BANDS = BL * BL / 2, G = 8 / BANDS;   // as in Quad
    static constexpr int RANGES = 2 * G, PER = P / RANGES;
    static constexpr int kNone = P * BYTES;        // tables of a particle that changes nothing
    static constexpr int kStage = kNone + BYTES;   // two batches of records and A
    static constexpr int kStageBytes = P * 36;
    static constexpr int kMask = kStage + 2 * kStageBytes;   // per block: the particles that reach it
    static constexpr int kLists = kMask + 16 * 8;
    static constexpr int LIST = 36;                // a block's particles of one range, padded
    static constexpr int kSmem = kLists + 8 * 4 * LIST;
    static_assert(kStage % 16 == 0 && kStageBytes % 16 == 0 && kMask % 16 == 0, "aligned");
    static_assert(G == 1 || G * 16 * W * W <= kNone, "the tables hold the warps' partials");
};
constexpr int kAbsorbCtas = 3;      // per SM: 80 registers; with 4 (64, more spilling) 8.31 ms

__device__ __forceinline__ void cp_async4(unsigned dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ float lds1(unsigned a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}

// Tabulate the particle (r0, r1, A), A > 0, into the block tab: thread q of its four fills column
// pairs and row pairs q, q + 4, ....
template <int W>
__device__ __forceinline__ void absorb_tabulate(float4 r0, float4 r1, float A, bool point, int x0, int y0,
                                                unsigned tab, int q) {
    using Q = Absorb<W>;
    if (q == 0) {
        const float inv = 1.f / A;
        const float e0 = r1.y * inv, e1 = r1.z * inv, e2 = r1.w * inv;
        sts2x2(tab + Q::SRC, pack2(e0, e0), pack2(e1, e1));
        sts2x2(tab + Q::SRC + 16, pack2(e2, e2), pack2(A, 0.f));
    }
    const int cx = unpack_xi(r0.x) - x0, cy = unpack_yi(r0.x) - y0;   // the point's pixel
    const float B = __fdividef(1048576.f, r1.x);
    const f32x2 nkq = pack2(-r0.w, -r0.w), B2 = pack2(B, B), AA = pack2(A, A);
    const float xf = (float)(2 * q - cx), yf = (float)(2 * q - cy);
    const f32x2 x2 = pack2(xf, xf + 1.f), y2 = pack2(yf, yf + 1.f);
    const f32x2 xh = pack2(0.5f - r0.y, 0.5f - r0.y), yh = pack2(0.5f - r0.z, 0.5f - r0.z);
    const f32x2 rr = pack2(r1.x, r1.x), one = pack2(1.f, 1.f), mone = pack2(-1.f, -1.f);
#pragma unroll
    for (int u = 0; u < W / 8; ++u) {
        const unsigned at = tab + 16 * q + 64 * u;
        if (point) {
            const int k = 2 * q + 8 * u;
            sts2x2(at, pack2(k == cx ? 1.f : 0.f, k + 1 == cx ? 1.f : 0.f), 0ull);
            sts2x2(at + Q::ROWS, pack2(k == cy ? A : 0.f, k + 1 == cy ? A : 0.f), pack2(2.f, 2.f));
            continue;
        }
        const f32x2 dx = add2(add2(x2, pack2(8.f * u, 8.f * u)), xh);
        const f32x2 dy = add2(add2(y2, pack2(8.f * u, 8.f * u)), yh);
        const f32x2 dx2 = mul2(dx, dx), dy2 = mul2(dy, dy);
        float ta, tb, wa, wb;
        unpack2(mul2(dx2, nkq), ta, tb);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
        sts2x2(at, pack2(wa, wb), mul2(dx2, B2));
        unpack2(mul2(dy2, nkq), ta, tb);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(ta));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(tb));
        sts2x2(at + Q::ROWS, mul2(AA, pack2(wa, wb)), fma2v(fma2v(dy2, mone, rr), B2, one));
    }
}

// 1 - exp(-tau) for tau >= 0, two values at once, with small relative error everywhere:
// below 1/16 the Taylor series to tau^5 (truncation < tau^5/720 relative, < 2e-9),
// above it one minus the hardware exp2 (relative error there < 16 * 2^-22).
// Computing 1 - exp(-tau) directly would lose all digits of a small tau.
__device__ __forceinline__ f32x2 one_minus_exp_neg2(f32x2 tau) {
    const f32x2 c5 = pack2(1.f / 120.f, 1.f / 120.f), c4 = pack2(-1.f / 24.f, -1.f / 24.f);
    const f32x2 c3 = pack2(1.f / 6.f, 1.f / 6.f), c2 = pack2(-0.5f, -0.5f);
    const f32x2 one = pack2(1.f, 1.f), mone = pack2(-1.f, -1.f);
    const f32x2 nl2e = pack2(-1.4426950408889634f, -1.4426950408889634f);
    f32x2 sr = fma2v(tau, c5, c4);
    sr = fma2v(tau, sr, c3);
    sr = fma2v(tau, sr, c2);
    sr = fma2v(tau, sr, one);
    sr = mul2(tau, sr);
    float u0, u1, e0, e1;
    unpack2(mul2(tau, nl2e), u0, u1);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(u0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(u1));
    const f32x2 ge = fma2v(pack2(e0, e1), mone, one);
    float t0, t1, s0, s1, g0, g1;
    unpack2(tau, t0, t1);
    unpack2(sr, s0, s1);
    unpack2(ge, g0, g1);
    return pack2(t0 < 0.0625f ? s0 : g0, t1 < 0.0625f ? s1 : g1);
}

// The same where tau <= 1, two values at once: tau (1 - tau / 2 + tau^2 q(tau)), q of degree 4
// fitted for the least relative error of the result on [0, 1], weighted eight times below 1/16
// (7.4e-10 there, 6.9e-9 on all of [0, 1]).  The first two coefficients are exact, so that a thin
// particle has no bias that a sum over many would add up.  In FP32 the error is that of the series
// below 1/16 (at most 9.0e-8, 3.1e-8 rms) and at most 1.4e-7 (4.2e-8 rms) up to 1, where the exp2
// form has 1.8e-6 (4.3e-7).  A particle with 0 <= A <= 1 never exceeds tau = 1, since its
// weights are at most 1, so that the choice is made once per warp step; per pixel pair it
// saves the hardware exp2s, the branch's two compares and selects and a packed operation.
// (A fit of one degree less, without the exact terms, biases thin particles by 6e-8: clustered
// 10M frame 2.73 ms, 2.78 so.)
__device__ __forceinline__ f32x2 one_minus_exp_neg2_unit(f32x2 tau) {
    f32x2 sr = fma2v(tau, pack2(0.000135529335f, 0.000135529335f), pack2(-0.00132052274f, -0.00132052274f));
    sr = fma2v(tau, sr, pack2(0.00829810929f, 0.00829810929f));
    sr = fma2v(tau, sr, pack2(-0.0416586585f, -0.0416586585f));
    sr = fma2v(tau, sr, pack2(0.166666105f, 0.166666105f));
    sr = fma2v(tau, sr, pack2(-0.5f, -0.5f));
    sr = fma2v(tau, sr, pack2(1.f, 1.f));
    return mul2(tau, sr);
}

// The step of one particle for a lane's 4 x 2 pixels, with either form of 1 - exp(-tau).
template <bool UNIT>
__device__ __forceinline__ void absorb_step(f32x2 (&tr)[4], f32x2 (&col)[4][3], const float (&wx)[4],
                                            const float (&dxb)[4], f32x2 aw, float rem_a, float rem_b,
                                            f32x2 s0, f32x2 s1, f32x2 s2) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const f32x2 clip = pack2(__saturatef(rem_a - dxb[k]), __saturatef(rem_b - dxb[k]));
        const f32x2 tau = mul2(mul2(pack2(wx[k], wx[k]), clip), aw);
        const f32x2 f = mul2(tr[k], UNIT ? one_minus_exp_neg2_unit(tau) : one_minus_exp_neg2(tau));
        fma2(col[k][0], f, s0);
        fma2(col[k][1], f, s1);
        fma2(col[k][2], f, s2);
        tr[k] = fma2v(f, pack2(-1.f, -1.f), tr[k]);
    }
}

// (C, T) of what lies in front, then of what lies behind it.
__device__ __forceinline__ float4 compose(float4 front, float4 back) {
    return make_float4(fmaf(front.w, back.x, front.x), fmaf(front.w, back.y, front.y),
                       fmaf(front.w, back.z, front.z), front.w * back.w);
}

// A segment behind others is left out once nothing in it can show: a.front holds, per
// segment (and part of a 64-pixel tile), log2 of the largest transmittance of its
// pixels, 0 until it is done, and kHidden when it is left out.  Where the segments in front
// come to less than kOpaque, the product of a pixel's transmittances there is below 2^-160:
// composed in FP32 it is 0 or, under factors above 1/2, stays at the smallest subnormal, so
// that the segment would add at most 2^-149 of its colour.  Whichever of
// the segments in front are done by then, only those count, so that the order of the items
// is free; they are taken by segment number (segment_order_kernel), so that
// the front ones of every tile are done first.  Clustered 10M / 1024^2, 29 segments per
// tile: 8.13 -> 1.17 ms with the order and the composition (1.24 since the polynomial of
// 1 - exp(-tau) has a term more).
constexpr float kOpaque = -160.f, kHidden = -1e30f;

template <int T>
__global__ void __launch_bounds__(kTileThreads, kAbsorbCtas) absorb_kernel(Views vs, TileArgs a,
                                                                           const int *item_offsets) {
    constexpr int W = T == 16 ? 16 : 32, SIDE = T / W, SUB = SIDE * SIDE;
    using Q = Absorb<W>;
    constexpr int P = Q::P, BL = Q::BL;
    extern __shared__ float4 smem_raw[];
    __shared__ int s_item[2];
    __shared__ float s_front;
    __shared__ unsigned s_most[2][kTileThreads / 32];
    volatile float *front = a.front;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_work = min(a.st->item_totals[0], a.items_cap) * SUB;
    const unsigned smem = (unsigned)__cvta_generic_to_shared(smem_raw);
    if (tid < Q::BYTES / 16) smem_raw[Q::kNone / 16 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int band = warp % Q::BANDS, group = warp / Q::BANDS;
    const int brow = band / (BL / 2), bcol = band % (BL / 2) * 2;     // left block of the pair
    const unsigned lt = (1u << lane) - 1u;
    const int quarter = lane >> 3, side = quarter >> 1, cg = lane & 1, rg = (lane >> 1) & 3;
    const bool behind = quarter & 1;               // this quarter's range of the pair 2 group, 2 group + 1
    const unsigned col_at = smem + (unsigned)((bcol + side) * 8 + 4 * cg) * 8u;
    const unsigned row_at = smem + Q::ROWS + (unsigned)(brow * 4 + rg) * 16u;
    const unsigned lists = smem + Q::kLists + (unsigned)(4 * warp) * Q::LIST;
    // threads 2p, 2p + 1 copy the halves of staged record p, thread 128 + p its A
    const int sp = tid < 2 * P ? tid >> 1 : tid - 2 * P;
    const bool copies = tid < 3 * P;
    const unsigned stage_at = smem + Q::kStage +
                              (tid < 2 * P ? (unsigned)(tid & 1) * (P * 16) + (unsigned)sp * 16u
                                           : (unsigned)(P * 32) + (unsigned)sp * 4u);
    int next = 0, done = -1;                       // the segment just finished, if it counts
    if (tid == 0) s_item[0] = atomicAdd(&a.st->item_counter[0], 1);
    for (int turn = 0;; turn ^= 1) {
        __syncthreads();
        if (tid == 0 && done >= 0) {
            unsigned most = 0;
            for (int k = 0; k < kTileThreads / 32; ++k) most = max(most, s_most[turn][k]);
            front[done] = most > 0x7f800000u ? 0.f : log2f(fmaxf(__uint_as_float(most), 1.17549435e-38f));
        }
        done = -1;
        const int it = s_item[turn];
        if (it >= n_work) break;
        if (tid == 0) next = atomicAdd(&a.st->item_counter[0], 1);
        const int idx = a.order ? a.order[it / SUB] : it / SUB, sub = it % SUB;
        const WorkItem w = a.items[idx];
        const int view = item_view(w), list = item_list(w);
        const FrameConst &fc = vs.fcs[view];
        if (front && list >= 0) {
            const int first = item_offsets[w.tile];
            if (warp == 0) {
                float sum = 0.f;
                for (int k = first + lane; k < idx; k += 32) sum += front[(size_t)k * SUB + sub];
#pragma unroll
                for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == 0) s_front = sum;
            }
            __syncthreads();
            if (s_front <= kOpaque) {
                if (tid == 0) {
                    front[(size_t)idx * SUB + sub] = kHidden;
                    s_item[turn ^ 1] = next;
                }
                continue;
            }
            done = idx * SUB + sub;
        }
        const int tile = w.tile - fc.tile_base, width = fc.width, height = fc.height;
        const int x0 = (tile % fc.ntx) * T + sub % SIDE * W, y0 = (tile / fc.ntx) * T + sub / SIDE * W;
        const float r_sml2 = fc.r_sml2;
        const int n_ent = SUB > 1 && (x0 >= width || y0 >= height) ? 0 : (int)(w.end - w.start);
        const unsigned *ent = a.entries + w.start;
        // the staged slot's range and place in it
        const int range = sp / Q::PER;
        const int e0 = (int)((long long)n_ent * range / Q::RANGES) + sp % Q::PER;
        const int e1 = (int)((long long)n_ent * (range + 1) / Q::RANGES);
        const int batches = ((n_ent + Q::RANGES - 1) / Q::RANGES + Q::PER - 1) / Q::PER;
        auto stage_copy = [&](unsigned id, unsigned buf) {
            if (tid < 2 * P)
                cp_async16(stage_at + buf * Q::kStageBytes,
                           reinterpret_cast<const char *>(a.recs + id) + (tid & 1) * 16);
            else
                cp_async4(stage_at + buf * Q::kStageBytes, &a.rec2[id].x);
        };
        f32x2 tr[4], col[4][3];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            tr[k] = pack2(1.f, 1.f);
            col[k][0] = col[k][1] = col[k][2] = 0ull;
        }
        unsigned id = 0, buf = 0;
        if (copies && e0 < e1) {
            stage_copy(ent[e0], 0u);
            if (e0 + Q::PER < e1) id = ent[e0 + Q::PER];
        }
#pragma unroll 1
        for (int b = 0; b < batches; ++b) {
            const unsigned st = smem + Q::kStage + buf * Q::kStageBytes;
            cp_async_wait();
            __syncthreads();
            const int en = e0 + (b + 1) * Q::PER;
            if (copies && en < e1) {
                stage_copy(id, buf ^ 1u);
                if (en + Q::PER < e1) id = ent[en + Q::PER];
            }
            {
                const int p = tid >> 2, q = tid & 3, rp = p / Q::PER;
                bool valid = (int)((long long)n_ent * rp / Q::RANGES) + p % Q::PER + b * Q::PER <
                             (int)((long long)n_ent * (rp + 1) / Q::RANGES);
                const float4 r0 = lds4(st + p * 16), r1 = lds4(st + P * 16 + p * 16);
                const float A = lds1(st + P * 32 + p * 4);
                // a particle with A <= 0 neither emits nor absorbs.  (A range starts at T = 1: those of
                // A < 0, last in the list, would raise T past the largest float there.)
                valid = valid && A > 0.f;
                // the blocks in row q of blocks that the particle reaches (a point: its
                // pixel's; a disc, with a margin, their pixel centres), as in the additive pass
                const bool point = r1.x <= r_sml2;
                const int cx = unpack_xi(r0.x) - x0, cy = unpack_yi(r0.x) - y0;
                const float r = r1.x * rsqrtf(r1.x) + 1e-3f;      // approximate: far inside the margin
                const float ax = (float)-cx + (0.5f - r0.y), ay = (float)(8 * q - cy) + (0.5f - r0.z);
                const float ny = fmaxf(ay, fminf(0.f, ay + 7.f)), room = r * r - ny * ny;
                unsigned bits = 0, any = 0;
#pragma unroll
                for (int u = 0; u < BL; ++u) {
                    const float nx = fmaxf(ax + (float)(8 * u), fminf(0.f, ax + (float)(8 * u + 7)));
                    const bool hit = point ? cx >> 3 == u && cy >> 3 == q : nx * nx <= room;
                    const unsigned h = __ballot_sync(0xffffffffu, valid && q < BL && hit);
                    if ((lane & (BL - 1)) == u) bits = h;
                    any |= h;
                }
                if (lane < BL * BL) {
                    const unsigned m = every_fourth(bits >> (lane / BL));
                    asm volatile("st.shared.u8 [%0], %1;" ::"r"(smem + Q::kMask + 8 * lane + warp), "r"(m)
                                 : "memory");
                }
                if (SUB > 1) valid = (any >> (lane & ~3)) & 0xfu;
                if (valid) absorb_tabulate<W>(r0, r1, A, point, x0, y0, smem + p * Q::BYTES, q);
            }
            __syncthreads();
            // per quarter: its block's particles of its range, in order, padded to the
            // longest of the warp's four
            const unsigned masks = smem + Q::kMask + 8u * (unsigned)(brow * BL + bcol);
            uint4 m;
            if (Q::G == 1) {
                m = ldsu4(masks);
            } else {
                const unsigned l = lds_u16(masks + 2 * group), r = lds_u16(masks + 8 + 2 * group);
                m = make_uint4(l & 0xffu, l >> 8, r & 0xffu, r >> 8);
            }
            const int first = 2 * group * Q::PER + lane;
            const int n0 = __popc(m.x), n1 = __popc(m.y), n2 = __popc(m.z), n3 = __popc(m.w);
            const int n = max(max(n0, n1), max(n2, n3));
            if (n0 + lane <= n) sts_u8(lists + n0 + lane, P);
            if (n1 + lane <= n) sts_u8(lists + Q::LIST + n1 + lane, P);
            if (n2 + lane <= n) sts_u8(lists + 2 * Q::LIST + n2 + lane, P);
            if (n3 + lane <= n) sts_u8(lists + 3 * Q::LIST + n3 + lane, P);
            if ((m.x >> lane) & 1u) sts_u8(lists + __popc(m.x & lt), first);
            if ((m.y >> lane) & 1u) sts_u8(lists + Q::LIST + __popc(m.y & lt), first + Q::PER);
            if ((m.z >> lane) & 1u) sts_u8(lists + 2 * Q::LIST + __popc(m.z & lt), first);
            if ((m.w >> lane) & 1u) sts_u8(lists + 3 * Q::LIST + __popc(m.w & lt), first + Q::PER);
            __syncwarp();
            unsigned at = lists + (unsigned)quarter * Q::LIST;
            unsigned off = lds_u8(at);
#pragma unroll 1
            for (int i = 0; i < n; ++i) {
                const unsigned tab = off * Q::BYTES;
                ++at;
                off = lds_u8(at);
                const float4 c0 = lds4(col_at + tab), c1 = lds4(col_at + tab + 16);
                f32x2 aw, rem, s0, s1, s2, av;
                lds2x2(row_at + tab, aw, rem);
                lds2x2(smem + Q::SRC + tab, s0, s1);
                lds2x2(smem + Q::SRC + 16 + tab, s2, av);
                const float wx[4] = {c0.x, c0.y, c1.x, c1.y}, dxb[4] = {c0.z, c0.w, c1.z, c1.w};
                float rem_a, rem_b, A, unused;
                unpack2(rem, rem_a, rem_b);
                unpack2(av, A, unused);
                if (__all_sync(0xffffffffu, A >= 0.f && A <= 1.f))
                    absorb_step<true>(tr, col, wx, dxb, aw, rem_a, rem_b, s0, s1, s2);
                else
                    absorb_step<false>(tr, col, wx, dxb, aw, rem_a, rem_b, s0, s1, s2);
            }
            buf ^= 1u;
        }
        // the quarters of a block compose their ranges: the front one keeps columns 0 and 1,
        // the one behind 2 and 3
        float4 px[2][2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float mine[2][4], theirs[2][4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const f32x2 a2 = c < 3 ? col[k][c < 3 ? c : 0] : tr[k], b2 = c < 3 ? col[k + 2][c < 3 ? c : 0] : tr[k + 2];
                float a0, a1, b0, b1;
                unpack2(a2, a0, a1);
                unpack2(b2, b0, b1);
                mine[0][c] = behind ? b0 : a0;
                mine[1][c] = behind ? b1 : a1;
                theirs[0][c] = __shfl_xor_sync(0xffffffffu, behind ? a0 : b0, 8);
                theirs[1][c] = __shfl_xor_sync(0xffffffffu, behind ? a1 : b1, 8);
            }
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const float4 u = make_float4(mine[y][0], mine[y][1], mine[y][2], mine[y][3]);
                const float4 v = make_float4(theirs[y][0], theirs[y][1], theirs[y][2], theirs[y][3]);
                px[k][y] = behind ? compose(v, u) : compose(u, v);
            }
        }
        float *image = a.images[view];
        unsigned most = 0;                         // the largest T: a NaN is larger than any
        auto put = [&](int row, int cx, float4 v) {
            if (y0 + row >= height || x0 + cx >= width) return;
            most = max(most, __float_as_uint(v.w));
            if (list < 0) {
                float *dst = image + 3 * ((int64_t)(y0 + row) * width + x0 + cx);
                dst[0] = v.x;
                dst[1] = v.y;
                dst[2] = v.z;
            } else {
                a.partial[(size_t)idx * (T * T) + (sub / SIDE * W + row) * T + sub % SIDE * W + cx] = v;
            }
        };
        const int row = brow * 8 + rg * 2, cx = (bcol + side) * 8 + cg * 4 + (behind ? 2 : 0);
        if constexpr (Q::G == 1) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int y = 0; y < 2; ++y) put(row + y, cx + k, px[k][y]);
        } else {
            // the warps that share a pair of blocks, in the order of their ranges
            float4 (*part)[W * W] = reinterpret_cast<float4 (*)[W * W]>(smem_raw);
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int y = 0; y < 2; ++y) part[group][(row + y) * W + cx + k] = px[k][y];
            __syncthreads();
            static_assert(Q::G == 1 || W * W == kTileThreads, "one pixel per thread");
            float4 v = part[0][tid];
#pragma unroll
            for (int g = 1; g < Q::G; ++g) v = compose(v, part[g][tid]);
            put(tid / W, tid % W, v);
        }
        most = __reduce_max_sync(0xffffffffu, most);
        if (lane == 0) s_most[turn ^ 1][warp] = most;
        if (tid == 0) s_item[turn ^ 1] = next;
    }
}

// Tiles cut into several items: compose the items' partials in list order.  A CTA
// takes 32 pixels of a tile; each of its eight warps composes an eighth of the
// items, and the eighths are composed in order (the composition is associative).
// Bound by the partials' traffic (16 B per pixel and item): a crowded tile has
// hundreds of items, and one thread per pixel running through all of them in four
// passes of a single CTA per tile was a chain of loads (597 us for the clustered
// 10M / 1024^2 frame; now 94 us).
template <int T>
__global__ void __launch_bounds__(256) absorb_combine_kernel(Views vs, const int *item_offsets,
                                                             const float4 *partial,
                                                             const float *front, float *const *images) {
    constexpr int GROUPS = T * T / 32, SIDE = T == 64 ? 2 : 1, SUB = SIDE * SIDE;
    __shared__ float4 part[8][32];
    __shared__ int s_n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long u = blockIdx.x; u < (long long)vs.total_tiles * GROUPS; u += gridDim.x) {
        const int g = (int)(u / GROUPS), px = (int)(u % GROUPS) * 32 + lane;
        const int i0 = item_offsets[g];
        int n = item_offsets[g + 1] - i0;
        if (n < 2) continue;                       // the same for the whole CTA
        if (front) {                               // up to the first segment left out
            const int first = (int)(u % GROUPS) * 32, sub = first / T / 32 * SIDE + first % T / 32;
            if (threadIdx.x == 0) s_n = n;
            __syncthreads();
            for (int k = threadIdx.x; k < n; k += 256)
                if (front[(size_t)(i0 + k) * SUB + (SUB > 1 ? sub : 0)] == kHidden) {
                    atomicMin(&s_n, k);
                    break;
                }
            __syncthreads();
            n = s_n;
        }
        const int a = i0 + (int)((long long)n * warp / 8), b = i0 + (int)((long long)n * (warp + 1) / 8);
        float c0 = 0.f, c1 = 0.f, c2 = 0.f, tr = 1.f;
#pragma unroll 4
        for (int it = a; it < b; ++it) {
            const float4 v = partial[(size_t)it * (T * T) + px];
            c0 = fmaf(tr, v.x, c0);
            c1 = fmaf(tr, v.y, c1);
            c2 = fmaf(tr, v.z, c2);
            tr *= v.w;
        }
        part[warp][lane] = make_float4(c0, c1, c2, tr);
        __syncthreads();
        if (warp == 0) {
            for (int k = 1; k < 8; ++k) {
                const float4 v = part[k][lane];
                c0 = fmaf(tr, v.x, c0);
                c1 = fmaf(tr, v.y, c1);
                c2 = fmaf(tr, v.z, c2);
                tr *= v.w;
            }
            const int view = view_of_tile(vs.fcs, vs.nviews, g);
            const FrameConst &fc = vs.fcs[view];
            const int tile = g - fc.tile_base;
            const int x = (tile % fc.ntx) * T + px % T, y = (tile / fc.ntx) * T + px / T;
            if (x < fc.width && y < fc.height) {
                float *dst = images[view] + 3 * ((int64_t)y * fc.width + x);
                dst[0] = c0;
                dst[1] = c1;
                dst[2] = c2;
            }
        }
        __syncthreads();
    }
}

// Every segment's place in a.front, and, unless the items have an order, their segment
// numbers as costs whose buckets put the first ones first.
__global__ void segment_order_kernel(const WorkItem *items, int items_cap, const DevStats *st,
                                     const int *item_offsets, int sub, float *front, float *cost) {
    const int n = min(st->item_totals[0], items_cap);
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < n; it += gridDim.x * blockDim.x) {
        for (int k = 0; k < sub; ++k) front[(size_t)it * sub + k] = 0.f;
        if (cost) cost[it] = bucket_cost(it - item_offsets[items[it].tile]);
    }
}

void launch_segment_order(const TileArgs &a, const int *item_offsets, int tile, float *cost, cudaStream_t s) {
    segment_order_kernel<<<256, 256, 0, s>>>(a.items, a.items_cap, a.st, item_offsets, tile == 64 ? 4 : 1,
                                             a.front, cost);
    ++g_launches;
}

template <int T>
static void launch_absorb_t(const Views &vs, const TileArgs &a, const int *item_offsets, int sms,
                            cudaStream_t s) {
    constexpr size_t bytes = Absorb<(T == 16 ? 16 : 32)>::kSmem;
    cudaFuncSetAttribute(absorb_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    absorb_kernel<T><<<sms * kAbsorbCtas, kTileThreads, bytes, s>>>(vs, a, item_offsets);
    ++g_launches;
    const long long units = (long long)vs.total_tiles * (T * T / 32);
    const int grid = (int)(units < sms * 8 ? units : sms * 8);
    if (grid > 0) {
        absorb_combine_kernel<T><<<grid, 256, 0, s>>>(vs, item_offsets, a.partial, a.front, a.images);
        ++g_launches;
    }
}

void launch_absorb_pass(const Views &vs, const TileArgs &a, const int *item_offsets, int sms,
                        cudaStream_t s) {
    if (vs.tile == 16)
        launch_absorb_t<16>(vs, a, item_offsets, sms, s);
    else if (vs.tile == 64)
        launch_absorb_t<64>(vs, a, item_offsets, sms, s);
    else
        launch_absorb_t<32>(vs, a, item_offsets, sms, s);
}

}  // namespace spl
