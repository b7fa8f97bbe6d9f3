// spl_raster.cu -- rasterisation (Sec. 2 "Processing and Rasterization",
// Sec. 4 one-thread-per-particle) and binning of particles into tile lists
// (the data organisation of Sec. 4, built with counts, a scan and a scatter
// instead of a radix sort by tile index; the absorption mode, whose lists are in
// depth order, sorts them by tile).
#include <cstddef>

#include "spl_geom.cuh"

namespace spl {

// ---------------------------------------------------------------------------
// double-float ("df") arithmetic in FP32: a value is hi + lo with |lo| <=
// ulp(hi)/2.  Error-free transforms: Knuth's two-sum, Dekker's fast two-sum
// (|a| >= |b|), and the FMA-based exact product.  The projection needs
// ~1e-9 relative accuracy (1e-6 px at a 1000 px offset); FP32 alone gives
// ~1e-4 px, which would cost ~1e-3 relative error on a 1 px Gaussian's tail.
// The kernel is bound by instruction issue: the rows of x_c and y_c, and the two screen
// coordinates, go through packed FP32x2 instructions, and a row's three products
// are summed with one compensation term (the Dot2 scheme of Ogita, Rump and Oishi)
// instead of a normalised df sum after each.  Clustered 10M: raster 0.358 -> 0.343 ms, with 5
// CTAs per SM (4 or 6: 0.364, 0.343).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float as_f(f32x2 v, int k) {
    float lo, hi;
    unpack2(v, lo, hi);
    return k ? hi : lo;
}
__device__ __forceinline__ f32x2 as2(float2 v) { return pack2(v.x, v.y); }
__device__ __forceinline__ float addv(float a, float b) { return __fadd_rn(a, b); }   // (never contracted)
__device__ __forceinline__ float mulv(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fmav(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float negv(float a) { return -a; }
__device__ __forceinline__ f32x2 addv(f32x2 a, f32x2 b) { return add2(a, b); }
__device__ __forceinline__ f32x2 mulv(f32x2 a, f32x2 b) { return mul2(a, b); }
__device__ __forceinline__ f32x2 fmav(f32x2 a, f32x2 b, f32x2 c) { return fma2v(a, b, c); }
__device__ __forceinline__ f32x2 negv(f32x2 a) { return a ^ 0x8000000080000000ull; }

// A df value, or two of them (V = f32x2).
template <typename V>
struct df { V hi, lo; };

template <typename V>
__device__ __forceinline__ df<V> two_sum(V a, V b) {
    const V s = addv(a, b);
    const V bb = addv(s, negv(a));
    return {s, addv(addv(a, negv(addv(s, negv(bb)))), addv(b, negv(bb)))};
}
template <typename V>
__device__ __forceinline__ df<V> fast_two_sum(V a, V b) {
    const V s = addv(a, b);
    return {s, addv(b, negv(addv(s, negv(a))))};
}

// R x - E for one row (or the pair of rows): products exact, their sum and the
// compensation carried in two floats.
template <typename V>
__device__ __forceinline__ df<V> row_times(const V *Rhi, const V *Rlo, V Ehi, V Elo, const V *x) {
    V s = mulv(Rhi[0], x[0]);
    V c = fmav(Rlo[0], x[0], fmav(Rhi[0], x[0], negv(s)));
#pragma unroll
    for (int k = 1; k < 3; ++k) {
        const V p = mulv(Rhi[k], x[k]);
        c = addv(fmav(Rlo[k], x[k], c), fmav(Rhi[k], x[k], negv(p)));
        const df<V> t = two_sum(s, p);
        s = t.hi;
        c = addv(c, t.lo);
    }
    const df<V> t = two_sum(s, negv(Ehi));
    c = addv(c, addv(t.lo, negv(Elo)));
    return fast_two_sum(t.hi, c);
}

// half + f a / b given rb ~ 1 / b.hi (a few ulp suffice): the first quotient's
// residual is exact (FMA) but for the low parts' rounding and is divided again, so
// that the quotient keeps df accuracy.
__device__ __forceinline__ df<f32x2> project(df<f32x2> a, df<float> b, float rb, f32x2 fhi, f32x2 flo,
                                             f32x2 half) {
    const f32x2 rb2 = pack2(rb, rb), bh = pack2(-b.hi, -b.hi), bl = pack2(-b.lo, -b.lo);
    const f32x2 q1 = mul2(a.hi, rb2);
    const f32x2 r = add2(fma2v(bh, q1, a.hi), fma2v(bl, q1, a.lo));
    const df<f32x2> q = fast_two_sum(q1, mul2(r, rb2));
    const f32x2 p = mul2(fhi, q.hi);
    const f32x2 e = fma2v(flo, q.hi, fma2v(fhi, q.lo, fma2v(fhi, q.hi, negv(p))));
    const df<f32x2> s = two_sum(half, p);
    return fast_two_sum(s.hi, add2(s.lo, e));
}

// Split x_s = xi + xf with xi integral (int16 range) and xf in [0, 1).
__device__ __forceinline__ void split_pos(df<float> v, int &xi, float &xf) {
    const float lim = 30000.f;
    if (v.hi < -lim || v.hi > lim) {       // far off screen: only a huge splat can reach
        float c = fminf(fmaxf(v.hi, -lim), lim);
        xi = (int)c;
        xf = (v.hi - c) + v.lo;
        return;
    }
    float fl = floorf(v.hi);
    xi = (int)fl;
    xf = (v.hi - fl) + v.lo;
    if (xf >= 1.f) { xf -= 1.f; xi += 1; }
    if (xf < 0.f) { xf += 1.f; xi -= 1; }
}

template <bool HALF>
__device__ __forceinline__ float load_attr(const void *p, int64_t i) {
    if (HALF) return __half2float(static_cast<const __half *>(p)[i]);
    return static_cast<const float *>(p)[i];
}

// Smoothing length of particle i: FP32 (ATTR 0, 2), binary16 (ATTR 1), or a
// 16-bit logarithmic code k with h = 2^(h_log2_min + k / 4096) (ATTR 3).
template <int ATTR>
__device__ __forceinline__ float load_h(const void *p, int64_t i, float h_log2_min) {
    if (ATTR == 3)
        return exp2f(fmaf((float)static_cast<const unsigned short *>(p)[i], 1.f / 4096.f, h_log2_min));
    return load_attr<ATTR == 1>(p, i);
}

// Rasterise one particle into its record; returns its class.  q2 receives
// (absorption coefficient A, depth key) for the absorption mode: A =
// absorption * brightness * I, the key z_c rounded to float (the double-float
// value's leading part).
__device__ __forceinline__ int raster_one(const FrameConst &fc, const float *spal, float x, float y,
                                          float z, float h, float inten, float s, const float *crgb,
                                          float4 &r0, float4 &r1, float2 &q2) {
    // roto-translation x_c = R x - R eye, in df
    const float pos[3] = {x, y, z};
    const f32x2 pos2[3] = {pack2(x, x), pack2(y, y), pack2(z, z)};
    const f32x2 Rh[3] = {as2(fc.Rxy_hi[0]), as2(fc.Rxy_hi[1]), as2(fc.Rxy_hi[2])};
    const f32x2 Rl[3] = {as2(fc.Rxy_lo[0]), as2(fc.Rxy_lo[1]), as2(fc.Rxy_lo[2])};
    const df<f32x2> cxy = row_times(Rh, Rl, as2(fc.Exy_hi), as2(fc.Exy_lo), pos2);
    const df<float> cz = row_times(fc.Rz_hi, fc.Rz_lo, fc.Ez_hi, fc.Ez_lo, pos);
    r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    r1 = make_float4(-1.f, 0.f, 0.f, 0.f);
    q2 = make_float2(0.f, 0.f);
    // non-finite inputs or a negative smoothing length: inactive
    // (0 v is zero for every finite v, NaN for the others)
    float zero = fmaf(0.f, x, fmaf(0.f, y, fmaf(0.f, z, fmaf(0.f, h, fmaf(0.f, inten, 0.f * s)))));
    if (crgb) zero = fmaf(0.f, crgb[0], fmaf(0.f, crgb[1], fmaf(0.f, crgb[2], zero)));
    if (!(zero == 0.f) || h < 0.f) return CLS_INACTIVE;
    const float zc = cz.hi;
    if (!(zc > fc.z_near)) return CLS_INACTIVE;
    // logarithms of processed quantities (Sec. 2)
    if (fc.log_flags & 1) {
        if (!(inten > 0.f)) return CLS_INACTIVE;
        inten = log10f(inten);
    }
    if (fc.log_flags & 2) {
        if (!(s > 0.f)) return CLS_INACTIVE;
        s = log10f(s);
    }
    // perspective projection
    const df<f32x2> sp = project(cxy, cz, 1.f / zc, as2(fc.f2_hi), as2(fc.f2_lo), as2(fc.half));
    int xi, yi;
    float xf, yf;
    split_pos({as_f(sp.hi, 0), as_f(sp.lo, 0)}, xi, xf);
    split_pos({as_f(sp.hi, 1), as_f(sp.lo, 1)}, yi, yf);
    // screen smoothing length and radius (Eq. 7)
    const float sig = fc.sig_fac * h * fc.fhi / zc;
    const float r = fc.chi * sig;
    // colour: normalise, palette look-up, scale by intensity (Sec. 2)
    float sn = fminf(fmaxf((s - fc.s_min) * fc.s_inv, 0.f), 1.f);
    float col[3];
    if (crgb) {
        col[0] = crgb[0]; col[1] = crgb[1]; col[2] = crgb[2];
    } else if (fc.npal == 1) {
        col[0] = spal[0]; col[1] = spal[1]; col[2] = spal[2];
    } else {
        float u = sn * (float)(fc.npal - 1);
        int k0 = min((int)floorf(u), fc.npal - 2);
        float t = u - (float)k0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float a = spal[3 * k0 + k], b = spal[3 * k0 + 3 + k];
            col[k] = a + t * (b - a);
        }
    }
    const float amp = fc.brightness * inten;
    // inactive when the disc's box misses the screen (Sec. 2, Fig. 4)
    const float xsf = (float)xi + xf, ysf = (float)yi + yf;
    if (xsf + r < 0.f || xsf - r >= (float)fc.width || ysf + r < 0.f || ysf - r >= (float)fc.height)
        return CLS_INACTIVE;
    r0 = make_float4(pack_xy(xi, yi), xf, yf, 1.4426950408889634f / (sig * sig));
    r1 = make_float4(r * r, amp * col[0], amp * col[1], amp * col[2]);
    q2 = make_float2(fc.absorption * amp, zc);
    return record_class(fc, r1.x);
}

// Tile footprint of one rasterised particle for the point / small / medium
// lists: a box of tiles [tx0, tx0 + bw) x [ty0, ty0 + nbox / bw) (nbox = 0:
// no entry); disc = 1 when a tile of the box must also be reached by the disc.
// Large particles are handled by large_tiles.  In the absorption mode
// points join the medium list, so that a tile's particles form one list that
// can be ordered by depth.
struct TileFoot { int list, tx0, ty0, bw, nbox, disc; float reach2; };

__device__ __forceinline__ TileFoot tile_footprint(const FrameConst &fc, int cls, float4 r0, float4 r1) {
    TileFoot f{-1, 0, 0, 1, 0, 0, 0.f};
    if (cls == CLS_POINT) {
        const int xi = unpack_xi(r0.x), yi = unpack_yi(r0.x);
        if (xi >= 0 && yi >= 0 && xi < fc.width && yi < fc.height) {
            f.list = fc.absorb ? L_MEDIUM : L_POINT;
            f.tx0 = xi >> fc.tile_shift; f.ty0 = yi >> fc.tile_shift; f.nbox = 1;
        }
        return f;
    }
    if (cls != CLS_SMALL && cls != CLS_MEDIUM) return f;
    PixBox b;
    if (!splat_box(fc, r0, r1.x, b)) return f;
    f.list = cls == CLS_SMALL ? L_SMALL : L_MEDIUM;
    f.disc = 1;
    f.reach2 = disc_reach2(r1.x);
    // the box is clamped to the image: non-negative pixel indices
    f.tx0 = b.i0 >> fc.tile_shift;
    f.ty0 = b.j0 >> fc.tile_shift;
    f.bw = (b.i1 >> fc.tile_shift) - f.tx0 + 1;
    f.nbox = f.bw * ((b.j1 >> fc.tile_shift) - f.ty0 + 1);
    return f;
}

// The (particle, box tile) pairs of a warp's 32 particles, taken 32 at a time
// across the lanes instead of one particle per lane: a lane with a wide
// footprint no longer holds the warp for as many rounds as it has tiles.
// Pairs are numbered particle by particle, each particle's box row by row.  The
// particles that have pairs leave their footprints in the warp's shared memory,
// closed up; the first pairs of the particles that start in a round, one bit each, tell
// every lane its particle by a count of the bits up to its own.  (A binary search over the
// lanes' prefix sums and nine shuffles of the owner's footprint, without the shared
// memory, took 3 % longer in the raster and, with a match of the warp's equal slots, 16 %
// longer in the list fill.)
struct FootWarp {
    int4 a[32];                // first pair, tile corner, (list + 1) | disc << 3 | lane << 4 | width << 9, 1 / width
    float4 b[32];              // r0.x, r0.y, r0.z, squared reach
};

struct FootPairs {
    int start, total, before;  // this lane's first pair (or -1), the warp's pairs, particles begun

    __device__ __forceinline__ FootPairs(const TileFoot &f, float4 r0, FootWarp &w, int lane) {
        int incl = f.nbox;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        total = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned have = __ballot_sync(0xffffffffu, f.nbox > 0);
        start = f.nbox > 0 ? incl - f.nbox : -1;
        before = 0;
        __syncwarp();                       // the previous particles' footprints are read
        if (f.nbox > 0) {
            const int k = __popc(have & ((1u << lane) - 1u));
            w.a[k] = make_int4(start, (f.tx0 & 0xFFFF) | (f.ty0 << 16),
                               (f.list + 1) | f.disc << 3 | lane << 4 | f.bw << 9,
                               __float_as_int(1.f / (float)f.bw));
            w.b[k] = make_float4(r0.x, r0.y, r0.z, f.reach2);
        }
        __syncwarp();
    }

    // Slot (list * ntiles + tile) of pair base + lane, or -1 when it is past the warp's
    // pairs or the disc misses that tile, and the owner lane.  Every lane of the warp
    // calls this, for base = 0, 32, ...
    __device__ __forceinline__ int slot(const FrameConst &fc, const FootWarp &w, int base, int lane,
                                        int &owner) {
        const int rel = start - base;
        const unsigned mine = start >= 0 && rel >= 0 && rel < 32 ? 1u << rel : 0u;
        const unsigned heads = __reduce_or_sync(0xffffffffu, mine);
        const int k = before + __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
        before += __popc(heads);
        const int j = base + lane;
        owner = 0;
        if (j >= total) return -1;
        const int4 a = w.a[k];
        owner = (a.z >> 4) & 31;
        // (t + 1/2) / bw is at least 1/(2 bw) away from an integer, far more than
        // the rounding of the product: the quotient is exact
        const int t = j - a.x, bw = a.z >> 9;
        const int ky = (int)(((float)t + 0.5f) * __int_as_float(a.w)), kx = t - ky * bw;
        const int tx = (a.y & 0xFFFF) + kx, ty = (a.y >> 16) + ky;
        if (a.z & 8) {
            const float4 b = w.b[k];
            if (!disc_meets_tile(fc, make_float4(b.x, b.y, b.z, 0.f), b.w, tx, ty)) return -1;
        }
        return ((a.z & 7) - 1) * fc.ntiles + ty * fc.ntx + tx;
    }
};

// ---------------------------------------------------------------------------
// Per-CTA aggregation of list slots.  A clustered particle set puts 1e5-1e6
// entries into single tiles; one global atomic per entry then serialises in
// L2.  Each CTA takes a contiguous chunk of particles and accumulates its
// entries in a small shared-memory hash table (open addressing, key = list *
// ntiles + tile), so that a hot slot receives one global atomic per CTA.  A key that finds no
// free place within kProbe probes falls back to global atomics; the table is
// never emptied while a CTA runs, so that choice is the same for every
// occurrence of the key within the CTA.
// ---------------------------------------------------------------------------
// kHashBits, kHash (slots) and kChunk (particles per CTA) are in spl_internal.cuh
constexpr int kProbe = 32;

__device__ __forceinline__ int hash_slot(const int *keys, int key, int bits, bool insert) {
    unsigned h = ((unsigned)key * 2654435761u) >> (32 - bits);
    for (int probe = 0; probe < kProbe; ++probe) {
        const int slot = (int)((h + (unsigned)probe) & ((1u << bits) - 1u));
        const int k = *(volatile const int *)&keys[slot];
        if (k == key) return slot;
        if (k == -1) {
            if (!insert) return -1;
            const int old = atomicCAS((int *)&keys[slot], -1, key);
            if (old == -1 || old == key) return slot;
        }
    }
    return -1;
}

// Count the slots of one round (one (particle, tile) pair per lane); a key
// with no room in the table is counted in ovf (placed through the cursors).
// Each lane adds its own pair: combining the warp's equal keys first (a match mask) cost
// more than it saved, here (clustered 10M / 1024^2 raster 0.425 -> 0.388 ms, 30M / 2048^2
// 1.462 -> 1.244 ms) and in the scatter, whose adds return the entry's rank (10M: 0.363 ->
// 0.314 ms).
__device__ __forceinline__ void count_round(int key, int bits, int *keys, int *vals, int *govf) {
    if (key >= 0) {
        const int slot = hash_slot(keys, key, bits, true);
        if (slot >= 0)
            atomicAdd(&vals[slot], 1);
        else
            atomicAdd(&govf[key], 1);
    }
}

__device__ __forceinline__ void hash_clear(int *keys, int *vals, int size) {
    for (int k = threadIdx.x; k < size; k += blockDim.x) {
        keys[k] = -1;
        vals[k] = 0;
    }
}

// Flush the CTA's hash table into the global slot counts, keep the table
// with every slot's offset inside its slot (tab: size entries) for the
// scatter, and clear it.
__device__ __forceinline__ void hash_flush(int *keys, int *vals, int size, int *gcounts, int2 *tab) {
    __syncthreads();
    for (int k = threadIdx.x; k < size; k += blockDim.x) {
        const int key = keys[k];
        int off = 0;
        if (key >= 0) off = atomicAdd(&gcounts[key], vals[k]);
        tab[k] = make_int2(key, off);
        keys[k] = -1;
        vals[k] = 0;
    }
    __syncthreads();
}

// Load view v's constants into shared memory (the whole CTA waits).
__device__ __forceinline__ void load_view(const FrameConst *fcs, int v, FrameConst *sfc) {
    __syncthreads();
    const int words = (int)(sizeof(FrameConst) / sizeof(int));
    for (int k = threadIdx.x; k < words; k += blockDim.x)
        reinterpret_cast<int *>(sfc)[k] = reinterpret_cast<const int *>(fcs + v)[k];
    __syncthreads();
}

// One thread per particle and view: the particle's chunk is rasterised for
// every view of the batch (its inputs are read from HBM once and then hit in
// L2), records are written to rec[view * n + id], list entries are counted.
// ATTR: 0 = h, I, s in FP32; 1 = all three in binary16; 2 = h in FP32, I and s
// in binary16; 3 = h as a 16-bit logarithmic code, I and s in binary16.  RGB:
// per-particle colour components replace the palette.
template <int ATTR, bool RGB>
__global__ void __launch_bounds__(256, 5) raster_kernel(Views vs, RasterArgs a) {
    __shared__ float spal[3 * kMaxPalette];
    __shared__ int keys[kHash], vals[kHash];
    __shared__ FootWarp feet[8];
    __shared__ unsigned long long bstat[5];
    __shared__ FrameConst sfc;
    const int bits = a.shape.hash_bits, size = 1 << bits;
    hash_clear(keys, vals, size);
    if (threadIdx.x < 5) bstat[threadIdx.x] = 0;
    const int lane = threadIdx.x & 31;
    unsigned n_act = 0, n_pt = 0, n_sm = 0, n_md = 0, n_lg = 0;
    const int64_t c0 = (int64_t)blockIdx.x * a.shape.chunk;
    const int64_t c1 = c0 + a.shape.chunk < a.n ? c0 + a.shape.chunk : a.n;
    for (int v = 0; v < vs.nviews; ++v) {
        load_view(vs.fcs, v, &sfc);
        const FrameConst &fc = sfc;
        for (int k = threadIdx.x; k < 3 * fc.npal; k += blockDim.x) spal[k] = a.pal[k];
        __syncthreads();
        // all lanes of a warp run the same number of iterations (warp collectives)
        for (int64_t base = c0; base < c1; base += blockDim.x) {
            const int64_t i = base + threadIdx.x;
            const bool valid = i < c1;
            int cls = CLS_INACTIVE;
            float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = make_float4(-1.f, 0.f, 0.f, 0.f);
            const int64_t rec = fc.rec_base + i;
            if (valid) {
                float2 q2;
                float crgb[3] = {0.f, 0.f, 0.f};
                if (RGB) {
                    crgb[0] = a.cr[i]; crgb[1] = a.cg[i]; crgb[2] = a.cb[i];
                }
                cls = raster_one(fc, spal, a.x[i], a.y[i], a.z[i], load_h<ATTR>(a.h, i, a.h_log2_min),
                                 load_attr<ATTR != 0>(a.I, i), load_attr<ATTR != 0>(a.s, i),
                                 RGB ? crgb : nullptr, r0, r1, q2);
                a.recs[rec] = Rec{r0, r1};
                if (a.rec2) a.rec2[rec] = q2;
            }
            const TileFoot foot = valid ? tile_footprint(fc, cls, r0, r1) : TileFoot{-1, 0, 0, 1, 0, 0, 0.f};
            FootPairs pairs(foot, r0, feet[threadIdx.x >> 5], lane);
            for (int base = 0; base < pairs.total; base += 32) {
                int owner;
                const int ls = pairs.slot(fc, feet[threadIdx.x >> 5], base, lane, owner);
                count_round(ls >= 0 ? fc.slot_base + ls : -1, bits, keys, vals, a.ovf);
            }
            n_act += cls != CLS_INACTIVE;
            n_pt += cls == CLS_POINT;
            n_sm += cls == CLS_SMALL;
            n_md += cls == CLS_MEDIUM;
            n_lg += cls == CLS_LARGE;
            // append large records to the large list (one atomic per warp)
            const unsigned big = __ballot_sync(0xffffffffu, cls == CLS_LARGE);
            if (big) {
                unsigned basek = 0;
                const int leader = __ffs(big) - 1;
                if (lane == leader) basek = atomicAdd(&a.st->n_large_ids, (unsigned)__popc(big));
                basek = __shfl_sync(0xffffffffu, basek, leader);
                if (cls == CLS_LARGE)
                    a.large_ids[basek + __popc(big & ((1u << lane) - 1u))] = (unsigned)rec;
            }
        }
        // one global atomic per distinct slot of this CTA and view
        hash_flush(keys, vals, size, a.counts, a.ctab + (((int64_t)blockIdx.x * vs.nviews + v) << bits));
    }
    n_act = __reduce_add_sync(0xffffffffu, n_act);
    n_pt = __reduce_add_sync(0xffffffffu, n_pt);
    n_sm = __reduce_add_sync(0xffffffffu, n_sm);
    n_md = __reduce_add_sync(0xffffffffu, n_md);
    n_lg = __reduce_add_sync(0xffffffffu, n_lg);
    if (lane == 0) {
        atomicAdd(&bstat[0], (unsigned long long)n_act);
        atomicAdd(&bstat[1], (unsigned long long)n_pt);
        atomicAdd(&bstat[2], (unsigned long long)n_sm);
        atomicAdd(&bstat[3], (unsigned long long)n_md);
        atomicAdd(&bstat[4], (unsigned long long)n_lg);
    }
    __syncthreads();
    if (threadIdx.x < 5 && bstat[threadIdx.x]) {
        // n_active .. n_large are consecutive fields of DevStats
        atomicAdd(&a.st->n_active + threadIdx.x, bstat[threadIdx.x]);
    }
}

void launch_raster(const Views &vs, RasterArgs a, int attr, int sms, cudaStream_t s) {
    if (a.n <= 0 || vs.nviews <= 0) return;
    a.shape = bin_shape(a.n, sms);
    const int64_t blocks = (a.n + a.shape.chunk - 1) / a.shape.chunk;
    const bool rgb = a.cr != nullptr;
    if (attr == 1) {
        if (rgb) raster_kernel<1, true><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
        else raster_kernel<1, false><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
    } else if (attr == 2) {
        if (rgb) raster_kernel<2, true><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
        else raster_kernel<2, false><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
    } else if (attr == 3) {
        if (rgb) raster_kernel<3, true><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
        else raster_kernel<3, false><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
    } else {
        if (rgb) raster_kernel<0, true><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
        else raster_kernel<0, false><<<(unsigned)blocks, 256, 0, s>>>(vs, a);
    }
    ++g_launches;
}

// ---------------------------------------------------------------------------
// Large particles: one warp per large record walks its (possibly thousands
// of) tiles.  mode 0 counts entries, mode 1 scatters record indices through
// the cursors.
// ---------------------------------------------------------------------------
template <int MODE>
__device__ __forceinline__ void large_tiles(const Views &vs, const BinArgs &a, unsigned block,
                                            unsigned nblocks) {
    const int lane = threadIdx.x & 31;
    const unsigned nl = a.st->n_large_ids;
    const unsigned warps = nblocks * (blockDim.x >> 5);
    for (unsigned w = block * (blockDim.x >> 5) + (threadIdx.x >> 5); w < nl; w += warps) {
        const unsigned rec = a.large_ids[w];
        const FrameConst &fc = vs.fcs[(int)(rec / (unsigned long long)vs.n)];
        const Rec rc = a.recs[rec];
        const float4 r0 = rc.r0, r1 = rc.r1;
        PixBox b;
        if (!splat_box(fc, r0, r1.x, b)) continue;
        const int tx0 = b.i0 >> fc.tile_shift, ty0 = b.j0 >> fc.tile_shift;
        const int ntx = (b.i1 >> fc.tile_shift) - tx0 + 1;
        const int nt = ntx * ((b.j1 >> fc.tile_shift) - ty0 + 1);
        const float reach2 = disc_reach2(r1.x);
        for (int k = lane; k < nt; k += 32) {
            const int tx = tx0 + k % ntx, ty = ty0 + k / ntx;
            if (!disc_meets_tile(fc, r0, reach2, tx, ty)) continue;
            const int slot = fc.slot_base + L_LARGE * fc.ntiles + ty * fc.ntx + tx;
            if (MODE == 0) {
                atomicAdd(&a.ovf[slot], 1);
            } else {
                // the entries that cover their tile go to the list's end (16-pixel
                // tiles have no use for them)
                const bool full = fc.tile > 16 && disc_covers_tile(fc, r0, r1.x, tx, ty);
                const long long pos =
                    full ? a.offsets[slot + 1] - 1 - atomicAdd(&a.full[fc.tile_base + ty * fc.ntx + tx], 1)
                         : (long long)atomicAdd(reinterpret_cast<unsigned long long *>(&a.cursor[slot]), 1ULL);
                if (pos < a.entries_cap)
                    a.entries[pos] = rec;
                else
                    atomicOr(&a.st->err, ERR_LIST_OVERFLOW);
            }
        }
    }
}

__global__ void __launch_bounds__(256) count_large_kernel(Views vs, BinArgs a) {
    large_tiles<0>(vs, a, blockIdx.x, gridDim.x);
}

void launch_count_large(const Views &vs, const BinArgs &a, int sms, cudaStream_t s) {
    if (vs.n <= 0) return;
    count_large_kernel<<<sms * 2, 256, 0, s>>>(vs, a);
    ++g_launches;
}

__global__ void slot_cursor_kernel(int m, const int *counts, const long long *offsets,
                                   long long *cursor, int *full) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < m; k += gridDim.x * blockDim.x) {
        cursor[k] = offsets[k] + counts[k];
        if (k < m / NLIST) full[k] = 0;
    }
}

// Exclusive scan of one value per thread over a block of 1024 threads (wsum: 33).
template <typename V>
__device__ __forceinline__ V block_scan(V v, V *wsum, V &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    V incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const V u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const V w = wsum[lane];
        V wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const V u = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += u;
        }
        wsum[lane] = wi - w;
        if (lane == 31) wsum[32] = wi;
    }
    __syncthreads();
    total = wsum[32];
    const V r = wsum[warp] + incl - v;
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------
// Exclusive scan: one CTA of 1024 threads, each owning a contiguous run.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) scan_kernel(int m, const int *in, int *out) {
    __shared__ int wsum[33];
    const int t = threadIdx.x, per = (m + 1023) / 1024;
    const int lo = min(t * per, m), hi = min(lo + per, m);
    int sum = 0;
    for (int k = lo; k < hi; ++k) sum += in[k];
    int total;
    int run = block_scan(sum, wsum, total);
    for (int k = lo; k < hi; ++k) {
        out[k] = run;
        run += in[k];
    }
    if (t == 0) out[m] = total;
}

void launch_scan(int m, const int *in, int *out, cudaStream_t s) {
    scan_kernel<<<1, 1024, 0, s>>>(m, in, out);
    ++g_launches;
}

void launch_slot_cursor(int m, const int *counts, const long long *offsets, long long *cursor,
                        int *full, cudaStream_t s) {
    const int grid = (m + 255) / 256 < 1024 ? (m + 255) / 256 : 1024;
    if (grid <= 0) return;
    slot_cursor_kernel<<<grid, 256, 0, s>>>(m, counts, offsets, cursor, full);
    ++g_launches;
}

// ---------------------------------------------------------------------------
// Work items: a light tile is one item (all its lists, pixels stored); a
// crowded tile is cut into segments of at most kSeg* entries per list (fewer on
// small frames), each its own item (pixels added).  Large-list entries always form separate
// items of the large pass.  item_counts = [tile-pass items | large items].
// ---------------------------------------------------------------------------
__device__ __forceinline__ int div_up(int a, int b) { return (a + b - 1) / b; }

// Entries per list of this frame, summed over the views (differences of the lists'
// first and last offsets), into tot[NLIST]; the whole block takes part.
__device__ __forceinline__ void list_totals(const Views &vs, const long long *off,
                                            unsigned long long *tot) {
    if (threadIdx.x < NLIST) tot[threadIdx.x] = 0ull;
    __syncthreads();
    for (int k = threadIdx.x; k < vs.nviews * NLIST; k += blockDim.x) {
        const FrameConst &fc = vs.fcs[k / NLIST];
        const int b = fc.slot_base + k % NLIST * fc.ntiles;
        atomicAdd(&tot[k % NLIST], (unsigned long long)(off[b + fc.ntiles] - off[b]));
    }
    __syncthreads();
}

// Segment lengths of a frame with these totals (see kSegShrink).  The weights are the
// lists' cost per entry in the tile pass, in medium entries.
__device__ __forceinline__ Segs frame_segs(const unsigned long long *tot, int sms) {
    const int full[NLIST] = {kSegPoint, kSegSmall, kSegMedium, kSegLarge};
    // CTAs of the passes: 4 per SM; two segments each
    const unsigned long long work = tot[L_MEDIUM] + tot[L_SMALL] / 8 + tot[L_POINT] / 64;
    Segs segs;
#pragma unroll
    for (int l = 0; l < NLIST; ++l) {
        const int whole = l == L_LARGE ? kSegLarge : kSegMedium;
        long long len = whole;
        if (sms > 0) {
            len = (long long)((l == L_LARGE ? tot[L_LARGE] : work) / (unsigned long long)(8 * sms));
            len = (len + 63) / 64 * 64;
            // longer large segments where there are plenty: fewer partial tiles (100M
            // heavy-tailed particles, large pass 3.71 -> 3.44 ms; 8 times: the same)
            const int most = l == L_LARGE ? 4 * whole : whole;
            len = len < whole / kSegShrink ? whole / kSegShrink : (len > most ? most : len);
        }
        segs.len[l] = (int)(full[l] / whole * len);
    }
    return segs;
}

// Items of global tile g: of the tile pass, and of the large pass in *large.
__device__ __forceinline__ int tile_items(const Views &vs, const long long *off, const Segs &segs, int g,
                                          int *large) {
    const FrameConst &fc = vs.fcs[view_of_tile(vs.fcs, vs.nviews, g)];
    const int nt = fc.ntiles;
    const long long *o = off + fc.slot_base + g - fc.tile_base;
    const int cp = (int)(o[L_POINT * nt + 1] - o[L_POINT * nt]);
    const int cs = (int)(o[L_SMALL * nt + 1] - o[L_SMALL * nt]);
    const int cm = (int)(o[L_MEDIUM * nt + 1] - o[L_MEDIUM * nt]);
    const int cl = (int)(o[L_LARGE * nt + 1] - o[L_LARGE * nt]);
    *large = div_up(cl, segs.len[L_LARGE]);
    if (cp + cs + cm == 0) return 0;
    if (cp <= segs.len[L_POINT] && cs <= segs.len[L_SMALL] && cm <= segs.len[L_MEDIUM]) return 1;
    return div_up(cp, segs.len[L_POINT]) + div_up(cs, segs.len[L_SMALL]) + div_up(cm, segs.len[L_MEDIUM]);
}

// ---------------------------------------------------------------------------
// From the slot counts to the list offsets and the item offsets.  Frames of up to
// kSlotChunk slots (1024 tiles) take one CTA and one launch; larger ones four
// launches of one chunk per CTA, each CTA adding up the chunks before its own.
// One CTA walking contiguous runs per thread, and a launch for each of the sum, scan,
// cursor, item count and item scan, took 10 us on a small frame and 170 us at 16384
// tiles (now 4 and 12 us).
// ---------------------------------------------------------------------------
constexpr int kSlotChunk = 4096, kItemChunk = 1024;

// This thread's four slots of a chunk: offsets and cursors from base.
__device__ __forceinline__ void put_slots(int k, int m, const int *c, const int *o, long long run,
                                          long long *offsets, long long *cursor) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (k + q < m) {
            offsets[k + q] = run;
            cursor[k + q] = run + c[q];
            run += c[q] + o[q];
        }
}

__device__ __forceinline__ long long get_slots(int k, int m, const int *counts, const int *ovf, int *c,
                                               int *o) {
    long long sum = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        c[q] = k + q < m ? counts[k + q] : 0;
        o[q] = k + q < m ? ovf[k + q] : 0;
        sum += c[q] + o[q];
    }
    return sum;
}

__global__ void __launch_bounds__(1024) slots_kernel(Views vs, int m, const int *counts, const int *ovf,
                                                     long long *offsets, long long *cursor, int *ioff,
                                                     DevStats *st, int sms) {
    __shared__ long long wsum[33];
    __shared__ int isum[33];
    __shared__ unsigned long long tot[NLIST];
    const int t = threadIdx.x;
    int c[4], o[4];
    long long total;
    const long long run = block_scan(get_slots(4 * t, m, counts, ovf, c, o), wsum, total);
    put_slots(4 * t, m, c, o, run, offsets, cursor);
    if (t == 0) {
        offsets[m] = total;
        st->slot_total = total;
    }
    __syncthreads();                       // the block's own offsets are visible to it
    list_totals(vs, offsets, tot);
    if (t < NLIST) st->totals[t] = (int)tot[t];
    const Segs segs = frame_segs(tot, sms);
    const int T = vs.total_tiles;
    int large = 0;
    const int n = t < T ? tile_items(vs, offsets, segs, t, &large) : 0;
    int n_tile, n_large;
    const int at = block_scan(n, isum, n_tile), lat = block_scan(large, isum, n_large);
    if (t < T) {
        ioff[t] = at;
        ioff[T + t] = n_tile + lat;
    }
    if (t == 0) {
        ioff[2 * T] = n_tile + n_large;
        st->item_totals[0] = n_tile;
        st->item_totals[1] = n_large;
    }
}

__global__ void __launch_bounds__(1024) slot_reduce_kernel(int m, const int *counts, const int *ovf,
                                                           long long *part) {
    __shared__ long long wsum[33];
    int c[4], o[4];
    long long total;
    block_scan(get_slots(blockIdx.x * kSlotChunk + 4 * threadIdx.x, m, counts, ovf, c, o), wsum, total);
    if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) slot_apply_kernel(int m, const int *counts, const int *ovf,
                                                          const long long *part, long long *offsets,
                                                          long long *cursor, DevStats *st) {
    __shared__ long long wsum[33];
    const int k = blockIdx.x * kSlotChunk + 4 * threadIdx.x;
    long long before = 0, base, total;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += 1024) before += part[b];
    block_scan(before, wsum, base);
    int c[4], o[4];
    const long long sum = get_slots(k, m, counts, ovf, c, o);
    const long long run = base + block_scan(sum, wsum, total);
    put_slots(k, m, c, o, run, offsets, cursor);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        offsets[m] = base + total;
        st->slot_total = base + total;
    }
}

__global__ void __launch_bounds__(kItemChunk) item_count_kernel(Views vs, const long long *off,
                                                                int *item_counts, int *part,
                                                                DevStats *st, int sms) {
    __shared__ unsigned long long tot[NLIST];
    __shared__ int isum[33];
    list_totals(vs, off, tot);
    if (blockIdx.x == 0 && threadIdx.x < NLIST) st->totals[threadIdx.x] = (int)tot[threadIdx.x];
    const Segs segs = frame_segs(tot, sms);
    const int T = vs.total_tiles, g = blockIdx.x * kItemChunk + threadIdx.x;
    int large = 0, n = 0, n_tile, n_large;
    if (g < T) {
        n = tile_items(vs, off, segs, g, &large);
        item_counts[g] = n;
        item_counts[T + g] = large;
    }
    block_scan(n, isum, n_tile);
    block_scan(large, isum, n_large);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = n_tile;
        part[gridDim.x + blockIdx.x] = n_large;
    }
}

__global__ void __launch_bounds__(kItemChunk) item_apply_kernel(int T, const int *item_counts,
                                                                const int *part, int *ioff,
                                                                DevStats *st) {
    __shared__ int isum[33];
    const int nb = gridDim.x, g = blockIdx.x * kItemChunk + threadIdx.x;
    int tb = 0, ta = 0, lb = 0;            // tile items before, tile items of all, large items before
    for (int b = threadIdx.x; b < nb; b += kItemChunk) {
        ta += part[b];
        if (b < (int)blockIdx.x) {
            tb += part[b];
            lb += part[nb + b];
        }
    }
    int tile_before, tile_all, large_before, n_tile, n_large;
    block_scan(tb, isum, tile_before);
    block_scan(ta, isum, tile_all);
    block_scan(lb, isum, large_before);
    const int at = block_scan(g < T ? item_counts[g] : 0, isum, n_tile);
    const int lat = block_scan(g < T ? item_counts[T + g] : 0, isum, n_large);
    if (g < T) {
        ioff[g] = tile_before + at;
        ioff[T + g] = tile_all + large_before + lat;
    }
    if ((int)blockIdx.x == nb - 1 && threadIdx.x == 0) {
        ioff[2 * T] = tile_all + large_before + n_large;
        st->item_totals[0] = tile_all;
        st->item_totals[1] = large_before + n_large;
    }
}

void launch_slots(const Views &vs, const SlotArgs &a, int sms, cudaStream_t s) {
    const int T = vs.total_tiles, m = NLIST * T;
    if (m <= kSlotChunk) {
        slots_kernel<<<1, 1024, 0, s>>>(vs, m, a.counts, a.ovf, a.offsets, a.cursor, a.item_offsets, a.st,
                                        sms);
        ++g_launches;
        return;
    }
    const int nb = (m + kSlotChunk - 1) / kSlotChunk, ni = (T + kItemChunk - 1) / kItemChunk;
    int *ipart = reinterpret_cast<int *>(a.part + nb);
    slot_reduce_kernel<<<nb, 1024, 0, s>>>(m, a.counts, a.ovf, a.part);
    slot_apply_kernel<<<nb, 1024, 0, s>>>(m, a.counts, a.ovf, a.part, a.offsets, a.cursor, a.st);
    item_count_kernel<<<ni, kItemChunk, 0, s>>>(vs, a.offsets, a.item_counts, ipart, a.st, sms);
    item_apply_kernel<<<ni, kItemChunk, 0, s>>>(T, a.item_counts, ipart, a.item_offsets, a.st);
    g_launches += 4;
}

size_t slot_parts(int tiles) {
    return (size_t)(NLIST * (int64_t)tiles / kSlotChunk + 1) + (size_t)tiles / kItemChunk + 1;
}

__device__ __forceinline__ void put_item(WorkItem *items, int cap, int pos, WorkItem w, DevStats *st) {
    if (pos < cap)
        items[pos] = w;
    else
        atomicOr(&st->err, ERR_LIST_OVERFLOW);
}

// One warp per tile: the lanes write the tile's segments side by side (a
// crowded tile has hundreds), in the same order as one thread would.
__device__ __forceinline__ void fill_items(const Views &vs, const long long *off, const int *ioff,
                                           WorkItem *items, int cap, DevStats *st, int sms, int block,
                                           int nblocks) {
    const int T = vs.total_tiles;
    __shared__ unsigned long long tot[NLIST];
    list_totals(vs, off, tot);
    const Segs segs = frame_segs(tot, sms);
    const int *seg = segs.len;
    const int lane = threadIdx.x & 31;
    const int warps = (nblocks * blockDim.x) >> 5;
    for (int g = (block * blockDim.x + threadIdx.x) >> 5; g < T; g += warps) {
        const int v = view_of_tile(vs.fcs, vs.nviews, g);
        const FrameConst &fc = vs.fcs[v];
        const int t = g - fc.tile_base, nt = fc.ntiles, sb = fc.slot_base;
        int w = ioff[g];
        const int nw = ioff[g + 1] - w;
        if (nw == 1) {
            if (lane == 0)
                put_item(items, cap, w, {g, (v << 8) | kAllLists, off[sb + L_MEDIUM * nt + t],
                                         off[sb + L_MEDIUM * nt + t + 1]}, st);
        } else if (nw > 1) {
            for (int l = 0; l < L_LARGE; ++l) {
                const long long b = off[sb + l * nt + t], e = off[sb + l * nt + t + 1];
                const int ns = (int)((e - b + seg[l] - 1) / seg[l]);
                for (int k = lane; k < ns; k += 32) {
                    const long long kb = b + (long long)k * seg[l];
                    put_item(items, cap, w + k, {g, (v << 8) | l, kb, kb + seg[l] < e ? kb + seg[l] : e}, st);
                }
                w += ns;
            }
        }
        const int wl = ioff[T + g];
        const long long b = off[sb + L_LARGE * nt + t], e = off[sb + L_LARGE * nt + t + 1];
        const int sl = seg[L_LARGE], ns = (int)((e - b + sl - 1) / sl);
        for (int k = lane; k < ns; k += 32) {
            const long long kb = b + (long long)k * sl;
            put_item(items, cap, wl + k,
                     {g, (v << 8) | (ns == 1 ? kSole : 0) | L_LARGE, kb,
                      kb + sl < e ? kb + sl : e}, st);
        }
    }
}

// ---------------------------------------------------------------------------
// Scatter particle ids of points, small and medium particles into their
// tiles' lists (order inside a tile follows the atomics, which is harmless:
// E_p = A_p makes the sum order-independent, Sec. 2).
// ---------------------------------------------------------------------------
__device__ __forceinline__ TileFoot load_foot(const FrameConst &fc, const BinArgs &a, int64_t rec,
                                              bool valid, float4 &r0, float4 &r1) {
    r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    r1 = make_float4(-1.f, 0.f, 0.f, 0.f);
    if (!valid) return TileFoot{-1, 0, 0, 1, 0, 0, 0.f};
    const Rec rc = a.recs[rec];
    r1 = rc.r1;
    const int cls = record_class(fc, r1.x);
    if (cls == CLS_INACTIVE || cls == CLS_LARGE) return TileFoot{-1, 0, 0, 1, 0, 0, 0.f};
    r0 = rc.r0;
    return tile_footprint(fc, cls, r0, r1);
}

// Scatter record indices of points, small and medium particles into their
// tiles' lists in one pass: per CTA and view, the rasteriser's table gives
// every slot the CTA used its range base offsets[slot] + offset; each entry
// goes to base + its rank among the CTA's entries of that slot (shared-memory
// counters).
// Keys that had no room in the table go through the cursors.  Order inside a
// tile follows the atomics, which is harmless: E_p = A_p makes the sum
// order-independent (Sec. 2); the absorption mode writes its lists in depth order
// (depth_entries_kernel) instead.
__device__ __forceinline__ void scatter_chunk(const Views &vs, const BinArgs &a, int block,
                                              long long *scatter_smem) {
    long long *bases = scatter_smem;                         // 2^hash_bits
    __shared__ FootWarp feet[8];
    const int bits = a.shape.hash_bits, size = 1 << bits;
    int *keys = reinterpret_cast<int *>(bases + size);       // size
    int *vals = keys + size;                                 // size
    __shared__ FrameConst sfc;
    const int lane = threadIdx.x & 31;
    const int64_t c0 = (int64_t)block * a.shape.chunk;
    const int64_t c1 = c0 + a.shape.chunk < vs.n ? c0 + a.shape.chunk : vs.n;
    for (int v = 0; v < vs.nviews; ++v) {
        load_view(vs.fcs, v, &sfc);     // (begins and ends with a barrier)
        const FrameConst &fc = sfc;
        const int2 *tab = a.ctab + (((int64_t)block * vs.nviews + v) << bits);
        for (int k = threadIdx.x; k < size; k += blockDim.x) {
            const int2 t = tab[k];
            keys[k] = t.x;
            vals[k] = 0;
            bases[k] = t.x >= 0 ? a.offsets[t.x] + t.y : 0;
        }
        __syncthreads();
        for (int64_t base = c0; base < c1; base += blockDim.x) {
            const int64_t i = base + threadIdx.x;
            const int64_t rec = fc.rec_base + i;
            float4 r0, r1;
            const TileFoot f = load_foot(fc, a, rec, i < c1, r0, r1);
            FootPairs pairs(f, r0, feet[threadIdx.x >> 5], lane);
            for (int pbase = 0; pbase < pairs.total; pbase += 32) {
                int owner;
                const int ls = pairs.slot(fc, feet[threadIdx.x >> 5], pbase, lane, owner);
                const unsigned orec = (unsigned)rec + (unsigned)(owner - lane);
                const int key = ls >= 0 ? fc.slot_base + ls : -1;
                if (key >= 0) {
                    const int slot = hash_slot(keys, key, bits, false);
                    const long long pos =
                        slot >= 0 ? bases[slot] + atomicAdd(&vals[slot], 1)
                                  : (long long)atomicAdd(reinterpret_cast<unsigned long long *>(&a.cursor[key]), 1ULL);
                    if (pos < a.entries_cap)
                        a.entries[pos] = orec;
                    else
                        atomicOr(&a.st->err, ERR_LIST_OVERFLOW);
                }
            }
        }
    }
}

// Everything that follows the offsets, in one launch, by the block's number: the large
// lists, the work items and the cleared images are a few blocks' work beside the
// scatter, and each was a launch of its own.  The images' blocks come last, so that small
// frames' chunks all start at once and the cleared pixels are still in L2 for the tile pass
// (200k particles: lists 29 -> 27 us; 1.3M: frame 1.089 -> 1.085 ms).
__global__ void __launch_bounds__(256, 6) lists_kernel(Views vs, BinArgs a, ListArgs l) {
    extern __shared__ long long lists_smem[];
    int b = blockIdx.x;
    if (b < l.large_blocks) {
        large_tiles<1>(vs, a, b, l.large_blocks);
        return;
    }
    b -= l.large_blocks;
    const int fill = (int)gridDim.x - l.large_blocks - l.item_blocks - l.zero_blocks;
    if (b < fill) {
        scatter_chunk(vs, a, b, lists_smem);
        return;
    }
    b -= fill;
    if (b < l.item_blocks) {
        fill_items(vs, a.offsets, l.item_offsets, l.items, l.items_cap, a.st, l.seg_sms, b, l.item_blocks);
        return;
    }
    b -= l.item_blocks;
    for (int v = 0; v < vs.nviews; ++v) {
        const int64_t n = (int64_t)3 * vs.fcs[v].width * vs.fcs[v].height;
        float *img = l.images[v];
        for (int64_t i = (int64_t)b * blockDim.x + threadIdx.x; i < n;
             i += (int64_t)l.zero_blocks * blockDim.x)
            img[i] = 0.f;
    }
}

void launch_lists(const Views &vs, BinArgs a, ListArgs l, bool zero, int sms, cudaStream_t s) {
    a.shape = bin_shape(vs.n, sms);
    const int64_t chunks = vs.n > 0 && l.scatter ? (vs.n + a.shape.chunk - 1) / a.shape.chunk : 0;
    // 8 to 32 KB by the set's size, beside 9 KB of static shared memory: within the 48 KB that need
    // no attribute.  (The attribute is the kernel's, not the launch's: a launch of another
    // thread that set it for a smaller set made this one fail.)
    const size_t smem = ((size_t)1 << a.shape.hash_bits) * (sizeof(long long) + 2 * sizeof(int));
    l.large_blocks = vs.n > 0 ? sms * 2 : 0;
    const int warps = (vs.total_tiles + 7) / 8;     // 8 warps of 256 threads, a warp per tile
    l.item_blocks = warps < sms * 4 ? warps : sms * 4;
    l.zero_blocks = zero ? sms * 2 : 0;
    const int64_t blocks = l.large_blocks + l.item_blocks + l.zero_blocks + chunks;
    lists_kernel<<<(unsigned)blocks, 256, smem, s>>>(vs, a, l);
    ++g_launches;
}

// ---------------------------------------------------------------------------
// The absorption mode's lists: the particles taken in depth order, every (particle,
// tile) pair as a key tile << 32 | particle, in that order.  A warp takes `run` of the
// particles; a first launch counts the pairs of each run, a second writes them from the
// scanned counts.  The footprints are worked out in both: kept, they would be more
// bytes than the records they come from.
// ---------------------------------------------------------------------------
template <bool WRITE>
__global__ void __launch_bounds__(256, 5) depth_entries_kernel(Views vs, const Rec *recs, const unsigned *by_depth,
                                                            int run, int *counts, unsigned long long *keys,
                                                            long long cap, DevStats *st) {
    __shared__ FrameConst sfc;
    __shared__ FootWarp feet[8];
    load_view(vs.fcs, 0, &sfc);
    const FrameConst &fc = sfc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t w = (int64_t)blockIdx.x * 8 + warp, k0 = w * run, k1 = k0 + run < vs.n ? k0 + run : vs.n;
    if (k0 >= vs.n) return;
    long long pos = WRITE ? counts[w] : 0;
    // the next 32 records are on their way while these are worked on, and the ids after them
    const Rec none{make_float4(0.f, 0.f, 0.f, 0.f), make_float4(-1.f, 0.f, 0.f, 0.f)};
    unsigned id1 = k0 + lane < k1 ? by_depth[k0 + lane] : 0u;
    Rec rc1 = k0 + lane < k1 ? recs[id1] : none;
    unsigned id2 = k0 + 32 + lane < k1 ? by_depth[k0 + 32 + lane] : 0u;
    for (int64_t k = k0; k < k1; k += 32) {
        const unsigned id = id1;
        const float4 r0 = rc1.r0, r1 = rc1.r1;
        id1 = id2;
        rc1 = k + 32 + lane < k1 ? recs[id2] : none;
        id2 = k + 64 + lane < k1 ? by_depth[k + 64 + lane] : 0u;
        const TileFoot f = tile_footprint(fc, record_class(fc, r1.x), r0, r1);
        FootPairs pairs(f, r0, feet[warp], lane);
        for (int base = 0; base < pairs.total; base += 32) {
            int owner;
            const int ls = pairs.slot(fc, feet[warp], base, lane, owner);
            const unsigned src = __shfl_sync(0xffffffffu, id, owner);
            const unsigned m = __ballot_sync(0xffffffffu, ls >= 0);
            const long long at = pos + __popc(m & lt);
            if (WRITE && ls >= 0) {
                if (at < cap)
                    keys[at] = (unsigned long long)(unsigned)(ls - L_MEDIUM * fc.ntiles) << 32 | src;
                else
                    atomicOr(&st->err, ERR_LIST_OVERFLOW);
            }
            pos += __popc(m);
        }
    }
    if (!WRITE && lane == 0) counts[w] = (int)pos;
}

// counts: the scan's input, output and block sums; the radix sort's scratch has them.
// Runs are short: 16384 of them leave the last wave of warps nearly empty (10M particles:
// count 0.218 and write 0.255 ms; with up to 65536 0.169 and 0.199).
constexpr int kDepthRuns = 65536;
void launch_depth_entries(const Views &vs, const Rec *recs, const unsigned *by_depth,
                          unsigned long long *keys, long long total, int *counts, DevStats *st,
                          cudaStream_t s) {
    int run = 32;
    while ((vs.n + run - 1) / run > kDepthRuns) run *= 2;
    const int runs = (int)((vs.n + run - 1) / run);
    const unsigned blocks = (unsigned)((runs + 7) / 8);
    int *bases = counts + runs + 1, *part = bases + runs + 1;
    depth_entries_kernel<false><<<blocks, 256, 0, s>>>(vs, recs, by_depth, run, counts, nullptr, 0, st);
    ++g_launches;
    launch_wide_scan(runs, counts, bases, part, s);
    depth_entries_kernel<true><<<blocks, 256, 0, s>>>(vs, recs, by_depth, run, bases, keys, total, st);
    ++g_launches;
}

// ---------------------------------------------------------------------------
// The start of a frame: the view's constants (a single view's travel as launch
// arguments) and everything that starts at zero.  Three memsets and two copies took
// as many slots of the stream.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) setup_kernel(const __grid_constant__ SetupArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    for (int k = i; k < a.slots; k += stride) {
        a.counts[k] = 0;
        a.ovf[k] = 0;
        if (k < a.slots / NLIST) a.full[k] = 0;
    }
    if (i < (int)(offsetof(DevStats, err) / sizeof(int))) reinterpret_cast<int *>(a.st)[i] = 0;
    if (a.fcs) {
        if (i < (int)(sizeof(FrameConst) / sizeof(int)))
            reinterpret_cast<int *>(a.fcs)[i] = reinterpret_cast<const int *>(&a.fc)[i];
        if (i == 0) *a.images = a.image;
    }
}

void launch_setup(const SetupArgs &a, int sms, cudaStream_t s) {
    const int blocks = (a.slots + 255) / 256;
    setup_kernel<<<blocks < 1 ? 1 : (blocks < sms * 4 ? blocks : sms * 4), 256, 0, s>>>(a);
    ++g_launches;
}

// ---------------------------------------------------------------------------
// Diagnostic: exact count of covered (particle, pixel) pairs per class, using
// the same FP32 clip test as the render passes.  Not part of a render.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) count_work_kernel(FrameConst fc, const Rec *recs, int64_t n,
                                                         unsigned long long *work) {
    unsigned long long acc[4] = {0, 0, 0, 0};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float4 r1 = recs[i].r1;
        const int cls = record_class(fc, r1.x);
        if (cls == CLS_INACTIVE) continue;
        const float4 r0 = recs[i].r0;
        const int xi = unpack_xi(r0.x), yi = unpack_yi(r0.x);
        if (cls == CLS_POINT) {
            acc[0] += (xi >= 0 && yi >= 0 && xi < fc.width && yi < fc.height);
            continue;
        }
        PixBox b;
        if (!splat_box(fc, r0, r1.x, b)) continue;
        unsigned long long cnt = 0;
        for (int j = b.j0; j <= b.j1; ++j) {
            const float dy = (float)(j - yi) + (0.5f - r0.z);
            const float rem = r1.x - dy * dy;
            if (rem < 0.f) continue;
            for (int i2 = b.i0; i2 <= b.i1; ++i2) {
                const float dx = (float)(i2 - xi) + (0.5f - r0.y);
                cnt += dx * dx <= rem;
            }
        }
        acc[cls] += cnt;
    }
    for (int k = 0; k < 4; ++k) {
        unsigned long long v = acc[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&work[k], v);
    }
}

void launch_count_work(const FrameConst &fc, const Rec *recs, int64_t n,
                       unsigned long long *work, int sms, cudaStream_t s) {
    if (n <= 0) return;
    int64_t blocks = (n + 255) / 256;
    blocks = blocks < (int64_t)sms * 8 ? blocks : (int64_t)sms * 8;
    count_work_kernel<<<(unsigned)blocks, 256, 0, s>>>(fc, recs, n, work);
    ++g_launches;
}

}  // namespace spl
