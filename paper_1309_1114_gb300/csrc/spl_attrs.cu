// spl_attrs.cu -- storage layouts of the per-particle attributes h, I, s.
//
// The memory-access model of Sec. 3.2 charges every particle its bytes once
// per frame; the smaller layouts store the same particles in fewer bytes.  The
// encoder converts FP32 attributes into any layout the rasteriser reads:
//   SPL_ATTR_F32      h, I, s FP32 (a copy)
//   SPL_ATTR_F16      h, I, s IEEE binary16, round to nearest even
//   SPL_ATTR_F16_IS   h FP32; I, s binary16
//   SPL_ATTR_LOGH16   I, s binary16; h as the 16-bit code
//                     k = round_half_even(4096 (log2 h - h_log2_min)) clamped to
//                     [0, 65535], formed in FP64 so that the code is the
//                     correctly rounded one except within ~1e-16 of a half
//                     step; the rasteriser decodes h = 2^(h_log2_min + k/4096).
// A smoothing length that no code can stand for (negative, NaN or infinite --
// a particle the FP32 layout renders inactive) keeps the particle inactive in
// the coded layout too: its I is stored as a binary16 NaN.
#include "spl_internal.cuh"

namespace spl {

// The code of h by FP64: the definition above.
__device__ __noinline__ unsigned short logh_code64(float h, float h_log2_min) {
    const double t = rint((log2((double)h) - (double)h_log2_min) * 4096.0);
    return (unsigned short)(t < 0.0 ? 0.0 : (t > 65535.0 ? 65535.0 : t));
}

// The same code by FP32 where FP32 can decide it.  With h = m 2^e, 1 <= m < 2,
// t = 4096 (e - h_log2_min) + 4096 log2(m): the first term is held exactly as a
// sum of two floats, and log2f(m) (within 1 ulp of a value below 1: 6e-8) moves t by
// less than 5e-4, so that the rounded value is the FP64 one unless t lies within
// 1e-3 of a half step.  Those (2 in 1000) and subnormal h take the FP64 path.
// FP64 throughput bounds the kernel otherwise: encoding 4M particles took 288 us with the
// FP64 logarithm for every h and takes 27 us (72 MB: 2.6 TB/s).
__device__ __forceinline__ unsigned short logh_code(float h, float h_log2_min) {
    const int bits = __float_as_int(h);
    const float e = (float)((bits >> 23) - 127), m = __int_as_float((bits & 0x007fffff) | 0x3f800000);
    const float s = e - h_log2_min, bb = s - e;                    // two-sum: s + err
    const float err = (e - (s - bb)) + (-h_log2_min - bb);
    const float a = s * 4096.f, b = log2f(m) * 4096.f;
    const float u = a + b, ub = u - a;                             // two-sum: u + v
    const float v = (a - (u - ub)) + (b - ub);
    const float k0 = rintf(u), d = (u - k0) + (v + err * 4096.f), adj = rintf(d);
    // (negated so that an overflowing h_log2_min's NaN goes to FP64, too)
    if (bits < 0x00800000 || !(fabsf(d - adj) < 0.499f)) return logh_code64(h, h_log2_min);
    const float k = k0 + adj;
    return (unsigned short)(k < 0.f ? 0.f : (k > 65535.f ? 65535.f : k));
}

template <int STORE>
__global__ void __launch_bounds__(256) encode_attrs_kernel(const float *h, const float *I, const float *s,
                                                           int64_t n, float h_log2_min, void *ho,
                                                           void *Io, void *so) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float hv = h[i], iv = I[i], sv = s[i];
        if (STORE == 0) {
            static_cast<float *>(ho)[i] = hv;
            static_cast<float *>(Io)[i] = iv;
            static_cast<float *>(so)[i] = sv;
            continue;
        }
        static_cast<__half *>(so)[i] = __float2half_rn(sv);
        if (STORE == 1) {
            static_cast<__half *>(ho)[i] = __float2half_rn(hv);
            static_cast<__half *>(Io)[i] = __float2half_rn(iv);
        } else if (STORE == 2) {
            static_cast<float *>(ho)[i] = hv;
            static_cast<__half *>(Io)[i] = __float2half_rn(iv);
        } else {
            const bool codable = isfinite(hv) && hv >= 0.f;
            static_cast<unsigned short *>(ho)[i] = codable && hv > 0.f ? logh_code(hv, h_log2_min) : 0;
            static_cast<__half *>(Io)[i] = codable ? __float2half_rn(iv) : __ushort_as_half(0x7E00);
        }
    }
}

void launch_encode_attrs(const float *h, const float *I, const float *s, int64_t n, int store,
                         float h_log2_min, void *ho, void *Io, void *so, int sms, cudaStream_t st) {
    if (n <= 0) return;
    int64_t blocks = (n + 255) / 256;
    blocks = blocks < (int64_t)sms * 8 ? blocks : (int64_t)sms * 8;
    const unsigned g = (unsigned)blocks;
    if (store == 0)
        encode_attrs_kernel<0><<<g, 256, 0, st>>>(h, I, s, n, h_log2_min, ho, Io, so);
    else if (store == 1)
        encode_attrs_kernel<1><<<g, 256, 0, st>>>(h, I, s, n, h_log2_min, ho, Io, so);
    else if (store == 2)
        encode_attrs_kernel<2><<<g, 256, 0, st>>>(h, I, s, n, h_log2_min, ho, Io, so);
    else
        encode_attrs_kernel<3><<<g, 256, 0, st>>>(h, I, s, n, h_log2_min, ho, Io, so);
    ++g_launches;
}

}  // namespace spl
