// The activation quantizer's arithmetic as the GEMM kernels that quantize their own tiles use it (Sec. 4.1).
#pragma once

#include "common.cuh"

namespace mixdq {
namespace i8 {

constexpr float kMagic = 12582912.f;  // 1.5 * 2^23: fma(x, inv, magic) rounds x * inv to nearest even

// Largest fp16 value c with c * inv < 127.5, i.e. the largest input whose code needs no clamping, provided the code
// of c itself is 127 (true whenever fp16 is finer than the quantization step around 127 steps, which fails only for
// scales below about 1e-7 or above 500): then clamping the fp16 input to [-c, c] -- one packed min and one packed max
// per two elements -- gives the same codes as clamping the rounded product to [-127, 127] (rounding is monotonic:
// inputs beyond c round to at least 127.5 -> 128 -> 127, and c rounds to 127).  false: no such value; the caller clamps the rounded product instead.
// qmax: 127, or the end of an asymmetric range (255 - zero, and zero for the other end).
__device__ __forceinline__ bool fp16_clamp_bound(float inv, __half* c_out, int qmax = 127)
{
    const float end = static_cast<float>(qmax) + 0.5f;
    const float t = __fdividef(end, inv);
    if (!(t > 0.f) || !(t < 65000.f)) return false;
    // whether v * inv < end: the fma rounds the exact difference once, so its sign is exact
    auto below = [&](unsigned bits) { return fmaf(__half2float(__ushort_as_half(static_cast<unsigned short>(bits))), inv, -end) < 0.f; };
    unsigned bits = __half_as_ushort(__float2half_rz(t));  // at most one off
    if (!below(bits))
        bits -= bits > 0;
    else if (below(bits + 1))
        ++bits;
    const float v = __half2float(__ushort_as_half(static_cast<unsigned short>(bits)));
    // ... and that it is the largest such value, and rounds to qmax (v * inv > qmax - 0.5)
    if (!below(bits) || below(bits + 1) || !(fmaf(v, inv, 1.f - end) > 0.f)) return false;
    *c_out = __ushort_as_half(static_cast<unsigned short>(bits));
    return true;
}

// Two products rounded to nearest even by one packed fma against 1.5 * 2^23 each.
__device__ __forceinline__ float2 fma2_magic(float2 v, float inv)
{
    uint64_t a, b, c, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(v.x), "f"(v.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(b) : "f"(inv));
    asm("mov.b64 %0, {%1, %1};" : "=l"(c) : "f"(kMagic));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}

// 16 fp16 values (two 16-byte chunks) to 16 code bytes: clamp(rne(x * inv), -127, 127), the arithmetic of the
// stand-alone quantization kernel (one rounding, by an fma against 1.5 * 2^23).  FAST: the input is clamped as
// fp16 (see fp16_clamp_bound), so the low byte of the fma's result is the code.
template <bool FAST>
__device__ __forceinline__ uint4 quantize_chunks(const uint4& v0, const uint4& v1, float inv, __half2 c2)
{
    const __half2* h0 = reinterpret_cast<const __half2*>(&v0);
    const __half2* h1 = reinterpret_cast<const __half2*>(&v1);
    const float lo = kMagic - 127.f, hi = kMagic + 127.f;
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        __half2 ha = j < 2 ? h0[2 * j] : h1[2 * j - 4];
        __half2 hb = j < 2 ? h0[2 * j + 1] : h1[2 * j - 3];
        uint32_t qa, qb, qc, qd;
        if (FAST) {
            ha = __hmin2(__hmax2(ha, __hneg2(c2)), c2);
            hb = __hmin2(__hmax2(hb, __hneg2(c2)), c2);
            const float2 ra = fma2_magic(__half22float2(ha), inv), rb = fma2_magic(__half22float2(hb), inv);
            qa = __float_as_uint(ra.x);
            qb = __float_as_uint(ra.y);
            qc = __float_as_uint(rb.x);
            qd = __float_as_uint(rb.y);
        } else {
            const float2 a = __half22float2(ha), b = __half22float2(hb);
            qa = __float_as_uint(fminf(fmaxf(fmaf(a.x, inv, kMagic), lo), hi));
            qb = __float_as_uint(fminf(fmaxf(fmaf(a.y, inv, kMagic), lo), hi));
            qc = __float_as_uint(fminf(fmaxf(fmaf(b.x, inv, kMagic), lo), hi));
            qd = __float_as_uint(fminf(fmaxf(fmaf(b.y, inv, kMagic), lo), hi));
        }
        w[j] = __byte_perm(__byte_perm(qa, qb, 0x0040), __byte_perm(qc, qd, 0x0040), 0x5410);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace i8
}  // namespace mixdq
