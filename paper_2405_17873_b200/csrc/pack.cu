// Offline side of the path: per-channel min-max parameters, weight quantization and
// packing (2 / 3 / 4 / 8 bits, canonical and device layouts) and the unpack parity hook.
#include "common.cuh"
#include "codes.cuh"

namespace mixdq {

namespace {

// round-half-even of the exact product w * inv (11-bit x 24-bit significands fit a double)
__device__ __forceinline__ long long rne_product(float w, float inv)
{
    double p = static_cast<double>(w) * static_cast<double>(inv);
    p = fmin(fmax(p, -1e15), 1e15);
    return __double2ll_rn(p);
}

__device__ __forceinline__ int clampi(long long v, int lo, int hi)
{
    return v < lo ? lo : (v > hi ? hi : static_cast<int>(v));
}

// Min / max of every output channel's row, then its scale and zero-point.  T threads per row: a warp for rows of up to
// 4096 weights (all its 16-byte loads in flight at once, no barrier), a CTA of 256 for longer ones.  Bound by reading W:
// 10240 x 1280 took 17 us with one CTA and two-byte loads per row.
constexpr int kRowWarp = 4096;

template <int T>
__global__ void __launch_bounds__(256)
weight_minmax_kernel(const __half* __restrict__ W, int64_t N, int64_t K, int bits, int symmetric,
                     float* __restrict__ scale_out, int32_t* __restrict__ zero_out)
{
    const int64_t n = blockIdx.x * static_cast<int64_t>(256 / T) + threadIdx.x / T;
    const int t = threadIdx.x % T;
    float lo = 0.f, hi = 0.f;
    if (n < N) {
        const __half* row = W + n * K;
        __half2 l2 = __half2half2(__ushort_as_half(0)), h2 = l2;
        int64_t done = 0;
        if ((reinterpret_cast<uintptr_t>(row) & 15) == 0) {
            const uint4* v4 = reinterpret_cast<const uint4*>(row);
            const int chunks = static_cast<int>(K >> 3);
#pragma unroll 8
            for (int c = t; c < chunks; c += T) {
                const uint4 v = __ldg(v4 + c);
                const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    l2 = __hmin2(l2, h[j]);
                    h2 = __hmax2(h2, h[j]);
                }
            }
            done = static_cast<int64_t>(chunks) << 3;
        }
        lo = fminf(__low2float(l2), __high2float(l2));
        hi = fmaxf(__low2float(h2), __high2float(h2));
        for (int64_t k = done + t; k < K; k += T) {
            const float w = __half2float(row[k]);
            lo = fminf(lo, w);
            hi = fmaxf(hi, w);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (T > 32) {
        __shared__ float s_lo[8], s_hi[8];
        if ((threadIdx.x & 31) == 0) {
            s_lo[threadIdx.x >> 5] = lo;
            s_hi[threadIdx.x >> 5] = hi;
        }
        __syncthreads();
        for (int i = 0; i < 8; ++i) {
            lo = fminf(lo, s_lo[i]);
            hi = fmaxf(hi, s_hi[i]);
        }
    }
    if (t == 0 && n < N) {
        if (symmetric) {
            const float amax = fmaxf(-lo, hi);
            const float qmax = static_cast<float>((1 << (bits - 1)) - 1);
            scale_out[n] = (amax == 0.f) ? 1.f : __fdiv_rn(amax, qmax);
            if (zero_out) zero_out[n] = 0;
        } else {
            const int L = (1 << bits) - 1;
            const float range = __fsub_rn(hi, lo);
            const float scale = (range == 0.f) ? 1.f : __fdiv_rn(range, static_cast<float>(L));
            scale_out[n] = scale;
            if (zero_out) zero_out[n] = clampi(rne_product(-lo, __fdiv_rn(1.f, scale)), 0, L);
        }
    }
}

// Quantize and pack: one thread per 32 consecutive codes of a row, read once (four 16-byte loads where rows are
// aligned) and written as the group's BITS words.  A code is clamp(rne(w * inv) [+ zero]): one fma against 1.5 * 2^23
// rounds the exact product to nearest even, the clamp acts on that float (it is monotonic, so a product too large
// for the trick clamps to the right end too), the code is the low bits of the result.  The form before this one made
// one thread per output WORD, so that a bit-plane layout computed every code once per plane, with products in double:
// 10240 x 1280 to 3 bits took 74 us.
template <int BITS>
__global__ void __launch_bounds__(256)
pack_kernel(const __half* __restrict__ W, int64_t N, int64_t K, int groups, const float* __restrict__ scale,
            const int32_t* __restrict__ zero, int layout, int64_t pitch, uint8_t* __restrict__ out)
{
    constexpr float kMagic = 12582912.f;
    const int64_t idx = blockIdx.x * static_cast<int64_t>(256) + threadIdx.x;
    if (idx >= N * groups) return;
    const int64_t n = idx / groups;
    const int g = static_cast<int>(idx - n * groups);
    const float inv = __fdiv_rn(1.f, scale[n]);
    const bool hz = zero != nullptr;
    const int z = hz ? zero[n] : 0;
    const float lo = kMagic + static_cast<float>(hz ? -z : -((1 << (BITS - 1)) - 1));
    const float hi = kMagic + static_cast<float>(hz ? (1 << BITS) - 1 - z : (1 << (BITS - 1)) - 1);
    const uint32_t offset = static_cast<uint32_t>(z) - 0x4B400000u;  // float bits of the clamped sum -> code
    // positions beyond K: the pad code (0 signed, zero-point unsigned); nothing in a canonical row's last nibble
    const uint32_t pad = (BITS == 4 && layout == MIXDQ_LAYOUT_CANONICAL) ? 0u : static_cast<uint32_t>(z);
    const int64_t k0 = 32ll * g;
    const __half* src = W + n * K + k0;
    const bool whole = k0 + 32 <= K && (reinterpret_cast<uintptr_t>(src) & 15) == 0;

    uint32_t nib[4];         // eight 4-bit fields of codes 8 s .. 8 s + 7, in the order the layout packs them
    uint32_t words[8];       // the group's packed words
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        float f[8];
        uint32_t c[8];
        if (whole) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(src) + s);
            const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 t = __half22float2(h[j]);
                f[2 * j] = t.x;
                f[2 * j + 1] = t.y;
            }
        } else {
            for (int j = 0; j < 8; ++j) f[j] = k0 + 8 * s + j < K ? __half2float(src[8 * s + j]) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            c[j] = __float_as_uint(fminf(fmaxf(fmaf(f[j], inv, kMagic), lo), hi)) + offset;
            if (!whole && k0 + 8 * s + j >= K) c[j] = pad;
        }
        if (BITS == 8) {
            words[2 * s] = __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
            words[2 * s + 1] = __byte_perm(__byte_perm(c[4], c[5], 0x0040), __byte_perm(c[6], c[7], 0x0040), 0x5410);
        } else {
            // fields in order, or (device layouts) field f = code f / 2 (f even), 4 + f / 2 (f odd)
            uint32_t w = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int fld = (j < 4) ? 2 * j : 2 * (j - 4) + 1;
                w |= (c[j] & 0xfu) << (4 * (layout == MIXDQ_LAYOUT_CANONICAL ? j : fld));
            }
            nib[s] = w;
            if (BITS == 4) words[s] = w;
        }
    }
    int64_t byte0 = 4ll * BITS * g, step = 4;  // where the group's words go in the row
    if (BITS <= 3) {
        if (layout == MIXDQ_LAYOUT_CANONICAL) {
            // plane p: bit j = bit p of code j.  Bit p of the eight fields, gathered into one byte per octet.
#pragma unroll
            for (int p = 0; p < BITS; ++p) {
                uint32_t w = 0;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    uint32_t x = (nib[s] >> p) & 0x11111111u;  // bits 0, 4, 8, ... -> 0 .. 7
                    x = (x | (x >> 3)) & 0x03030303u;
                    x = (x | (x >> 6)) & 0x000f000fu;
                    x = (x | (x >> 12)) & 0xffu;
                    w |= x << (8 * s);
                }
                words[p] = w;
            }
        } else {
            // blocks of 128 codes, 16 bytes per plane: bit 4 f + s of the word is field f's bit of octet s
#pragma unroll
            for (int p = 0; p < BITS; ++p) {
                uint32_t w = 0;
#pragma unroll
                for (int s = 0; s < 4; ++s) w |= ((nib[s] >> p) & 0x11111111u) << s;
                words[p] = w;
            }
            byte0 = (g >> 2) * 16ll * BITS + (g & 3) * 4;
            step = 16;
        }
    }
    uint8_t* row = out + n * pitch;
    if (BITS >= 4 && (pitch & 15) == 0) {
#pragma unroll
        for (int i = 0; i < BITS; i += 4)
            if (byte0 + 4 * i < pitch)
                *reinterpret_cast<uint4*>(row + byte0 + 4 * i) = make_uint4(words[i], words[i + 1], words[i + 2], words[i + 3]);
    } else if ((pitch & 3) == 0) {
#pragma unroll
        for (int i = 0; i < BITS; ++i)
            if (byte0 + i * step < pitch) *reinterpret_cast<uint32_t*>(row + byte0 + i * step) = words[i];
    } else {
        // odd-sized canonical rows: byte by byte, the last word may be partial
#pragma unroll
        for (int i = 0; i < BITS; ++i)
            for (int b = 0; b < 4; ++b)
                if (byte0 + i * step + b < pitch) row[byte0 + i * step + b] = static_cast<uint8_t>(words[i] >> (8 * b));
    }
}

template <int BITS>
void launch_pack(const __half* W, int64_t N, int64_t K, const float* scale, const int32_t* zero, int layout, int64_t pitch,
                 uint8_t* out, cudaStream_t st)
{
    // groups of 32 codes that cover the row's packed bytes (blocks of 128 codes in the device's bit-plane layouts)
    const int64_t groups = ceil_div(pitch, 4 * BITS);
    pack_kernel<BITS><<<static_cast<unsigned>(ceil_div(N * groups, 256)), 256, 0, st>>>(
        W, N, K, static_cast<int>(groups), scale, zero, layout, pitch, out);
}

// One thread per code.
__global__ void unpack_kernel(const uint8_t* __restrict__ packed, int64_t N, int64_t K, int bits,
                              int is_signed, int layout, int64_t pitch, int16_t* __restrict__ codes)
{
    const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (idx >= N * K) return;
    const int64_t n = idx / K;
    const int64_t k = idx - n * K;
    codes[idx] = static_cast<int16_t>(decode_code(packed + n * pitch, k, bits, is_signed, layout));
}

// One CTA of 128 threads per output channel: sum over k of its signed codes.
__global__ void code_sums_kernel(const uint8_t* __restrict__ packed, int64_t K, int bits, int64_t pitch,
                                 int32_t* __restrict__ sums)
{
    __shared__ int part[4];
    const uint8_t* row = packed + blockIdx.x * pitch;
    int s = 0;
    for (int64_t k = threadIdx.x; k < K; k += blockDim.x) s += decode_code(row, k, bits, 1, MIXDQ_LAYOUT_DEVICE);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) sums[blockIdx.x] = part[0] + part[1] + part[2] + part[3];
}

bool width_ok(int bits) { return bits == 2 || bits == 3 || bits == 4 || bits == 8; }

}  // namespace

}  // namespace mixdq

using namespace mixdq;

// The layer kernels load a layer's constants (packed weights, scales, zero-points, code sums) before they
// wait for earlier kernels of the stream, so a kernel that WRITES such constants must be complete, not merely
// finishing, when a layer kernel behind it starts.  The entry points below that produce constants therefore leave a
// note for the stream, and the library's next kernel on it is launched plainly, without the programmatic overlap
// (launch_ex).  Where no note can be left (while the stream captures, on the per-thread stream), this empty kernel,
// launched plainly, stands between the two.  (It used to end every one of these calls: two launches and some 3 us of a
// 10240 x 1280 layer's preparation.)
__global__ void constants_complete_kernel() {}

static int finish_constants(cudaStream_t st)
{
    if (cudaGetLastError() != cudaSuccess) return MIXDQ_ERR_CUDA;
    if (note_constants_written(st)) return MIXDQ_OK;
    constants_complete_kernel<<<1, 32, 0, st>>>();
    return check_launch();
}

extern "C" int mixdq_packed_bytes(int64_t N, int64_t K, int bits, int layout, size_t* out)
{
    if (!out || N <= 0 || K <= 0) return MIXDQ_ERR_INVALID_ARG;
    if (layout != MIXDQ_LAYOUT_CANONICAL && layout != MIXDQ_LAYOUT_DEVICE) return MIXDQ_ERR_INVALID_ARG;
    if (!width_ok(bits)) return MIXDQ_ERR_UNSUPPORTED;
    if (layout == MIXDQ_LAYOUT_CANONICAL) {
        *out = static_cast<size_t>(N * row_pitch_bytes(K, bits, layout));
    } else {
        // device buffers are read in whole 16-byte units
        *out = static_cast<size_t>(round_up(N * row_pitch_bytes(K, bits, layout), 16));
    }
    return MIXDQ_OK;
}

extern "C" int mixdq_weight_minmax_params(const void* W, int64_t N, int64_t K, int bits, int symmetric,
                                          float* scale_out, int32_t* zero_out, void* stream)
{
    if (!W || !scale_out || N <= 0 || K <= 0) return MIXDQ_ERR_INVALID_ARG;
    if (bits < 2 || bits > 8) return MIXDQ_ERR_UNSUPPORTED;
    if (!symmetric && !zero_out) return MIXDQ_ERR_INVALID_ARG;
    if (K <= kRowWarp)
        weight_minmax_kernel<32><<<static_cast<unsigned>(ceil_div(N, 8)), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __half*>(W), N, K, bits, symmetric, scale_out, zero_out);
    else
        weight_minmax_kernel<256><<<static_cast<unsigned>(N), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __half*>(W), N, K, bits, symmetric, scale_out, zero_out);
    return finish_constants(static_cast<cudaStream_t>(stream));
}

extern "C" int mixdq_pack_weights(const void* W, int64_t N, int64_t K, int bits, const float* scale,
                                  const int32_t* zero, int layout, void* packed_out, void* stream)
{
    if (!W || !scale || !packed_out || N <= 0 || K <= 0) return MIXDQ_ERR_INVALID_ARG;
    if (layout != MIXDQ_LAYOUT_CANONICAL && layout != MIXDQ_LAYOUT_DEVICE) return MIXDQ_ERR_INVALID_ARG;
    if (!width_ok(bits)) return MIXDQ_ERR_UNSUPPORTED;
    if (bits <= 3 && !zero) return MIXDQ_ERR_UNSUPPORTED;  // bit-plane codes are unsigned only
    if (reinterpret_cast<uintptr_t>(packed_out) & 15) return MIXDQ_ERR_ALIGNMENT;
    const int64_t pitch = row_pitch_bytes(K, bits, layout);
    const __half* w = static_cast<const __half*>(W);
    uint8_t* out = static_cast<uint8_t*>(packed_out);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    switch (bits) {
        case 2: launch_pack<2>(w, N, K, scale, zero, layout, pitch, out, st); break;
        case 3: launch_pack<3>(w, N, K, scale, zero, layout, pitch, out, st); break;
        case 4: launch_pack<4>(w, N, K, scale, zero, layout, pitch, out, st); break;
        default: launch_pack<8>(w, N, K, scale, zero, layout, pitch, out, st);
    }
    return finish_constants(static_cast<cudaStream_t>(stream));
}

extern "C" int mixdq_unpack_weights(const void* packed, int64_t N, int64_t K, int bits, int is_signed,
                                    int layout, int16_t* codes_out, void* stream)
{
    if (!packed || !codes_out || N <= 0 || K <= 0) return MIXDQ_ERR_INVALID_ARG;
    if (layout != MIXDQ_LAYOUT_CANONICAL && layout != MIXDQ_LAYOUT_DEVICE) return MIXDQ_ERR_INVALID_ARG;
    if (!width_ok(bits)) return MIXDQ_ERR_UNSUPPORTED;
    if (bits <= 3 && is_signed) return MIXDQ_ERR_UNSUPPORTED;
    const int64_t pitch = row_pitch_bytes(K, bits, layout);
    unpack_kernel<<<static_cast<unsigned>(ceil_div(N * K, 256)), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const uint8_t*>(packed), N, K, bits, is_signed, layout, pitch, codes_out);
    return check_launch();
}

extern "C" int mixdq_weight_code_sums(const void* packed_W, int64_t N, int64_t K, int bits, int32_t* sums_out,
                                      void* stream)
{
    if (!packed_W || !sums_out || N <= 0 || K <= 0) return MIXDQ_ERR_INVALID_ARG;
    if (bits != 4 && bits != 8) return MIXDQ_ERR_UNSUPPORTED;
    const int64_t pitch = row_pitch_bytes(K, bits, MIXDQ_LAYOUT_DEVICE);
    code_sums_kernel<<<static_cast<unsigned>(N), 128, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const uint8_t*>(packed_W), K, bits, pitch, sums_out);
    return finish_constants(static_cast<cudaStream_t>(stream));
}
