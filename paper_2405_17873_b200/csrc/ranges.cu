// Per-tensor activation ranges (max |x|, or min and max with 0 included) and the 8-bit quantizer's parameters that
// follow from them: one call per layer and step where activation scales are dynamic.
#include "common.cuh"

namespace mixdq {

namespace {

enum : int { R_ABSMAX = 0, R_SCALE = 1, R_MINMAX = 2, R_PARAMS = 3 };  // what becomes of the range

__host__ __device__ constexpr bool one_sided(int mode) { return mode == R_ABSMAX || mode == R_SCALE; }

// out0 / out1: max |x|; the symmetric scale max |x| / 127 (1 for an all-zero tensor); {lo, hi} at out0[0 .. 1]; or
// scale = (hi - lo) / 255 and zero = clamp(rne(-lo / scale), 0, 255) (an all-zero tensor: scale 1, zero 0).
template <int MODE>
__device__ __forceinline__ void store_range(float lo, float hi, float* out0, int32_t* out1)
{
    if (MODE == R_ABSMAX) {
        out0[0] = hi;
    } else if (MODE == R_SCALE) {
        out0[0] = (hi == 0.f) ? 1.f : __fdiv_rn(hi, 127.f);
    } else if (MODE == R_MINMAX) {
        out0[0] = lo;
        out0[1] = hi;
    } else if (hi == lo) {
        out0[0] = 1.f;
        out1[0] = 0;
    } else {
        const float s = __fdiv_rn(__fsub_rn(hi, lo), 255.f);
        const float inv = __fdiv_rn(1.f, s);
        // -lo * inv <= 255 * (1 + 2^-22): the magic-number addition rounds the exact product to nearest even
        const float t = __fmaf_rn(-lo, inv, 12582912.f);
        const int z = static_cast<int>(__float_as_uint(t)) - 0x4B400000;
        out0[0] = s;
        out1[0] = z < 0 ? 0 : (z > 255 ? 255 : z);
    }
}

__device__ __forceinline__ void fold(__half2& lo, __half2& hi, uint4 v, bool abs)
{
    const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (abs) {
            hi = __hmax2(hi, __habs2(h[j]));
        } else {
            lo = __hmin2(lo, h[j]);
            hi = __hmax2(hi, h[j]);
        }
    }
}

// This thread's share of X, every `step`-th of its 16-byte chunks from `first` on, eight in flight at a time.  lo and hi
// start at 0.  skip_mod > 0 leaves out rows whose index is a multiple of it.
template <bool ABS>
__device__ __forceinline__ void scan(const __half* __restrict__ X, long long rows, long long cols, long long stride, int skip_mod,
                                     long long first, long long step, float& lo_out, float& hi_out)
{
    float lo = 0.f, hi = 0.f;
    if (((cols | stride) & 7) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0) {
        __half2 l2 = __half2half2(__ushort_as_half(0)), h2 = l2;
        const uint4* base = reinterpret_cast<const uint4*>(X);
        const long long per_row = cols >> 3, total = rows * per_row;
        if (stride == cols && skip_mod <= 0) {
            long long i = first;
            for (; i + 7 * step < total; i += 8 * step) {
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = __ldg(base + i + u * step);
#pragma unroll
                for (int u = 0; u < 8; ++u) fold(l2, h2, v[u], ABS);
            }
            for (; i < total; i += step) fold(l2, h2, __ldg(base + i), ABS);
        } else {
            const long long stride8 = stride >> 3;
#pragma unroll 4
            for (long long i = first; i < total; i += step) {
                const long long r = total <= 0x7fffffff ? static_cast<uint32_t>(i) / static_cast<uint32_t>(per_row) : i / per_row;
                if (skip_mod > 0 && r % skip_mod == 0) continue;
                fold(l2, h2, __ldg(base + r * stride8 + (i - r * per_row)), ABS);
            }
        }
        lo = fminf(__low2float(l2), __high2float(l2));
        hi = fmaxf(__low2float(h2), __high2float(h2));
    } else {
        const long long total = rows * cols;
        for (long long i = first; i < total; i += step) {
            const long long r = i / cols;
            if (skip_mod > 0 && r % skip_mod == 0) continue;
            const float f = __half2float(X[r * stride + (i - r * cols)]);
            lo = fminf(lo, f);
            hi = fmaxf(hi, ABS ? fabsf(f) : f);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    lo_out = lo < 0.f ? lo : 0.f;  // (+0, never -0)
    hi_out = hi > 0.f ? hi : 0.f;
}

// Tensors of up to kClusterBytes: ONE launch of one cluster of up to 16 CTAs, whose partial ranges meet in the first
// CTA's shared memory; nothing has to be cleared beforehand and no atomics are needed.  Sixteen SMs read some 2 TB/s from
// L2, so the whole device would scan faster only where the scan outweighs the two further launches (clear, finish)
// that a grid needs to agree on one number.
constexpr int kClusterThreads = 1024;
constexpr int kClusterMax = 16;
constexpr long long kClusterBytes = 8ll << 20;

template <int MODE>
__global__ void __launch_bounds__(kClusterThreads)
range_cluster_kernel(const __half* __restrict__ X, long long rows, long long cols, long long stride, int skip_mod,
                     float* __restrict__ out0, int32_t* __restrict__ out1)
{
    __shared__ float2 s_warp[kClusterThreads / 32];
    __shared__ float2 s_cta[kClusterMax];
    cluster_arrive();  // "this CTA runs": its shared memory may be written to from then on
    pdl_launch_dependents();
    pdl_wait();
    const int rank = static_cast<int>(blockIdx.x), ctas = static_cast<int>(gridDim.x);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float lo, hi;
    scan<one_sided(MODE)>(X, rows, cols, stride, skip_mod, rank * kClusterThreads + tid, static_cast<long long>(ctas) * kClusterThreads,
                          lo, hi);
    if (lane == 0) s_warp[warp] = make_float2(lo, hi);
    __syncthreads();
    cluster_wait();
    if (warp == 0) {
        lo = s_warp[lane].x;
        hi = s_warp[lane].y;
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (lane == 0) {
            const uint32_t there = map_to_cta(smem_u32(&s_cta[rank]), 0);
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(there), "f"(lo), "f"(hi) : "memory");
        }
    }
    cluster_sync();
    if (rank == 0 && tid == 0) {
        for (int i = 0; i < ctas; ++i) {
            lo = fminf(lo, s_cta[i].x);
            hi = fmaxf(hi, s_cta[i].y);
        }
        store_range<MODE>(lo, hi, out0, out1);
    }
}

// Larger tensors: clear, scan with the whole device, finish.  The running range lives in the outputs themselves, as
// integers that order like the floats (negative ones with their magnitude bits flipped) and are 0 for +0.
__device__ __forceinline__ int order_key(float f)
{
    const int b = __float_as_int(f);
    return b < 0 ? b ^ 0x7fffffff : b;
}

template <int MODE>
__device__ __forceinline__ int* second_slot(float* out0, int32_t* out1)
{
    return MODE == R_MINMAX ? reinterpret_cast<int*>(out0 + 1) : out1;
}

template <int MODE>
__global__ void range_clear_kernel(float* out0, int32_t* out1)
{
    pdl_launch_dependents();
    pdl_wait();
    out0[0] = 0.f;
    if (!one_sided(MODE)) *second_slot<MODE>(out0, out1) = 0;
}

template <int MODE>
__global__ void __launch_bounds__(256)
range_scan_kernel(const __half* __restrict__ X, long long rows, long long cols, long long stride, int skip_mod, float* out0,
                  int32_t* out1)
{
    pdl_launch_dependents();
    pdl_wait();
    float lo, hi;
    scan<one_sided(MODE)>(X, rows, cols, stride, skip_mod, blockIdx.x * 256ll + threadIdx.x, gridDim.x * 256ll, lo, hi);
    if ((threadIdx.x & 31) == 0) {
        int* first = reinterpret_cast<int*>(out0);
        if (one_sided(MODE)) {
            if (hi > 0.f) atomicMax(first, order_key(hi));
        } else {
            if (lo < 0.f) atomicMin(first, order_key(lo));
            if (hi > 0.f) atomicMax(second_slot<MODE>(out0, out1), order_key(hi));
        }
    }
}

template <int MODE>
__global__ void range_finish_kernel(float* out0, int32_t* out1)
{
    pdl_launch_dependents();
    pdl_wait();
    const int a = __float_as_int(out0[0]);
    if (one_sided(MODE)) {
        store_range<MODE>(0.f, __int_as_float(a), out0, out1);
    } else {
        const int b = *second_slot<MODE>(out0, out1);
        store_range<MODE>(__int_as_float(a < 0 ? a ^ 0x7fffffff : a), __int_as_float(b), out0, out1);
    }
}

template <int MODE>
int run_range(const void* X, int64_t rows, int64_t cols, int64_t stride, int skip_mod, float* out0, int32_t* out1, void* stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const __half* x = static_cast<const __half*>(X);
    const long long r = rows, c = cols, s = stride, bytes = 2ll * rows * cols;
    if (bytes <= kClusterBytes) {
        auto kernel = range_cluster_kernel<MODE>;
        unsigned ctas = 1;  // at least 16 KB each: one 16-byte chunk per thread
        while (ctas < kClusterMax && bytes > static_cast<long long>(ctas) * 16 * kClusterThreads) ctas *= 2;
        if (allow_large_clusters(reinterpret_cast<const void*>(kernel)) != MIXDQ_OK) return MIXDQ_ERR_CUDA;
        return launch_ex(kernel, dim3(ctas), dim3(kClusterThreads), 0, st, ctas, 1, x, r, c, s, skip_mod, out0, out1);
    }
    int rc = launch_ex(range_clear_kernel<MODE>, dim3(1), dim3(1), 0, st, 1, 1, out0, out1);
    if (rc != MIXDQ_OK) return rc;
    const unsigned grid = static_cast<unsigned>(8 * (sm_count() > 0 ? sm_count() : 1));
    rc = launch_ex(range_scan_kernel<MODE>, dim3(grid), dim3(256), 0, st, 1, 1, x, r, c, s, skip_mod, out0, out1);
    if (rc != MIXDQ_OK || MODE == R_ABSMAX) return rc;
    return launch_ex(range_finish_kernel<MODE>, dim3(1), dim3(1), 0, st, 1, 1, out0, out1);
}

template <int MODE>
__global__ void params_from_range_kernel(const float* __restrict__ range, float* __restrict__ out0, int32_t* __restrict__ out1)
{
    pdl_launch_dependents();
    pdl_wait();
    if (MODE == R_SCALE)
        store_range<MODE>(0.f, range[0], out0, out1);
    else
        store_range<MODE>(range[0], range[1], out0, out1);
}

}  // namespace

}  // namespace mixdq

using namespace mixdq;

static bool range_args_ok(const void* X, int64_t rows, int64_t cols, int64_t row_stride)
{
    return X && rows > 0 && cols > 0 && row_stride >= cols;
}

extern "C" int mixdq_act_absmax(const void* X, int64_t rows, int64_t cols, int64_t row_stride, int skip_rows_mod,
                                float* amax_out, void* stream)
{
    if (!range_args_ok(X, rows, cols, row_stride) || !amax_out || skip_rows_mod < 0) return MIXDQ_ERR_INVALID_ARG;
    return run_range<R_ABSMAX>(X, rows, cols, row_stride, skip_rows_mod, amax_out, nullptr, stream);
}

extern "C" int mixdq_act_scale(const void* X, int64_t rows, int64_t cols, int64_t row_stride, int skip_rows_mod,
                               float* scale_out, void* stream)
{
    if (!range_args_ok(X, rows, cols, row_stride) || !scale_out || skip_rows_mod < 0) return MIXDQ_ERR_INVALID_ARG;
    return run_range<R_SCALE>(X, rows, cols, row_stride, skip_rows_mod, scale_out, nullptr, stream);
}

extern "C" int mixdq_act_scale_from_absmax(const float* amax, float* scale_out, void* stream)
{
    if (!amax || !scale_out) return MIXDQ_ERR_INVALID_ARG;
    return launch_ex(params_from_range_kernel<R_SCALE>, dim3(1), dim3(1), 0, static_cast<cudaStream_t>(stream), 1, 1, amax,
                     scale_out, static_cast<int32_t*>(nullptr));
}

extern "C" int mixdq_act_minmax(const void* X, int64_t rows, int64_t cols, int64_t row_stride, float* minmax_out, void* stream)
{
    if (!range_args_ok(X, rows, cols, row_stride) || !minmax_out) return MIXDQ_ERR_INVALID_ARG;
    return run_range<R_MINMAX>(X, rows, cols, row_stride, 0, minmax_out, nullptr, stream);
}

extern "C" int mixdq_act_asym_params(const void* X, int64_t rows, int64_t cols, int64_t row_stride, float* scale_out,
                                     int32_t* zero_out, void* stream)
{
    if (!range_args_ok(X, rows, cols, row_stride) || !scale_out || !zero_out) return MIXDQ_ERR_INVALID_ARG;
    return run_range<R_PARAMS>(X, rows, cols, row_stride, 0, scale_out, zero_out, stream);
}

extern "C" int mixdq_act_asym_params_from_minmax(const float* minmax, float* scale_out, int32_t* zero_out, void* stream)
{
    if (!minmax || !scale_out || !zero_out) return MIXDQ_ERR_INVALID_ARG;
    return launch_ex(params_from_range_kernel<R_PARAMS>, dim3(1), dim3(1), 0, static_cast<cudaStream_t>(stream), 1, 1, minmax,
                     scale_out, zero_out);
}
