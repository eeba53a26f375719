// Tensor-map (TMA descriptor) encoding.  The driver entry point is looked up through the
// runtime so that the library has no link-time dependency on libcuda and still loads on
// a machine without a GPU driver.
#include <atomic>
#include <mutex>
#include <new>
#include <unordered_set>

#include "common.cuh"

namespace mixdq {

namespace {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);
using EncodeIm2colFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const int*, const int*, cuuint32_t, cuuint32_t, const cuuint32_t*,
                                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                    CUtensorMapFloatOOBfill);

void* driver_entry(const char* name)
{
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess) return p;
    (void)cudaGetLastError();
    return nullptr;
}

EncodeTiledFn get_encode_fn()
{
    static const EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(driver_entry("cuTensorMapEncodeTiled"));
    return fn;
}

EncodeIm2colFn get_encode_im2col_fn()
{
    static const EncodeIm2colFn fn = reinterpret_cast<EncodeIm2colFn>(driver_entry("cuTensorMapEncodeIm2col"));
    return fn;
}

}  // namespace

int encode_tmap_2d_u8(CUtensorMap* map, const void* base, uint64_t row_bytes, uint64_t rows,
                      uint64_t pitch_bytes, uint32_t box_bytes, uint32_t box_rows, int swizzle)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return MIXDQ_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (pitch_bytes & 15)) return MIXDQ_ERR_ALIGNMENT;
    cuuint64_t dims[2] = {row_bytes, rows};
    cuuint64_t strides[1] = {pitch_bytes};
    cuuint32_t box[2] = {box_bytes, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swizzle == SWIZZLE_128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                           : (swizzle == SWIZZLE_64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE),
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? MIXDQ_OK : MIXDQ_ERR_CUDA;
}

int encode_tmap_2d_f16(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows,
                       uint64_t pitch_elems, uint32_t box_cols, uint32_t box_rows, bool swizzle64)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return MIXDQ_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15) || ((pitch_elems * 2) & 15)) return MIXDQ_ERR_ALIGNMENT;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {pitch_elems * 2};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? MIXDQ_OK : MIXDQ_ERR_CUDA;
}


static int encode_tmap_4d(CUtensorMap* map, CUtensorMapDataType dtype, const void* base, const uint64_t dims[4],
                          const uint64_t strides_bytes[3], const uint32_t box[4], uint32_t hw_step);

int encode_tmap_4d_u8(CUtensorMap* map, const void* base, const uint64_t dims[4], const uint64_t strides_bytes[3],
                      const uint32_t box[4], uint32_t hw_step)
{
    return encode_tmap_4d(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, base, dims, strides_bytes, box, hw_step);
}

int encode_tmap_4d_f16(CUtensorMap* map, const void* base, const uint64_t dims[4], const uint64_t strides_bytes[3],
                       const uint32_t box[4], uint32_t hw_step)
{
    return encode_tmap_4d(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, base, dims, strides_bytes, box, hw_step);
}

static int encode_tmap_4d(CUtensorMap* map, CUtensorMapDataType dtype, const void* base, const uint64_t dims[4],
                          const uint64_t strides_bytes[3], const uint32_t box[4], uint32_t hw_step)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return MIXDQ_ERR_CUDA;
    if (reinterpret_cast<uintptr_t>(base) & 15) return MIXDQ_ERR_ALIGNMENT;
    cuuint64_t d[4], st[3];
    // hw_step > 1 (strided convolution): the box takes every hw_step-th pixel along W and H; the
    // encoder wants the traversed extent, of which it loads ceil(extent / step) elements
    cuuint32_t b[4], estr[4] = {1, hw_step, hw_step, 1};
    for (int i = 0; i < 4; ++i) {
        d[i] = dims[i];
        b[i] = (i == 1 || i == 2) ? box[i] * hw_step : box[i];
        if (b[i] > 256) return MIXDQ_ERR_UNSUPPORTED;
    }
    for (int i = 0; i < 3; ++i) {
        if (strides_bytes[i] & 15) return MIXDQ_ERR_ALIGNMENT;
        st[i] = strides_bytes[i];
    }
    CUresult r = fn(map, dtype, 4, const_cast<void*>(base), d, st, b, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? MIXDQ_OK : MIXDQ_ERR_CUDA;
}

int encode_tmap_im2col3x3(CUtensorMap* map, const void* base, bool f16, int B, int H, int W, int C, int pad, int stride,
                          int channels, int pixels)
{
    EncodeIm2colFn fn = get_encode_im2col_fn();
    if (!fn) return MIXDQ_ERR_CUDA;
    const cuuint64_t row = static_cast<cuuint64_t>(C) * (f16 ? 2 : 1);
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (row & 15)) return MIXDQ_ERR_ALIGNMENT;
    const cuuint64_t d[4] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(W), static_cast<cuuint64_t>(H),
                             static_cast<cuuint64_t>(B)};
    const cuuint64_t st[3] = {row, row * W, row * W * H};
    // the filter's corner pixel runs over [-1, W - 2] (a border that is part of the image moves it by one)
    const int lower[2] = {pad - 1, pad - 1}, upper[2] = {-1 - pad, -1 - pad};
    const cuuint32_t step[4] = {1, static_cast<cuuint32_t>(stride), static_cast<cuuint32_t>(stride), 1};
    CUresult r = fn(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(base),
                    d, st, lower, upper, static_cast<cuuint32_t>(channels), static_cast<cuuint32_t>(pixels), step,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? MIXDQ_OK : MIXDQ_ERR_CUDA;
}

namespace {

constexpr int kMaxDevices = 64;

// Function attributes and device properties belong to a device: everything cached here is keyed by it.
int current_device()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    return (dev >= 0 && dev < kMaxDevices) ? dev : -1;
}

}  // namespace

namespace {

// Sets a function attribute once per (device, kernel).
int set_once(const void* kernel, cudaFuncAttribute attribute, int value, std::mutex& mu, std::unordered_set<const void*> (&done)[kMaxDevices])
{
    const int dev = current_device();
    if (dev < 0) return MIXDQ_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev].count(kernel)) return MIXDQ_OK;
    MIXDQ_CUDA_TRY(cudaFuncSetAttribute(kernel, attribute, value));
    try {
        done[dev].insert(kernel);
    } catch (const std::bad_alloc&) {
        // set all the same, and again by the next call: nothing may be thrown through the C interface
    }
    return MIXDQ_OK;
}

}  // namespace

int prefer_max_shared_carveout(const void* kernel)
{
    static std::mutex mu;
    static std::unordered_set<const void*> done[kMaxDevices];
    return set_once(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared, mu, done);
}

int ensure_dynamic_smem(const void* kernel, int bytes)
{
    static std::mutex mu;
    static std::unordered_set<const void*> done[kMaxDevices];
    return set_once(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes, mu, done);
}

int allow_large_clusters(const void* kernel)
{
    static std::mutex mu;
    static std::unordered_set<const void*> done[kMaxDevices];
    return set_once(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1, mu, done);
}

namespace {

// Notes by (device, handle): a handle alone does not name a stream, the default stream is handle 0 on every device.  (A
// stream's id would do, but asking for it ends a capture with an error.)  A destroyed stream's handle may come back: the
// new stream's first launch then is a plain one for nothing.
struct Note {
    int device;
    cudaStream_t stream;
    uint64_t serial;  // another one each time: a launch takes the note that it saw, not one left since
};

constexpr size_t kMaxNotes = 64;
std::mutex g_notes_mutex;
Note g_notes[kMaxNotes];
std::atomic<size_t> g_note_count{0};  // read without the lock by every launch
uint64_t g_note_serial = 0;

bool capturing(cudaStream_t stream)
{
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &status) == cudaSuccess) return status != cudaStreamCaptureStatusNone;
    (void)cudaGetLastError();
    return true;  // (the default stream while another one captures: nothing can be launched on it)
}

// The default stream has two handles.
cudaStream_t one_handle(cudaStream_t stream) { return stream == cudaStreamLegacy ? nullptr : stream; }

// With the lock held.
Note* find_note(int device, cudaStream_t stream)
{
    for (size_t i = 0, n = g_note_count.load(std::memory_order_relaxed); i < n; ++i)
        if (g_notes[i].device == device && g_notes[i].stream == stream) return &g_notes[i];
    return nullptr;
}

}  // namespace

bool note_constants_written(cudaStream_t stream)
{
    // The per-thread handle is another stream in every thread.  While a stream captures, nothing runs: a note left then
    // would be spent on a kernel of another graph or of none.
    const int device = current_device();
    if (device < 0 || stream == cudaStreamPerThread || capturing(stream)) return false;
    std::lock_guard<std::mutex> lock(g_notes_mutex);
    Note* note = find_note(device, one_handle(stream));
    if (!note) {
        const size_t n = g_note_count.load(std::memory_order_relaxed);
        if (n == kMaxNotes) return false;
        note = &g_notes[n];
        note->device = device;
        note->stream = one_handle(stream);
        g_note_count.store(n + 1, std::memory_order_release);
    }
    note->serial = ++g_note_serial;
    return true;
}

ConstantsNote standing_constants_note(cudaStream_t stream)
{
    ConstantsNote r;
    if (g_note_count.load(std::memory_order_acquire) == 0) return r;
    const int device = current_device();
    std::lock_guard<std::mutex> lock(g_notes_mutex);
    if (const Note* note = find_note(device, one_handle(stream))) {
        r.plain = true;
        r.serial = capturing(stream) ? 0 : note->serial;
    }
    return r;
}

void take_constants_note(const ConstantsNote& note)
{
    if (note.serial == 0) return;
    std::lock_guard<std::mutex> lock(g_notes_mutex);
    const size_t n = g_note_count.load(std::memory_order_relaxed);
    for (size_t i = 0; i < n; ++i)
        if (g_notes[i].serial == note.serial) {
            g_notes[i] = g_notes[n - 1];
            g_note_count.store(n - 1, std::memory_order_release);
            return;
        }
}

int sm_count()
{
    static std::mutex mu;
    static int count[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (!count[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        count[dev] = n;
    }
    return count[dev];
}

}  // namespace mixdq
