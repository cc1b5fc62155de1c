// kd_noalloc.cu -- presort of one small cloud that allocates no memory.
//
// kd_presort takes its workspace from the context's stream-ordered pool.
// Some callers cannot let a library allocate at call time: a process that
// has already handed all device memory to its own allocator (a call would
// then fail with KD_ENOMEM), or a latency-bound loop where a growing pool or
// a cudaFree would stall the device for every stream.  kd_presort_noalloc
// serves them for clouds of up to KD_NOALLOC_MAX_N tuples: its only
// workspace is one file-scope device array (NA_BYTES), set up once per
// device, and its outputs go to buffers the caller owns.  The sorts are
// those of kd_small.cu.
//
// It computes what kd_presort + kd_handle_arrays compute (Section 2.1: the
// k index arrays sorted by the cyclic super keys x_d : x_{d+1} : ... and
// duplicate tuples removed, the smallest index of a run surviving).
//
// The one static array per device is shared by every call on that device
// that uses it (more than 2048 tuples, or outputs that overlap the
// coordinates of a call that reads these while it writes, which it copies
// there first): two such calls whose kernels can overlap (different streams,
// or different threads without ordering between them) race on it.  Order
// such calls on one stream.
#include <mutex>
#include <string>

#include "kd_internal.cuh"
#include "kdtree.h"

namespace kd {
// Context access (kd_api.cu).
int ctx_device(const kd_ctx* ctx);
cudaStream_t ctx_stream(const kd_ctx* ctx);
void ctx_set_error(kd_ctx* ctx, const std::string& msg);
void ctx_add_launches(kd_ctx* ctx, int n);
cudaError_t launch_small_arrays(int dtype, const void* coords, int n, int k, void* work, int32_t* rows, int32_t* m_out,
                                cudaStream_t s);
size_t small_arrays_bytes(int n, int k);
int small_sort_launches(int64_t n);
bool small_reads_while_writing(int64_t n);
}  // namespace kd

namespace {

constexpr int NA_MAX_N = KD_NOALLOC_MAX_N;

// The chunked sort's workspace at the largest cloud of 64-bit keys (keys,
// indices and places of k rows, a bit per place, a word per chunk), which
// exceeds the coordinates of any cloud.
constexpr size_t NA_BYTES = (size_t)KD_MAX_K * NA_MAX_N * (8 + 4 + 4) + (size_t)KD_MAX_K * NA_MAX_N / 8 + 1024;
static __device__ __align__(256) unsigned char na_scratch[NA_BYTES];

// Per-device set-up, once per device with that device current: the address
// of the static array.
std::mutex na_mu;
unsigned char* na_ws[64] = {};

cudaError_t noalloc_setup(int device, unsigned char** ws) {
    std::lock_guard<std::mutex> lk(na_mu);
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (!na_ws[device]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, na_scratch);
        if (e != cudaSuccess) return e;
        na_ws[device] = static_cast<unsigned char*>(p);
    }
    *ws = na_ws[device];
    return cudaSuccess;
}

// Device (or managed) memory owned by `device`: a buffer on another GPU
// would be read or written through peer access, which need not be enabled.
bool on_device_memory(const void* p, int device) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();  // the query's own error, raised just now
        return false;
    }
    return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == device;
}

bool overlap(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + nb && y < x + na;
}

kd_status na_fail(kd_ctx* ctx, kd_status code, const std::string& msg) {
    kd::ctx_set_error(ctx, "kd_presort_noalloc: " + msg);
    return code;
}

}  // namespace

extern "C" kd_status kd_presort_noalloc(kd_ctx* ctx, const kd_cloud* cloud, int32_t* arrays_out, int32_t* m_out) {
    if (!ctx) return KD_EINVAL;
    if (!cloud || !m_out) return na_fail(ctx, KD_EINVAL, "null cloud or m_out");
    const int64_t n = cloud->n;
    const int k = cloud->k;
    if (k < 1 || k > KD_MAX_K) return na_fail(ctx, KD_EINVAL, "k must be in 1.." + std::to_string(KD_MAX_K));
    if (n < 0 || n > NA_MAX_N)
        return na_fail(ctx, KD_EINVAL,
                       "n = " + std::to_string(n) + " exceeds the static workspace limit of " +
                           std::to_string(NA_MAX_N) + " tuples (KD_NOALLOC_MAX_N); use kd_presort");
    if (cloud->dtype != KD_I32 && cloud->dtype != KD_I64 && cloud->dtype != KD_F32)
        return na_fail(ctx, KD_EINVAL, "bad dtype");
    if (!cloud->on_device) return na_fail(ctx, KD_EINVAL, "coordinates must be device memory (on_device = 1)");
    const int dev = kd::ctx_device(ctx);
    cudaError_t e = cudaSetDevice(dev);
    if (e != cudaSuccess) return na_fail(ctx, KD_EDEVICE, cudaGetErrorString(e));
    if (!on_device_memory(m_out, dev))
        return na_fail(ctx, KD_EINVAL, "m_out must be device memory on the context's device");
    if (n > 0 && (!cloud->coords || !arrays_out || !on_device_memory(cloud->coords, dev) ||
                  !on_device_memory(arrays_out, dev)))
        return na_fail(ctx, KD_EINVAL, "coords and arrays_out must be non-null device memory on the context's device");
    unsigned char* ws = nullptr;
    e = noalloc_setup(dev, &ws);
    if (e != cudaSuccess) return na_fail(ctx, KD_EDEVICE, std::string("set-up: ") + cudaGetErrorString(e));
    cudaStream_t s = kd::ctx_stream(ctx);
    if (n == 0) {
        e = cudaMemsetAsync(m_out, 0, sizeof(int32_t), s);
        return e == cudaSuccess ? KD_OK : na_fail(ctx, KD_EDEVICE, cudaGetErrorString(e));
    }
    const void* coords = cloud->coords;
    const size_t bytes = (size_t)n * k * (cloud->dtype == KD_I64 ? 8 : 4);
    if (kd::small_reads_while_writing(n) &&
        (overlap(coords, bytes, arrays_out, (size_t)n * k * 4) || overlap(coords, bytes, m_out, 4))) {
        e = cudaMemcpyAsync(ws, coords, bytes, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return na_fail(ctx, KD_EDEVICE, cudaGetErrorString(e));
        coords = ws;
    }
    if (kd::small_arrays_bytes((int)n, k) > NA_BYTES) return na_fail(ctx, KD_EINVAL, "internal: workspace");
    e = kd::launch_small_arrays(cloud->dtype, coords, (int)n, k, ws, arrays_out, m_out, s);
    if (e != cudaSuccess) return na_fail(ctx, KD_EDEVICE, std::string("launch: ") + cudaGetErrorString(e));
    kd::ctx_add_launches(ctx, kd::small_sort_launches(n));
    return KD_OK;
}
