// mqr_noalloc.cu -- mqr_sort_objects_noalloc: the Morton-key computation and
// radix sort of the objects, for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc: embedders that own all device memory
// (a fixed budget or their own pool) and latency-critical loops that cannot
// afford the device-wide synchronisation cudaMalloc / cudaFree may cause.
// This entry point needs no allocation at all: its scratch (sort ping-pong
// buffers, digit counts) is one file-scope __device__
// array of fixed size (about 4.3 MB for MQR_NOALLOC_MAX_OBJECTS objects),
// which every GPU that loads the library holds until the process exits.  The
// caller passes only inputs and outputs.
#include <cuda_runtime.h>

#include <mutex>
#include <string>

#include "../../include/mqr.h"
#include "mqr_internal.cuh"

using namespace mqr;

namespace {

constexpr uint32_t kMaxN = MQR_NOALLOC_MAX_OBJECTS;
constexpr uint32_t kTiles = (kMaxN + kSortTile - 1) / kSortTile;

// Layout of the scratch array (byte offsets, each 256-byte aligned).
constexpr size_t kOffKeysA = 0;
constexpr size_t kOffKeysB = kOffKeysA + (size_t)kMaxN * 8;
constexpr size_t kOffErr = kOffKeysB + (size_t)kMaxN * 8;             // error word
constexpr size_t kOffGroup = kOffErr + 256;                            // coarse digit counts of the four passes
constexpr size_t kOffTile = kOffGroup + 4 * sort_group_words(kMaxN) * 4;
constexpr size_t kZeroBytes = kOffTile - kOffErr;
constexpr size_t kScratchBytes = kOffTile + (size_t)256 * kTiles * 4;  // the pass's tile digit counts

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
unsigned char *g_dev_ptr[kMaxDevices] = {};
bool g_dev_small[kMaxDevices] = {};          // the one-launch sort can run there

mqr_status nfail(mqr_status s, const std::string &m) {
    set_last_error(m);   // reported by mqr_last_error()
    return s;
}

// Device address of the scratch array on the current device, looked up once
// per device (cudaGetSymbolAddress must run with that device current).
mqr_status scratch_ptr(unsigned char **out, bool *small) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return nfail(MQR_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return nfail(MQR_ERR_INTERNAL, "device index out of range");
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_dev_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr)
            return nfail(MQR_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        g_dev_ptr[dev] = static_cast<unsigned char *>(p);
        g_dev_small[dev] = small_sort_ready();
    }
    *out = g_dev_ptr[dev];
    *small = g_dev_small[dev];
    return MQR_OK;
}

}  // namespace

extern "C" mqr_status mqr_sort_objects_noalloc(mqr_rect bounds, const float *xy_dev, uint32_t n,
                                               uint32_t *keys_out_dev, uint32_t *ids_out_dev,
                                               void *cuda_stream) {
    if (n > kMaxN)
        return nfail(MQR_ERR_INVALID_ARG, "n exceeds MQR_NOALLOC_MAX_OBJECTS (" + std::to_string(kMaxN) + ")");
    if (n > 0 && (!xy_dev || !keys_out_dev || !ids_out_dev))
        return nfail(MQR_ERR_INVALID_ARG, "xy_dev / keys_out_dev / ids_out_dev is NULL");
    if (!(bounds.xmax > bounds.xmin) || !(bounds.ymax > bounds.ymin))
        return nfail(MQR_ERR_INVALID_ARG, "bounds must have xmax > xmin and ymax > ymin");
    if (n > 0 && ((reinterpret_cast<uintptr_t>(xy_dev) & 7u) ||
                  ((reinterpret_cast<uintptr_t>(keys_out_dev) | reinterpret_cast<uintptr_t>(ids_out_dev)) & 3u)))
        return nfail(MQR_ERR_INVALID_ARG, "xy_dev must be 8-byte and keys_out_dev / ids_out_dev 4-byte aligned");
    if (n == 0) return MQR_OK;
    unsigned char *s = nullptr;
    bool small = false;
    mqr_status st = scratch_ptr(&s, &small);
    if (st != MQR_OK) return st;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    volatile float wx = bounds.xmax - bounds.xmin, wy = bounds.ymax - bounds.ymin;
    volatile float sx = 32768.0f / wx, sy = 32768.0f / wy;

    const float2 *xy = reinterpret_cast<const float2 *>(xy_dev);
    if (small && n <= kSmallSortMax) {           // one launch, no scratch
        cudaError_t e = launch_small_sort(stream, xy, nullptr, n, bounds.xmin, bounds.ymin, sx, sy, Worlds{},
                                          keys_out_dev, ids_out_dev, nullptr, nullptr);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return nfail(MQR_ERR_CUDA, std::string("stream: ") + cudaGetErrorString(e));
        return MQR_OK;
    }
    // The array keeps the previous call's contents: clear the error word and
    // the coarse digit counts.
    cudaError_t e = cudaMemsetAsync(s + kOffErr, 0, kZeroBytes, stream);
    if (e != cudaSuccess) return nfail(MQR_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
    unsigned long long *a = reinterpret_cast<unsigned long long *>(s + kOffKeysA);
    unsigned long long *b = reinterpret_cast<unsigned long long *>(s + kOffKeysB);
    unsigned long long *err = reinterpret_cast<unsigned long long *>(s + kOffErr);
    uint32_t *group = reinterpret_cast<uint32_t *>(s + kOffGroup);
    uint32_t *tile = reinterpret_cast<uint32_t *>(s + kOffTile);
    launch_morton_keys(stream, xy, nullptr, n, bounds.xmin, bounds.ymin, sx, sy, Worlds{}, a, tile, group, nullptr);
    for (int p = 0; p < 4; ++p) {
        launch_sort_pass(stream, a, b, n, 32 + 8 * p, tile, group + sort_group_words(n) * p, p == 0, err,
                         p == 3, nullptr, keys_out_dev, ids_out_dev, nullptr);
        unsigned long long *t = a; a = b; b = t;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return nfail(MQR_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
    unsigned long long herr = 0;
    e = cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return nfail(MQR_ERR_CUDA, std::string("stream: ") + cudaGetErrorString(e));
    if (herr) return nfail(MQR_ERR_INTERNAL, "device index out of range in the sort");
    return MQR_OK;
}
