// Per-device facts the launch plans depend on, looked up once per device ordinal.
#include "common.cuh"

#include <atomic>
#include <mutex>
#include <stdlib.h>
#include <string.h>

namespace vptq {

namespace {
constexpr int kMaxDevices = 64;
std::atomic<int> g_sm_count[kMaxDevices];     // 0 = not looked up yet
std::atomic<unsigned long long> g_wait_limit{0};
}

unsigned long long debug_wait_limit() { return g_wait_limit.load(std::memory_order_relaxed); }
void set_debug_wait_limit(unsigned long long cycles) { g_wait_limit.store(cycles, std::memory_order_relaxed); }

// Streaming multiprocessors of the CURRENT device (every persistent grid and every row split is sized by
// it, so a plan made with one device current must be launched with that device current).  Without a
// usable device (size queries on a machine with no GPU) the answer is that of a B200.
int device_sm_count()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 148;
    if (dev < kMaxDevices) {
        const int cached = g_sm_count[dev].load(std::memory_order_relaxed);
        if (cached > 0) return cached;
    }
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) return 148;
    if (dev < kMaxDevices) g_sm_count[dev].store(v, std::memory_order_relaxed);
    return v;
}

// What has been allowed so far, per (kernel, device): a small open-addressed table that only ever grows and is read without
// a lock (a slot's key is written last).  More kernels than slots fall back to setting the attribute at every launch.
namespace {
struct SmemSlot {
    std::atomic<const void *> kernel{nullptr};
    int dev;
    std::atomic<size_t> bytes{0};
};
constexpr int kSmemSlots = 1024;
SmemSlot g_smem[kSmemSlots];
std::mutex g_smem_mutex;
}

cudaError_t allow_dynamic_smem(const void *kernel, size_t bytes)
{
    if (bytes <= 40 * 1024) return cudaSuccess;           // with its static part inside the 48 KB every kernel may use
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const size_t h = ((size_t)kernel >> 4) * 31 + (size_t)dev;
    for (int i = 0; i < kSmemSlots; i++) {
        SmemSlot &s = g_smem[(h + i) % kSmemSlots];
        const void *k = s.kernel.load(std::memory_order_acquire);
        if (k == nullptr) break;
        if (k == kernel && s.dev == dev) {
            if (s.bytes.load(std::memory_order_acquire) >= bytes) return cudaSuccess;
            break;
        }
    }
    std::lock_guard<std::mutex> lock(g_smem_mutex);
    SmemSlot *slot = nullptr;
    for (int i = 0; i < kSmemSlots && slot == nullptr; i++) {
        SmemSlot &s = g_smem[(h + i) % kSmemSlots];
        const void *k = s.kernel.load(std::memory_order_relaxed);
        if (k == nullptr || (k == kernel && s.dev == dev)) slot = &s;
    }
    if (slot != nullptr && slot->kernel.load(std::memory_order_relaxed) == kernel && slot->bytes.load(std::memory_order_relaxed) >= bytes)
        return cudaSuccess;                                // another thread was faster
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && slot != nullptr) {
        slot->dev = dev;
        slot->bytes.store(bytes, std::memory_order_release);
        slot->kernel.store(kernel, std::memory_order_release);
    }
    return e;
}

namespace {
struct ClusterSlot { const void *kernel; int dev, size, answer; };
ClusterSlot g_clusters[256];
std::atomic<int> g_n_clusters{0};
std::mutex g_clusters_mutex;
}

int max_resident_clusters(const void *kernel, int size, int threads, size_t smem)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 148 / size;      // size queries without a device: those of a B200
    auto find = [&](int n) {
        for (int i = 0; i < n; i++)
            if (g_clusters[i].kernel == kernel && g_clusters[i].dev == dev && g_clusters[i].size == size) return g_clusters[i].answer;
        return -1;
    };
    int a = find(g_n_clusters.load(std::memory_order_acquire));
    if (a >= 0) return a;
    std::lock_guard<std::mutex> lock(g_clusters_mutex);
    const int n = g_n_clusters.load(std::memory_order_relaxed);
    if ((a = find(n)) >= 0) return a;
    a = 0;
    if (allow_dynamic_smem(kernel, smem) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)size * 1024u);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = attr; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&a, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); a = 0; }
    }
    if (n < 256) {
        g_clusters[n] = {kernel, dev, size, a};
        g_n_clusters.store(n + 1, std::memory_order_release);
    }
    return a;
}

bool pdl_enabled(const char *family)
{
    static const char *off = getenv("VPTQ_NO_PDL");          // read once
    if (off == nullptr || off[0] == 0) return true;
    return strstr(off, "all") == nullptr && strstr(off, family) == nullptr;
}

}  // namespace vptq
