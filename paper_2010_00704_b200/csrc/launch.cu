// Per-process caches behind launch.cuh.
#include "launch.cuh"
#include "tensor_map.cuh"

namespace bcnn {

namespace {

constexpr int MAX_DEVICES = 64;
constexpr int SLOTS = 1024;               // open-addressed, insert-only; a full table only costs the repeated query

struct Slot {
    std::atomic<uint64_t> key{0};
    std::atomic<int> value{0};
};

// the value stored for `key`, or 0
int find(const Slot (&t)[SLOTS], uint64_t key)
{
    for (uint32_t i = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 54), n = 0; n < 16; ++n, i = (i + 1) % SLOTS) {
        const uint64_t k = t[i].key.load(std::memory_order_acquire);
        if (k == key) return t[i].value.load(std::memory_order_acquire);
        if (k == 0) return 0;
    }
    return 0;
}

// values are never 0; a reader that meets the key before its value takes the slow path once more
void insert(Slot (&t)[SLOTS], uint64_t key, int value)
{
    for (uint32_t i = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 54), n = 0; n < 16; ++n, i = (i + 1) % SLOTS) {
        uint64_t expected = 0;
        if (t[i].key.compare_exchange_strong(expected, key) || expected == key) {
            t[i].value.store(value, std::memory_order_release);
            return;
        }
    }
}

int current_device()
{
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess ? dev : -1;
}

// kernel addresses fit 48 bits
uint64_t kernel_key(const void *kernel, int dev) { return ((uint64_t)reinterpret_cast<uintptr_t>(kernel) << 6) | (uint64_t)(dev & 63); }

}  // namespace

EncodeTiledFn encode_tiled_fn()
{
    static std::atomic<EncodeTiledFn> fn{nullptr};
    EncodeTiledFn f = fn.load(std::memory_order_relaxed);
    if (!f) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess && qres == cudaDriverEntryPointSuccess)
            f = reinterpret_cast<EncodeTiledFn>(ptr);
        fn.store(f, std::memory_order_relaxed);
    }
    return f;
}

int sm_count()
{
    static std::atomic<int> cache[MAX_DEVICES];
    const int dev = current_device();
    if (dev < 0 || dev >= MAX_DEVICES) return 148;
    int sms = cache[dev].load(std::memory_order_relaxed);
    if (sms == 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 148;
        cache[dev].store(sms, std::memory_order_relaxed);
    }
    return sms;
}

int blocks_per_sm(const void *kernel, int threads, size_t smem)
{
    static Slot table[SLOTS];
    const int dev = current_device();
    // one thread count per kernel; two kernels that met on one key would only size their grids differently
    const uint64_t key = (kernel_key(kernel, dev) * 0xD6E8FEB86659FD93ull ^ (uint64_t)smem * 0xA24BAED4963EE407ull) | 1u;
    int n = find(table, key);
    if (n > 0) return n;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        return 1;
    }
    if (dev >= 0 && dev < MAX_DEVICES) insert(table, key, n);
    return n;
}

int max_clusters(const void *kernel, int cluster, int threads, size_t smem)
{
    static Slot table[SLOTS];
    const int dev = current_device();
    // one cluster size, thread count and size of shared memory per kernel
    const uint64_t key = kernel_key(kernel, dev);
    int n = find(table, key);
    if (n > 0) return n;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cluster);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        return 0;
    }
    if (dev >= 0 && dev < MAX_DEVICES) insert(table, key, n);
    return n;
}

bool allow_smem(const void *kernel, int bytes)
{
    static Slot table[SLOTS];
    const int dev = current_device();
    const uint64_t key = kernel_key(kernel, dev);
    if (find(table, key) == bytes) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    if (dev >= 0 && dev < MAX_DEVICES) insert(table, key, bytes);
    return true;
}

}  // namespace bcnn
