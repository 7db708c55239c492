// Device memory of the weight handles.
//
// A handle's arrays lie in two blocks (the codes; everything small).  cudaMalloc and cudaFree cost 0.1 - 1 ms each (they map and
// unmap memory and may synchronise the device): a handle of six separate allocations took 0.9 - 8 ms to prepare and 0.6 - 12 ms to
// free, 20 to 100 times the work on the GPU.  A freed block is therefore kept for the next handle of a similar size: at most
// kMaxBytes and kMaxBlocks per device, the rest goes back to the driver at once, and all of it does when an allocation fails.
// A block comes here only after the device was synchronised without an error (qvggt_free_weights), so whoever takes it next may use
// it on any stream.  One mutex serves all threads; nothing is kept by the address or the contents of a caller's buffer.
// A block serves only the context that it was allocated in: after a device reset the addresses of the old one mean nothing, and its
// entries, which must not be freed either, wait here for others to take their places.
#include <cuda.h>

#include <mutex>

#include "qvggt_internal.cuh"
#include "tensor_map.cuh"

namespace {

constexpr size_t kSmall = 1 << 20;          // up to here sizes are rounded up to kSmallGranule, beyond to the driver's 2 MB
constexpr size_t kSmallGranule = 16 << 10, kGranule = 2 << 20;
constexpr size_t kMaxBytes = 64 << 20;      // kept per device: the codes of one block's four linears, one per byte, take 12 MB
constexpr int kMaxBlocks = 64;

struct DeviceBlocks {
    QvggtBlock kept[kMaxBlocks];
    int n = 0;
};

std::mutex g_mutex;
DeviceBlocks g_blocks[kQvggtMaxDevices];

// Identity of the context that the runtime uses on this thread, never used again in this process; 0 where the driver does not tell.
unsigned long long current_context()
{
    using GetIdFn = CUresult (*)(CUcontext, unsigned long long *);
    static const GetIdFn get_id = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) p = nullptr;
        return reinterpret_cast<GetIdFn>(p);
    }();
    unsigned long long id = 0;
    if (!get_id) return 0;
    if (get_id(nullptr, &id) == CUDA_SUCCESS) return id;
    if (cudaFree(nullptr) != cudaSuccess) cudaGetLastError();      // a thread's first call: binds the device's context
    return get_id(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

// Frees everything kept for a context of a device.  The caller holds the mutex.
void drop_all(DeviceBlocks &d, unsigned long long context)
{
    for (int i = d.n - 1; i >= 0; --i)
        if (d.kept[i].context == context) {
            cudaFree(d.kept[i].p);
            d.kept[i] = d.kept[--d.n];
        }
}

}  // namespace

cudaError_t qvggt_block_acquire(int device, size_t bytes, QvggtBlock *block)
{
    *block = QvggtBlock();
    if (device < 0 || device >= kQvggtMaxDevices) return cudaErrorInvalidDevice;
    const size_t granule = bytes <= kSmall ? kSmallGranule : kGranule;
    bytes = (bytes + granule - 1) / granule * granule;
    const unsigned long long context = current_context();
    DeviceBlocks &d = g_blocks[device];
    if (context) {
        std::lock_guard<std::mutex> lock(g_mutex);
        int best = -1;
        for (int i = 0; i < d.n; ++i) {     // the smallest that is large enough and not wasteful
            const QvggtBlock &k = d.kept[i];
            if (k.context == context && k.bytes >= bytes && k.bytes <= bytes + bytes / 4 + granule && (best < 0 || k.bytes < d.kept[best].bytes)) best = i;
        }
        if (best >= 0) {
            *block = d.kept[best];
            d.kept[best] = d.kept[--d.n];
            return cudaSuccess;
        }
    }
    cudaError_t e = cudaMalloc(&block->p, bytes);
    if (e == cudaErrorMemoryAllocation && context) {
        cudaGetLastError();
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            drop_all(d, context);
        }
        e = cudaMalloc(&block->p, bytes);
    }
    if (e != cudaSuccess) block->p = nullptr;
    block->bytes = bytes;
    block->context = context;
    return e;
}

void qvggt_block_release(int device, const QvggtBlock &block, bool idle)
{
    if (!block.p) return;
    const unsigned long long context = current_context();
    if (block.context && context && block.context != context) return;      // it went with its context
    if (idle && context && block.context && device >= 0 && device < kQvggtMaxDevices) {
        std::lock_guard<std::mutex> lock(g_mutex);
        DeviceBlocks &d = g_blocks[device];
        size_t bytes = block.bytes;
        int at = d.n;
        for (int i = 0; i < d.n; ++i) {
            if (d.kept[i].context == context) bytes += d.kept[i].bytes;
            else if (d.n == kMaxBlocks) at = i;
        }
        if (at < kMaxBlocks && bytes <= kMaxBytes) {
            d.kept[at] = block;
            if (at == d.n) ++d.n;
            return;
        }
    }
    if (cudaFree(block.p) != cudaSuccess) cudaGetLastError();
}
