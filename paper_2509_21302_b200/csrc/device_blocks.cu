// Device memory of the weight handles.
//
// A handle's arrays lie in two blocks (the codes; everything small).  cudaMalloc and cudaFree cost 0.1 - 1 ms each (they map and
// unmap memory and may synchronise the device): a handle of six separate allocations took 0.9 - 8 ms to prepare and 0.6 - 12 ms to
// free, 20 to 100 times the work on the GPU.  A freed block is therefore kept for the next handle of a similar size: at most
// kMaxBytes and kMaxBlocks per device, the rest goes back to the driver at once, and all of it does when an allocation fails.
// A block comes here only after the device was synchronised without an error (qvggt_free_weights), so whoever takes it next may use
// it on any stream.  One mutex serves all threads; nothing is kept by the address or the contents of a caller's buffer.
#include <mutex>

#include "qvggt_internal.cuh"
#include "tensor_map.cuh"

namespace {

constexpr size_t kSmall = 1 << 20;          // up to here sizes are rounded up to kSmallGranule, beyond to the driver's 2 MB
constexpr size_t kSmallGranule = 16 << 10, kGranule = 2 << 20;
constexpr size_t kMaxBytes = 64 << 20;      // kept per device: the codes of one block's four linears, one per byte, take 12 MB
constexpr int kMaxBlocks = 64;

struct Kept {
    void *p;
    size_t bytes;
};
struct DeviceBlocks {
    Kept kept[kMaxBlocks];
    int n = 0;
    size_t bytes = 0;
};

std::mutex g_mutex;
DeviceBlocks g_blocks[kQvggtMaxDevices];

// Frees everything kept for a device.  The caller holds the mutex.
void drop_all(DeviceBlocks &d)
{
    for (int i = 0; i < d.n; ++i) cudaFree(d.kept[i].p);
    d.n = 0;
    d.bytes = 0;
}

}  // namespace

cudaError_t qvggt_block_acquire(int device, size_t bytes, void **block, size_t *block_bytes)
{
    *block = nullptr;
    if (device < 0 || device >= kQvggtMaxDevices) return cudaErrorInvalidDevice;
    const size_t granule = bytes <= kSmall ? kSmallGranule : kGranule;
    bytes = (bytes + granule - 1) / granule * granule;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        DeviceBlocks &d = g_blocks[device];
        int best = -1;
        for (int i = 0; i < d.n; ++i)       // the smallest that is large enough and not wasteful
            if (d.kept[i].bytes >= bytes && d.kept[i].bytes <= bytes + bytes / 4 + granule && (best < 0 || d.kept[i].bytes < d.kept[best].bytes)) best = i;
        if (best >= 0) {
            *block = d.kept[best].p;
            *block_bytes = d.kept[best].bytes;
            d.bytes -= d.kept[best].bytes;
            d.kept[best] = d.kept[--d.n];
            return cudaSuccess;
        }
    }
    *block_bytes = bytes;
    cudaError_t e = cudaMalloc(block, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            drop_all(g_blocks[device]);
        }
        e = cudaMalloc(block, bytes);
    }
    if (e != cudaSuccess) *block = nullptr;
    return e;
}

void qvggt_block_release(int device, void *block, size_t block_bytes)
{
    if (!block) return;
    if (device >= 0 && device < kQvggtMaxDevices) {
        std::lock_guard<std::mutex> lock(g_mutex);
        DeviceBlocks &d = g_blocks[device];
        if (d.n < kMaxBlocks && d.bytes + block_bytes <= kMaxBytes) {
            d.kept[d.n++] = Kept{block, block_bytes};
            d.bytes += block_bytes;
            return;
        }
    }
    cudaFree(block);
}
