// Scratch of the synchronous entry points: a few fixed device slots instead of
// an allocation per call.  A stream-ordered allocation is mapped and unmapped
// again around every call that waits for its stream (about 190 us per call on
// GB300, most of a small call); a slot costs an atomic on the host.
//
// A slot is held from acquire to release by one call, which has waited for its
// stream in between, so calls on any streams and host threads have slots of
// their own; when all are taken, or the call needs more than a slot, it
// allocates as before.  A slot holds the 2-opt's neighbour lists for tours of up
// to 4000 viewpoints.  Every GPU that loads the library holds the slots (8 MiB)
// until the process exits.
#include <atomic>

#include "common.cuh"

namespace dpso {
namespace {

constexpr int kSlots = 8, kMaxDevices = 32;
static __device__ __align__(256) unsigned char g_slots[kSlots][kScratchSlotBytes];
std::atomic<unsigned> g_taken[kMaxDevices];  // bit per slot, by device

}  // namespace

cudaError_t Scratch::acquire_slot(size_t bytes, cudaStream_t st) {
    stream = st;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || bytes > kScratchSlotBytes || dev >= kMaxDevices) return e;
    for (int k = 0; k < kSlots; ++k) {
        if (g_taken[dev].fetch_or(1u << k, std::memory_order_acquire) >> k & 1) continue;
        void* base = nullptr;
        e = cudaGetSymbolAddress(&base, g_slots);
        if (e != cudaSuccess) {
            g_taken[dev].fetch_and(~(1u << k), std::memory_order_release);
            return e;
        }
        device = dev;
        slot = k;
        p = static_cast<unsigned char*>(base) + k * kScratchSlotBytes;
        break;
    }
    return cudaSuccess;
}

cudaError_t Scratch::acquire(size_t bytes, cudaStream_t st) {
    cudaError_t e = acquire_slot(bytes, st);
    if (e != cudaSuccess || p) return e;
    e = cudaMallocAsync(&p, bytes, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    return cudaSuccess;
}

void Scratch::release() {
    if (!p) return;
    if (slot >= 0) g_taken[device].fetch_and(~(1u << slot), std::memory_order_release);
    else cudaFreeAsync(p, stream);
    p = nullptr;
    slot = -1;
}

}  // namespace dpso
