// Which of a caller's field arrays the kernels may read or write where they lie; the others go through a
// copy.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>

namespace cmlbm {

typedef CUresult (*PointerGetAttributes)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);

// The driver's query, looked up through the runtime (no link against libcuda); null if it cannot be had.
inline PointerGetAttributes pointer_get_attributes() {
    static std::atomic<void*> known{nullptr};
    void* p = known.load(std::memory_order_relaxed);
    if (!p) {
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        cudaGetLastError();
        known.store(p, std::memory_order_relaxed);
    }
    return reinterpret_cast<PointerGetAttributes>(p);
}

inline bool overlap(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

// `bytes` bytes of floats at p are whole in one allocation of device memory of device dev.  Host, managed
// and other devices' memory and floats off their 4-byte alignment are copied.  An array that ends before its
// allocation does is copied too: the copy checks its range and refuses it, a kernel would not.
inline bool in_place(const void* p, size_t bytes, int dev) {
    if (reinterpret_cast<uintptr_t>(p) & 3) return false;
    const PointerGetAttributes get = pointer_get_attributes();
    if (!get) return false;
    unsigned int type = 0, managed = 0;
    int device = -1;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* into[5] = {&type, &managed, &device, &start, &size};
    const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p);
    if (get(5, what, into, at) != CUDA_SUCCESS) return false;
    return type == CU_MEMORYTYPE_DEVICE && !managed && device == dev && at >= start && at - start <= size && size - (at - start) >= bytes;
}

// there[k] = outs[k] for the outputs of `bytes` bytes each that the kernels may write where they lie: clear of
// the population store they read, and of the other outputs (which are then copied in their order), else null.
inline void direct_outputs(float* const (&outs)[4], size_t bytes, int dev, const void* store, size_t store_bytes, float* (&there)[4]) {
    for (int k = 0; k < 4; ++k) {
        there[k] = nullptr;
        bool clear = outs[k] && in_place(outs[k], bytes, dev) && !overlap(outs[k], bytes, store, store_bytes);
        for (int j = 0; clear && j < 4; ++j) clear = j == k || !outs[j] || !overlap(outs[k], bytes, outs[j], bytes);
        if (clear) there[k] = outs[k];
    }
}

}  // namespace cmlbm
