// Whether a device allocation is long enough for what a kernel is about to
// read through a caller's pointer. A copy of a range that leaves its allocation
// is refused by the driver; a kernel (or a library transform) that reads it in
// place would fault, so the range is looked up first (about 1 us).
#pragma once

#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace spg {

enum class Extent { holds, too_short, unknown };

template <class F>
F driver_entry(const char *name, unsigned version)
{
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion(name, &p, version, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return reinterpret_cast<F>(p);
}

// `bytes` from p on, for memory of the current device; unknown for other
// memory. Memory mapped in pieces (virtual memory management) may go on behind
// the piece that p lies in: unknown.
inline Extent device_extent(const void *p, size_t bytes)
{
    static const auto query = driver_entry<PFN_cuPointerGetAttributes_v7000>("cuPointerGetAttributes", 7000);
    static const auto retain = driver_entry<PFN_cuMemRetainAllocationHandle_v11000>("cuMemRetainAllocationHandle", 11000);
    static const auto release = driver_entry<PFN_cuMemRelease_v10020>("cuMemRelease", 10020);
    if (!query || !retain || !release) return Extent::unknown;
    unsigned type = 0, managed = 0;
    int ordinal = -1, dev = -1;
    CUdeviceptr base = 0;
    size_t size = 0;
    const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p);
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                  CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *to[] = {&type, &managed, &ordinal, &base, &size};
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return Extent::unknown;
    }
    if (query(5, what, to, at) != CUDA_SUCCESS || type != CU_MEMORYTYPE_DEVICE || managed || ordinal != dev || !base ||
        at < base)
        return Extent::unknown;
    const size_t before = (size_t)(at - base);
    if (before <= size && bytes <= size - before) return Extent::holds;
    CUmemGenericAllocationHandle h;
    if (retain(&h, const_cast<void *>(p)) == CUDA_SUCCESS) {
        release(h);
        return Extent::unknown;
    }
    return Extent::too_short;
}

}  // namespace spg
