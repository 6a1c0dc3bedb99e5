// rd_extent.h -- whether a caller's device buffer is as long as it should be.
#pragma once

#include <cuda.h>
#include <stddef.h>

namespace rdk {

// How [p, p + bytes) lies in the driver's allocations.
enum class Extent {
    kOne,       // inside one
    kSeveral,   // inside several that adjoin (mapped pieces of one buffer, or
                // neighbours), or the driver does not know p
    kShort      // it ends past the last allocation
};

// ``range`` is cuMemGetAddressRange or a stand-in with its contract: base and
// size of the allocation that holds an address, an error where none does.
template <class RangeFn>
Extent extent_of(RangeFn range, CUdeviceptr p, size_t bytes) {
    for (CUdeviceptr at = p;;) {
        CUdeviceptr base = 0;
        size_t size = 0;
        if (range(&base, &size, at) != CUDA_SUCCESS) return at == p ? Extent::kSeveral
                                                                    : Extent::kShort;
        const CUdeviceptr end = base + size;
        if (end <= at) return Extent::kSeveral;
        if (bytes <= end - p) return at == p ? Extent::kOne : Extent::kSeveral;
        at = end;
    }
}

}  // namespace rdk
