// The fixed scratch of headcast_dense_attend_noalloc.
#pragma once
#include <cuda_runtime.h>

namespace hc {

constexpr size_t NOALLOC_SCRATCH_BYTES = size_t(38) << 20;

// Its address on the current device.
cudaError_t noalloc_scratch_address(void** ptr);

}  // namespace hc
