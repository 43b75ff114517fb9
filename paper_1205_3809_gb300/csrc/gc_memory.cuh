// Device memory shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

namespace gc {

// cudaMalloc; when that is refused, once more after the memory kept from
// destroyed batch plans on this device has been given back.
cudaError_t malloc_device(void** p, size_t bytes);

}  // namespace gc
