// Device memory of handles and the encoder on the GPU (us_load.cu).
#pragma once
#include <cuda_runtime.h>

#include "us_host.h"

namespace us {

// Device memory from the library's pool on `device` (the current device): stream ordered on pool_stream(device).
// pool_free expects that no work using p is in flight on any other stream.
cudaError_t pool_alloc(int device, void** p, size_t bytes);
void pool_free(int device, void* p);
cudaStream_t pool_stream(int device);   // after the first pool_alloc

struct DeviceMatrix {
    uint8_t* blob = nullptr;
    uint32_t* item_off = nullptr;
    int32_t* row_order = nullptr;
};

// The tiles of a matrix whose layout encode_layout has laid down, built on the GPU: fills what encode_host would have
// filled in but the blob itself (h->blob stays empty). Enqueued on pool_stream(device).
us_status encode_device(const int8_t* W, int device, uint32_t flags, HostMatrix* h, DeviceMatrix* out);

}  // namespace us
