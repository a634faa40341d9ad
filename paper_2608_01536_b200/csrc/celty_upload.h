// Copies of packed images to the GPU (celty_upload.cpp).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime_api.h>

namespace celty {

// Enqueues the copy, and the clearing of another buffer, on st; from has been read when it returns.
cudaError_t upload(void *to, const uint8_t *from, size_t bytes, void *clear, size_t clear_bytes, cudaStream_t st);

// Gives back the memory that upload keeps.
cudaError_t release_staging();

}  // namespace celty
