// Lossless entropy stage over the records of a compressed state (order-0
// byte-wise rANS; the layout and the coder are described in entropy.cu).
#pragma once
#include <cuda_runtime.h>

namespace wcs {
// Host memory for the coded state once its size is known (null: none wanted).
typedef void* (*entropy_sink)(void* user, long long nbytes);
// Codes the npatch records at arena (table tab: offset << 24 | bytes; all
// below arena + live), decodes them again on the device and sets *mismatches
// to the number of bytes that did not come back; if there are none, copies the
// coded state to the memory that sink gives for it.  Synchronises the stream.
cudaError_t entropy_code_state(const unsigned char* arena, const unsigned long long* tab, int npatch,
                               unsigned long long live, cudaStream_t stream, entropy_sink sink, void* user,
                               long long* nbytes, unsigned long long* mismatches);
}  // namespace wcs
