// Digests of byte ranges (mpt_hash_device, mpt_hash_ranges_noalloc): hash.cu.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mpt {

// Add the digest of [ptrs[i], ptrs[i] + bytes[i]) to out[i] for every i < n (device memory,
// zeroed by the caller beforehand) on stream s: a launch for up to 160 neighbouring ranges of
// one memory kind (device or host).  Allocates nothing.
cudaError_t launch_hash(const void* const* ptrs, const uint64_t* bytes, uint32_t n, unsigned long long* out, int sms,
                        cudaStream_t s);

}  // namespace mpt
