// Digests of byte ranges (mpt_hash_device, mpt_hash_ranges_noalloc): hash.cu.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mpt {

// Where the digest of a single range goes when the kernel delivers it itself: `result` is the
// device address of a host word, `count` a device word.  The accumulator and the
// count are zero between launches (the kernel leaves them so).
struct HashResult {
  unsigned long long* result;
  uint32_t* count;
};

// Add the digest of [ptrs[i], ptrs[i] + bytes[i]) to out[i] for every i < n (device memory,
// zeroed by the caller beforehand) on stream s: a launch for up to 160 neighbouring ranges of
// one memory kind (device or host).  With `to` (n is 1 and bytes[0] above 0), the digest is
// written to to->result instead and out[0] is zero again afterwards.  Allocates nothing.
cudaError_t launch_hash(const void* const* ptrs, const uint64_t* bytes, uint32_t n, unsigned long long* out, int sms,
                        cudaStream_t s, const HashResult* to = nullptr);

}  // namespace mpt
