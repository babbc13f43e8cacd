// Hop two of the host-to-device staged path (Algorithm 2 StageHostCopy: a chunk's second
// hop runs after its first).  Copy-engine nodes fill the chunks of a device stage from the
// host buffer, and a memset node after each raises that chunk's ready flag.  This one
// consumer kernel, launched beside them in the same graph, walks the chunks' 64 KiB tiles,
// waits (bounded) for each chunk's flag, and moves the tile from the stage to its
// destination.
//
// Flags and tile counters are put back to 0 by a memset node at the head of every replay,
// ordered before the copy-engine nodes and before this kernel.  A replay therefore never
// sees a flag raised by an earlier one, even when an earlier replay's wait gave up part way
// (its CTAs return at once, leaving raised flags and partial counts behind).
//
// The stage is written by copy engines while this kernel runs, so its bytes are read with
// coherent loads after an acquire of the flag, never through the read-only (.nc) path.
#include "copy_device.cuh"
#include "kernels.cuh"

namespace mpt {

namespace {

// The whole CTA copies n bytes s -> o: bytes until o is 16-byte aligned, 16-byte words
// (straight when s is then aligned too, else assembled from two aligned source words), and the
// remaining tail bytes.  Reads never leave the 16-byte blocks that hold source bytes.
__device__ __forceinline__ void cta_copy(const uint8_t* s, uint8_t* o, uint64_t n) {
  const uint32_t tid = threadIdx.x, bd = blockDim.x;
  const uint64_t skew = (16u - (uint32_t)(reinterpret_cast<uintptr_t>(o) & 15)) & 15u;
  const uint64_t head = skew < n ? skew : n;
  if (tid < head) o[tid] = s[tid];
  const uint8_t* s1 = s + head;
  uint8_t* o1 = o + head;
  const uint64_t n1 = n - head;
  const uint64_t nv = n1 >> 4;
  uint4* ov = reinterpret_cast<uint4*>(o1);
  const uint32_t m = (uint32_t)(reinterpret_cast<uintptr_t>(s1) & 15);
  uint64_t v = tid;
  if (m == 0) {
    const uint4* sv = reinterpret_cast<const uint4*>(s1);
    for (; v + 3ull * bd < nv; v += 4ull * bd) {
      const uint4 r0 = ld_plain(sv + v), r1 = ld_plain(sv + v + bd), r2 = ld_plain(sv + v + 2 * bd),
                  r3 = ld_plain(sv + v + 3 * bd);
      st_plain(ov + v, r0);
      st_plain(ov + v + bd, r1);
      st_plain(ov + v + 2 * bd, r2);
      st_plain(ov + v + 3 * bd, r3);
    }
    for (; v < nv; v += bd) st_plain(ov + v, ld_plain(sv + v));
  } else {
    const uint4* sw = reinterpret_cast<const uint4*>(s1 - m);
    const uint32_t k = m >> 2, r = (m & 3u) * 8u;
#pragma unroll 2
    for (; v < nv; v += bd) st_plain(ov + v, shift16(ld_plain(sw + v), ld_plain(sw + v + 1), k, r));
  }
  for (uint64_t b = (nv << 4) + tid; b < n1; b += bd) o1[b] = s1[b];
}

}  // namespace

__global__ void __launch_bounds__(kVecThreads) k_stage_consume(StageArgs a) {
  __shared__ int ok;
  constexpr uint64_t kTile = kStageTile;
  const uint32_t total = a.nchunks * a.tiles_per_chunk;
  const uint32_t tid = threadIdx.x;
  for (uint32_t t = blockIdx.x; t < total; t += gridDim.x) {
    const uint32_t k = t / a.tiles_per_chunk;
    const uint32_t lt = t - k * a.tiles_per_chunk;
    if (tid == 0) {
      const uint64_t limit = a.wait_ns ? *(volatile const uint64_t*)a.wait_ns : a.timeout_ns;
      const uint64_t deadline = global_ns() + limit;
      int seen = 0;
      while (true) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.ready + k) : "memory");
        if (v != 0) {
          seen = 1;
          break;
        }
        if (global_ns() > deadline) break;
        __nanosleep(128);
      }
      ok = seen;
      if (!seen) record_timeout(a.status, kSiteStageFlag);
    }
    // thread 0's acquire, then the barrier, orders every thread's stage loads after the flag
    __syncthreads();
    if (!ok) return;
    const StageChunk c = a.chunks[k];
    const uint64_t off = (uint64_t)lt * kTile;
    if (off < c.bytes) {
      const uint64_t n = c.bytes - off < kTile ? c.bytes - off : kTile;
      cta_copy(a.stage + c.stage_off + off, a.dst + c.dst_off + off, n);
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(a.done + k, 1u);  // tiles of chunk k moved (read back by tests and tools)
    }
  }
}

}  // namespace mpt
