// Device-side copy helpers shared by the copy kernels: 128-bit loads and stores, and the
// assembly of a destination-aligned 16-byte word from two aligned source words when source
// and destination differ modulo 16 (so no path ever falls back to byte-by-byte copies).
#pragma once
#include <cstdint>

namespace mpt {

// Programmatic dependent launch.  A copy kernel launched with programmatic stream
// serialization may start while the kernel before it on the stream is finishing; it waits
// here, before touching memory, until that kernel has completed and its writes are visible,
// then lets the next such kernel begin its own launch.  Launched without the attribute
// (graph nodes, plain launches) both instructions are no-ops.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Global timer in nanoseconds: the clock every bounded device-side wait measures against.
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// A wait ran out: record (site << 8) | MPT_ETIMEDOUT in the context's status word, unless
// an earlier failure is already recorded there.
__device__ __forceinline__ void record_timeout(uint32_t* status, uint32_t site) {
  constexpr uint32_t kTimedOut = 4;  // MPT_ETIMEDOUT
  if (status) atomicCAS(status, 0u, (site << 8) | kTimedOut);
}

// A kernel refused its arguments: record (site << 8) | MPT_EINVAL the same way.
__device__ __forceinline__ void record_invalid(uint32_t* status, uint32_t site) {
  constexpr uint32_t kInvalid = 1;  // MPT_EINVAL
  if (status) atomicCAS(status, 0u, (site << 8) | kInvalid);
}

__device__ __forceinline__ uint4 ld_plain(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Coherent as ld_plain, for bytes that are read once: not kept in L1.
__device__ __forceinline__ uint4 ld_once(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// 32 bytes in one instruction, for both ends 32-byte aligned.  Coherent, and not through the
// read-only path on the device either: a kernel launched with programmatic stream serialization
// starts while the one ahead may still be writing its source.
struct Wide {
  uint32_t w[8];
};

__device__ __forceinline__ Wide ld_wide(const void* p) {
  Wide v;
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]),
                 "=r"(v.w[7])
               : "l"(p));
  return v;
}

__device__ __forceinline__ void st_wide(void* p, const Wide& v) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]),
               "r"(v.w[3]), "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7])
               : "memory");
}

__device__ __forceinline__ void st_plain(uint4* p, const uint4& v) {
  asm volatile("st.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

// Index of the range that launch tile t belongs to (ranges are few: a linear scan).
template <typename Args>
__device__ __forceinline__ int find_range(const Args& a, uint32_t t) {
  int r = 0;
  while (r + 1 < (int)a.nranges && t >= a.tile_start[r + 1]) ++r;
  return r;
}

// Head (bytes before the destination-aligned body) and tail (bytes after it) of a range;
// threads 0..31 copy the head, threads 32..63 the tail (of at most 31 bytes each).
template <typename Range>
__device__ __forceinline__ void copy_edges(const uint8_t* s, uint8_t* o, const Range& d, uint64_t body_bytes) {
  const uint32_t tid = threadIdx.x;
  if (tid < d.head) o[tid] = s[tid];
  const uint64_t tail_start = d.head + body_bytes;
  const uint32_t tail = (uint32_t)(d.bytes - tail_start);
  if (tid >= 32 && tid < 32 + tail) o[tail_start + (tid - 32)] = s[tail_start + (tid - 32)];
}

__device__ __forceinline__ uint4 shfl4(const uint4& v, uint32_t from) {
  return make_uint4(__shfl_sync(0xffffffffu, v.x, from), __shfl_sync(0xffffffffu, v.y, from),
                    __shfl_sync(0xffffffffu, v.z, from), __shfl_sync(0xffffffffu, v.w, from));
}

// Bytes [4k + r/8, 4k + r/8 + 16) of the 32-byte little-endian concatenation w0 | w1
// (k in 0..3 words, r in {0, 8, 16, 24} bits): each output word is a funnel shift of two
// neighbouring input words.
__device__ __forceinline__ uint4 shift16(const uint4& w0, const uint4& w1, uint32_t k, uint32_t r) {
  const uint32_t a[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
  uint4 o;
  switch (k) {
    case 0:
      o = make_uint4(__funnelshift_r(a[0], a[1], r), __funnelshift_r(a[1], a[2], r), __funnelshift_r(a[2], a[3], r),
                     __funnelshift_r(a[3], a[4], r));
      break;
    case 1:
      o = make_uint4(__funnelshift_r(a[1], a[2], r), __funnelshift_r(a[2], a[3], r), __funnelshift_r(a[3], a[4], r),
                     __funnelshift_r(a[4], a[5], r));
      break;
    case 2:
      o = make_uint4(__funnelshift_r(a[2], a[3], r), __funnelshift_r(a[3], a[4], r), __funnelshift_r(a[4], a[5], r),
                     __funnelshift_r(a[5], a[6], r));
      break;
    default:
      o = make_uint4(__funnelshift_r(a[3], a[4], r), __funnelshift_r(a[4], a[5], r), __funnelshift_r(a[5], a[6], r),
                     __funnelshift_r(a[6], a[7], r));
      break;
  }
  return o;
}

}  // namespace mpt
