// The digest kernel: H = mix64(N) + sum_i mix64(w_i XOR i * gamma) mod 2^64 over the 8-byte
// little-endian words of a range, the last one zero-padded; the sum's order does not matter.
//
// Bound: reading the range once from HBM.  One launch covers many ranges.  Their 16 KiB tiles
// are numbered through, and each CTA takes a run of neighbouring ones, so that it reduces its
// threads' sums and issues an atomic once per range that its run meets, not once per tile.  A
// thread holds four 16-byte vectors of a tile and loads the next tile's before it mixes them.
// With 8-byte loads one at a time and a launch per range, as before, too few bytes were in
// flight (1.7 TB/s on 32 MiB) and every launch cost 4 us: 64 ranges of 4 KiB to 64 MiB (302 MB)
// took 448 us a call, now 92 (the kernel 53 to 54 from a cold L2; its bytes at 6.76 TB/s 45);
// 1 GiB takes 174 us (6.2 TB/s), 206 off a 16-byte boundary.  Measured against it, 1 GiB
// aligned / not: loads not ahead of the mixing 191 / 273 (64 registers), two vectors a tile
// 175 / 217, 64 registers instead of 80 173 / 277 (spills), 8 CTAs per SM 177 / 210.
//
// A call with one range (mpt_hash_device) is bound by its round trip: the last CTA writes the sum
// to host memory and puts the accumulator back to zero, instead of a memset before
// and a copy after the kernel: 16 B to 4 KiB 17.1 -> 12.0 us a call, 64 KiB
// 17.0 -> 13.5, 8 MiB 19.8 -> 14.8.
#include "hash.cuh"

#include <cuda.h>

#include <algorithm>

#include "copy_device.cuh"

namespace mpt {
namespace {

constexpr uint32_t kHashThreads = 256;
constexpr uint32_t kHashUnroll = 4;
constexpr uint32_t kTilePairs = kHashThreads * kHashUnroll;  // a pair: two words, 16 bytes
constexpr uint32_t kHashCtasPerSm = 16;  // of them three resident
// CTAs of a launch over host memory: 32 keep 1 MiB of loads in flight, enough for the host
// link's rate, while a full grid's 15 MiB is a queue of 70 us on the link that everything else
// crossing it waits behind (serving at 50k requests/s beside the digests of 1 % of them: p99
// 700 us with a full grid, 235 with 32 CTAs, 283-345 with the kernel that had one 8-byte load
// in flight per thread).
constexpr uint32_t kHashHostCtas = 32;
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;

// kCap ranges by value: a launch copies its whole argument, so one range alone takes the small
// one; 160 ranges are 3.2 KiB of the 4 that a launch's arguments may take on any path.
template <int kCap>
struct HashArgs {
  uint32_t n;
  uint32_t per_cta, extra;  // tiles of every CTA; the first `extra` take one more
  unsigned long long* out;
  HashResult to;
  const uint8_t* ptr[kCap];
  uint64_t bytes[kCap];
  uint32_t first_tile[kCap + 1];
};
constexpr int kHashRanges = 160;
static_assert(sizeof(HashArgs<kHashRanges>) <= 4096, "kernel argument size");

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The words of pair v, g = gamma times the index of the first.
__device__ __forceinline__ uint64_t mix_pair(const uint4& v, uint64_t g) {
  return mix64((((uint64_t)v.y << 32) | v.x) ^ g) + mix64((((uint64_t)v.w << 32) | v.z) ^ (g + kGamma));
}

// A warp's vectors of one tile: lane l holds vectors 32 u + l of its 128; `end` (lane 31, only
// where the range starts off a 16-byte boundary) the one after the last.
struct TileVecs {
  uint4 x[kHashUnroll], end;
};

template <bool kShift>
__device__ __forceinline__ TileVecs load_tile(const uint4* v, bool last_lane) {
  TileVecs t;
#pragma unroll
  for (uint32_t u = 0; u < kHashUnroll; ++u) t.x[u] = __ldcs(v + 32 * u);
  if (kShift && last_lane) t.end = __ldcs(v + 32 * (kHashUnroll - 1) + 1);
  return t;
}

// Pair u of this lane.  Off a 16-byte boundary a pair lies in two neighbouring vectors, the
// second of them in the next lane, or for lane 31 in lane 0 of the next u.
template <bool kShift>
__device__ __forceinline__ uint64_t mix_tile(const TileVecs& t, uint32_t lane, uint32_t m, uint64_t g, uint32_t npairs) {
  uint64_t acc = 0;
  uint4 rot;
  if (kShift) rot = shfl4(t.x[0], lane + 1);
#pragma unroll
  for (uint32_t u = 0; u < kHashUnroll; ++u) {
    uint4 v = t.x[u];
    if (kShift) {
      uint4 next = t.end;
      if (u + 1 < kHashUnroll) next = shfl4(t.x[u + 1 < kHashUnroll ? u + 1 : u], lane + 1);
      v = shift16(v, lane == 31 ? next : rot, m >> 2, (m & 3u) * 8u);
      rot = next;
    }
    if (32 * u + lane < npairs) acc += mix_pair(v, g + 64ull * u * kGamma);
  }
  return acc;
}

// This thread's part of tiles [t0, t1) of a range: whole pairs, and after the last of them the
// up to 15 bytes that are left.  Only vectors that hold bytes of a whole pair are read.  The
// next tile's loads are issued before a tile is mixed.
template <bool kShift>
__device__ __forceinline__ uint64_t hash_tiles(const uint8_t* p, uint64_t n, uint32_t t0, uint32_t t1) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t m = kShift ? (uint32_t)(reinterpret_cast<uintptr_t>(p) & 15) : 0u;
  const uint64_t np = n >> 4;
  const uint64_t w = (uint64_t)t0 * kTilePairs + (threadIdx.x - lane) * kHashUnroll;  // the warp's first pair
  const uint4* v = reinterpret_cast<const uint4*>(p - m) + w + lane;
  uint64_t g = 2 * (w + lane) * kGamma, acc = 0;
  const uint64_t nfull = np / kTilePairs;
  const uint32_t tf = (uint32_t)(nfull < t1 ? nfull : t1);  // whole tiles end here
  uint32_t t = t0;
  if (t < tf) {
    TileVecs cur = load_tile<kShift>(v, lane == 31);
    while (true) {
      TileVecs next;
      const bool more = t + 1 < tf;
      if (more) next = load_tile<kShift>(v + kTilePairs, lane == 31);
      acc += mix_tile<kShift>(cur, lane, m, g, ~0u);
      v += kTilePairs;
      g += 2ull * kTilePairs * kGamma;
      ++t;
      if (!more) break;
      cur = next;
    }
  }
  if (t == t1) return acc;
  // the range's last tile, not a whole one
  const uint64_t first = (uint64_t)t * kTilePairs + (threadIdx.x - lane) * kHashUnroll;
  const uint32_t left = (uint32_t)(np > first ? (np - first < 32 * kHashUnroll ? np - first : 32 * kHashUnroll) : 0);
  TileVecs last;
#pragma unroll
  for (uint32_t u = 0; u < kHashUnroll; ++u) {
    last.x[u] = make_uint4(0, 0, 0, 0);
    if (32 * u + lane < left + (kShift && left ? 1u : 0u)) last.x[u] = __ldcs(v + 32 * u);
  }
  last.end = make_uint4(0, 0, 0, 0);
  if (kShift && lane == 31 && left == 32 * kHashUnroll) last.end = __ldcs(v + 32 * (kHashUnroll - 1) + 1);
  return acc + mix_tile<kShift>(last, lane, m, g, left);
}

// Words w and w + 1 after the whole pairs of a range, zero-padded (threads 0 and 1).
__device__ __forceinline__ uint64_t hash_tail(const uint8_t* p, uint64_t n) {
  const uint64_t w = 2 * (n >> 4) + threadIdx.x;
  if (threadIdx.x >= 2 || 8 * w >= n) return 0;
  uint64_t v = 0;
  for (uint32_t b = 0; b < 8; ++b)
    if (8 * w + b < n) v |= (uint64_t)p[8 * w + b] << (8 * b);
  return mix64(v ^ (w * kGamma));
}

template <int kCap>
__global__ void __launch_bounds__(kHashThreads, 3) k_hash(const __grid_constant__ HashArgs<kCap> a) {
  __shared__ uint64_t warp_sum[kHashThreads / 32];
  const uint32_t tid = threadIdx.x;
  uint32_t t = blockIdx.x * a.per_cta + min(blockIdx.x, a.extra);
  const uint32_t t1 = t + a.per_cta + (blockIdx.x < a.extra ? 1u : 0u);
  uint32_t lo = 0, hi = a.n - 1;  // the range of tile t: the last one that starts at or before it
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (a.first_tile[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  while (t < t1) {
    const uint32_t first = a.first_tile[lo], end = min(a.first_tile[lo + 1], t1);
    const uint8_t* p = a.ptr[lo];
    const uint64_t n = a.bytes[lo];
    uint64_t acc = t == first ? hash_tail(p, n) + (tid == 0 ? mix64(n) : 0) : 0;
    acc += (reinterpret_cast<uintptr_t>(p) & 15) ? hash_tiles<true>(p, n, t - first, end - first)
                                                 : hash_tiles<false>(p, n, t - first, end - first);
    t = end;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((tid & 31) == 0) warp_sum[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
      uint64_t s = 0;
#pragma unroll
      for (uint32_t i = 0; i < kHashThreads / 32; ++i) s += warp_sum[i];
      if (!a.to.result) {
        atomicAdd(a.out + lo, (unsigned long long)s);
      } else if (gridDim.x == 1) {
        *a.to.result = s;
      } else {  // one range: the last CTA takes the sum and leaves both words zero
        atomicAdd(a.out, (unsigned long long)s);
        __threadfence();
        if (atomicAdd(a.to.count, 1u) == gridDim.x - 1) {
          __threadfence();
          *a.to.result = atomicExch(a.out, 0ull);
          *a.to.count = 0;
        }
      }
    }
    __syncthreads();
    ++lo;
  }
}

template <int kCap>
cudaError_t launch(const void* const* ptrs, const uint64_t* bytes, uint32_t n, unsigned long long* out, uint32_t ctas,
                   cudaStream_t s, const HashResult* to) {
  HashArgs<kCap> a;
  a.n = n;
  a.out = out;
  a.to = to ? *to : HashResult{nullptr, nullptr};
  uint64_t tiles = 0;
  for (uint32_t i = 0; i < n; ++i) {
    a.ptr[i] = static_cast<const uint8_t*>(ptrs[i]);
    a.bytes[i] = bytes[i];
    a.first_tile[i] = (uint32_t)tiles;
    tiles += bytes[i] ? std::max<uint64_t>(1, ((bytes[i] >> 4) + kTilePairs - 1) / kTilePairs) : 0;
  }
  if (tiles >= (1ull << 32)) return cudaErrorInvalidValue;
  for (uint32_t i = n; i <= (uint32_t)kCap; ++i) a.first_tile[i] = (uint32_t)tiles;
  if (tiles == 0) return cudaSuccess;  // empty ranges: the digest of no bytes is 0
  const uint32_t grid = (uint32_t)std::min<uint64_t>(tiles, ctas);
  a.per_cta = (uint32_t)tiles / grid;
  a.extra = (uint32_t)tiles % grid;
  // the launch's own status: the runtime's last error may be an earlier call's of the caller's
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kHashThreads);
  cfg.stream = s;
  return cudaLaunchKernelEx(&cfg, k_hash<kCap>, a);
}

// Memory kind of one range after another; ranges inside the allocation of the last query, the
// usual case, are answered without another one.
class HostSide {
 public:
  bool operator()(const void* p, uint64_t n) {
    const uint64_t a = (uint64_t)(uintptr_t)p;
    if (n == 0) return host_;
    if (a >= lo_ && a + n <= hi_) return host_;
    lo_ = hi_ = 0;
    host_ = true;  // not known to CUDA: pageable host memory
    CUmemorytype type{};
    CUdeviceptr base = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* into[] = {&type, &base, &size};
    static const auto query = entry();
    if (query && query(3, what, into, (CUdeviceptr)a) == CUDA_SUCCESS && type != 0) {
      host_ = type == CU_MEMORYTYPE_HOST;
      if (base) {
        lo_ = base;
        hi_ = base + size;
      }
    }
    return host_;
  }

 private:
  using Query = CUresult (*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
  static Query entry() {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    return reinterpret_cast<Query>(f);
  }
  uint64_t lo_ = 0, hi_ = 0;
  bool host_ = true;
};

}  // namespace

cudaError_t launch_hash(const void* const* ptrs, const uint64_t* bytes, uint32_t n, unsigned long long* out, int sms,
                        cudaStream_t s, const HashResult* to) {
  // a call that reads no more than the host launches keep in flight need not be told apart
  uint64_t total = 0;
  for (uint32_t i = 0; i < n; ++i) total += bytes[i];
  const bool ask = total > (1ull << 20);
  HostSide host_side;
  const auto is_host = [&](uint32_t i) { return ask && host_side(ptrs[i], bytes[i]); };
  for (uint32_t i = 0; i < n;) {
    const bool host = is_host(i);
    uint32_t k = 1;
    while (i + k < n && k < (uint32_t)kHashRanges && is_host(i + k) == host) ++k;
    const uint32_t ctas = host ? kHashHostCtas : kHashCtasPerSm * (uint32_t)sms;
    const cudaError_t e = k <= 4 ? launch<4>(ptrs + i, bytes + i, k, out + i, ctas, s, to)
                                 : launch<kHashRanges>(ptrs + i, bytes + i, k, out + i, ctas, s, to);
    if (e != cudaSuccess) return e;
    i += k;
  }
  return cudaSuccess;
}

}  // namespace mpt
