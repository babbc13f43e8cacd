// Data-moving kernels of the transfer paths, written for sm_103a.
//
//  k_sm_copy_vec   SM copy kernel: each CTA walks tiles of the ranges it is given, every thread
//                  keeping kU 32-byte vectors in flight.  The device-to-device path the SMs add
//                  next to the copy engines (Sec. 4.3's horizontal split over paths).
//  k_zc_copy       zero-copy kernel: the same loop without the first tile's prefetch, used on
//                  mapped page-locked host memory for host<->device transfers.
//
// The bulk-copy variant of the SM copy kernel (cp.async.bulk through shared memory) is in
// copy_bulk.cu.
#include "kernels.cuh"
#include "bulk_config.h"
#include "copy_device.cuh"

#include <algorithm>

namespace mpt {

namespace {

// 32-byte units of a range's body before its first one in their 128-byte line; tiles begin on
// lines, tile 0 that much before the body.
__host__ __device__ __forceinline__ uint32_t lead_units(uintptr_t src, uintptr_t dst, bool src_lines) {
  return (uint32_t)((src_lines ? src : dst) >> 5) & 3u;
}

// Before waiting on the kernel ahead (programmatic dependent launch), one thread asks L2 for
// the source bytes of the CTA's first tile.  This is only a hint to L2, the GPU's point of
// coherence: if the kernel ahead writes those bytes before the wait returns, its stores
// update the lines in L2, and the loads after the wait, which miss L1, read the new bytes.
// No data reaches registers before the wait.  The short messages of a stream of copies then
// find their source in L2 instead of HBM once the kernel ahead completes.
template <uint32_t kTile, typename Args>
__device__ __forceinline__ void prefetch_first_tile(const Args& a) {
  if (threadIdx.x != 0 || blockIdx.x >= a.ntiles) return;
  const int r = find_range(a, blockIdx.x);
  const RangeDesc& d = a.r[r];
  const uint64_t lt = blockIdx.x - a.tile_start[r];
  // bytes of the range this tile reads, at most: from the range start (tile 0 also copies the
  // head) or a line and a unit before the tile's place, to a unit past it
  const uint64_t lo = lt == 0 ? 0 : d.head + lt * kTile - 160;
  const uint64_t end = d.head + (lt + 1) * kTile + 32;
  const uint64_t hi = end < d.bytes ? end : d.bytes;
  if (hi <= lo) return;
  // whole 16-byte blocks around [lo, hi): each holds a source byte, so it is mapped memory
  const uintptr_t base = reinterpret_cast<uintptr_t>(a.src + d.src_off);
  const uintptr_t p0 = (base + lo) & ~(uintptr_t)15, p1 = (base + hi + 15) & ~(uintptr_t)15;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p0), "r"((uint32_t)(p1 - p0)) : "memory");
}

// The loops below move units [lo, hi) of one tile, s and o the addresses of its unit 0: all of
// them but in a range's first and last tile.  o is 32-byte aligned.

// Source and destination agree modulo 32: kU units a thread.
template <int kU>
__device__ __forceinline__ void copy_units(const uint8_t* s, uint8_t* o, int lo, int hi) {
  const int i0 = (int)threadIdx.x;
  s += 32 * i0;
  o += 32 * i0;
  Wide x[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u)
    if (i0 + kVecThreads * u >= lo && i0 + kVecThreads * u < hi) x[u] = ld_wide(s + kVecTile * u);
#pragma unroll
  for (int u = 0; u < kU; ++u)
    if (i0 + kVecThreads * u >= lo && i0 + kVecThreads * u < hi) st_wide(o + kVecTile * u, x[u]);
}

// They differ, s - m (0 < m < 32) being aligned: a destination unit is bytes [m, m + 32) of two
// neighbouring source units, the second of them in the next lane, or for lane 31 in lane 0 of the
// next u (which loads the one after the warp's last for it).  Each warp moves a run of 32 kU.
// kK words and, with kBits, r more bits of shift.
template <int kK, bool kBits, int kU>
__device__ __forceinline__ void store_shifted(const Wide (&x)[kU + 1], uint8_t* o, uint32_t r, uint32_t lane, int i0,
                                              int lo, int hi) {
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = x[u].w[i];
#pragma unroll
    for (int i = 0; i < kK + (kBits ? 1 : 0); ++i)
      w[8 + i] = __shfl_sync(0xffffffffu, lane == 0 ? x[u + 1].w[i] : x[u].w[i], lane + 1);
    Wide y;
#pragma unroll
    for (int i = 0; i < 8; ++i) y.w[i] = kBits ? __funnelshift_r(w[kK + i], w[kBits ? kK + i + 1 : 0], r) : w[kK + i];
    if (i0 + 32 * u >= lo && i0 + 32 * u < hi) st_wide(o + 1024 * u, y);
  }
}

template <int kU>
__device__ __forceinline__ void copy_shifted(const uint8_t* s, uint8_t* o, uint32_t m, int lo, int hi) {
  const uint32_t lane = threadIdx.x & 31u;
  const int i0 = (int)((threadIdx.x - lane) * kU + lane);
  s = s + 32 * i0 - m;
  o += 32 * i0;
  const int last = lo < hi ? hi : lo - 1;  // unit hi holds the last bytes of destination unit hi - 1
  Wide x[kU + 1];
#pragma unroll
  for (int u = 0; u <= kU; ++u)
    if (i0 + 32 * u >= lo && i0 + 32 * u <= last && (u < kU || lane == 0)) x[u] = ld_wide(s + 1024 * u);
  const uint32_t r = (m & 3u) * 8u;
  switch (m) {
    case 4: store_shifted<1, false, kU>(x, o, 0, lane, i0, lo, hi); return;
    case 8: store_shifted<2, false, kU>(x, o, 0, lane, i0, lo, hi); return;
    case 16: store_shifted<4, false, kU>(x, o, 0, lane, i0, lo, hi); return;
  }
  switch (m >> 2) {
    case 0: store_shifted<0, true, kU>(x, o, r, lane, i0, lo, hi); break;
    case 1: store_shifted<1, true, kU>(x, o, r, lane, i0, lo, hi); break;
    case 2: store_shifted<2, true, kU>(x, o, r, lane, i0, lo, hi); break;
    case 3: store_shifted<3, true, kU>(x, o, r, lane, i0, lo, hi); break;
    case 4: store_shifted<4, true, kU>(x, o, r, lane, i0, lo, hi); break;
    case 5: store_shifted<5, true, kU>(x, o, r, lane, i0, lo, hi); break;
    case 6: store_shifted<6, true, kU>(x, o, r, lane, i0, lo, hi); break;
    default: store_shifted<7, true, kU>(x, o, r, lane, i0, lo, hi); break;
  }
}

template <bool kAny, int kU, typename Args>
__device__ __forceinline__ void copy_tiles(const Args& a) {
  constexpr int64_t kUnits = (int64_t)kVecThreads * kU;
  for (uint32_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
    const int r = find_range(a, t);
    const uint32_t lt = t - a.tile_start[r];
    const RangeDesc& d = a.r[r];
    const uint8_t* s = a.src + d.src_off;
    uint8_t* o = a.dst + d.dst_off;
    const int64_t units = (int64_t)((d.bytes - d.head) >> 5);
    if (lt == 0) copy_edges(s, o, d, (uint64_t)units << 5);
    s += d.head;
    o += d.head;
    const int64_t u0 = lt * kUnits - lead_units(reinterpret_cast<uintptr_t>(s), reinterpret_cast<uintptr_t>(o),
                                                a.src_lines != 0);  // the tile's first unit
    const int lo = u0 < 0 ? (int)-u0 : 0, hi = units - u0 < kUnits ? (int)(units - u0) : (int)kUnits;
    s += 32 * u0;
    o += 32 * u0;
    if (kAny && d.shift) copy_shifted<kU>(s, o, d.shift, lo, hi);
    else copy_units<kU>(s, o, lo, hi);
  }
}

}  // namespace

// Bound by HBM from some 30 MiB on, below that by what a launch costs beside its bytes: the first
// loads' latency and the last wave.  32-byte accesses move more per request than the 16-byte ones
// of before (us per message, back to back, 16-byte against 32-byte: 24 MiB 9.0 / 8.5, 64 MiB 21.2 /
// 20.4, 1 GiB 307 / 303; as the tuner's grids have it 6 MiB 3.8 / 2.8, 12 MiB 4.7 / 4.2).  Where
// source and destination differ modulo 32, a shuffle hands each unit on instead of a second load,
// and the kernel keeps two CTAs per SM instead of one: 3 bytes apart, 12 MiB 7.2 / 5.0, 64 MiB
// 25.4 / 20.2, 1 GiB 362 / 303.  The arguments of a single range are 88 bytes instead of 650.
template <int kU, bool kAny, int kN>
__global__ void __launch_bounds__(kVecThreads, kAny ? 4 - kU : kU == 4 ? 2 : 4) k_sm_copy_vec(const __grid_constant__ CopyArgsT<kN> a) {
  prefetch_first_tile<kVecTile * kU>(a);
  pdl_enter();
  copy_tiles<kAny, kU>(a);
}

template <bool kAny, int kN>
__global__ void __launch_bounds__(kVecThreads) k_zc_copy(const __grid_constant__ CopyArgsT<kN> a) {
  pdl_enter();
  copy_tiles<kAny, 4>(a);
}

// ---- host side -------------------------------------------------------------------------

namespace {

template <int kU, bool kAny>
void* vec_fn(bool one) {
  return one ? reinterpret_cast<void*>(&k_sm_copy_vec<kU, kAny, 1>)
             : reinterpret_cast<void*>(&k_sm_copy_vec<kU, kAny, kInlineRanges>);
}

template <bool kAny>
void* zc_fn(bool one) {
  return one ? reinterpret_cast<void*>(&k_zc_copy<kAny, 1>) : reinterpret_cast<void*>(&k_zc_copy<kAny, kInlineRanges>);
}

}  // namespace

void* vec_copy_fn(const CopyArgs& a, bool zero_copy) {
  const bool one = a.nranges == 1, any = a.any_shift != 0;
  if (zero_copy) return any ? zc_fn<true>(one) : zc_fn<false>(one);
  switch (a.piece / kVecTile) {
    case 1: return any ? vec_fn<1, true>(one) : vec_fn<1, false>(one);
    case 2: return any ? vec_fn<2, true>(one) : vec_fn<2, false>(one);
    default: return vec_fn<4, false>(one);
  }
}

int make_copy_args(CopyArgs& a, const void* src, void* dst, const RangeDesc* ranges, int n, int variant,
                   uint32_t* status, uint32_t bulk_cfg, uint32_t ctas, uint32_t sms, bool src_lines) {
  a.src = static_cast<const uint8_t*>(src);
  a.dst = static_cast<uint8_t*>(dst);
  a.status = status;
  a.bulk_cfg = variant == 1 ? bulk_cfg : 0;
  a.src_lines = variant == 2 && src_lines ? 1 : 0;
  a.nranges = 0;
  a.any_shift = 0;
  uint64_t total = 0;
  for (int i = 0; i < n && i < kInlineRanges; ++i) {
    const uint64_t apart = reinterpret_cast<uintptr_t>(src) + ranges[i].src_off - reinterpret_cast<uintptr_t>(dst) - ranges[i].dst_off;
    total += ranges[i].bytes;
    if (ranges[i].bytes && (apart & 31)) a.any_shift = 1;
  }
  // Tiles of the vector kernel.  Up to one wave of the grid the smallest tile that fits it, as it
  // spreads the message over most SMs; past one wave of the largest, smaller ones fill the last
  // wave better until there are many.  Measured on GB300 at 16 / 32 / 64 KiB (us per message, back
  // to back): 4 MiB 2.5 / 2.7 / 2.7, 8 MiB 3.2 / 3.7 / 3.1-4.0, 12 MiB 4.8 / 4.5 / 4.2, 16 MiB
  // 6.1 / 5.4 / 5.2, 20 MiB 7.0 / 7.1 / 7.6, 24 MiB 8.3 / 8.0 / 8.6, 32 MiB 10.7 / 10.6 / 10.5,
  // 1 GiB 307 / 307 / 304.  Off 32-byte boundaries 64 KiB tiles would leave one CTA per SM.
  const auto fits = [&](uint64_t tile, uint32_t per_sm) { return total <= tile * std::min(ctas, per_sm * sms); };
  if (variant == 1) a.piece = bulk_config(bulk_cfg).stage_bytes;
  else if (variant == 2) a.piece = 4 * kVecTile;
  else if (variant == 3 || fits(kVecTile, 4)) a.piece = kVecTile;
  else if (a.any_shift) a.piece = 2 * kVecTile;
  else if (fits(4 * kVecTile, 2)) a.piece = 4 * kVecTile;
  else if (fits(2 * kVecTile, 7)) a.piece = 2 * kVecTile;
  else a.piece = 4 * kVecTile;
  uint64_t tiles = 0;
  a.tile_start[0] = 0;
  for (int i = 0; i < n && i < kInlineRanges; ++i) {
    RangeDesc d = ranges[i];
    if (d.bytes == 0) continue;
    const uintptr_t s = reinterpret_cast<uintptr_t>(src) + d.src_off;
    const uintptr_t o = reinterpret_cast<uintptr_t>(dst) + d.dst_off;
    const uint32_t unit = variant == 1 ? 16 : 32;
    d.head = (uint32_t)std::min<uint64_t>(d.bytes, (unit - (o & (unit - 1))) & (unit - 1));
    d.shift = (uint32_t)((s + d.head) - (o + d.head)) & (unit - 1);
    if (variant == 1 && d.shift) return kArgsNeedVec;
    const uint64_t body = (d.bytes - d.head) / unit * unit;
    const uint64_t lead = variant == 1 ? 0 : 32 * lead_units(s + d.head, o + d.head, a.src_lines != 0);
    uint64_t t = body ? (body + lead + a.piece - 1) / a.piece : 0;
    if (t == 0) t = 1;  // a range too short for a body still needs its edge bytes copied
    a.r[a.nranges] = d;
    tiles += t;
    a.tile_start[a.nranges + 1] = (uint32_t)tiles;
    a.nranges++;
  }
  for (uint32_t i = a.nranges + 1; i <= (uint32_t)kInlineRanges; ++i) a.tile_start[i] = (uint32_t)tiles;
  a.ntiles = (uint32_t)tiles;
  return tiles < (1ull << 31) ? kArgsOk : kArgsTooLarge;
}

}  // namespace mpt
