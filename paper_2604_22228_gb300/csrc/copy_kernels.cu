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
#include <type_traits>

namespace mpt {

namespace {

// Bytes of a range's 128-byte line before its body, in units of `unit`; tiles begin on lines, tile 0
// that much before the body.
__host__ __device__ __forceinline__ uint32_t lead_bytes(uintptr_t src, uintptr_t dst, bool src_lines, uint32_t unit) {
  return (uint32_t)(src_lines ? src : dst) & (128u - unit);
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
// them but in a range's first and last tile.  o is aligned to a unit.

__device__ __forceinline__ void load(Wide& v, const uint8_t* p) { v = ld_wide(p); }
__device__ __forceinline__ void load(uint4& v, const uint8_t* p) { v = ld_once(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ void store(uint8_t* p, const Wide& v) { st_wide(p, v); }
__device__ __forceinline__ void store(uint8_t* p, const uint4& v) { st_plain(reinterpret_cast<uint4*>(p), v); }

// Source and destination agree modulo a unit (Wide: 32 bytes, uint4: a word of 16): kU a thread.
template <typename Unit, int kU>
__device__ __forceinline__ void copy_units(const uint8_t* s, uint8_t* o, int lo, int hi) {
  constexpr int kUnit = sizeof(Unit);
  const int i0 = (int)threadIdx.x;
  s += kUnit * i0;
  o += kUnit * i0;
  Unit x[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u)
    if (i0 + kVecThreads * u >= lo && i0 + kVecThreads * u < hi) load(x[u], s + kVecThreads * kUnit * u);
#pragma unroll
  for (int u = 0; u < kU; ++u)
    if (i0 + kVecThreads * u >= lo && i0 + kVecThreads * u < hi) store(o + kVecThreads * kUnit * u, x[u]);
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

// kB: bytes of a tile per thread.
template <uint32_t kMove, int kB, typename Args>
__device__ __forceinline__ void copy_tiles(const Args& a) {
  constexpr int kUnit = kMove == kMoveWords ? 16 : 32;
  constexpr int64_t kUnits = (int64_t)kVecThreads * kB / kUnit;
  for (uint32_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
    const int r = find_range(a, t);
    const uint32_t lt = t - a.tile_start[r];
    const RangeDesc& d = a.r[r];
    const uint8_t* s = a.src + d.src_off;
    uint8_t* o = a.dst + d.dst_off;
    const int64_t units = (int64_t)((d.bytes - d.head) / kUnit);
    if (lt == 0) copy_edges(s, o, d, (uint64_t)units * kUnit);
    s += d.head;
    o += d.head;
    const uint32_t lead = lead_bytes(reinterpret_cast<uintptr_t>(s), reinterpret_cast<uintptr_t>(o), a.src_lines != 0, kUnit);
    const int64_t u0 = lt * kUnits - lead / kUnit;  // the tile's first unit
    const int lo = u0 < 0 ? (int)-u0 : 0, hi = units - u0 < kUnits ? (int)(units - u0) : (int)kUnits;
    s += kUnit * u0;
    o += kUnit * u0;
    if constexpr (kMove == kMoveWords) {
      copy_units<uint4, kB / 16>(s, o, lo, hi);
    } else {
      if (kMove == kMoveShifted && d.shift) copy_shifted<kB / 32>(s, o, d.shift, lo, hi);
      else copy_units<Wide, kB / 32>(s, o, lo, hi);
    }
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
template <int kB, uint32_t kMove, int kN>
__global__ void __launch_bounds__(kVecThreads, kMove == kMoveShifted ? (kB == 128 ? 1 : 4 - kB / 32) : kB == 128 ? 2 : 4)
    k_sm_copy_vec(const __grid_constant__ CopyArgsT<kN> a) {
  prefetch_first_tile<kVecThreads * kB>(a);
  pdl_enter();
  copy_tiles<kMove, kB>(a);
}

template <uint32_t kMove, int kN>
__global__ void __launch_bounds__(kVecThreads) k_zc_copy(const __grid_constant__ CopyArgsT<kN> a) {
  pdl_enter();
  copy_tiles<kMove, 128>(a);
}

// ---- host side -------------------------------------------------------------------------

namespace {

template <int kB, uint32_t kMove>
void* vec_fn(bool one) {
  return one ? reinterpret_cast<void*>(&k_sm_copy_vec<kB, kMove, 1>)
             : reinterpret_cast<void*>(&k_sm_copy_vec<kB, kMove, kInlineRanges>);
}

template <uint32_t kMove>
void* zc_fn(bool one) {
  return one ? reinterpret_cast<void*>(&k_zc_copy<kMove, 1>) : reinterpret_cast<void*>(&k_zc_copy<kMove, kInlineRanges>);
}

}  // namespace

void* vec_copy_fn(const CopyArgs& a, bool zero_copy) {
  const bool one = a.nranges == 1;
  if (zero_copy)
    return a.move == kMoveUnits ? zc_fn<kMoveUnits>(one) : a.move == kMoveWords ? zc_fn<kMoveWords>(one) : zc_fn<kMoveShifted>(one);
  const uint32_t per_thread = a.piece / kVecThreads;
  if (per_thread == 16) return vec_fn<16, kMoveWords>(one);
  const auto fn = [&](auto move) {
    constexpr uint32_t kMove = decltype(move)::value;
    return per_thread == 32 ? vec_fn<32, kMove>(one) : per_thread == 64 ? vec_fn<64, kMove>(one) : vec_fn<128, kMove>(one);
  };
  if (a.move == kMoveUnits) return fn(std::integral_constant<uint32_t, kMoveUnits>());
  if (a.move == kMoveWords) return fn(std::integral_constant<uint32_t, kMoveWords>());
  return fn(std::integral_constant<uint32_t, kMoveShifted>());
}

int make_copy_args(CopyArgs& a, const void* src, void* dst, const RangeDesc* ranges, int n, int variant,
                   uint32_t* status, uint32_t bulk_cfg, uint32_t ctas, uint32_t sms, bool src_lines) {
  a.src = static_cast<const uint8_t*>(src);
  a.dst = static_cast<uint8_t*>(dst);
  a.status = status;
  a.bulk_cfg = variant == 1 ? bulk_cfg : 0;
  a.src_lines = variant == 2 && src_lines ? 1 : 0;
  a.nranges = 0;
  uint64_t total = 0;
  uint32_t apart = 0;  // source minus destination, modulo 32, of all ranges together
  for (int i = 0; i < n && i < kInlineRanges; ++i) {
    if (ranges[i].bytes == 0) continue;
    total += ranges[i].bytes;
    apart |= (uint32_t)(reinterpret_cast<uintptr_t>(src) + ranges[i].src_off - reinterpret_cast<uintptr_t>(dst) - ranges[i].dst_off) & 31u;
  }
  // Words or units.  Up to 1 MiB words are at least as fast where source and destination agree
  // modulo 16, and leave tiles of 8 KiB to choose.  Beyond, 32-byte units win, shifted ones too from
  // HBM (64 MiB, 16 apart: 19.7 us shifted, 21.8 in words; from L2 19.5 and 15.7).  Over the host link
  // words are ahead where units would be shifted (16 apart, 16 KiB host-to-device 2.87 us in units,
  // 2.28 in words; 1 MiB 7.5 and 7.8) and in short messages whose destination begins inside a unit
  // (4 KiB 2.56 and 2.13; 256 KiB 3.4 and 3.6).
  const bool half = (apart & 15) == 0 && ((reinterpret_cast<uintptr_t>(dst) + ranges[0].dst_off) & 31) == 16;
  const bool words = variant == 2 ? (apart ? total < (1u << 20) : half && total <= 2 * kVecTile) : total <= (1u << 20);
  a.move = (apart & 15) ? kMoveShifted : words ? kMoveWords : apart ? kMoveShifted : kMoveUnits;
  // Tiles of the vector kernel.  Up to one wave of the grid the smallest tile that fits it, as it
  // spreads the message over most SMs; past one wave of the largest, smaller ones fill the last
  // wave better until there are many.  Measured on GB300 at 16 / 32 / 64 KiB (us per message, back
  // to back): 4 MiB 2.5 / 2.7 / 2.7, 8 MiB 3.2 / 3.7 / 3.1-4.0, 12 MiB 4.8 / 4.5 / 4.2, 16 MiB
  // 6.1 / 5.4 / 5.2, 20 MiB 7.0 / 7.1 / 7.6, 24 MiB 8.3 / 8.0 / 8.6, 32 MiB 10.7 / 10.6 / 10.5,
  // 1 GiB 307 / 307 / 304; 4 MiB on a grid of 152 CTAs 3.4 / 2.3 / 2.8.  Words at 8 / 16 / 32 KiB:
  // 100 bytes 1.35 / 1.35 / 1.09, 16 KiB 1.40 / 1.58 / 1.37, 64 KiB 1.48 / 1.60 / 1.65, 256 KiB
  // 1.48 / 1.60 / 1.81, 1 MiB 1.71 / 1.71 / 1.89.  Shifted units at 16 / 32 / 64 KiB: 100 bytes
  // 1.50 / 1.35 / 1.60, 16 KiB 1.75 / 1.54 / 1.76, 64 KiB 1.68 / 1.80 / 2.65, 2 MiB 1.94 / 2.04 /
  // 2.78, 3 MiB 2.50 / 2.09 / 2.81, 8 MiB 3.93 / 3.27 / 3.22, 16 MiB 6.1 / 6.1 / 6.3; at 64 KiB one CTA
  // fits an SM, which is the better way on a grid that small: 8 MiB on 152 CTAs 5.8 / 4.8 / 3.4, on 16
  // CTAs 25 / 15.3 / 12.5.
  const auto fits = [&](uint64_t tile, uint32_t per_sm) { return total <= tile * std::min(ctas, per_sm * sms); };
  const bool tiny = total <= kVecTile;
  if (variant == 1) a.piece = bulk_config(bulk_cfg).stage_bytes;
  else if (variant == 2) a.piece = 4 * kVecTile;
  else if (a.move == kMoveShifted)
    a.piece = tiny ? 2 * kVecTile : fits(kVecTile, 1) ? kVecTile : ctas > sms || fits(2 * kVecTile, 1) ? 2 * kVecTile : 4 * kVecTile;
  else if (a.move == kMoveWords)
    a.piece = tiny ? 2 * kVecTile : fits(kVecTile / 2, 4) ? kVecTile / 2 : fits(kVecTile, 4) ? kVecTile : fits(2 * kVecTile, 4) ? 2 * kVecTile : 4 * kVecTile;
  else if (variant == 3 || fits(kVecTile, 4)) a.piece = kVecTile;
  else if (fits(2 * kVecTile, 1)) a.piece = 2 * kVecTile;
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
    const uint32_t unit = variant == 1 || a.move == kMoveWords ? 16 : 32;
    d.head = (uint32_t)std::min<uint64_t>(d.bytes, (unit - (o & (unit - 1))) & (unit - 1));
    d.shift = (uint32_t)((s + d.head) - (o + d.head)) & (unit - 1);
    if (variant == 1 && d.shift) return kArgsNeedVec;
    const uint64_t body = (d.bytes - d.head) / unit * unit;
    const uint64_t lead = variant == 1 ? 0 : lead_bytes(s + d.head, o + d.head, a.src_lines != 0, unit);
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
