// Interface of the batched-transfer kernels (persistent descriptor-table kernel and the
// completion kernel of its copy-engine lanes) between batch.cu and the runtime.  Kept apart
// from kernels.cuh, which the copy kernels are compiled from.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mpt {

// ---- batched transfers: persistent descriptor-table kernel --------------------------
constexpr uint32_t kDescHostDst = 1;   // destination is host memory: publish with system fences
constexpr uint32_t kDescHostSide = 2;  // one side is host memory: coherent loads, no read-only path

// Tiles come in two classes, each numbered from 0 and claimed through its own cursor: link
// tiles (one side in host memory: they move over the host link) and device tiles (both sides
// in this GPU's memory).  CTAs [0, link_ctas) claim link tiles first and move to device
// tiles when those run out; the others claim device tiles only.  The link, which bounds a
// mixed batch, stays busy from the start while the device tiles run beside it, and no more
// of its traffic is in flight than the link group keeps there.
struct BatchHeader {
  uint32_t n;            // descriptors with tiles: link class first, then the device class
  uint32_t n_link;       // of them in the link class
  uint32_t link_tiles;   // tiles of each class
  uint32_t dev_tiles;
  uint32_t link_tile;    // bytes of a tile of each class
  uint32_t dev_tile;
  uint32_t epoch;        // value written to a finished descriptor's host flag
  uint32_t link_ctas;    // CTAs that may take link tiles (the first ones of the grid)
};

struct BatchDesc {
  uint64_t src, dst, bytes;
  uint32_t first_tile;  // prefix sum of tiles before this descriptor, within its class
  uint32_t ntiles;      // max(1, ceil(bytes / tile))
  uint32_t flags;
  uint32_t index;       // the transfer's place in the caller's batch: its flag, count and time
};

// Device table of one batch, packed so that a batch of n transfers is one copy of its first
// bytes: header | DMA-lane map | desc[n] | first[n], where first repeats the descriptors'
// first_tile for the search (its address follows from hdr->n; transfers of a DMA lane have no
// descriptor).
//
// The launch counters (cursors, per-transfer tile counts, exited CTAs, start times) are zero
// when a launch begins and the kernel leaves them zero: the warp that counts a transfer's last
// tile clears that transfer's count, and the last CTA to exit, once no warp can claim any
// more, clears the rest.  No reset node runs between launches.
struct BatchArgs {
  const BatchHeader* hdr;
  const BatchDesc* desc;
  uint32_t* cursor;              // next link tile to claim
  uint32_t* cursor_dev;          // next device tile to claim
  unsigned long long* start_inv; // ~(first CTA's start time) while CTAs exit
  unsigned long long* start_last;  // last CTA's start time while CTAs exit
  unsigned long long* start_out; // the launch's ~(start time), kept after the launch
  uint32_t* done;                // tiles finished per transfer
  unsigned long long* times;     // completion time per transfer (global timer, ns)
  uint32_t* host_flags;          // device alias of page-locked flags, one per transfer
  uint32_t* exited;              // CTAs that have stopped claiming
  unsigned long long* host_stamps;  // device alias of page-locked [first, last] CTA start times
};

// A short batch carries its table in the kernel's arguments.
constexpr uint32_t kInlineXfers = 8;
struct BatchInline {
  BatchArgs args;
  BatchHeader hdr;
  BatchDesc desc[kInlineXfers];
};

// Completion of one DMA-lane item: dma_map[item] is the descriptor its copy-engine node
// moved (~0 when the item is unused); stamps its time and raises its host flag.
__global__ void k_batch_dma_done(BatchArgs a, const uint32_t* dma_map, uint32_t item);

// k_batch needs every transfer's source and destination to agree modulo 16; k_batch_any copies
// any alignment.
__global__ void k_batch(BatchArgs a);
__global__ void k_batch_any(BatchArgs a);

}  // namespace mpt
