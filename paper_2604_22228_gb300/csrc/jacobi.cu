// Compute for the compute-plus-communication demonstration: one Jacobi sweep over a
// subdomain with halo rows, the workload of the paper's application study (Sec. 5.4: a
// Jacobi solver whose subdomains exchange boundary rows with their two neighbours, a ring).
// The paper puts only the transfers into CUDA graphs and expects larger gains once kernels
// join them; this kernel lets a caller capture stencil sweeps and multi-path halo
// exchanges into one graph.
//
// Layout: (rows + 2) x cols fp32, row-major, row 0 and row rows+1 the halos.  For interior
// rows r and columns 1..cols-2:
//   out[r][c] = ((in[r-1][c] + in[r+1][c]) + (in[r][c-1] + in[r][c+1])) * 0.25
// in that operation order, each step rounded to fp32 (so a CPU program in the same order
// reproduces it bit for bit); columns 0 and cols-1 are copied unchanged; halo rows of
// `out` are not written.
#include <algorithm>
#include <cstdlib>

#include "copy_device.cuh"
#include "internal.h"

namespace mpt {
namespace {

constexpr uint32_t kThreads = 256;

// Strip heights.  A strip of kR rows reads kR + 2, so taller strips read less, while shorter
// ones give a small grid more warps.  Measured on GB300 (us a sweep, sweeps rotating over
// 400 MB of buffers), 16-byte rows at kR = 2 / 4 / 8: 512 x 1024 points 1.89 / 1.99 / 2.35;
// 1024 x 1024 2.81 / 2.53 / 2.75; 2048 x 2048 5.43 / 4.84 / 5.53; 2048 x 4096 8.90 / 8.10 /
// 8.15; 4096 x 4096 22.9 / 20.9 / 19.2; 8 x 16 Mi 223 / 189 / 173 (kR = 16: 181).  Other rows
// with a point per thread and at kR x kG = 2x4 / 4x4: 64 x 33 1.18 / 1.68 / -; 1000 x 97 1.57 / 1.94
// / -; 1000 x 193 1.86 / 1.99 / -; 300 x 1023 2.11 / 2.08 / -; 500 x 513 2.40 / 2.04 / -;
// 2047 x 2047 - / 7.33 / 6.80; 2 x (1 Mi + 1) - / 5.70 / 6.62.
constexpr uint64_t kTinyGrid = 3ull << 16, kSmallGrid = 3ull << 18, kLargeGrid = 1ull << 23;

// Rows of at most 32 columns leave most of a warp's 128 idle, and with many of them it is the count
// of warps that costs: one group of columns and tall strips there (us a sweep at kR x kG = 8x1 /
// 4x4: 100,000 x 3 6.7 / 13.8; 2,000,000 x 3 103 / 240; 2,000,000 x 25 127 / 273; with a point per
// thread, as in the first layout, 13.9, 119 and 232).
constexpr uint64_t kNarrow = 32;
constexpr uint32_t kNarrowRows = 4096;

__device__ __forceinline__ float jacobi_point(float up, float down, float left, float right) {
  return __fmul_rn(__fadd_rn(__fadd_rn(up, down), __fadd_rn(left, right)), 0.25f);
}

// Plain loads that stay where they are written, behind the wait for the kernel ahead: that kernel
// may still be writing the rows while this one starts, so they are no read-only data.
__device__ __forceinline__ float4 ld4(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

__device__ __forceinline__ float ld1(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Both kernels cut the rows into strips of kR and give a strip of some columns to each warp.
// The sweep is bound by memory, so a warp issues every load of its strip (kR + 2 rows) before
// the first point is computed: that keeps enough bytes in flight, each row is read once from
// HBM (the rows two strips share come from L2), and a grid of any aspect ratio fills the SMs.
// One thread walking down all rows of its columns, the layout before, left the GPU to the 4
// blocks that the width gives a 1024 x 4096 subdomain: 514 us a sweep over grids of 400 MB in
// turns and 243 over one that stays in L2, against 6.9 and 4.3 now (its bytes at 6.76 TB/s: 5.0 us);
// 16384 x 16384 8385 us against 302 (317).

// 16-byte aligned rows: a lane owns four columns as one float4, a warp 128.  Horizontal
// neighbours come from the adjacent lanes (shuffles); the two lanes at the warp's edges read
// their outside neighbour from global memory.
template <int kR>
__global__ void __launch_bounds__(kThreads) k_jacobi_v4(const float* in, float* out,
                                                        uint32_t rows, uint64_t cols) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t nq = cols / 4;
  const uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  pdl_enter();
  if (q - lane >= nq) return;  // a warp past the row's end
  const bool active = q < nq;
  const uint64_t c0 = 4 * (active ? q : nq - 1);  // idle lanes shadow the last quad (shuffles need them)
  const bool edge = (lane == 0 && c0 > 0) || (lane == 31 && c0 + 4 < cols);
  const uint64_t ec = lane == 0 ? c0 - 1 : c0 + 4;  // the neighbour column outside the warp
  const uint32_t nstrips = rows / kR + (rows % kR != 0);
  for (uint32_t s = blockIdx.y * blockDim.y + threadIdx.y; s < nstrips; s += gridDim.y * blockDim.y) {
    const uint32_t r0 = s * kR;  // the strip writes rows r0 + 1 .. r0 + n
    const uint32_t n = rows - r0 < (uint32_t)kR ? rows - r0 : (uint32_t)kR;
    const float* ip = in + (uint64_t)r0 * cols;
    float4 x[kR + 2];
    float e[kR];
#pragma unroll
    for (int i = 0; i < kR + 2; ++i)
      if (i < 2 || (uint32_t)i < n + 2) x[i] = ld4(ip + (uint64_t)i * cols + c0);
#pragma unroll
    for (int i = 0; i < kR; ++i) e[i] = edge && (uint32_t)i < n ? ld1(ip + (uint64_t)(i + 1) * cols + ec) : 0.0f;
#pragma unroll
    for (int i = 0; i < kR; ++i) {
      if ((uint32_t)i >= n) break;
      const float4 up = x[i], mid = x[i + 1], down = x[i + 2];
      float left = __shfl_up_sync(0xffffffffu, mid.w, 1);
      float right = __shfl_down_sync(0xffffffffu, mid.x, 1);
      if (lane == 0) left = e[i];
      if (lane == 31) right = e[i];
      // (a quad whose right neighbour lies past the row ends in column cols-1, copied as is)
      float4 o;
      o.x = c0 == 0 ? mid.x : jacobi_point(up.x, down.x, left, mid.y);
      o.y = jacobi_point(up.y, down.y, mid.x, mid.z);
      o.z = jacobi_point(up.z, down.z, mid.y, mid.w);
      o.w = c0 + 4 == cols ? mid.w : jacobi_point(up.w, down.w, mid.z, right);
      if (active) *reinterpret_cast<float4*>(out + (uint64_t)(r0 + i + 1) * cols + c0) = o;
    }
  }
}

// Small grids of any column count or alignment: a point per thread.  Their time is the latency of
// one chain of loads, which strips with their shuffles make longer (1000 x 97, sweeps following
// each other in a graph: 1.57 us, 1.99 as strips of two rows).
__global__ void __launch_bounds__(kThreads) k_jacobi_point(const float* in, float* out, uint32_t rows, uint64_t cols) {
  const uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  pdl_enter();
  if (c >= cols) return;
  for (uint32_t r = blockIdx.y * blockDim.y + threadIdx.y; r < rows; r += gridDim.y * blockDim.y) {
    const float* p = in + (uint64_t)(r + 1) * cols + c;
    out[(uint64_t)(r + 1) * cols + c] =
        c == 0 || c + 1 == cols ? ld1(p) : jacobi_point(ld1(p - cols), ld1(p + cols), ld1(p - 1), ld1(p + 1));
  }
}

// Any column count or alignment: a warp owns kG groups of 32 neighbouring columns, a lane one
// column of each, so that every access is a coalesced 4-byte one and only the two ends of the
// warp's 32 * kG columns need a load of their own.  With one group (or one point per thread, as
// before) too few bytes are in flight: 16384 x 16381 took 847 us, 543 with kG = 1, 359 now.
template <int kR, int kG>
__global__ void __launch_bounds__(kThreads) k_jacobi(const float* in, float* out,
                                                     uint32_t rows, uint64_t cols) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x - lane) * kG;  // the warp's first column
  pdl_enter();
  if (w0 >= cols) return;
  const uint64_t c0 = w0 + lane;
  const uint64_t w1 = w0 + 32 * kG;  // one past its last column
  const bool edge = (lane == 0 && w0 > 0) || (lane == 31 && w1 < cols);
  const uint64_t ec = lane == 0 ? w0 - 1 : w1;
  const uint32_t nstrips = rows / kR + (rows % kR != 0);
  for (uint32_t s = blockIdx.y * blockDim.y + threadIdx.y; s < nstrips; s += gridDim.y * blockDim.y) {
    const uint32_t r0 = s * kR;
    const uint32_t n = rows - r0 < (uint32_t)kR ? rows - r0 : (uint32_t)kR;
    const float* ip = in + (uint64_t)r0 * cols;
    float x[kR + 2][kG];
    float e[kR];
#pragma unroll
    for (int i = 0; i < kR + 2; ++i)
#pragma unroll
      for (int g = 0; g < kG; ++g)
        x[i][g] = (i < 2 || (uint32_t)i < n + 2) && c0 + 32 * g < cols ? ld1(ip + (uint64_t)i * cols + c0 + 32 * g) : 0.0f;
#pragma unroll
    for (int i = 0; i < kR; ++i) e[i] = edge && (uint32_t)i < n ? ld1(ip + (uint64_t)(i + 1) * cols + ec) : 0.0f;
#pragma unroll
    for (int i = 0; i < kR; ++i) {
      if ((uint32_t)i >= n) break;
      float* op = out + (uint64_t)(r0 + i + 1) * cols;
      float before = e[i], after = __shfl_sync(0xffffffffu, x[i + 1][0], lane + 1);
#pragma unroll
      for (int g = 0; g < kG; ++g) {
        // rotations: lane 0 receives lane 31's value (the left neighbour of the next group's
        // first column) and lane 31 lane 0's (the right neighbour of the last group's last)
        const float mid = x[i + 1][g];
        const float up1 = __shfl_sync(0xffffffffu, mid, lane + 31);
        const float next = g + 1 < kG ? __shfl_sync(0xffffffffu, x[i + 1][g + 1 < kG ? g + 1 : g], lane + 1) : e[i];
        const float left = lane == 0 ? before : up1;
        const float right = lane == 31 ? next : after;
        before = up1;
        after = next;
        const uint64_t c = c0 + 32 * g;
        if (c < cols) op[c] = c == 0 || c + 1 == cols ? mid : jacobi_point(x[i][g], x[i + 2][g], left, right);
      }
    }
  }
}

// MPT_PDL=0 turns overlapped launches off, here as for a context's direct copies; a sweep has no
// context to ask, so the environment is read at the process's first one.
bool overlap_allowed() {
  static const bool allowed = [] {
    const char* v = std::getenv("MPT_PDL");
    if (!v || !*v) return true;
    char* end = nullptr;
    return std::strtoull(v, &end, 0) != 0 || *end != 0;
  }();
  return allowed;
}

// Blocks of 8 warps: across a row where it is wide enough, else over strips of rows too.  Outside a
// stream capture the launch overlaps the end of the kernel ahead, as the copy kernels' does; each
// waits for that kernel before it touches memory (a ring of four 1024 x 4096 subdomains, two
// iterations with their halo copies: 91.7 us without, 78.3 with; 8 x 4 Mi 460 and 438).
template <typename Kernel>
cudaError_t launch(Kernel k, uint32_t warp_cols, uint32_t strip, const float* in, float* out, uint32_t rows,
                   uint64_t cols, cudaStream_t s) {
  const uint64_t nxw = (cols + warp_cols - 1) / warp_cols;  // warps across a row
  uint32_t bx = 1;
  while (bx < kThreads / 32 && bx < nxw) bx <<= 1;
  const uint32_t by = kThreads / 32 / bx;
  const uint32_t nstrips = rows / strip + (rows % strip != 0);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
    cudaGetLastError();
    cap = cudaStreamCaptureStatusActive;
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((uint32_t)((nxw + bx - 1) / bx), std::min<uint32_t>((nstrips + by - 1) / by, 65535u));
  cfg.blockDim = dim3(32 * bx, by);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone && overlap_allowed() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, in, out, rows, cols);
}

}  // namespace
}  // namespace mpt

extern "C" MPT_API mpt_status mpt_demo_jacobi_step(const float* in, float* out, uint32_t rows, uint64_t cols,
                                                   void* stream) {
  if (!in || !out || rows == 0 || cols < 2) return mpt::fail(MPT_EINVAL, "mpt_demo_jacobi_step: bad argument");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool vec = cols % 4 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  const uint64_t blocks = ((vec ? cols / 4 : cols) + mpt::kThreads - 1) / mpt::kThreads;
  if (blocks > 0x7fffffffull) return mpt::fail(MPT_EINVAL, "mpt_demo_jacobi_step: %llu columns", (unsigned long long)cols);
  using namespace mpt;
  const uint64_t points = (uint64_t)rows * cols;
  cudaError_t e;
  if (vec) {
    if (rows == 1) e = launch(k_jacobi_v4<1>, 128, 1, in, out, rows, cols, s);
    else if (rows == 2 || points < kSmallGrid) e = launch(k_jacobi_v4<2>, 128, 2, in, out, rows, cols, s);
    else if (rows <= 4 || points < kLargeGrid) e = launch(k_jacobi_v4<4>, 128, 4, in, out, rows, cols, s);
    else e = launch(k_jacobi_v4<8>, 128, 8, in, out, rows, cols, s);
  } else {
    if (cols <= kNarrow && rows >= kNarrowRows) e = launch(k_jacobi<8, 1>, 32, 8, in, out, rows, cols, s);
    else if (points < kTinyGrid) e = launch(k_jacobi_point, 32, 1, in, out, rows, cols, s);
    else if (rows <= 3 || points < kSmallGrid) e = launch(k_jacobi<2, 4>, 128, 2, in, out, rows, cols, s);
    else e = launch(k_jacobi<4, 4>, 128, 4, in, out, rows, cols, s);
  }
  if (e != cudaSuccess) return fail(MPT_ECUDA, "mpt_demo_jacobi_step: %s", cudaGetErrorString(e));
  return MPT_OK;
}
