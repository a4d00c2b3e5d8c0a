// Row compaction for the tensor-core log-prob path: the forward skips rows
// whose row_mask is 0 and the backward skips rows whose incoming gradient is
// 0 (observation and masked tokens), by running the GEMMs on a compacted,
// zero-padded copy of the active rows of H. The active count stays on the
// device; the persistent GEMM kernels read it at start-up.
#include <cuda_bf16.h>
#include <stdint.h>

#include "rows.cuh"
#include "sao_common.cuh"
#include "sao_internal.h"

namespace sao {
namespace {

constexpr int kScanThreads = 256;
constexpr int kRowsPerThread = 16;
constexpr int kRowsPerBlock = kScanThreads * kRowsPerThread;  // 4096
// Up to this many blocks (2^23 rows) each scatter CTA adds the counts of the
// blocks before it; above, a scan runs between the two passes.
constexpr int kAddBlocks = 2048;

// Bit i set when row t0 + i is active (t0 a multiple of 16): the mask byte, or
// the gradient, is not 0. 16-byte loads where the 16 rows are in range and the
// array aligned.
__device__ __forceinline__ uint32_t active_rows16(const uint8_t *mask, const float *g, int64_t N, int64_t t0) {
  if (t0 >= N) return 0u;
  uint32_t bits = 0u;
  const bool whole = t0 + kRowsPerThread <= N;
  if (mask != nullptr && whole && aligned16_dev(mask)) {
    const uint4 q = ld(reinterpret_cast<const uint4 *>(mask + t0));
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t h = (((w[k] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w[k]) & 0x80808080u;
      bits |= ((h * 0x00204081u) >> 28) << (4 * k);
    }
  } else if (mask == nullptr && whole && aligned16_dev(g)) {
    float4 x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = ld(reinterpret_cast<const float4 *>(g + t0) + k);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      bits |= uint32_t((x[k].x != 0.f) | (x[k].y != 0.f) << 1 | (x[k].z != 0.f) << 2 | (x[k].w != 0.f) << 3)
              << (4 * k);
  } else {
    for (int i = 0; i < kRowsPerThread && t0 + i < N; ++i)
      bits |= uint32_t(mask ? mask[t0 + i] != 0 : g[t0 + i] != 0.f) << i;
  }
  return bits;
}

// Active rows per 4096-row block.
__global__ void __launch_bounds__(kScanThreads) compact_count_kernel(const uint8_t *mask, const float *g,
                                                                     int64_t N, int *block_count) {
  grid_wait();
  const int64_t t0 = int64_t(blockIdx.x) * kRowsPerBlock + int64_t(threadIdx.x) * kRowsPerThread;
  const int c = __reduce_add_sync(0xffffffffu, __popc(active_rows16(mask, g, N, t0)));
  __shared__ int sh[kScanThreads / 32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) s += sh[w];
    block_count[blockIdx.x] = s;
  }
}

// Exclusive scan of the block counts (one CTA) and the total.
__global__ void __launch_bounds__(1024) compact_scan_kernel(int *block_count, int nblocks, int *total) {
  grid_wait();
  __shared__ int sh[1024];
  const int per = (nblocks + 1023) / 1024;
  const int b0 = threadIdx.x * per;
  int s = 0;
  for (int i = 0; i < per; ++i)
    if (b0 + i < nblocks) s += block_count[b0 + i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int v = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
    __syncthreads();
    sh[threadIdx.x] += v;
    __syncthreads();
  }
  int run = threadIdx.x ? sh[threadIdx.x - 1] : 0;
  for (int i = 0; i < per; ++i)
    if (b0 + i < nblocks) {
      const int c = block_count[b0 + i];
      block_count[b0 + i] = run;
      run += c;
    }
  if (threadIdx.x == 1023) *total = sh[1023];
}

// idx[compact] = row and pos[row] = compact (or -1), in row order. `scanned`:
// the counts already hold prefix sums; otherwise this CTA adds those before it
// and the last one writes the total. A thread lists its 16 consecutive rows
// (with 16 rounds of 256 rows and three barriers each, and the scan as a launch
// of its own, listing 65,536 rows took 20 us).
__global__ void __launch_bounds__(kScanThreads) compact_scatter_kernel(const uint8_t *mask, const float *g,
                                                                       int64_t N, const int *block_count, bool scanned,
                                                                       int *idx, int *pos, int *total) {
  grid_wait();
  const int64_t t0 = int64_t(blockIdx.x) * kRowsPerBlock + int64_t(threadIdx.x) * kRowsPerThread;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int before = 0;  // active rows of the blocks before this one: this thread's share
  if (scanned)
    before = threadIdx.x == 0 ? block_count[blockIdx.x] : 0;
  else
    for (int i = threadIdx.x; i < int(blockIdx.x); i += kScanThreads) before += block_count[i];
  const uint32_t bits = active_rows16(mask, g, N, t0);
  const int c = __popc(bits);
  int x = c;  // inclusive prefix over the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  __shared__ int sh[kScanThreads / 32], sh_before[kScanThreads / 32];
  if (lane == 31) sh[warp] = x;
  if (lane == 0) sh_before[warp] = before;
  __syncthreads();
  int off = x - c, all = 0;
#pragma unroll
  for (int w = 0; w < kScanThreads / 32; ++w) {
    off += sh_before[w] + (w < warp ? sh[w] : 0);
    all += sh_before[w] + sh[w];
  }
  if (!scanned && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = all;
  if (t0 >= N) return;
  int p[kRowsPerThread];
#pragma unroll
  for (int i = 0; i < kRowsPerThread; ++i) {
    const bool a = (bits >> i) & 1u;
    p[i] = a ? off : -1;
    if (a) idx[off++] = int(t0 + i);
  }
  if (t0 + kRowsPerThread <= N) {  // pos starts 256-byte aligned
#pragma unroll
    for (int k = 0; k < kRowsPerThread / 4; ++k)
      reinterpret_cast<int4 *>(pos + t0)[k] = make_int4(p[4 * k], p[4 * k + 1], p[4 * k + 2], p[4 * k + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < kRowsPerThread; ++i)
      if (t0 + i < N) pos[t0 + i] = p[i];
  }
}

// H_c[i] = H[idx[i]] for i < count; rows [count, round_up(count, 128)) = 0.
__global__ void gather_rows_kernel(const __nv_bfloat16 *H, int h, const int *idx, const int *count,
                                   __nv_bfloat16 *Hc, int64_t rows_cap) {
  grid_wait();
  const int n = *count;
  const int64_t pad = (int64_t(n) + 127) / 128 * 128;
  const int vec = h / 8;  // 16-byte vectors per row (h % 8 == 0)
  const int64_t total = (pad < rows_cap ? pad : rows_cap) * vec;
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = e / vec;
    const int v = int(e - i * vec);
    uint4 val = make_uint4(0u, 0u, 0u, 0u);
    if (i < n) val = reinterpret_cast<const uint4 *>(H + int64_t(idx[i]) * h)[v];
    reinterpret_cast<uint4 *>(Hc + i * h)[v] = val;
  }
}

// Sum over the parts of columns [4v, 4v + 4) of row i (fixed order). kOne: one
// part, without the loop, which kept the loads of several elements from
// overlapping (65,536 rows of h = 2048: 176 us with it, 113 without).
template <bool kOne>
__device__ __forceinline__ float4 row_sum(const float *acc, int parts, int64_t part_stride, int64_t i, int h, int v) {
  const float *src = acc + i * h + 4 * v;
  float4 x = *reinterpret_cast<const float4 *>(src);
  if constexpr (kOne) return x;
#pragma unroll 4
  for (int k = 1; k < parts; ++k) {
    const float4 o = *reinterpret_cast<const float4 *>(src + k * part_stride);
    x = make_float4(x.x + o.x, x.y + o.y, x.z + o.z, x.w + o.w);
  }
  return x;
}
// x times its row's scale (null: none), which is applied to the whole sum: a scaled
// part may be infinite where the sum is not, or of the other sign. A zero scale gives
// zeros whatever the sum holds.
__device__ __forceinline__ float4 scaled(const float4 &x, const float *scale, int64_t i) {
  if (scale == nullptr) return x;
  const float s = ld(scale + i);
  return s == 0.f ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(x.x * s, x.y * s, x.z * s, x.w * s);
}
__device__ __forceinline__ void store_bf16x4(__nv_bfloat16 *dst, const float4 &x) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
  uint2 w;
  w.x = *reinterpret_cast<const uint32_t *>(&a);
  w.y = *reinterpret_cast<const uint32_t *>(&b);
  *reinterpret_cast<uint2 *>(dst) = w;
}

// dH[t] = bf16(sum of the parts of row pos[t]) for active rows; the others get 0.
template <bool kOne>
__global__ void scatter_rows_f32_to_bf16_kernel(const float *acc, const DhParts d, int h, const float *scale,
                                                const int *pos, const int *count, int64_t N, __nv_bfloat16 *dH) {
  grid_wait();
  const int rows = *count, parts = kOne ? 1 : dh_parts(d, rows);
  const int64_t part_stride = int64_t(rows) * h;
  const int vec = h / 4;
  const int64_t total = N * vec;
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t t = e / vec;
    const int v = int(e - t * vec);
    const int i = pos[t];
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i >= 0) x = scaled(row_sum<kOne>(acc, parts, part_stride, i, h, v), scale, i);
    store_bf16x4(dH + t * h + 4 * v, x);
  }
}

// dH[idx[i]] = bf16(sum of the parts of row i) for the active rows i < count only.
template <bool kOne>
__global__ void scatter_active_f32_to_bf16_kernel(const float *acc, const DhParts d, int h, const int *idx,
                                                  const int *count, __nv_bfloat16 *dH) {
  grid_wait();
  const int rows = *count, parts = kOne ? 1 : dh_parts(d, rows);
  const int64_t part_stride = int64_t(rows) * h;
  const int vec = h / 4;
  const int64_t total = int64_t(rows) * vec;
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = e / vec;
    const int v = int(e - i * vec);
    store_bf16x4(dH + int64_t(idx[i]) * h + 4 * v, row_sum<kOne>(acc, parts, part_stride, i, h, v));
  }
}

}  // namespace

size_t list_ws_bytes(int64_t N) {
  const int64_t nblocks = (N + kRowsPerBlock - 1) / kRowsPerBlock;
  return round256(sizeof(int) * (nblocks + 1)) + round256(sizeof(int) * 4) + round256(sizeof(int) * N) * 2;
}

size_t compact_ws_bytes(int64_t N, int32_t h) {
  const int64_t cap = (N + 127) / 128 * 128;
  return list_ws_bytes(N) + round256(size_t(cap) * size_t(h) * 2);
}

sao_status list_rows(const uint8_t *mask, const float *g, int64_t N, RowList *out, Carver &c, cudaStream_t s) {
  const int64_t nblocks = (N + kRowsPerBlock - 1) / kRowsPerBlock;
  int *block = c.take<int>(size_t(nblocks) + 1);
  int *count = c.take<int>(4);
  out->idx = c.take<int>(size_t(N));
  out->pos = c.take<int>(size_t(N));
  out->count = count;
  if (!c.ok()) return fail(SAO_ERR_WORKSPACE, "workspace too small for row compaction");
  int slot = launch_begin("compact_rows", s);
  pdl(compact_count_kernel, unsigned(nblocks), kScanThreads, 0, s)(mask, g, N, block);
  SAO_TRY(launch_end(slot, s));
  slot = launch_begin("compact_rows", s);
  const bool scan = nblocks > kAddBlocks;
  if (scan) {
    pdl(compact_scan_kernel, 1, 1024, 0, s)(block, int(nblocks), count);
    SAO_TRY(launch_end(slot, s));
    slot = launch_begin("compact_rows", s);
  }
  pdl(compact_scatter_kernel, unsigned(nblocks), kScanThreads, 0, s)(mask, g, N, block, scan, out->idx, out->pos,
                                                                     count);
  return launch_end(slot, s);
}

sao_status compact_rows(const uint8_t *mask, const float *g, int64_t N, const __nv_bfloat16 *H, int32_t h,
                        CompactRows *out, Carver &c, cudaStream_t s) {
  const int64_t cap = (N + 127) / 128 * 128;
  SAO_TRY(list_rows(mask, g, N, out, c, s));
  out->Hc = c.take<__nv_bfloat16>(size_t(cap) * size_t(h));
  out->cap = cap;
  if (!c.ok()) return fail(SAO_ERR_WORKSPACE, "workspace too small for row compaction");
  DeviceInfo di;
  SAO_TRY(device_info(&di));
  int slot = launch_begin("gather_rows", s);
  pdl(gather_rows_kernel, unsigned(di.sm_count * 8), 256, 0, s)(H, h, out->idx, out->count, out->Hc, cap);
  return launch_end(slot, s);
}

sao_status scatter_rows_to_bf16(const float *acc, const DhParts &parts, int32_t h, const float *scale,
                                const int *pos, const int *idx, const int *count, int64_t N, __nv_bfloat16 *dH,
                                bool all_rows, cudaStream_t s) {
  DeviceInfo di;
  SAO_TRY(device_info(&di));
  const bool one = parts.cap_rows == 0;
  int slot = launch_begin("scatter_dH", s);
  if (all_rows)
    pdl(one ? scatter_rows_f32_to_bf16_kernel<true> : scatter_rows_f32_to_bf16_kernel<false>,
        unsigned(di.sm_count * 8), 256, 0, s)(acc, parts, h, scale, pos, count, N, dH);
  else
    pdl(one ? scatter_active_f32_to_bf16_kernel<true> : scatter_active_f32_to_bf16_kernel<false>,
        unsigned(di.sm_count * 8), 256, 0, s)(acc, parts, h, idx, count, dH);
  return launch_end(slot, s);
}

}  // namespace sao
