// Merge of the vocabulary-tile softmax partials into lse and logp (Eq. 1-2).
#include <math.h>

#include "logprobs_common.cuh"
#include "sao_common.cuh"

namespace sao {
namespace {

// kSub threads per row: thread k of a row merges tiles k, k + kSub, ... in one
// online pass with several loads in flight, then the (max, sum) pairs are
// combined by a fixed shuffle tree. Eight per row (four rows per warp): each
// warp load is four consecutive rows of eight tiles, eight full 32-byte
// sectors. With few rows the latency of a thread's own tiles is the time (517
// rows of 594 tiles: 18 rounds of four loads, 18 us), so a whole warp takes a row.
constexpr int64_t kWarpRows = 8192;  // rows up to which a warp takes one

template <int kSub>
__global__ void __launch_bounds__(256) lse_merge_kernel(const float2 *part, int nvt,
                                                        const float *zy, const int32_t *y,
                                                        const uint8_t *row_mask,
                                                        const int *pos, int64_t N, int V,
                                                        float *logp, float *lse, unsigned int *err) {
  grid_wait();
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t row = t / kSub;
  const int sub = int(t % kSub);
  // a row's threads are consecutive lanes of one warp; rows past N only join the shuffles
  const bool live = row < N;
  bool skip = !live || (row_mask != nullptr && row_mask[row] == 0);
  // partials of a compacted forward are stored at the row's compact index
  int64_t src = row;
  if (!skip && pos != nullptr) {
    const int i = pos[row];
    if (i < 0)
      skip = true;
    else
      src = i;
  }
  // (m, s) = running maximum and sum of exp(z - m); the larger of the two
  // maxima has factor exp(0), so one exponential serves both sides
  float m = -INFINITY, s = 0.f;
  auto merge = [&](float pm, float ps) {
    const bool up = pm > m;
    const float mn = up ? pm : m;
    if (mn == -INFINITY) return;  // nothing merged on either side yet
    const float e = expf((up ? m : pm) - mn);
    s = up ? fmaf(s, e, ps) : fmaf(ps, e, s);
    m = mn;
  };
  if (!skip) {
    constexpr int kU = kSub == 32 ? 8 : 4;  // loads in flight
    int j = sub;
    for (; j + (kU - 1) * kSub < nvt; j += kU * kSub) {
      float2 p[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) p[u] = __ldcs(part + int64_t(j + u * kSub) * N + src);
#pragma unroll
      for (int u = 0; u < kU; ++u) merge(p[u].x, p[u].y);
    }
    for (; j < nvt; j += kSub) {
      const float2 p = __ldcs(part + int64_t(j) * N + src);
      merge(p.x, p.y);
    }
  }
#pragma unroll
  for (int o = 1; o < kSub; o <<= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, m, o), os = __shfl_xor_sync(0xffffffffu, s, o);
    merge(om, os);
  }
  if (!live || sub != 0) return;
  if (skip) {
    logp[row] = 0.f;
    lse[row] = 0.f;
    return;
  }
  const float l = m + logf(s);
  lse[row] = l;
  const int yy = y[row];
  if (yy >= 0 && yy < V) {
    logp[row] = zy[src] - l;
  } else {
    logp[row] = __int_as_float(0x7fc00000);
    raise_device_error(err, SAO_DEVERR_TOKEN_ID);
  }
}

}  // namespace

sao_status lse_merge_launch(const float2 *part, int nvt, const float *zy, const int32_t *y,
                            const uint8_t *row_mask, const int *pos, int64_t N, int32_t V, float *logp, float *lse,
                            unsigned int *err, cudaStream_t s) {
  const int sub = N <= kWarpRows ? 32 : 8;
  const int64_t grid = (N * sub + 255) / 256;
  int slot = launch_begin("lse_merge", s);
  pdl(sub == 32 ? lse_merge_kernel<32> : lse_merge_kernel<8>, unsigned(grid), 256, 0, s)(
      part, nvt, zy, y, row_mask, pos, N, V, logp, lse, err);
  return launch_end(slot, s);
}

}  // namespace sao
