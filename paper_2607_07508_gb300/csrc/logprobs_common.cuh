// Pieces shared by the fp32 and tensor-core log-prob paths.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sao.h"

namespace sao {

// Parts that a contraction over K elements is cut into when its product has
// `tiles` output tiles: the fewest (of at most `most`, each part at least 512
// elements) for which the waves of work items on 152 SMs take at most 6 % more
// than the least time, an item costing K / parts elements plus `fixed` for filling
// the pipeline and writing its part. From two waves of whole tiles on the product
// is left alone (8,192 tokens of the moe head, 3.4 waves of dH: 3 parts 2.61 ms
// against 2.46). A function of sizes alone, so every device gives the same bits.
__host__ __device__ inline bool may_split(int64_t tiles) { return tiles < 2 * 152; }
__host__ __device__ inline unsigned split_cost(unsigned tiles, unsigned K, unsigned fixed, unsigned s) {
  return ((tiles * s + 151u) / 152u) * ((K / s + fixed) / 2u);
}
__host__ __device__ inline bool split_near(unsigned cost, unsigned least) {
  return 94ull * cost <= 100ull * least;
}
inline int k_splits(int64_t tiles, int64_t K, unsigned fixed, int most) {
  if (!may_split(tiles)) return 1;
  const unsigned n = unsigned(tiles), k = unsigned(K);
  unsigned least = ~0u, s = 1;
  for (s = 1; s <= unsigned(most) && (s == 1 || k / s >= 512u); ++s) {
    const unsigned c = split_cost(n, k, fixed, s);
    least = c < least ? c : least;
  }
  for (s = 1; !split_near(split_cost(n, k, fixed, s), least); ++s) {
  }
  return int(s);
}

// The parts of a dH product (rows x nN tiles of 128 x 256, contraction over K)
// whose scratch holds cap_rows output rows over all its parts. The rows are the
// active ones, whose number only the device knows: the GEMM and the kernel that
// adds the parts each work it out, a lane per number of parts (one thread's
// loop: 8 us). (517 rows of the moe head, 388 of them active: 7 parts, chosen
// for all rows, are two waves of 7 x 32 items, 300 us; 4 parts, chosen for the
// active ones, one wave, 220 us.)
struct DhParts {
  int64_t cap_rows;  // 0: one part
  int nN;
  int64_t K;
};
constexpr int kMostDhParts = 16;
constexpr unsigned kDhPartCost = 2000;  // elements of K that an item's start, its 128 KB of output and their sum cost
// (called by whole warps)
__device__ __forceinline__ int dh_parts(const DhParts &d, int rows) {
  if (d.cap_rows == 0 || rows <= 0) return 1;
  const int64_t tiles = int64_t(rows + 127) / 128 * d.nN;
  if (!may_split(tiles)) return 1;
  const unsigned s = (threadIdx.x & 31) + 1, k = unsigned(d.K);
  const bool fits = s == 1 || (s <= unsigned(kMostDhParts) && int64_t(s) * rows <= d.cap_rows && k / s >= 512u);
  const unsigned c = fits ? split_cost(unsigned(tiles), k, kDhPartCost, s) : ~0u;
  const unsigned least = __reduce_min_sync(0xffffffffu, c);
  return __ffs(__ballot_sync(0xffffffffu, split_near(c, least)));
}

// Merges per-(vocab tile, row) partials part[j * N + i] = (max_j, sumexp_j)
// into lse[row] = log sum_v e^z and logp[row] = zy[i] - lse[row], where i is
// the row itself, or pos[row] when the forward ran on compacted rows (pos < 0:
// a skipped row, logp = lse = 0). Rows with row_mask == 0 also get zeros.
// Token ids outside [0, V) give logp = NaN.
sao_status lse_merge_launch(const float2 *part, int nvt, const float *zy, const int32_t *y,
                            const uint8_t *row_mask, const int *pos, int64_t N, int32_t V, float *logp, float *lse,
                            unsigned int *err, cudaStream_t s);

size_t f32_ws_bytes(int64_t N, int32_t h, int32_t V);
sao_status f32_fwd(const float *H, const float *W, const int32_t *y, const uint8_t *row_mask, int64_t N,
                    int32_t h, int32_t V, float *logp, float *lse, unsigned int *err, void *ws, size_t ws_bytes,
                    cudaStream_t s);
sao_status f32_bwd(const float *H, const float *W, const int32_t *y, const float *lse, const float *G,
                    int64_t N, int32_t h, int32_t V, float *dH, float *dW, int accumulate, unsigned int *err,
                    void *ws, size_t ws_bytes, cudaStream_t s);

// The forward's stored probabilities (tensor-core path). For forward row f
// (token idx[f]) with shift kappa[f] = z[f, y] + kKappaOffset, where z[f, y]
// is the sampled token's logit from a pre-pass, e[f, v] = exp(z[f, v] -
// kappa[f]) in bf16, except at v = y, which holds e[f, y] - exp(lse - kappa)
// once the forward has lse. Then dZ[f, .] = -G exp(kappa - lse) e[f, .]: the
// backward is two GEMMs on e with a per-row scale. flag[f] marks a row where
// some z - kappa exceeded kFlagExponent (its stored values were clamped); the
// backward recomputes those rows' logits instead.
constexpr float kKappaOffset = 20.f;
constexpr float kFlagExponent = 40.f;
struct LogprobCache {
  __nv_bfloat16 *e;   // [rows, lde]
  int64_t lde, rows;
  int *idx;           // [N] forward row -> token
  int *pos;           // [N] token -> forward row, or -1 (not computed)
  int *count;         // device scalar: forward rows
  float *kappa;       // [N] per forward row
  uint8_t *flag;      // [N] per forward row
  size_t bytes;       // total size of the cache buffer
};
LogprobCache logprob_cache_view(void *base, int64_t N, int32_t V);

size_t tc_ws_bytes(int64_t N, int32_t h, int32_t V);
sao_status tc_fwd(const void *H, const void *W, const int32_t *y, const uint8_t *row_mask, int64_t N,
                  int32_t h, int32_t V, float *logp, float *lse, unsigned int *err, void *ws, size_t ws_bytes,
                  const LogprobCache *cache, cudaStream_t s);
sao_status tc_bwd(const void *H, const void *W, const int32_t *y, const float *lse, const float *G,
                  int64_t N, int32_t h, int32_t V, void *dH, float *dW, int accumulate, unsigned int *err,
                  void *ws, size_t ws_bytes, const LogprobCache *cache, cudaStream_t s);

}  // namespace sao
