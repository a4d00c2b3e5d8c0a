// Row compaction helpers of the tensor-core log-prob path (see rows.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "logprobs_common.cuh"
#include "sao_common.cuh"

namespace sao {

struct RowList {
  int *idx;            // [N] compact index -> original row
  int *pos;            // [N] original row -> compact index, or -1
  int *count;          // device scalar: number of active rows
};

struct CompactRows : RowList {
  __nv_bfloat16 *Hc;   // [cap, h] active rows of H, zero-padded to a multiple of 128
  int64_t cap;         // rows allocated in Hc (N rounded up to 128)
};

size_t list_ws_bytes(int64_t N);
size_t compact_ws_bytes(int64_t N, int32_t h);

// Active rows are those with mask[t] != 0 (mask given) or g[t] != 0.
sao_status list_rows(const uint8_t *mask, const float *g, int64_t N, RowList *out, Carver &c, cudaStream_t s);
// The list, and the active rows of H gathered in its order.
sao_status compact_rows(const uint8_t *mask, const float *g, int64_t N, const __nv_bfloat16 *H, int32_t h,
                        CompactRows *out, Carver &c, cudaStream_t s);

// dH[t] = bf16(sum over the parts k of acc[(k * count + pos[t]) * h ..]) on the
// active rows, times scale[pos[t]] where a scale is given (all_rows only); inactive
// rows get zeros when all_rows (a sweep over all N rows), else keep their contents (a sweep over the `*count` active rows idx[0..count)
// only). The parts are those that the GEMM which wrote them took.
sao_status scatter_rows_to_bf16(const float *acc, const DhParts &parts, int32_t h, const float *scale,
                                const int *pos, const int *idx, const int *count, int64_t N, __nv_bfloat16 *dH,
                                bool all_rows, cudaStream_t s);

}  // namespace sao
