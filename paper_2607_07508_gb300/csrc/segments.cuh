// Helpers for kernels that walk packed trajectories (cu_seqlens) in warp
// chunks of kSegChunk tokens: the trajectory of a token, a view of a chunk's
// cu_seqlens slice staged in shared memory, and the number of action tokens per
// trajectory.
//
// A warp finds the trajectories of its own tokens by searching cu_seqlens, 32
// entries a step (2 steps of one L2 latency for a thousand trajectories, hidden
// by the other warps). A table of every chunk's first trajectory written by a
// pass of its own cost a launch in each call, and with a thread per trajectory
// 12 us at 2^24 tokens in 256 trajectories, where each thread wrote 64 entries.
#pragma once

#include <stdint.h>

#include "sao_common.cuh"

namespace sao {
namespace seg {

constexpr int kItems = 32;               // tokens per lane (one bit each in a uint32)
constexpr int kSegChunk = 32 * kItems;   // tokens per warp chunk
constexpr int kCuCap = 128;              // cu_seqlens entries staged per warp
constexpr int kCountChunks = 8;          // chunks per warp in action_count_kernel, at most
constexpr int kCastChunks = 2;           // chunks per warp in traj_broadcast_kernel

// Chunks per warp and CTAs (of 8 warps) of action_count_kernel for nchunks
// chunks: up to 8 while 32 warps of each of 152 SMs have one (8 at 2^20 tokens, 16
// CTAs, took 3 us longer than 1). The counts are integers, the same for any split.
__host__ __device__ constexpr int count_chunks(int nchunks) {
  const int c = nchunks / (152 * 32);
  return c < 1 ? 1 : c > kCountChunks ? kCountChunks : c;
}
__host__ __device__ constexpr unsigned action_count_grid(int nchunks) {
  return unsigned((nchunks + 8 * count_chunks(nchunks) - 1) / (8 * count_chunks(nchunks)));
}
// CTAs (of 8 warps) of traj_broadcast_kernel for nchunks chunks.
__host__ __device__ constexpr unsigned broadcast_grid(int nchunks) {
  return unsigned((nchunks + 8 * kCastChunks - 1) / (8 * kCastChunks));
}

// cu_seqlens entries [blo, blo + n) of one chunk, read from shared memory
// when the slice fits there, else from global memory.
struct CuView {
  const int32_t *g;
  const int32_t *s;
  int blo;
  bool in_smem;
  __device__ __forceinline__ int64_t operator[](int b) const { return in_smem ? s[b - blo] : ld(g + b); }
  // largest b in [lo, hi] with cu[b] <= t
  __device__ __forceinline__ int find(int lo, int hi, int64_t t) const {
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((*this)[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  }
};

// Stages the cu_seqlens slice of warp chunk q into `s_cu` (kCuCap entries) and
// returns the view; blo/bhi are the first/last trajectories the chunk can touch.
__device__ __forceinline__ CuView stage_chunk(const int32_t *cu, int B, int nchunks, const int *chunk_first, int q,
                                              int lane, int32_t *s_cu, int &blo, int &bhi) {
  blo = ld(chunk_first + q);
  bhi = q + 1 < nchunks ? ld(chunk_first + q + 1) : B - 1;
  const int ncu = bhi - blo + 2;  // cu[blo .. bhi + 1]
  const CuView v{cu, s_cu, blo, ncu <= kCuCap};
  if (v.in_smem)
    for (int i = lane; i < ncu; i += 32) s_cu[i] = ld(cu + blo + i);
  __syncwarp();
  return v;
}

// The kernels below get internal linkage: each translation unit that
// includes this header launches its own copy.
namespace {

// The largest b in [lo, B) with cu[b] <= t (lo, or 0 when not given, when there is
// none), by the whole warp; lo is taken to satisfy it. With a valid cu_seqlens it is the
// trajectory of token t; with any other contents it is still an index.
__device__ __forceinline__ int find_traj(const int32_t *cu, int B, int64_t t, int lane, int lo = -1) {
  // from a given lo the 32 entries next to it first (a later chunk's trajectory
  // is near), then even steps
  int n = lo < 0 ? B : B - lo;  // candidates lo .. lo + n - 1
  int step = lo < 0 ? (n + 31) / 32 : 1;
  lo = lo < 0 ? 0 : lo;
  while (n > 1) {
    const int64_t i = int64_t(lo) + int64_t(lane + 1) * step;
    const bool le = i < int64_t(lo) + n && int64_t(ld(cu + i)) <= t;
    const int c = __popc(__ballot_sync(0xffffffffu, le));
    const int used = c * step;
    lo += used;
    n -= used;
    if (c < 32 && n > step) n = step;  // the answer lies before the next probe
    step = (n + 31) / 32;
  }
  return lo;
}
// Number of action tokens per trajectory; nact must start at zero. One warp
// per count_chunks(nchunks) consecutive chunks, 8 warps per CTA (grid:
// action_count_grid). A lane's 4 tokens inside its current trajectory are
// counted with one byte-wise popcount; only groups that cross a trajectory
// end take the per-token walk. Each lane adds its count to a trajectory's
// total when it leaves it, and the lanes that end in the same trajectory add
// theirs together. chunk_first (nullable) receives each chunk's first trajectory.
__device__ __forceinline__ void count_warp(const uint8_t *m, const int32_t *cu_g, int B, int64_t N, int nchunks, int q0,
                                           int lane, int32_t *s_cu, int *chunk_first, int *nact) {
  const int per = count_chunks(nchunks);
  const int q1 = q0 + per < nchunks ? q0 + per : nchunks;
  const int blo = find_traj(cu_g, B, int64_t(q0) * kSegChunk, lane);
  const int bhi = q1 < nchunks ? find_traj(cu_g, B, int64_t(q1) * kSegChunk, lane, blo) : B - 1;
  const int ncu = bhi - blo + 2;  // cu[blo .. bhi + 1]
  const CuView cu{cu_g, s_cu, blo, ncu <= kCuCap};
  if (cu.in_smem)
    for (int i = lane; i < ncu; i += 32) s_cu[i] = ld(cu_g + blo + i);
  __syncwarp();
  if (chunk_first && q0 + lane < q1) chunk_first[q0 + lane] = cu.find(blo, bhi, int64_t(q0 + lane) * kSegChunk);
  const int64_t c0 = int64_t(q0) * kSegChunk;
  const int64_t c1 = int64_t(q1) * kSegChunk < N ? int64_t(q1) * kSegChunk : N;
  int b = blo;
  int64_t next_end = cu[b + 1];
  int cnt = 0;
  const bool aligned = (reinterpret_cast<uintptr_t>(m) & 3u) == 0;
  // 128-token groups, lane l taking tokens 4l .. 4l+3 (each warp load reads 128
  // contiguous bytes); the mask words of 8 groups are loaded together, so a
  // warp waits for one load latency per 1024 tokens; a lane's tokens only
  // increase, so its walk only moves forward
#pragma unroll 1
  for (int64_t base = c0; base < c1; base += 8 * 128) {
    uint32_t u[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int64_t t0 = base + j * 128 + int64_t(lane) * 4;
      u[j] = (aligned && t0 + 4 <= c1) ? ld(reinterpret_cast<const uint32_t *>(m + t0)) : 0u;
    }
    if (aligned && base + 8 * 128 <= c1 && base + 8 * 128 <= next_end) {
      // the whole window inside the lane's current trajectory (the common case)
#pragma unroll
      for (int j = 0; j < 8; ++j) cnt += __popc(((u[j] & 0x7f7f7f7fu) + 0x7f7f7f7fu | u[j]) & 0x80808080u);
      continue;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int64_t t0 = base + j * 128 + int64_t(lane) * 4;
      if (t0 >= c1) break;
      if (aligned && t0 + 4 <= c1 && t0 + 4 <= next_end) {  // all 4 tokens in trajectory b
        cnt += __popc(((u[j] & 0x7f7f7f7fu) + 0x7f7f7f7fu | u[j]) & 0x80808080u);
        continue;
      }
      for (int k = 0; k < 4; ++k) {
        const int64_t t = t0 + k;
        if (t >= c1) break;
        if (t >= next_end) {
          const int nb0 = b;
          while (b < bhi && t >= next_end) {
            ++b;
            next_end = cu[b + 1];
          }
          if (b != nb0 && cnt) {
            atomicAdd(nact + nb0, cnt);
            cnt = 0;
          }
        }
        cnt += m[t] != 0;
      }
    }
  }
  const unsigned peers = __match_any_sync(0xffffffffu, b);
  const int tot = __reduce_add_sync(peers, cnt);
  if (lane == __ffs(peers) - 1 && tot) atomicAdd(nact + b, tot);
}
__global__ void __launch_bounds__(256, 6) action_count_kernel(const uint8_t *m, const int32_t *cu_g, int B, int64_t N,
                                                           int nchunks, int *chunk_first, int *nact) {
  grid_wait();
  __shared__ int32_t s_cu_all[8][kCuCap];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q0 = (blockIdx.x * 8 + warp) * count_chunks(nchunks);
  if (q0 < nchunks) count_warp(m, cu_g, B, N, nchunks, q0, lane, s_cu_all[warp], chunk_first, nact);
}

// 0 = cu[0] <= cu[1] <= ... <= cu[B] = N, at trajectory b.
__device__ __forceinline__ void check_cu(const int32_t *cu, int b, int B, int64_t N, unsigned int *err) {
  if ((b == 0 && cu[0] != 0) || cu[b + 1] < cu[b] || (b == B - 1 && int64_t(cu[B]) != N))
    raise_device_error(err, SAO_DEVERR_CU_SEQLENS);
}

// adv[t] = a_traj[b] on the action tokens of trajectory b, 0 on every other
// token; every token below N is written (cu_seqlens covers [0, N)). Grid:
// broadcast_grid, kCastChunks chunks per warp (its stores run in one short
// wave per chunk pair, so small units keep the SMs busy to the end); in 128-token
// groups lane l takes 4 tokens (a 4-byte mask load, a float4 store); a group
// inside the lane's current trajectory takes no per-token work.
// kValues: also ret[t] = a_traj[b] and adv[t] = a_traj[b] - values[t] on the
// action tokens (0 elsewhere): the GAE of a trajectory whose recursion
// telescopes (gamma = lambda = 1: the advantage is its reward minus the
// value, the return its reward), with the values read by float4 as well; and
// cu_seqlens is checked.
template <bool kValues>
__global__ void __launch_bounds__(256) traj_broadcast_kernel(const float *a_traj, const uint8_t *m,
                                                             const int32_t *cu_g, int B, int64_t N, int nchunks,
                                                             float *adv, const float *values, float *ret,
                                                             unsigned int *err) {
  grid_wait();
  __shared__ int32_t s_cu_all[8][kCuCap];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (kValues)  // no other pass of the call looks at cu_seqlens
    for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < B; i += int64_t(gridDim.x) * 256)
      check_cu(cu_g, int(i), B, N, err);
  const int q0 = (blockIdx.x * 8 + warp) * kCastChunks;
  if (q0 >= nchunks) return;
  const int q1 = q0 + kCastChunks < nchunks ? q0 + kCastChunks : nchunks;
  const int blo = find_traj(cu_g, B, int64_t(q0) * kSegChunk, lane);
  const int bhi = q1 < nchunks ? find_traj(cu_g, B, int64_t(q1) * kSegChunk, lane, blo) : B - 1;
  const int ncu = bhi - blo + 2;  // cu[blo .. bhi + 1]
  const CuView cu{cu_g, s_cu_all[warp], blo, ncu <= kCuCap};
  if (cu.in_smem)
    for (int i = lane; i < ncu; i += 32) s_cu_all[warp][i] = ld(cu_g + blo + i);
  __syncwarp();
  const int64_t c0 = int64_t(q0) * kSegChunk;
  const int64_t c1 = int64_t(q1) * kSegChunk < N ? int64_t(q1) * kSegChunk : N;
  int b = blo;
  int64_t next_end = cu[b + 1];
  float v = ld(a_traj + b);
  uintptr_t al = reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(adv);
  if (kValues) al |= reinterpret_cast<uintptr_t>(values) | reinterpret_cast<uintptr_t>(ret);
  const bool aligned = (al & 15u) == 0;
  // 128-token groups: lane l takes tokens 4l .. 4l+3, so each warp load reads
  // 128 contiguous bytes and each warp store writes 512; the mask words of 8
  // groups are loaded together, so a warp waits for one load latency per
  // 1024 tokens instead of one per group
#pragma unroll 1
  for (int64_t base = c0; base < c1; base += 8 * 128) {
    uint32_t u[8];
    float4 x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int64_t t0 = base + j * 128 + int64_t(lane) * 4;
      const bool full = aligned && t0 + 4 <= c1;
      u[j] = full ? ld(reinterpret_cast<const uint32_t *>(m + t0)) : 0u;
      if (kValues) x[j] = full ? __ldcs(reinterpret_cast<const float4 *>(values + t0)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int64_t t0 = base + j * 128 + int64_t(lane) * 4;
      if (t0 >= c1) break;
      if (aligned && t0 + 4 <= c1 && t0 + 4 <= next_end) {  // all 4 tokens in trajectory b
        const uint32_t w = u[j];
        const bool a0 = (w & 0xffu) != 0u, a1 = (w & 0xff00u) != 0u, a2 = (w & 0xff0000u) != 0u,
                   a3 = (w & 0xff000000u) != 0u;
        if (kValues) {
          __stcs(reinterpret_cast<float4 *>(adv + t0),
                 make_float4(a0 ? __fsub_rn(v, x[j].x) : 0.f, a1 ? __fsub_rn(v, x[j].y) : 0.f,
                             a2 ? __fsub_rn(v, x[j].z) : 0.f, a3 ? __fsub_rn(v, x[j].w) : 0.f));
          __stcs(reinterpret_cast<float4 *>(ret + t0), make_float4(a0 ? v : 0.f, a1 ? v : 0.f, a2 ? v : 0.f,
                                                                   a3 ? v : 0.f));
        } else {
          __stcs(reinterpret_cast<float4 *>(adv + t0), make_float4(a0 ? v : 0.f, a1 ? v : 0.f, a2 ? v : 0.f,
                                                                   a3 ? v : 0.f));
        }
        continue;
      }
      for (int k = 0; k < 4; ++k) {
        const int64_t t = t0 + k;
        if (t >= c1) break;
        if (t >= next_end) {
          while (b < bhi && t >= next_end) {
            ++b;
            next_end = cu[b + 1];
          }
          v = ld(a_traj + b);
        }
        const bool act = m[t] != 0;
        if (kValues) {
          adv[t] = act ? __fsub_rn(v, values[t]) : 0.f;
          ret[t] = act ? v : 0.f;
        } else {
          adv[t] = act ? v : 0.f;
        }
      }
    }
  }
}

}  // namespace

}  // namespace seg
}  // namespace sao
