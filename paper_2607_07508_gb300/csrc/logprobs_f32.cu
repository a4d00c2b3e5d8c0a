// fp32 path of the LM-head log-probs (Eq. 1-2) and their gradient, on the
// tensor cores by splitting each fp32 operand into three bf16 pieces.
//
// a = a0 + a1 + a2 exactly (8 + 8 + 8 significand bits, each piece rounded to
// nearest) for 2^-110 <= |a| < 2^100; below, the last piece falls under bf16's
// smallest step, 2^-133, and a is off by up to 2^-134: negligible next to operands of
// ordinary size, but a dZ that is nowhere above 2^-110 (incoming gradients of 1e-31
// and less) loses precision that fp32 products would keep. So
//   a b = a0 b0 + (a0 b1 + a1 b0) + (a0 b2 + a1 b1 + a2 b0)
// up to terms below 2^-26 |a b|: six bf16 products with exact fp32 results stand in
// for one fp32 product (the splitting is the one of Henry, Tang and Heinecke,
// "Leveraging the bfloat16 Artificial Intelligence Datatype For
// Higher-Precision Computations", 2019). Tensor-core accumulation truncates,
// which over a long contraction costs more than fp32 FMA rounding, so the
// accumulator is emptied every 32 elements of the contraction: within those,
// the small products come first and only the last two MMAs (a0 b0) add at full
// scale; the 32-element sums are then added in fp32 registers, rounded to
// nearest.
//
// Measured at N = 4099 (3,074 active rows), h = 1024, V = 32000 against 64x64
// fp32 FMA tiles: forward and backward 43.9 -> 3.1 ms (the four products
// 0.67-0.83 ms each, 1.45-1.8 PFLOP/s of bf16 products); relative error of dH
// against fp64 3.2e-6 -> 2.2e-7, of log-probs below 6e-8 on both sides.
//
//   split     H (active rows) and a chunk of W -> three bf16 planes each
//   forward   Z = H W^T tiles -> per-(row, 64-column quarter tile) (max, sum-exp)
//             partials and the sampled token's logit, merged by lse_merge
//   backward  per vocabulary chunk: dZ = G (1[v == y] - exp(z - lse)) written as
//             three planes, then dH (+)= dZ W and dW (+)= dZ^T H
//
// Pieces of opposite signs must not overflow to opposite infinities where fp32
// gives one infinity or none. So each operand's largest magnitude is kept on the
// device as a class (below 2^26, 2^62, 2^100, or beyond: NaN and infinities too),
// and a GEMM whose two classes allow a product of 2^126 or more runs its tiles with
// fp32 FMA on the original arrays instead (dZ, held as planes only, keeps
// infinities and NaN in its first plane).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <stdint.h>

#include "logprobs_common.cuh"
#include "per_device.h"
#include "rows.cuh"
#include "sao_common.cuh"
#include "sao_internal.h"
#include "tc_ptx.cuh"

namespace sao {
namespace {

using namespace tc;

constexpr int TM = 128, TN = 256;            // output tile
constexpr int KB = 32;                       // contraction elements per stage
constexpr int PL = 3;                        // bf16 planes per operand
constexpr uint32_t PLANE_A = TM * KB * 2, PLANE_B = TN * KB * 2;  // one K-major plane: rows of 64 bytes
constexpr uint32_t MN_BOX = PL * KB * 128;   // MN-major: 64 MN elements (128 bytes) x 32 k rows x 3 planes
constexpr uint32_t A_BYTES = PL * PLANE_A, B_BYTES = PL * PLANE_B;
static_assert(A_BYTES == TM / 64 * MN_BOX && B_BYTES == TN / 64 * MN_BOX, "both majors take the same bytes");
constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int STAGES = 3;
constexpr int ACCS = 2;                      // accumulators of 256 TMEM columns
constexpr uint32_t TMEM_COLS = ACCS * TN;
constexpr size_t SMEM_BYTES = 1024 + size_t(STAGES) * STAGE_BYTES + 256;
static_assert(SMEM_BYTES <= 232448, "shared memory of an SM");
constexpr int NUM_THREADS = 640;             // warp 0 TMA, warp 1 MMA, warps 4-19 accumulate and finish
constexpr int HN = TN / 4;                   // columns per accumulating warp: four warps (128 rows) per quarter
// Registers: the kernel starts with 96 a thread (61,440 for its 20 warps); the
// first four warps hand theirs to the sixteen that hold 64 sums a thread.
constexpr int LAUNCH_REGS = 96, ISSUE_REGS = 40, SUM_REGS = 104;
static_assert(128 * ISSUE_REGS + 512 * SUM_REGS <= NUM_THREADS * LAUNCH_REGS, "split within the launch's registers");
constexpr float CLASS_LIMIT[3] = {0x1p26f, 0x1p62f, 0x1p100f};
constexpr unsigned SAFE_CLASSES = 2;  // 2^26 x 2^100, 2^62 x 2^62: products up to 2^126
enum Operand : int { kOpH = 0, kOpW = 1, kOpDZ = 2, kOperands = 3 };
constexpr int64_t MAX_ROWS = int64_t(65535) * 64;

enum Kind : int { kLogits = 0, kDLogits = 1, kDH = 2, kDW = 3 };

struct F32Params {
  int nM, nN, nK;     // tiles along M and N, 32-element steps along K
  int splits;         // K is cut in this many parts (kDH, kDW)
  int group_m;        // raster: M tiles per group, M fastest inside
  int64_t rows;       // M extent (rows of H; kDW: columns of the chunk)
  int cols;           // N extent
  const int *m_count; // kLogits, kDLogits, kDH: active rows (null: rows)
  const int *k_count; // kDW: active rows
  const int *row_idx; // compact row -> token (null: the row itself)
  const float *H, *W; // the fp32 operands (W at the chunk's first row)
  int h, vc;          // hidden size, vocabulary columns of the chunk
  const int32_t *y;
  int v0;             // first vocabulary index of the chunk
  int tile0;          // kLogits: partial index of the chunk's first quarter tile
  float2 *part;       // [quarter tiles][part_ld]
  int64_t part_ld;
  float *zy;
  const float *lse, *G;
  __nv_bfloat16 *dz;  // three planes [rows][ldz]
  int64_t ldz, dz_plane;
  float *out;         // kDH, kDW: [split][M][ldo]
  int64_t ldo, out_split;
  int accumulate;
  // classes of H, W (raised by the split passes) and dZ (raised by kDLogits, read
  // by kDH and kDW). A kernel takes its path from words that no CTA of its own
  // launch writes: one that starts late, on an SM that other work held, would else
  // take the other path's tiles.
  unsigned int *range;
  unsigned int *err;
};

struct __align__(8) SmemCtl {
  uint64_t full[STAGES], empty[STAGES], acc_full[ACCS], acc_empty[ACCS];
  uint32_t tmem_base;
  int abort;
};

// a = p0 + p1 + p2, for |a| below 2^100
__device__ __forceinline__ void split3(float a, float &p0, float &p1, float &p2) {
  p0 = __bfloat162float(__float2bfloat16_rn(a));
  const float r = a - p0;
  p1 = __bfloat162float(__float2bfloat16_rn(r));
  p2 = r - p1;
}
// Largest magnitude (NaN if there is one), and its class.
__device__ __forceinline__ float larger(float most, float a) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(most), "f"(fabsf(a)));
  return r;
}
__device__ __forceinline__ void raise_class(unsigned int *word, float most) {
  const unsigned c = !(most < CLASS_LIMIT[0]) + !(most < CLASS_LIMIT[1]) + !(most < CLASS_LIMIT[2]);
  if (c > 0) atomicMax(word, c);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// ---------------------------------------------------------------------------
// splitting
// ---------------------------------------------------------------------------
struct SplitSrc {
  const float *src;    // rows of h floats
  const int *idx;      // row -> source row (null: itself)
  const int *count;    // rows on the device (null: rows)
  int64_t rows, pad;   // rows, and rows written (zeros past the count, up to its next multiple of 128)
  __nv_bfloat16 *dst;  // planes [pad][hp]
  int64_t plane;
};

__device__ __forceinline__ float split_rows(const SplitSrc &a, int h, int hp, int64_t tid, int64_t stride) {
  const int64_t n = a.count ? int64_t(*a.count) : a.rows;
  int64_t pad = (n + TM - 1) / TM * TM;
  if (pad > a.pad) pad = a.pad;
  const int vec = hp / 4;
  const bool wide = (h % 4) == 0 && aligned16_dev(a.src);
  float most = 0.f;
  for (int64_t e = tid; e < pad * vec; e += stride) {
    const int64_t i = e / vec;
    const int k = int(e - i * vec) * 4;
    float x[4] = {0.f, 0.f, 0.f, 0.f};
    if (i < n) {
      const float *r = a.src + (a.idx ? int64_t(ld(a.idx + i)) : i) * h + k;
      if (wide && k < h) {
        const float4 v = ld(reinterpret_cast<const float4 *>(r));
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (k + j < h) x[j] = ld(r + j);
      }
    }
    float p[PL][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      most = larger(most, x[j]);
      split3(x[j], p[0][j], p[1][j], p[2][j]);
    }
#pragma unroll
    for (int q = 0; q < PL; ++q)
      *reinterpret_cast<uint2 *>(a.dst + q * a.plane + i * hp + k) =
          make_uint2(pack2(p[q][0], p[q][1]), pack2(p[q][2], p[q][3]));
  }
  return most;
}

// Both operands in one launch: the first `blocks_a` CTAs take a, the rest b.
__global__ void __launch_bounds__(256) f32_split_kernel(SplitSrc a, SplitSrc b, int blocks_a, int h, int hp,
                                                        unsigned int *range) {
  grid_wait();
  const bool first = int(blockIdx.x) < blocks_a;
  const int blk = first ? int(blockIdx.x) : int(blockIdx.x) - blocks_a;
  const int blocks = first ? blocks_a : int(gridDim.x) - blocks_a;
  raise_class(range + (first ? kOpH : kOpW),
              split_rows(first ? a : b, h, hp, int64_t(blk) * 256 + threadIdx.x, int64_t(blocks) * 256));
}

// ---------------------------------------------------------------------------
// shared-memory and TMA helpers of this kernel's layouts
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int32_t x, int32_t y,
                                            int32_t z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// 32 TMEM lanes x 16 consecutive 32-bit columns (lane i: row i).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// K-major operand of 64-byte rows (32 bf16) under the 64-byte swizzle: 8-row
// groups 512 bytes apart, swizzle mode 4 in bits 61-63.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t addr) {
  return uint64_t((addr >> 4) & 0x3FFFu) | (uint64_t(1) << 16) | (uint64_t(512 >> 4) << 32) | (uint64_t(1) << 46) |
         (uint64_t(4) << 61);
}

__device__ __forceinline__ void tile_of(int L, const F32Params &p, int nM, int &m, int &n) {
  const int per_group = p.group_m * p.nN;
  const int g = L / per_group;
  const int within = L - g * per_group;
  const int m0 = g * p.group_m;
  const int gm = min(p.group_m, nM - m0);
  m = m0 + within % gm;
  n = within / gm;
}

// ---------------------------------------------------------------------------
// fp32 FMA tiles, for operands that the splitting cannot represent: the tiles,
// raster and parts of the tensor-core path. Warps 0-3 bring 16 elements of K of
// both operands into one of two shared-memory buffers while warps 4-19 work on
// the other one, 8x8 outputs per thread: warp w takes 32 rows and 64 columns (as it
// does of a TMEM accumulator), lane l rows 8 (l / 8) + i and columns 4 (l % 8) + j of
// each 32. Bound by the FMAs and their shared-memory reads: 4,099 x 32,000 x 1,024
// with 3,074 active rows, forward and backward, 30 ms (27 TFLOP/s of executed
// products); with 128x128 tiles whose operands the computing threads fetched
// element by element 56; FMA kernels of 64x64 tiles over all rows 43.8.
// ---------------------------------------------------------------------------
constexpr int FK = 16, FBAR = 1;
constexpr int FLD_A = TM + 4, FLD_B = TN + 4;
constexpr int FBUF = FK * (FLD_A + FLD_B);  // floats of one buffer

// Elements c .. c + 3 of a row of `limit` floats, zeros past its end. `wide`: rows start 16-byte aligned.
__device__ __forceinline__ float4 fma_load(const float *row, int64_t c, int64_t limit, bool wide) {
  if (wide && c + 4 <= limit) return ld(reinterpret_cast<const float4 *>(row + c));
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < limit) v.x = ld(row + c);
  if (c + 1 < limit) v.y = ld(row + c + 1);
  if (c + 2 < limit) v.z = ld(row + c + 2);
  if (c + 3 < limit) v.w = ld(row + c + 3);
  return v;
}
// The same of a row of dZ, from its planes (pitch a multiple of the tile, c of 4).
__device__ __forceinline__ float4 fma_load_dz(const F32Params &p, int64_t row, int64_t c, int64_t limit) {
  uint2 u[PL];
#pragma unroll
  for (int q = 0; q < PL; ++q)
    u[q] = *reinterpret_cast<const uint2 *>(p.dz + q * p.dz_plane + row * p.ldz + c);
  float v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float d[PL];
#pragma unroll
    for (int q = 0; q < PL; ++q) {
      const uint32_t w = j < 2 ? u[q].x : u[q].y;
      d[q] = __uint_as_float((j & 1) ? w & 0xffff0000u : w << 16);
    }
    // an infinity or a NaN stands alone (its remainder is a NaN)
    v[j] = c + j >= limit ? 0.f : isfinite(d[0]) ? (d[0] + d[1]) + d[2] : d[0];
  }
  return make_float4(v[0], v[1], v[2], v[3]);
}

// Operand `kOpA`'s rows [r0, r0 + kRows) of this slab, K elements [k0, k0 + FK) with
// zeros from kend on, to dst[k][row]. By warps 0-3.
template <int kKind, bool kOpA>
__device__ __forceinline__ void fma_fill(const F32Params &p, float *dst, int64_t r0, int64_t k0, int64_t M,
                                         int64_t kend, bool wide) {
  constexpr int kRows = kOpA ? TM : TN, kLd = kOpA ? FLD_A : FLD_B;
  // contiguous along K: H and W of the logits, dZ of dH
  constexpr bool kAlongK = kKind == kLogits || kKind == kDLogits || (kKind == kDH && kOpA);
  constexpr int kPer = kAlongK ? FK / 4 : kRows / 4;  // 4-element pieces of a source row
  constexpr int kPieces = kRows * FK / 4 / 128;       // per thread
  constexpr int kU = 4;
#pragma unroll 1
  for (int u0 = 0; u0 < kPieces; u0 += kU) {
    float4 x[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = (u0 + u) * 128 + threadIdx.x;
      const int i = e / kPer, c = e % kPer * 4;  // source row of the slab, first element
      x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (kKind == kLogits || kKind == kDLogits) {
        const int64_t r = r0 + i;
        if (kOpA ? r < M : r < p.cols) {
          const int64_t t = kOpA && p.row_idx ? int64_t(ld(p.row_idx + r)) : r;
          x[u] = fma_load((kOpA ? p.H : p.W) + t * p.h, k0 + c, kend, wide);
        }
      } else if constexpr (kKind == kDH && kOpA) {
        if (r0 + i < M) x[u] = fma_load_dz(p, r0 + i, k0 + c, kend);
      } else if (k0 + i < kend) {
        if constexpr (kKind == kDH)
          x[u] = fma_load(p.W + (k0 + i) * p.h, r0 + c, p.cols, wide);
        else if constexpr (kOpA)
          x[u] = fma_load_dz(p, k0 + i, r0 + c, M);
        else
          x[u] = fma_load(p.H + (p.row_idx ? int64_t(ld(p.row_idx + k0 + i)) : k0 + i) * p.h, r0 + c, p.cols, wide);
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = (u0 + u) * 128 + threadIdx.x;
      const int i = e / kPer, c = e % kPer * 4;
      if constexpr (kAlongK) {
        dst[c * kLd + i] = x[u].x;
        dst[(c + 1) * kLd + i] = x[u].y;
        dst[(c + 2) * kLd + i] = x[u].z;
        dst[(c + 3) * kLd + i] = x[u].w;
      } else {
        *reinterpret_cast<float4 *>(dst + i * kLd + c) = x[u];
      }
    }
  }
}

// Work item `it`: its tile's first row and column, its part and that part's elements of K.
struct FmaItem {
  int sp;
  int64_t m0, n0, kbeg, kend;
};
__device__ __forceinline__ FmaItem fma_item(const F32Params &p, int it, int nM, int64_t K) {
  const int64_t steps = (K + KB - 1) / KB;
  FmaItem t;
  t.sp = it % p.splits;
  int m, n;
  tile_of(it / p.splits, p, nM, m, n);
  t.m0 = int64_t(m) * TM;
  t.n0 = int64_t(n) * TN;
  t.kbeg = steps * t.sp / p.splits * KB;
  t.kend = min(K, steps * (t.sp + 1) / p.splits * KB);
  return t;
}

// Both roles are out of line: inlined, they cost the tensor-core path's epilogues
// registers (688 bytes of spill loads in dlogits against 64; a step of the tiny
// configuration 175 us against 157). The buffers start 1,024-byte aligned in the
// kernel's dynamic shared memory, named here so that they are read as such.
__device__ __forceinline__ float *fma_buffers() {
  extern __shared__ uint8_t smem_raw[];
  return reinterpret_cast<float *>(smem_raw + (-smem_u32(smem_raw) & 1023u));
}
template <int kKind>
__device__ __noinline__ void fma_produce(const F32Params &p, int64_t M, int64_t K, int nM, int items) {
  float *sm = fma_buffers();
  const float *other = kKind == kDW ? p.H : p.W;  // the fp32 operands share h, so one test serves both
  const bool wide = (p.h & 3) == 0 && aligned16_dev(other) && aligned16_dev(p.H);
  int buf = 0;
#pragma unroll 1
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const FmaItem t = fma_item(p, it, nM, K);
#pragma unroll 1
    for (int64_t k0 = t.kbeg; k0 < t.kend; k0 += FK, buf ^= 1) {
      float *dst = sm + buf * FBUF;
      fma_fill<kKind, true>(p, dst, t.m0, k0, M, t.kend, wide);
      fma_fill<kKind, false>(p, dst + FK * FLD_A, t.n0, k0, M, t.kend, wide);
      // full; and the other buffer, which was full at the barrier before, is free
      named_barrier(FBAR, NUM_THREADS);
    }
  }
}

template <int kKind>
__device__ __noinline__ void fma_consume(const F32Params &p, int64_t M, int64_t K, int nM, int items) {
  const float *sm = fma_buffers();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r_in = 32 * (warp & 3) + 8 * (lane >> 3), quarter = (warp - 4) >> 2;
  const int c_in = HN * quarter + 4 * (lane & 7);  // columns c_in + j and c_in + 32 + j, j < 4
  int buf = 0;
#pragma unroll 1
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const FmaItem t = fma_item(p, it, nM, K);
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 1
    for (int64_t k0 = t.kbeg; k0 < t.kend; k0 += FK, buf ^= 1) {
      named_barrier(FBAR, NUM_THREADS);
      const float *sa = sm + buf * FBUF + r_in, *sb = sm + buf * FBUF + FK * FLD_A + c_in;
#pragma unroll 2
      for (int k = 0; k < FK; ++k) {
        float a[8], b[8];
        *reinterpret_cast<float4 *>(a) = *reinterpret_cast<const float4 *>(sa + k * FLD_A);
        *reinterpret_cast<float4 *>(a + 4) = *reinterpret_cast<const float4 *>(sa + k * FLD_A + 4);
        *reinterpret_cast<float4 *>(b) = *reinterpret_cast<const float4 *>(sb + k * FLD_B);
        *reinterpret_cast<float4 *>(b + 4) = *reinterpret_cast<const float4 *>(sb + k * FLD_B + 32);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
    }
    if (t.n0 + HN * quarter >= p.cols) continue;
    [[maybe_unused]] float most = 0.f;  // of dZ
    auto col = [&](int j) { return t.n0 + c_in + (j >> 2) * 32 + (j & 3); };
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t row = t.m0 + r_in + i;
      const bool ok = row < M;
      const int64_t tok = (ok && p.row_idx) ? int64_t(ld(p.row_idx + row)) : row;
      if constexpr (kKind == kLogits) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (col(j) < p.cols) mx = fmaxf(mx, acc[i][j]);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (col(j) < p.cols) s += expf(acc[i][j] - mx);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (ok) {
          if ((lane & 7) == 0)
            p.part[int64_t(p.tile0 + 4 * int(t.n0 / TN) + quarter) * p.part_ld + row] = make_float2(mx, s);
          const int yy = ld(p.y + tok) - p.v0;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (col(j) == yy && yy < p.cols) p.zy[row] = acc[i][j];
        }
      } else if constexpr (kKind == kDLogits) {
        if (row >= p.rows) continue;
        const float g = ok ? ld(p.G + tok) : 0.f, l = ok ? ld(p.lse + tok) : 0.f;
        const int yy = ok ? ld(p.y + tok) - p.v0 : -1;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (col(j) >= p.cols) continue;
          float d = 0.f;
          if (g != 0.f) d = g * ((col(j) == yy ? 1.f : 0.f) - expf(acc[i][j] - l));
          most = larger(most, d);
          float p0, p1, p2;  // (a NaN remainder where d is infinite or rounds to infinity)
          split3(d, p0, p1, p2);
          __nv_bfloat16 *dst = p.dz + row * p.ldz + col(j);
          dst[0] = __float2bfloat16_rn(p0);
          dst[p.dz_plane] = __float2bfloat16_rn(p1);
          dst[2 * p.dz_plane] = __float2bfloat16_rn(p2);
        }
      } else if (ok) {
        float *dst = p.out + t.sp * p.out_split + row * p.ldo;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (col(j) < p.cols) dst[col(j)] = p.accumulate ? dst[col(j)] + acc[i][j] : acc[i][j];
      }
    }
    if constexpr (kKind == kDLogits) raise_class(p.range + kOpDZ, most);
  }
}

// ---------------------------------------------------------------------------
// the GEMM
// ---------------------------------------------------------------------------
// One persistent CTA per SM, 128x256 output tiles. A stage holds 32 elements
// of K of both operands, three planes each (72 KB, 3 stages), and feeds 12 MMAs
// of 128x256x16. Each stage accumulates into its own one of two 256-column
// TMEM accumulators; sixteen warps read it back (64 columns of a row per
// thread), add it to fp32 registers and finish the tile, while the MMA warp
// fills the other one. Their code is unrolled over the sums a thread holds, so
// 64 columns a thread and sixteen warps (against 128 and eight) halve it and
// double the warps that hide its latencies. 128x128 tiles (4 stages, 4 accumulators) were bound by
// the issuing thread: 12 MMAs of 64 cycles take it 750 cycles to issue, and the
// waits and commits of a stage another 550 that nothing overlapped.
template <int kKind>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    f32_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                    const F32Params p) {
  constexpr bool kAMN = kKind == kDW, kBMN = kKind == kDH || kKind == kDW;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t *gbase = smem_raw + (base - raw);
  SmemCtl *ctl = reinterpret_cast<SmemCtl *>(gbase + size_t(STAGES) * STAGE_BYTES);
  volatile int *abort = &ctl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int a = 0; a < ACCS; ++a) {
      mbar_init(smem_u32(&ctl->acc_full[a]), 1);
      mbar_init(smem_u32(&ctl->acc_empty[a]), 512);
    }
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), TMEM_COLS);
    tmem_relinquish();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_map(&map_a);
    tma_prefetch_map(&map_b);
  }
  grid_wait_long();
  if (threadIdx.x == 0) {
    const unsigned ca = p.range[kKind == kDH || kKind == kDW ? kOpDZ : kOpH];
    const unsigned cb = p.range[kKind == kDW ? kOpH : kOpW];
    ctl->abort = ca + cb > SAFE_CLASSES;
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = ctl->tmem_base;
  const bool use_fma = ctl->abort != 0;

  int nM = p.nM, nK = p.nK;
  int64_t rows = p.rows;
  if (p.m_count) {
    rows = *p.m_count;
    nM = int((rows + TM - 1) / TM);
  }
  int64_t K = kKind == kDH ? p.vc : p.h;
  if constexpr (kKind == kDW) {
    K = *p.k_count;
    nK = int((K + KB - 1) / KB);
  }
  const bool nothing = kKind == kDW && nK == 0 && p.accumulate;  // an empty contraction adds nothing
  const int all_items = nothing ? 0 : nM * p.nN * p.splits;
  const int items = use_fma ? 0 : all_items;
  // 64-column boxes of B that tile n of an MN-major B holds: the last tile of
  // an odd extent loads and multiplies only those (K-major B: always 4)
  auto boxes = [&](int n) { return kBMN ? min(TN / 64, (p.cols - n * TN + 63) / 64) : TN / 64; };

  if (warp < 4) {
    if (use_fma) fma_produce<kKind>(p, rows, K, nM, all_items);
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(ISSUE_REGS));
    if (warp == 0 && lane == 0) {
      // ---------------------------------------------------------- TMA producer
      int stage = 0;
      uint32_t phase = 0, issued = 0, issued_phase = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const int sp = it % p.splits;
        int m, n;
        tile_of(it / p.splits, p, nM, m, n);
        const int nb = boxes(n);
        const int kend = int(int64_t(nK) * (sp + 1) / p.splits);
        for (int kb = int(int64_t(nK) * sp / p.splits); kb < kend; ++kb) {
          if (!mbar_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort, p.err)) {
            ok = false;
            break;
          }
          const uint32_t fb = smem_u32(&ctl->full[stage]);
          issued |= 1u << stage;
          issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
          mbar_arrive_expect_tx(fb, A_BYTES + uint32_t(nb) * MN_BOX);
          const uint32_t sa = base + uint32_t(stage) * STAGE_BYTES, sb = sa + A_BYTES;
          const int k0 = kb * KB;
          if constexpr (kAMN) {
            tma_load_3d(sa, &map_a, fb, m * TM, k0, 0);
            tma_load_3d(sa + MN_BOX, &map_a, fb, m * TM + 64, k0, 0);
          } else {
            tma_load_3d(sa, &map_a, fb, k0, m * TM, 0);
          }
          if constexpr (kBMN) {
            for (int j = 0; j < nb; ++j) tma_load_3d(sb + j * MN_BOX, &map_b, fb, n * TN + 64 * j, k0, 0);
          } else {
            tma_load_3d(sb, &map_b, fb, k0, n * TN, 0);
          }
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) {
        // let the copies already in flight land before the CTA can exit
        for (int s = 0; s < STAGES; ++s) {
          if (!((issued >> s) & 1u)) continue;
          const uint32_t par = (issued_phase >> s) & 1u;
          const uint64_t t0 = globaltimer_ns();
          while (!mbar_try_wait(smem_u32(&ctl->full[s]), par) && globaltimer_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
    if (warp == 1 && lane == 0) {
      // ---------------------------------------------------------- MMA issuer
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const int sp = it % p.splits;
        int m, n;
        tile_of(it / p.splits, p, nM, m, n);
        const uint32_t idesc = idesc_bf16(TM, 64 * boxes(n), kAMN, kBMN);
        const int kend = int(int64_t(nK) * (sp + 1) / p.splits);
        for (int kb = int(int64_t(nK) * sp / p.splits); kb < kend; ++kb) {
          if (!mbar_wait(smem_u32(&ctl->acc_empty[acc]), acc_phase ^ 1u, abort, p.err) ||
              !mbar_wait(smem_u32(&ctl->full[stage]), phase, abort, p.err)) {
            ok = false;
            break;
          }
          fence_after_sync();
          const uint32_t sa = base + uint32_t(stage) * STAGE_BYTES, sb = sa + A_BYTES;
          const uint32_t d = tmem_base + uint32_t(acc) * TN;
          // smallest products first
          constexpr int pa[6] = {0, 2, 1, 0, 1, 0}, pb[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
          for (int q = 0; q < 6; ++q) {
#pragma unroll
            for (int kk = 0; kk < KB / 16; ++kk) {
              const uint64_t ad = kAMN ? sdesc_sw128(sa + pa[q] * (KB * 128u) + kk * 2048u, MN_BOX, 1024u)
                                       : sdesc_sw64(sa + pa[q] * PLANE_A + kk * 32u);
              const uint64_t bd = kBMN ? sdesc_sw128(sb + pb[q] * (KB * 128u) + kk * 2048u, MN_BOX, 1024u)
                                       : sdesc_sw64(sb + pb[q] * PLANE_B + kk * 32u);
              mma_bf16(d, ad, bd, idesc, (q | kk) != 0 ? 1u : 0u);
            }
          }
          mma_commit(smem_u32(&ctl->empty[stage]));
          mma_commit(smem_u32(&ctl->acc_full[acc]));
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
          if (++acc == ACCS) {
            acc = 0;
            acc_phase ^= 1u;
          }
        }
      }
    }
  } else {
    if (use_fma) fma_consume<kKind>(p, rows, K, nM, all_items);
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(SUM_REGS));
    // ------------------------------------------------------------ accumulate and finish
    const int quad = warp & 3;  // TMEM lane quadrant this warp may access
    const int quarter = (warp - 4) >> 2;
    const int r = quad * 32 + lane;
    int a = 0;
    uint32_t a_phase = 0;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
      const int sp = it % p.splits;
      int m, n;
      tile_of(it / p.splits, p, nM, m, n);
      const int64_t row0 = int64_t(m) * TM, row = row0 + r;
      const bool row_ok = row < rows;
      const int col0 = n * TN + quarter * HN;
      const bool live = col0 < p.cols;  // a ragged last tile: this quarter may hold no column
      float z[HN];
#pragma unroll
      for (int j = 0; j < HN; ++j) z[j] = 0.f;
      bool ok = true;
      const int kend = int(int64_t(nK) * (sp + 1) / p.splits);
#pragma unroll 1
      for (int kb = int(int64_t(nK) * sp / p.splits); kb < kend; ++kb) {
        if (!mbar_wait(smem_u32(&ctl->acc_full[a]), a_phase, abort, p.err)) {
          ok = false;
          break;
        }
        fence_after_sync();
        const uint32_t taddr = tmem_base + (uint32_t(quad * 32) << 16) + uint32_t(a) * TN + uint32_t(quarter * HN);
        if (live) {
#pragma unroll
          for (int c = 0; c < HN; c += 16) {
            uint32_t u[16];
            tmem_ld16(taddr + c, u);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) z[c + j] += __uint_as_float(u[j]);
          }
        }
        fence_before_sync();
        mbar_arrive(smem_u32(&ctl->acc_empty[a]));
        if (++a == ACCS) {
          a = 0;
          a_phase ^= 1u;
        }
      }
      if (!ok) break;
      if (!live) continue;
      const int64_t tok = (row_ok && p.row_idx) ? int64_t(ld(p.row_idx + row)) : row;

      if constexpr (kKind == kLogits) {
        const int valid = p.cols - col0;  // > 0
        const int rel = row_ok ? ld(p.y + tok) - p.v0 - col0 : -1;
        if (rel >= 0 && rel < HN && rel < valid) {
          float v = z[0];
#pragma unroll
          for (int j = 1; j < HN; ++j) v = j == rel ? z[j] : v;
          p.zy[row] = v;
        }
        if (valid < HN) {
#pragma unroll
          for (int j = 0; j < HN; ++j) z[j] = j < valid ? z[j] : -INFINITY;
        }
        float mx = z[0];
#pragma unroll
        for (int j = 1; j < HN; ++j) mx = fmaxf(mx, z[j]);
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < HN; ++j) s[j & 3] += expf(z[j] - mx);
        if (row_ok)
          p.part[int64_t(p.tile0 + 4 * n + quarter) * p.part_ld + row] = make_float2(mx, (s[0] + s[1]) + (s[2] + s[3]));
      } else if constexpr (kKind == kDLogits) {
        float g = 0.f, l = 0.f;
        int yy = -1;
        if (row_ok) {
          g = ld(p.G + tok);
          l = ld(p.lse + tok);
          yy = ld(p.y + tok) - p.v0 - col0;
        }
        float most = 0.f;
#pragma unroll
        for (int j = 0; j < HN; ++j) {
          z[j] = g != 0.f ? g * ((j == yy ? 1.f : 0.f) - expf(z[j] - l)) : 0.f;
          most = larger(most, z[j]);
        }
        raise_class(p.range + kOpDZ, most);
        // a thread's 16 columns of a plane are one 32-byte sector; the planes'
        // pitch is a multiple of the tile, and every row of a tile exists
        __nv_bfloat16 *dst = p.dz + row * p.ldz + col0;
#pragma unroll
        for (int c = 0; c < HN; c += 16) {
#pragma unroll
          for (int q = 0; q < PL; ++q) {
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float &x0 = z[c + 2 * i], &x1 = z[c + 2 * i + 1];
              pk[i] = pack2(x0, x1);
              if (q < 2) {
                x0 -= __uint_as_float(pk[i] << 16);
                x1 -= __uint_as_float(pk[i] & 0xffff0000u);
              }
            }
            store_sector(dst + q * p.dz_plane + c, pk);
          }
        }
      } else if (row_ok) {
        float *dst = p.out + sp * p.out_split + row * p.ldo + col0;
        const int valid = min(HN, p.cols - col0);
        // rows of whole 32-byte sectors: 8 floats per access
        const bool sectors = (p.ldo & 7) == 0 && (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0;
#pragma unroll
        for (int c = 0; c < HN; c += 8) {
          if (sectors && c + 8 <= valid) {
            if (p.accumulate) {
              uint32_t o[8];
              load_sector(dst + c, o);
#pragma unroll
              for (int i = 0; i < 8; ++i) z[c + i] += __uint_as_float(o[i]);
            }
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) pk[i] = __float_as_uint(z[c + i]);
            store_sector(dst + c, pk);
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (c + i < valid) dst[c + i] = p.accumulate ? dst[c + i] + z[c + i] : z[c + i];
          }
        }
      }
    }
  }

  fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    fence_after_sync();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// out[t][c] (+)= sum over the splits of part[split][row of t][c] (fixed order);
// pos (nullable): token -> row, or -1 (zeros). A warp per token; rows of part
// are 16-byte aligned.
__global__ void __launch_bounds__(256) f32_reduce_kernel(const float *part, int splits, int64_t split_stride,
                                                         int64_t ldp, const int *pos, int64_t rows, int h, float *out,
                                                         int accumulate) {
  grid_wait();
  const int lane = threadIdx.x & 31;
  const bool wide = (h & 3) == 0 && aligned16_dev(out);
  for (int64_t t = int64_t(blockIdx.x) * 8 + (threadIdx.x >> 5); t < rows; t += int64_t(gridDim.x) * 8) {
    const int64_t i = pos ? int64_t(ld(pos + t)) : t;
    const float *src = part + i * ldp;
    float *dst = out + t * h;
    for (int c = lane * 4; c < h; c += 128) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i >= 0) {
        s = __ldcs(reinterpret_cast<const float4 *>(src + c));
        for (int k = 1; k < splits; ++k) {
          const float4 v = __ldcs(reinterpret_cast<const float4 *>(src + k * split_stride + c));
          s.x += v.x;
          s.y += v.y;
          s.z += v.z;
          s.w += v.w;
        }
      }
      if (wide) {
        if (accumulate) {
          const float4 o = *reinterpret_cast<const float4 *>(dst + c);
          s = make_float4(o.x + s.x, o.y + s.y, o.z + s.z, o.w + s.w);
        }
        *reinterpret_cast<float4 *>(dst + c) = s;
      } else {
        const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c + j < h) dst[c + j] = accumulate ? dst[c + j] + v[j] : v[j];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// Planes [3][rows][pitch] (bf16), loaded in boxes of box_x x box_y elements of
// all three planes.
sao_status plane_map(CUtensorMap *m, const void *ptr, int64_t inner, int64_t rows, int64_t pitch, int64_t plane,
                     uint32_t box_x, uint32_t box_y) {
  auto fn = tensor_map_encoder();
  if (!fn) return fail(SAO_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  cuuint64_t dims[3] = {cuuint64_t(inner), cuuint64_t(rows), PL};
  cuuint64_t strides[2] = {cuuint64_t(pitch) * 2, cuuint64_t(plane) * 2};
  cuuint32_t box[3] = {box_x, box_y, PL};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapSwizzle sw = box_x * 2 == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(SAO_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", int(r));
  return SAO_OK;
}

template <int kKind>
sao_status launch_f32(const char *name, const CUtensorMap &ma, const CUtensorMap &mb, const F32Params &p,
                      cudaStream_t s) {
  DeviceInfo di;
  SAO_TRY(device_info(&di));
  static PerDevice<cudaError_t> set_up;
  const cudaError_t e = set_up.get(di.device, [] {
    return cudaFuncSetAttribute(f32_gemm_kernel<kKind>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SMEM_BYTES));
  });
  if (e != cudaSuccess) return fail(SAO_ERR_CUDA, "kernel set-up: %s", cudaGetErrorString(e));
  const int64_t items = int64_t(p.nM) * p.nN * p.splits;
  if (items == 0) return SAO_OK;
  const int grid = items < di.sm_count ? int(items) : di.sm_count;
  int slot = launch_begin(name, s);
  pdl(f32_gemm_kernel<kKind>, grid, NUM_THREADS, SMEM_BYTES, s)(ma, mb, p);
  return launch_end(slot, s);
}

int64_t up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Sizes of the fp32 path for one problem, from N, h, V and the dZ budget alone
// (the same on every device, so the results are too).
struct F32Plan {
  int64_t cap;    // rows of the H and dZ planes: N rounded up to the tile
  int hp;         // plane pitch of H and W: h rounded up to 8 elements (TMA row pitch)
  int hq;         // pitch of the partial outputs
  int vc_fwd;     // vocabulary rows of W split at a time by the forward ...
  int vc_bwd;     // ... and columns of dZ held by the backward: multiples of the tile
  int s_dh, s_dw; // parts that K is cut into
  bool dw_parts;  // dW through a padded buffer: several parts, or rows that are not whole 32-byte sectors
};

F32Plan f32_plan(int64_t N, int32_t h, int32_t V) {
  F32Plan q;
  q.cap = up(N > 0 ? N : 1, TM);
  q.hp = int(up(h, 8));
  q.hq = int(up(h, 8));
  const int64_t vpad = up(V, TN);
  const int64_t budget = int64_t(dz_budget());
  auto chunk = [&](int64_t row_bytes) {
    int64_t v = budget / row_bytes / TN * TN;
    return int(v < TN ? TN : v > vpad ? vpad : v);
  };
  q.vc_fwd = chunk(int64_t(PL) * 2 * q.hp);
  // the backward holds a chunk of W as well: with fewer rows than h that is the larger
  q.vc_bwd = chunk(int64_t(PL) * 2 * (q.cap > q.hp ? q.cap : int64_t(q.hp)));
  const int64_t nm = q.cap / TM, nh = up(h, TN) / TN, nv = up(q.vc_bwd, TM) / TM;
  q.s_dh = k_splits(nm * nh, q.vc_bwd < V ? q.vc_bwd : V, 300, 16);
  q.s_dw = k_splits(nv * nh, N, 300, 16);
  q.dw_parts = q.s_dw > 1 || (h & 7) != 0;
  return q;
}

}  // namespace

size_t f32_ws_bytes(int64_t N, int32_t h, int32_t V) {
  const F32Plan q = f32_plan(N, h, V);
  const int64_t nvt = (int64_t(V) + HN - 1) / HN;
  const size_t hplanes = round256(size_t(PL) * size_t(q.cap) * size_t(q.hp) * 2);
  const size_t common = 256 + list_ws_bytes(N) + hplanes;
  const size_t fwd = common + round256(size_t(PL) * size_t(q.vc_fwd) * size_t(q.hp) * 2) +
                     round256(sizeof(float2) * size_t(nvt) * size_t(N)) + round256(sizeof(float) * size_t(N));
  size_t bwd = common + round256(size_t(PL) * size_t(q.vc_bwd) * size_t(q.hp) * 2) +
               round256(size_t(PL) * size_t(q.cap) * size_t(q.vc_bwd) * 2) +
               round256(sizeof(float) * size_t(q.s_dh) * size_t(q.cap) * size_t(q.hq));
  if (q.dw_parts) bwd += round256(sizeof(float) * size_t(q.s_dw) * size_t(q.vc_bwd) * size_t(q.hq));
  return fwd > bwd ? fwd : bwd;
}

namespace {

// Planes of the rows of H listed in `list` (all of them without one) and of
// W[v0 .. v0 + vc).
sao_status split_launch(const float *H, const RowList *list, int64_t N, const float *W, int vc, int vcap, int h,
                        const F32Plan &q, __nv_bfloat16 *hpl, __nv_bfloat16 *wpl, bool with_h, unsigned int *range,
                        cudaStream_t s) {
  DeviceInfo di;
  SAO_TRY(device_info(&di));
  const int64_t per = int64_t(256) * 4;
  const int64_t most = int64_t(di.sm_count) * 8;
  auto blocks = [&](int64_t rows) {
    const int64_t b = (rows * (q.hp / 4) + per - 1) / per;
    return int(b < 1 ? 1 : b > most ? most : b);
  };
  SplitSrc a{H, list ? list->idx : nullptr, list ? list->count : nullptr, N, q.cap, hpl, q.cap * q.hp};
  SplitSrc b{W, nullptr, nullptr, vc, vc, wpl, int64_t(vcap) * q.hp};
  const int ba = with_h ? blocks(q.cap) : 0;
  int slot = launch_begin("f32_split", s);
  pdl(f32_split_kernel, unsigned(ba + blocks(vc)), 256, 0, s)(a, b, ba, h, q.hp, range);
  return launch_end(slot, s);
}

}  // namespace

sao_status f32_fwd(const float *H, const float *W, const int32_t *y, const uint8_t *row_mask, int64_t N, int32_t h,
                   int32_t V, float *logp, float *lse, unsigned int *err, void *ws, size_t ws_bytes,
                   cudaStream_t s) {
  if (N > MAX_ROWS) return fail(SAO_ERR_SHAPE, "fp32 path supports at most %lld tokens", (long long)MAX_ROWS);
  const F32Plan q = f32_plan(N, h, V);
  const int nvt = (V + HN - 1) / HN;  // partials: quarter tiles that hold a column
  Carver c(ws, ws_bytes);
  unsigned int *range = c.take<unsigned int>(kOperands);
  RowList list{};
  SAO_TRY(clear_scratch(range, kOperands * sizeof(unsigned int), s));
  // Rows left out save nothing while all of them fit in one wave of 152 tiles, and listing
  // them is two launches (200 rows of h = 96, V = 1000: 19.3 us with the list, 14.5
  // without); the merge then skips them.
  const bool listed = row_mask && q.cap / TM * ((int64_t(V) + TN - 1) / TN) > 152;
  if (listed) SAO_TRY(list_rows(row_mask, nullptr, N, &list, c, s));
  __nv_bfloat16 *hpl = c.take<__nv_bfloat16>(size_t(PL) * size_t(q.cap) * size_t(q.hp));
  __nv_bfloat16 *wpl = c.take<__nv_bfloat16>(size_t(PL) * size_t(q.vc_fwd) * size_t(q.hp));
  float2 *part = c.take<float2>(size_t(nvt) * size_t(N));
  float *zy = c.take<float>(size_t(N));
  if (!c.ok()) return fail(SAO_ERR_WORKSPACE, "workspace too small for the fp32 log-prob forward");
  CUtensorMap ma, mb;
  SAO_TRY(plane_map(&ma, hpl, h, q.cap, q.hp, q.cap * q.hp, KB, TM));
  for (int v0 = 0; v0 < V; v0 += q.vc_fwd) {
    const int vc = V - v0 < q.vc_fwd ? V - v0 : q.vc_fwd;
    SAO_TRY(split_launch(H, listed ? &list : nullptr, N, W + int64_t(v0) * h, vc, q.vc_fwd, h, q, hpl, wpl, v0 == 0,
                         range, s));
    SAO_TRY(plane_map(&mb, wpl, h, vc, q.hp, int64_t(q.vc_fwd) * q.hp, KB, TN));
    F32Params p{};
    p.nM = int(q.cap / TM);
    p.nN = (vc + TN - 1) / TN;
    p.nK = (h + KB - 1) / KB;
    p.splits = 1;
    p.group_m = 32;
    p.rows = N;
    p.cols = vc;
    p.m_count = listed ? list.count : nullptr;
    p.row_idx = listed ? list.idx : nullptr;
    p.H = H;
    p.W = W + int64_t(v0) * h;
    p.h = h;
    p.vc = vc;
    p.y = y;
    p.v0 = v0;
    p.tile0 = v0 / HN;
    p.part = part;
    p.part_ld = N;
    p.zy = zy;
    p.range = range;
    p.err = err;
    SAO_TRY((launch_f32<kLogits>("f32_logits_fwd", ma, mb, p, s)));
  }
  return lse_merge_launch(part, nvt, zy, y, listed ? nullptr : row_mask, listed ? list.pos : nullptr, N, V, logp, lse,
                          err, s);
}

sao_status f32_bwd(const float *H, const float *W, const int32_t *y, const float *lse, const float *G, int64_t N,
                   int32_t h, int32_t V, float *dH, float *dW, int accumulate, unsigned int *err, void *ws,
                   size_t ws_bytes, cudaStream_t s) {
  if (N > MAX_ROWS || (int64_t(h) + 63) / 64 > 65535) return fail(SAO_ERR_SHAPE, "fp32 path size limit exceeded");
  const F32Plan q = f32_plan(N, h, V);
  Carver c(ws, ws_bytes);
  unsigned int *range = c.take<unsigned int>(kOperands);
  RowList list{};
  SAO_TRY(clear_scratch(range, kOperands * sizeof(unsigned int), s));
  SAO_TRY(list_rows(nullptr, G, N, &list, c, s));
  __nv_bfloat16 *hpl = c.take<__nv_bfloat16>(size_t(PL) * size_t(q.cap) * size_t(q.hp));
  __nv_bfloat16 *wpl = c.take<__nv_bfloat16>(size_t(PL) * size_t(q.vc_bwd) * size_t(q.hp));
  __nv_bfloat16 *dz = c.take<__nv_bfloat16>(size_t(PL) * size_t(q.cap) * size_t(q.vc_bwd));
  float *dh_part = c.take<float>(size_t(q.s_dh) * size_t(q.cap) * size_t(q.hq));
  float *dw_part = q.dw_parts ? c.take<float>(size_t(q.s_dw) * size_t(q.vc_bwd) * size_t(q.hq)) : nullptr;
  if (!c.ok()) return fail(SAO_ERR_WORKSPACE, "workspace too small for the fp32 log-prob backward");
  const int64_t hplane = q.cap * q.hp, wplane = int64_t(q.vc_bwd) * q.hp, zplane = q.cap * int64_t(q.vc_bwd);
  CUtensorMap mH_K, mH_MN, mW_K, mW_MN, mZ_K, mZ_MN;
  SAO_TRY(plane_map(&mH_K, hpl, h, q.cap, q.hp, hplane, KB, TM));
  SAO_TRY(plane_map(&mH_MN, hpl, h, q.cap, q.hp, hplane, 64, KB));
  DeviceInfo di;
  SAO_TRY(device_info(&di));

  F32Params b{};
  b.H = H;
  b.h = h;
  b.y = y;
  b.lse = lse;
  b.G = G;
  b.row_idx = list.idx;
  b.dz = dz;
  b.ldz = q.vc_bwd;
  b.dz_plane = zplane;
  b.range = range;
  b.err = err;
  for (int v0 = 0; v0 < V; v0 += q.vc_bwd) {
    const int vc = V - v0 < q.vc_bwd ? V - v0 : q.vc_bwd;
    const float *Wc = W + int64_t(v0) * h;
    SAO_TRY(split_launch(H, &list, N, Wc, vc, q.vc_bwd, h, q, hpl, wpl, v0 == 0, range, s));
    SAO_TRY(plane_map(&mW_K, wpl, h, vc, q.hp, wplane, KB, TN));
    SAO_TRY(plane_map(&mW_MN, wpl, h, vc, q.hp, wplane, 64, KB));
    SAO_TRY(plane_map(&mZ_K, dz, vc, q.cap, q.vc_bwd, zplane, KB, TM));
    SAO_TRY(plane_map(&mZ_MN, dz, vc, q.cap, q.vc_bwd, zplane, 64, KB));
    b.W = Wc;
    b.vc = vc;
    b.v0 = v0;
    {  // dZ, active rows x chunk
      F32Params p = b;
      p.nM = int(q.cap / TM);
      p.nN = (vc + TN - 1) / TN;
      p.nK = (h + KB - 1) / KB;
      p.splits = 1;
      p.group_m = 32;
      p.rows = q.cap;
      p.cols = vc;
      p.m_count = list.count;
      SAO_TRY((launch_f32<kDLogits>("f32_dlogits", mH_K, mW_K, p, s)));
    }
    {  // dH parts (+)= dZ W
      F32Params p = b;
      p.nM = int(q.cap / TM);
      p.nN = (h + TN - 1) / TN;
      p.nK = (vc + KB - 1) / KB;
      p.splits = q.s_dh;
      p.group_m = 1;
      p.rows = q.cap;
      p.cols = h;
      p.m_count = list.count;
      p.out = dh_part;
      p.ldo = q.hq;
      p.out_split = q.cap * int64_t(q.hq);
      p.accumulate = v0 > 0;
      SAO_TRY((launch_f32<kDH>("f32_dH_gemm", mZ_K, mW_MN, p, s)));
    }
    {  // dW[v0 ..) (+)= dZ^T H
      F32Params p = b;
      p.nM = (vc + TM - 1) / TM;
      p.nN = (h + TN - 1) / TN;
      p.nK = int(q.cap / KB);
      p.splits = q.s_dw;
      p.group_m = 1;
      p.rows = vc;
      p.cols = h;
      p.k_count = list.count;
      float *dst = dW + int64_t(v0) * h;
      p.out = q.dw_parts ? dw_part : dst;
      p.ldo = q.dw_parts ? q.hq : h;
      p.out_split = int64_t(q.vc_bwd) * q.hq;
      p.accumulate = q.dw_parts ? 0 : accumulate;
      SAO_TRY((launch_f32<kDW>("f32_dW_gemm", mZ_MN, mH_MN, p, s)));
      if (q.dw_parts) {
        int slot = launch_begin("f32_reduce", s);
        pdl(f32_reduce_kernel, unsigned(di.sm_count * 8), 256, 0, s)(dw_part, q.s_dw, p.out_split, q.hq, nullptr, vc, h,
                                                                    dst, accumulate);
        SAO_TRY(launch_end(slot, s));
      }
    }
  }
  int slot = launch_begin("f32_reduce", s);
  pdl(f32_reduce_kernel, unsigned(di.sm_count * 8), 256, 0, s)(dh_part, q.s_dh, q.cap * int64_t(q.hq), q.hq, list.pos,
                                                              N, h, dH, 0);
  return launch_end(slot, s);
}

}  // namespace sao
