// Policy loss (Eq. 1-3, §3.1), the decoupled three-policy objective that DIS
// simplifies (§3.1) and value loss (Preliminaries, §4.4) kernels.
//
// Each loss is an operation on one token (struct Policy, Decoupled, Value) run
// by one of two kernels:
//   - token_cluster_kernel, few tokens: one cluster of 8 CTAs counts the action
//     tokens (the normaliser, unless the caller passes its own), runs over the
//     tokens and adds its partial sums through distributed shared memory, one
//     launch in all;
//   - token_kernel: 16-byte vector loads of four tokens at a time, a grid of a
//     few CTAs per SM striding over the input, per-CTA partial sums written to
//     the workspace and added in a fixed order by the CTA that finishes last.
//     When the normaliser is not given, a count pass (1 byte per token) runs
//     first, so the per-token outputs are scaled in the pass that computes them.
// Every result is deterministic.
//
// These calls at the size of a training step are launches and latencies, not
// bytes; see kClusterTokens for both sides of the line.
#include <stdint.h>

#include <atomic>

#include "sao_common.cuh"
#include "sao_internal.h"

namespace sao {
namespace {

constexpr int kThreads = 256;
constexpr int kCluster = 8, kClusterThreads = 1024;

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
// s = a + b rounded, e = the rounding error (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// Compensated fp32 accumulator: sums a thread's terms with about twice fp32 precision.
struct Acc2 {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    float e;
    two_sum(hi, x, hi, e);
    lo = __fadd_rn(lo, e);
  }
};
// A thread's sum as hi + lo + c: adding two of them loses about 2^-72 of their size.
struct Acc3 {
  float hi, lo, c;
  __device__ __forceinline__ void merge(const Acc3 &o) {
    float e, f, g;
    two_sum(hi, o.hi, hi, e);
    two_sum(lo, o.lo, lo, f);
    two_sum(lo, e, lo, g);
    c = __fadd_rn(__fadd_rn(c, o.c), __fadd_rn(f, g));
  }
};

// Sums over a CTA in fp64, whose range and 53 bits the results keep (merged as fp32
// pairs, the EV sums of 65,536 tokens were 2.8e-15 off against 8.5e-16, and NaN
// above 3.4e38). GB300 adds or converts fp64 at two lanes a clock and SM, idle
// lanes included: a value from every thread goes through shared memory, and kN / 8
// full lanes add eight each, where a shuffle tree would spend 32 lanes on each of
// its steps. The sum of v[k] is returned in lane 0 of warp k.
template <int kN>
__device__ __forceinline__ double pairwise(const double *v, int stride) {
  if constexpr (kN == 1) return *v;
  else return pairwise<kN / 2>(v, stride) + pairwise<kN / 2>(v + kN / 2 * stride, stride);
}
template <int kN, int kS, int kLd>
__device__ __forceinline__ double column_sums(double (&v)[kS][kLd]) {
  constexpr int kLeft = kN >= 256 ? kN / 8 : kN;
  const int t = threadIdx.x, w = t >> 5, l = t & 31;
  __syncthreads();
  if constexpr (kLeft < kN) {
    if (t < kS * kLeft) {
      double *c = &v[t / kLeft][t % kLeft];
      *c = pairwise<8>(c, kLeft);
    }
    __syncthreads();
  }
  double r = 0.0;
  if (w < kS) {
    r = pairwise<kLeft / 32>(&v[w][l], 32);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;
}
template <int kT, int kS>
__device__ __forceinline__ double block_sums(const double (&x)[kS]) {
  __shared__ double v[kS][kT];
#pragma unroll
  for (int k = 0; k < kS; ++k) v[k][threadIdx.x] = x[k];
  return column_sums<kT>(v);
}
// Four sums held in fp32 parts: those of four threads are merged in fp32 first (a
// quarter of each where a warp holds large ones, so that the sum overflows no earlier
// than one of them; small ones whole, a quarter might not be exact), each of the threads taking one sum of the four, which it turns into fp64. (Value loss of
// 65,536 tokens by one cluster, every thread converting its four sums: 14.3 us.)
template <int kT>
__device__ __forceinline__ double block_sums(const Acc3 (&x)[4]) {
  constexpr int kN = kT / 4;
  __shared__ double v[4][kN + 8];  // (padded: a warp's four rows in different banks)
  const int t = threadIdx.x;
  uint32_t bits = 0u;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    bits |= __float_as_uint(x[k].hi) | __float_as_uint(x[k].lo) | __float_as_uint(x[k].c);
  double r = 0.0;
  if (__any_sync(0xffffffffu, bits != 0u)) {  // (most warps of a short call hold zeros)
    const float most = fmaxf(fmaxf(fabsf(x[0].hi), fabsf(x[1].hi)), fmaxf(fabsf(x[2].hi), fabsf(x[3].hi)));
    const bool large = __any_sync(0xffffffffu, most >= 0x1p100f);
    const float q = large ? 0.25f : 1.f;
    auto part = [q](const Acc3 &a) { return Acc3{q * a.hi, q * a.lo, q * a.c}; };
    auto either = [](bool first, const Acc3 &a, const Acc3 &b) {
      return Acc3{first ? a.hi : b.hi, first ? a.lo : b.lo, first ? a.c : b.c};
    };
    auto from = [](const Acc3 &a, int o) {
      return Acc3{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o),
                  __shfl_xor_sync(0xffffffffu, a.c, o)};
    };
    Acc3 y[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {  // odd lanes go on with sums 2 and 3, even ones with 0 and 1
      const Acc3 a = part(x[i]), b = part(x[2 + i]);
      y[i] = either(t & 1, b, a);
      y[i].merge(from(either(t & 1, a, b), 1));
    }
    Acc3 z = either(t & 2, y[1], y[0]);
    z.merge(from(either(t & 2, y[0], y[1]), 2));
    r = double(z.hi) + (double(z.lo) + double(z.c));
    if (large) r *= 4.0;
  }
  v[2 * (t & 1) + (t >> 1 & 1)][t >> 2] = r;
  return column_sums<kN>(v);
}

// Per-CTA totals of kS sums and kC counts, in shared memory: written by every
// thread of the CTA together, complete after the last barrier in here.
template <int kS, int kC>
struct Totals {
  double s[kS];
  long long c[kC];
};
template <int kT, class S, class C, int kS, int kC>
__device__ __forceinline__ void block_totals(const S (&s)[kS], const C (&c)[kC], Totals<kS, kC> &out) {
  __shared__ long long sh_c[kC][kT / 32];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kC; ++k) {
    long long v;
    if constexpr (sizeof(C) == 4) {
      v = __reduce_add_sync(0xffffffffu, c[k]);
    } else {  // in two parts, whose sums over a warp fit in 32 bits (counts are below 2^31)
      v = (long long)__reduce_add_sync(0xffffffffu, unsigned(c[k] & 0xffff)) +
          ((long long)__reduce_add_sync(0xffffffffu, unsigned(c[k] >> 16)) << 16);
    }
    if (l == 0) sh_c[k][w] = v;
  }
  const double r = block_sums<kT>(s);  // (its barriers also order sh_c)
  if (l == 0 && w < kS) out.s[w] = r;
  if (threadIdx.x < kC) {
    long long v = 0;
#pragma unroll
    for (int i = 0; i < kT / 32; ++i) v += sh_c[threadIdx.x][i];
    out.c[threadIdx.x] = v;
  }
  __syncthreads();
}

// Mask bytes that are not 0 among 16 (or 4).
__device__ __forceinline__ int nonzero_bytes(uint32_t w) {
  return __popc(((w & 0x7f7f7f7fu) + 0x7f7f7f7fu | w) & 0x80808080u);
}

// Action tokens among this thread's share of the mask: 16 bytes at a time between
// the bytes before the first 16-byte boundary and those after the last. (Byte by byte
// off alignment, 65,536 tokens by 4 CTAs took 4 us more.)
__device__ __forceinline__ long long count_share(const uint8_t *m, int64_t N, int64_t tid, int64_t stride) {
  long long c = 0;
  const int64_t to_boundary = int64_t(-reinterpret_cast<uintptr_t>(m) & 15u);
  const int64_t head = to_boundary < N ? to_boundary : N;
  if (tid < head) c = m[tid] != 0;
  const int64_t n16 = (N - head) / 16;
  const uint4 *m16 = reinterpret_cast<const uint4 *>(m + head);
  auto count16 = [](const uint4 q) {
    return nonzero_bytes(q.x) + nonzero_bytes(q.y) + nonzero_bytes(q.z) + nonzero_bytes(q.w);
  };
  int64_t i = tid;
  // four independent 16-byte loads in flight per thread
  for (; i + 3 * stride < n16; i += 4 * stride) {
    uint4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = ld(m16 + i + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) c += count16(q[u]);
  }
  for (; i < n16; i += stride) c += count16(ld(m16 + i));
  for (int64_t t = head + n16 * 16 + tid; t < N; t += stride) c += m[t] != 0;
  return c;
}

// Sum over the CTA of one integer per thread, in every thread.
template <int kT>
__device__ __forceinline__ long long block_count(long long v) {
  __shared__ long long sh[kT / 32];
  __shared__ long long total;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    long long x = threadIdx.x < kT / 32 ? sh[threadIdx.x] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (threadIdx.x == 0) total = x;
  }
  __syncthreads();
  return total;
}

// The same for a cluster's counts of one thread each, in thread 0.
__device__ __forceinline__ int block_total(int v) {
  __shared__ int sh[kClusterThreads / 32];
  v = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  return threadIdx.x < 32 ? __reduce_add_sync(0xffffffffu, sh[threadIdx.x]) : 0;
}

// 1 / n rounded once to fp32 (0 for n = 0). Below 2^24 the fp32 division of the
// exact n gives the same bits as the fp64 one.
__device__ __forceinline__ float inverse(long long n) {
  return n <= 0 ? 0.f : n < (1 << 24) ? __fdiv_rn(1.f, float(n)) : float(1.0 / double(n));
}
// The same in every thread of the CTA. One thread divides: an fp64 division in
// each of an SM's 2,048 threads took 10 us.
__device__ __forceinline__ float block_inverse(long long n) {
  __shared__ float inv;
  if (threadIdx.x == 0) inv = inverse(n);
  __syncthreads();
  return inv;
}

// Action-token count (n_valid), one partial per CTA; clears the ticket of the
// pass that follows.
__global__ void __launch_bounds__(kThreads) count_mask_kernel(const uint8_t *m, int64_t N,
                                                             long long *partial, unsigned int *ticket) {
  grid_wait();
  const long long c = block_count<kThreads>(
      count_share(m, N, int64_t(blockIdx.x) * kThreads + threadIdx.x, int64_t(gridDim.x) * kThreads));
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = c;
    if (blockIdx.x == 0) *ticket = 0u;
  }
}

// ---------------------------------------------------------------------------
// policy loss, Eq. 1-3
// ---------------------------------------------------------------------------
struct PLToken {
  float coef;
  uint8_t flag;
};

// One token: ratio (Eq. 2), strict mask (Eq. 3), contribution to the
// surrogate -f(r) A and its derivative with f detached.
__device__ __forceinline__ PLToken pl_token(float lp, float old, float a, uint8_t m, float lo,
                                            float hi, float inv_n, float &contrib, int &n_low,
                                            int &n_high, int &n_nonfin) {
  PLToken t{0.f, SAO_FLAG_NOT_ACTION};
  if (!m) return t;
  const float d = lp - old;
  if (!isfinite(d) || !isfinite(a)) {
    t.flag = SAO_FLAG_NONFINITE;
    n_nonfin++;
    return t;
  }
  const float r = expf(d);
  if (r <= lo) {
    t.flag = SAO_FLAG_LOW;
    n_low++;
  } else if (r >= hi) {
    t.flag = SAO_FLAG_HIGH;
    n_high++;
  } else {
    const float c = r * a;
    contrib += c;
    t.flag = SAO_FLAG_IN;
    t.coef = -c * inv_n;
  }
  return t;
}

// Every operation has: kSums sums (held as Sum) and kCounts counts (the last one
// counts the action tokens); kReduce, whether they are used; vec(), whether four
// tokens can be taken with 16-byte accesses; load() and four(), or load_one() and
// one(), the tokens; sums(), the thread's sums; and finish(), which writes the
// call's results.
template <bool kBwd>
struct Policy {
  static constexpr int kSums = 1, kCounts = 4;  // sum of kept r A; low, high, non-finite, action
  static constexpr bool kReduce = !kBwd;
  using Sum = double;
  const float *logp, *old, *adv;
  float lo, hi;
  float *coef;              // may be null
  uint8_t *flags;           // may be null
  const float *grad_scale;  // bwd: device scalar
  float *loss;
  int64_t *counts;
  struct State {
    float inv_n, gscale;
    double acc = 0.0;
    int n[kCounts] = {0, 0, 0, 0};
  };
  __device__ __forceinline__ void begin(State &s, float inv_n) const {
    s.inv_n = inv_n;
    s.gscale = kBwd ? ld(grad_scale) : 1.f;
  }
  __device__ __forceinline__ bool vec(const uint8_t *m) const {
    return aligned16_dev(logp) && aligned16_dev(old) && aligned16_dev(adv) &&
           ((reinterpret_cast<uintptr_t>(m) & 3u) == 0) && (coef == nullptr || aligned16_dev(coef)) &&
           (flags == nullptr || (reinterpret_cast<uintptr_t>(flags) & 3u) == 0);
  }
  struct Four {
    float4 lp, od, ad;
    uint32_t mw;
  };
  __device__ __forceinline__ Four load(const uint8_t *m, int64_t i) const {
    return Four{ld(reinterpret_cast<const float4 *>(logp) + i), ld(reinterpret_cast<const float4 *>(old) + i),
                ld(reinterpret_cast<const float4 *>(adv) + i), ld(reinterpret_cast<const uint32_t *>(m) + i)};
  }
  __device__ __forceinline__ void four(State &s, const Four &f, int64_t i) const {
    const float4 &lp = f.lp, &od = f.od, &ad = f.ad;
    const uint32_t mw = f.mw;
    if (kReduce) s.n[3] += nonzero_bytes(mw);
    float contrib = 0.f;
    const PLToken t0 = pl_token(lp.x, od.x, ad.x, uint8_t(mw), lo, hi, s.inv_n, contrib, s.n[0], s.n[1], s.n[2]);
    const PLToken t1 = pl_token(lp.y, od.y, ad.y, uint8_t(mw >> 8), lo, hi, s.inv_n, contrib, s.n[0], s.n[1], s.n[2]);
    const PLToken t2 = pl_token(lp.z, od.z, ad.z, uint8_t(mw >> 16), lo, hi, s.inv_n, contrib, s.n[0], s.n[1], s.n[2]);
    const PLToken t3 = pl_token(lp.w, od.w, ad.w, uint8_t(mw >> 24), lo, hi, s.inv_n, contrib, s.n[0], s.n[1], s.n[2]);
    if (kReduce) s.acc += double(contrib);
    if (coef)
      reinterpret_cast<float4 *>(coef)[i] =
          make_float4(t0.coef * s.gscale, t1.coef * s.gscale, t2.coef * s.gscale, t3.coef * s.gscale);
    if (flags) reinterpret_cast<uchar4 *>(flags)[i] = make_uchar4(t0.flag, t1.flag, t2.flag, t3.flag);
  }
  struct One {
    float lp, od, ad;
    uint8_t m;
  };
  __device__ __forceinline__ One load_one(const uint8_t *m, int64_t i) const {
    return One{ld(logp + i), ld(old + i), ld(adv + i), ld(m + i)};
  }
  __device__ __forceinline__ void one(State &s, const One &f, int64_t i) const {
    float contrib = 0.f;
    if (kReduce) s.n[3] += f.m != 0;
    const PLToken t = pl_token(f.lp, f.od, f.ad, f.m, lo, hi, s.inv_n, contrib, s.n[0], s.n[1], s.n[2]);
    if (kReduce) s.acc += double(contrib);
    if (coef) coef[i] = t.coef * s.gscale;
    if (flags) flags[i] = t.flag;
  }
  __device__ __forceinline__ void sums(const State &s, double (&out)[kSums]) const { out[0] = s.acc; }
  __device__ __forceinline__ void finish(const Totals<kSums, kCounts> &t, int64_t n_norm) const {
    const long long n = n_norm > 0 ? n_norm : t.c[3];
    *loss = n > 0 ? float(-t.s[0] / double(n)) : 0.f;
    counts[0] = t.c[3];
    counts[1] = t.c[0];
    counts[2] = t.c[1];
    counts[3] = t.c[2];
  }
};

// ---------------------------------------------------------------------------
// decoupled three-policy objective (§3.1)
// ---------------------------------------------------------------------------
struct DLBounds {
  float lo, hi, wlo, whi;
};

struct DLCounts {
  int low = 0, high = 0, nonfin = 0, wlow = 0, whigh = 0;
};

// One token: the mismatch weight w = pi_old/pi_rollout must lie strictly
// inside (wlo, whi); then the clipped surrogate of r = pi_theta/pi_old, scaled
// by w. Adds the token's -loss contribution to `contrib`.
__device__ __forceinline__ PLToken dl_token(float lp, float px, float ro, float a, uint8_t m, const DLBounds &A,
                                            float inv_n, float &contrib, DLCounts &c) {
  PLToken t{0.f, SAO_FLAG_NOT_ACTION};
  if (!m) return t;
  const float d = lp - px, e = px - ro;
  if (!isfinite(d) || !isfinite(e) || !isfinite(a)) {
    t.flag = SAO_FLAG_NONFINITE;
    c.nonfin++;
    return t;
  }
  const float w = expf(e);
  if (w <= A.wlo) {
    t.flag = SAO_FLAG_MISMATCH_LOW;
    c.wlow++;
    return t;
  }
  if (w >= A.whi) {
    t.flag = SAO_FLAG_MISMATCH_HIGH;
    c.whigh++;
    return t;
  }
  const float r = expf(d);
  if (a > 0.f && r > A.hi) {
    t.flag = SAO_FLAG_HIGH;
    c.high++;
    contrib += w * (A.hi * a);
  } else if (a < 0.f && r < A.lo) {
    t.flag = SAO_FLAG_LOW;
    c.low++;
    contrib += w * (A.lo * a);
  } else {
    const float v = w * (r * a);
    contrib += v;
    t.flag = SAO_FLAG_IN;
    t.coef = -v * inv_n;
  }
  return t;
}

template <bool kBwd>
struct Decoupled {
  static constexpr int kSums = 1, kCounts = 6;  // low, high, non-finite, mismatch low, mismatch high, action
  static constexpr bool kReduce = !kBwd;
  using Sum = double;
  const float *logp, *prox, *roll, *adv;
  DLBounds b;
  float *coef;              // may be null
  uint8_t *flags;           // may be null
  const float *grad_scale;  // bwd: device scalar
  float *loss;
  int64_t *counts;
  struct State {
    float inv_n, gscale;
    double acc = 0.0;
    DLCounts c;
    int n[kCounts] = {0, 0, 0, 0, 0, 0};
  };
  __device__ __forceinline__ void begin(State &s, float inv_n) const {
    s.inv_n = inv_n;
    s.gscale = kBwd ? ld(grad_scale) : 1.f;
  }
  __device__ __forceinline__ bool vec(const uint8_t *m) const {
    return aligned16_dev(logp) && aligned16_dev(prox) && aligned16_dev(roll) && aligned16_dev(adv) &&
           ((reinterpret_cast<uintptr_t>(m) & 3u) == 0) && (coef == nullptr || aligned16_dev(coef)) &&
           (flags == nullptr || (reinterpret_cast<uintptr_t>(flags) & 3u) == 0);
  }
  struct Four {
    float4 lp, px, ro, ad;
    uint32_t mw;
  };
  __device__ __forceinline__ Four load(const uint8_t *m, int64_t i) const {
    return Four{__ldcs(reinterpret_cast<const float4 *>(logp) + i), __ldcs(reinterpret_cast<const float4 *>(prox) + i),
                __ldcs(reinterpret_cast<const float4 *>(roll) + i), __ldcs(reinterpret_cast<const float4 *>(adv) + i),
                __ldcs(reinterpret_cast<const uint32_t *>(m) + i)};
  }
  __device__ __forceinline__ void four(State &s, const Four &f, int64_t i) const {
    const float4 &lp = f.lp, &px = f.px, &ro = f.ro, &ad = f.ad;
    const uint32_t mw = f.mw;
    if (kReduce) s.n[5] += nonzero_bytes(mw);
    float contrib = 0.f;
    const PLToken t0 = dl_token(lp.x, px.x, ro.x, ad.x, uint8_t(mw), b, s.inv_n, contrib, s.c);
    const PLToken t1 = dl_token(lp.y, px.y, ro.y, ad.y, uint8_t(mw >> 8), b, s.inv_n, contrib, s.c);
    const PLToken t2 = dl_token(lp.z, px.z, ro.z, ad.z, uint8_t(mw >> 16), b, s.inv_n, contrib, s.c);
    const PLToken t3 = dl_token(lp.w, px.w, ro.w, ad.w, uint8_t(mw >> 24), b, s.inv_n, contrib, s.c);
    if (kReduce) s.acc += double(contrib);
    if (coef)
      __stcs(reinterpret_cast<float4 *>(coef) + i,
             make_float4(t0.coef * s.gscale, t1.coef * s.gscale, t2.coef * s.gscale, t3.coef * s.gscale));
    if (flags) reinterpret_cast<uchar4 *>(flags)[i] = make_uchar4(t0.flag, t1.flag, t2.flag, t3.flag);
  }
  struct One {
    float lp, px, ro, ad;
    uint8_t m;
  };
  __device__ __forceinline__ One load_one(const uint8_t *m, int64_t i) const {
    return One{ld(logp + i), ld(prox + i), ld(roll + i), ld(adv + i), ld(m + i)};
  }
  __device__ __forceinline__ void one(State &s, const One &f, int64_t i) const {
    float contrib = 0.f;
    if (kReduce) s.n[5] += f.m != 0;
    const PLToken t = dl_token(f.lp, f.px, f.ro, f.ad, f.m, b, s.inv_n, contrib, s.c);
    if (kReduce) s.acc += double(contrib);
    if (coef) coef[i] = t.coef * s.gscale;
    if (flags) flags[i] = t.flag;
  }
  __device__ __forceinline__ void sums(State &s, double (&out)[kSums]) const {
    out[0] = s.acc;
    s.n[0] = s.c.low;
    s.n[1] = s.c.high;
    s.n[2] = s.c.nonfin;
    s.n[3] = s.c.wlow;
    s.n[4] = s.c.whigh;
  }
  __device__ __forceinline__ void finish(const Totals<kSums, kCounts> &t, int64_t n_norm) const {
    const long long n = n_norm > 0 ? n_norm : t.c[5];
    *loss = n > 0 ? float(-t.s[0] / double(n)) : 0.f;
    counts[0] = t.c[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) counts[1 + j] = t.c[j];
  }
};

// ---------------------------------------------------------------------------
// value loss
// ---------------------------------------------------------------------------
// Per-token terms of the value loss and the EV sums, exact up to the final
// additions: d = V - R as an fp32 pair (two-sum), its square and R^2 as a
// rounded product plus the product's remainder (fused multiply-add), so the
// sums are fp64-grade although every operation is fp32.
struct VLTerms {
  Acc2 d2, e, r, r2;  // sum d^2 (= sum (R - V)^2), sum (R - V), sum R, sum R^2: leading parts
  float d2_lo = 0.f, e_lo = 0.f, r2_lo = 0.f;  // their small remainders, summed plainly
  __device__ __forceinline__ void add(float v, float rt) {
    const float dh = __fsub_rn(v, rt);
    const float bb = __fsub_rn(dh, v);
    const float dl = __fsub_rn(__fsub_rn(v, __fsub_rn(dh, bb)), __fadd_rn(rt, bb));  // v - rt = dh + dl exactly
    const float p = __fmul_rn(dh, dh);
    d2.add(p);
    d2_lo = __fadd_rn(d2_lo, __fmaf_rn(2.f * dh, dl, __fmaf_rn(dh, dh, -p)));
    e.add(-dh);
    e_lo = __fsub_rn(e_lo, dl);
    r.add(rt);
    const float q = __fmul_rn(rt, rt);
    r2.add(q);
    r2_lo = __fadd_rn(r2_lo, __fmaf_rn(rt, rt, -q));
  }
};

struct Value {
  static constexpr int kSums = 4, kCounts = 1;  // sum d^2, e, R, R^2; action
  static constexpr bool kReduce = true;
  using Sum = Acc3;
  const float *v, *ret;
  float *grad;
  float *loss;
  double *ev;  // may be null
  struct State {
    float two_over_n;
    VLTerms acc;
    int n[kCounts] = {0};
  };
  __device__ __forceinline__ void begin(State &s, float inv_n) const { s.two_over_n = 2.f * inv_n; }
  __device__ __forceinline__ bool vec(const uint8_t *m) const {
    return aligned16_dev(v) && aligned16_dev(ret) && aligned16_dev(grad) &&
           ((reinterpret_cast<uintptr_t>(m) & 3u) == 0);
  }
  static __device__ __forceinline__ float token(State &s, float x, float r, bool act) {
    if (!act) return 0.f;
    s.acc.add(x, r);
    return s.two_over_n * (x - r);
  }
  struct Four {
    float4 x, r;
    uint32_t mw;
  };
  __device__ __forceinline__ Four load(const uint8_t *m, int64_t i) const {
    return Four{ld(reinterpret_cast<const float4 *>(v) + i), ld(reinterpret_cast<const float4 *>(ret) + i),
                ld(reinterpret_cast<const uint32_t *>(m) + i)};
  }
  __device__ __forceinline__ void four(State &s, const Four &f, int64_t i) const {
    const float4 &x = f.x, &r = f.r;
    const uint32_t mw = f.mw;
    s.n[0] += nonzero_bytes(mw);
    float4 g;
    g.x = token(s, x.x, r.x, (mw & 0xffu) != 0u);
    g.y = token(s, x.y, r.y, (mw & 0xff00u) != 0u);
    g.z = token(s, x.z, r.z, (mw & 0xff0000u) != 0u);
    g.w = token(s, x.w, r.w, (mw & 0xff000000u) != 0u);
    reinterpret_cast<float4 *>(grad)[i] = g;
  }
  struct One {
    float x, r;
    uint8_t m;
  };
  __device__ __forceinline__ One load_one(const uint8_t *m, int64_t i) const {
    return One{ld(v + i), ld(ret + i), ld(m + i)};
  }
  __device__ __forceinline__ void one(State &s, const One &f, int64_t i) const {
    s.n[0] += f.m != 0;
    grad[i] = token(s, f.x, f.r, f.m != 0);
  }
  static __device__ __forceinline__ Acc3 joined(const Acc2 &a, float lo) {
    Acc3 r;
    r.hi = a.hi;
    two_sum(a.lo, lo, r.lo, r.c);
    return r;
  }
  __device__ __forceinline__ void sums(const State &s, Acc3 (&out)[kSums]) const {
    out[0] = joined(s.acc.d2, s.acc.d2_lo);
    out[1] = joined(s.acc.e, s.acc.e_lo);
    out[2] = Acc3{s.acc.r.hi, s.acc.r.lo, 0.f};
    out[3] = joined(s.acc.r2, s.acc.r2_lo);
  }
  __device__ __forceinline__ void finish(const Totals<kSums, kCounts> &t, int64_t n_norm) const {
    const long long n = n_norm > 0 ? n_norm : t.c[0];
    *loss = n > 0 ? float(t.s[0] / double(n)) : 0.f;
    if (ev) {
      ev[0] = t.s[1];
      ev[1] = t.s[0];  // sum (R - V)^2 = sum d^2
      ev[2] = t.s[2];
      ev[3] = t.s[3];
    }
  }
};

// ---------------------------------------------------------------------------
// the two kernels
// ---------------------------------------------------------------------------
// This thread's share of the tokens; `first` (kHave): its first four, loaded
// already where the arrays allow vectors.
template <bool kHave, class Op>
__device__ __forceinline__ void run_tokens(const Op &op, typename Op::State &s, const uint8_t *m, int64_t N,
                                           int64_t tid, int64_t stride, const typename Op::Four &first) {
  int64_t done = 0;
  if (op.vec(m)) {
    const int64_t n4 = N / 4;
    int64_t i = tid;
    if (i < n4) {
      // the next four tokens are on their way while these are worked on (value loss,
      // 2^24 tokens: 57 -> 51 us; without it the policy backward's loads wait behind
      // the stores: 4 million tokens 11.9 us against 10.5)
      typename Op::Four cur = kHave ? first : op.load(m, i);
      while (i + stride < n4) {
        const typename Op::Four next = op.load(m, i + stride);
        op.four(s, cur, i);
        cur = next;
        i += stride;
      }
      op.four(s, cur, i);
    }
    done = n4 * 4;
  }
  // the tail, or arrays off 16-byte alignment: tokens one by one, four on their way
  // (2^24 tokens off alignment, policy loss backward: 61 us, 136 with one)
  int64_t i = done + tid;
  for (; i + 3 * stride < N; i += 4 * stride) {
    typename Op::One f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) f[u] = op.load_one(m, i + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) op.one(s, f[u], i + u * stride);
  }
  for (; i < N; i += stride) op.one(s, op.load_one(m, i), i);
}

struct TokenArgs {
  const uint8_t *m;
  int64_t N;
  int64_t n_norm;              // > 0: the caller's normaliser
  const long long *cnt_partial;  // else the count pass's partials
  int n_cnt;
  unsigned int *ticket;        // CTAs that have written their partials (cleared before the launch)
  double *part_s;              // [kSums][CTAs]
  long long *part_c;           // [kCounts][CTAs]
};

template <class Op>
__global__ void __launch_bounds__(kThreads) token_kernel(const Op op, const TokenArgs a) {
  grid_wait();
  long long n = a.n_norm;
  if (n <= 0) {  // every CTA adds the same partials
    long long c = 0;
    for (int i = threadIdx.x; i < a.n_cnt; i += kThreads) c += a.cnt_partial[i];
    n = block_count<kThreads>(c);
  }
  typename Op::State s;
  op.begin(s, block_inverse(n));
  run_tokens<false>(op, s, a.m, a.N, int64_t(blockIdx.x) * kThreads + threadIdx.x, int64_t(gridDim.x) * kThreads, {});
  if constexpr (Op::kReduce) {
    __shared__ Totals<Op::kSums, Op::kCounts> t;
    {
      typename Op::Sum sums[Op::kSums];
      op.sums(s, sums);
      block_totals<kThreads>(sums, s.n, t);
    }
    __shared__ bool last;
    const int g = gridDim.x;
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 0; k < Op::kSums; ++k) a.part_s[k * g + blockIdx.x] = t.s[k];
#pragma unroll
      for (int k = 0; k < Op::kCounts; ++k) a.part_c[k * g + blockIdx.x] = t.c[k];
      __threadfence();
      last = atomicAdd(a.ticket, 1u) == unsigned(g) - 1u;
    }
    __syncthreads();
    if (!last) return;
    // the last CTA adds every CTA's partials: thread i takes i, i + 256, ...
    __threadfence();
    double sums[Op::kSums];
#pragma unroll
    for (int k = 0; k < Op::kSums; ++k) sums[k] = 0.0;
    long long c[Op::kCounts];
#pragma unroll
    for (int k = 0; k < Op::kCounts; ++k) c[k] = 0;
    for (int i = threadIdx.x; i < g; i += kThreads) {
#pragma unroll
      for (int k = 0; k < Op::kSums; ++k) sums[k] += __ldcg(a.part_s + k * g + i);
#pragma unroll
      for (int k = 0; k < Op::kCounts; ++k) c[k] += __ldcg(a.part_c + k * g + i);
    }
    block_totals<kThreads>(sums, c, t);
    if (threadIdx.x == 0) op.finish(t, a.n_norm);
  }
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The same shared variable in the CTA of cluster rank `rank`.
template <class T>
__device__ __forceinline__ T *peer_shared(T *p, unsigned rank) {
  uint64_t out;
  asm("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
  return reinterpret_cast<T *>(out);
}

// One cluster of kCluster CTAs does the whole call. A chain of latencies: the
// count, a cluster barrier, the tokens, the sums, a second barrier. So a thread's
// first tokens are loaded before the count, and what a rank reads from the others
// it reads with a lane per rank (rank after rank: about 1 us; every warp reading
// the counts for itself: as much again).
template <class Op>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kClusterThreads)
    token_cluster_kernel(const Op op, const uint8_t *m, int64_t N, int64_t n_norm) {
  grid_wait();
  __shared__ int my_count;
  __shared__ float inv;
  __shared__ Totals<Op::kSums, Op::kCounts> mine;
  const int lane = threadIdx.x & 31;
  // warps of the CTAs in turn: a short call's fp64 sums are spread over the SMs
  // (8,192 tokens in the first two CTAs: value loss 8.9 us)
  const int64_t tid = int64_t(threadIdx.x - lane) * kCluster + blockIdx.x * 32 + lane;
  constexpr int64_t stride = int64_t(kCluster) * kClusterThreads;
  typename Op::Four first{};
  if (op.vec(m) && tid < N / 4) first = op.load(m, tid);
  if (n_norm <= 0) {
    const int c = block_total(int(count_share(m, N, tid, stride)));
    if (threadIdx.x == 0) my_count = c;
    cluster_barrier();
  }
  if (threadIdx.x < 32) {
    long long n = n_norm;
    if (n <= 0) n = __reduce_add_sync(0xffffffffu, lane < kCluster ? *peer_shared(&my_count, lane) : 0);
    if (lane == 0) inv = inverse(n);
  }
  __syncthreads();
  typename Op::State s;
  op.begin(s, inv);
  run_tokens<true>(op, s, m, N, tid, stride, first);
  if constexpr (Op::kReduce) {
    typename Op::Sum sums[Op::kSums];
    op.sums(s, sums);
    block_totals<kClusterThreads>(sums, s.n, mine);
    cluster_barrier();
    if (blockIdx.x == 0 && threadIdx.x < 32) {
      // rank by rank in a fixed tree over the first lanes
      const Totals<Op::kSums, Op::kCounts> *o = peer_shared(&mine, lane % kCluster);
      Totals<Op::kSums, Op::kCounts> t;
#pragma unroll
      for (int k = 0; k < Op::kSums; ++k) {
        double v = o->s[k];
#pragma unroll
        for (int d = kCluster / 2; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        t.s[k] = v;
      }
#pragma unroll
      for (int k = 0; k < Op::kCounts; ++k)
        t.c[k] = __reduce_add_sync(0xffffffffu, lane < kCluster ? int(o->c[k]) : 0);
      if (lane == 0) op.finish(t, n_norm);
    }
  }
  cluster_barrier();  // no CTA leaves while its shared memory may still be read
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
constexpr int kMaxGrid = 4096;
constexpr int kMaxCountGrid = 1024;
// Tokens up to which one cluster does the whole call. On the GPU alone (us, one
// cluster / count pass and full grid; policy loss forward, backward, value loss,
// decoupled loss):
//   8,192    5.9 / 7.5   3.3 / 4.0   6.2 / 7.3   6.3 / 7.8
//   32,768   6.5 / 7.4   3.9 / 4.1   8.7 / 7.4   7.3 / 7.9
//   49,152   7.4 / 7.5   4.9 / 4.1   8.5 / 7.5   8.5 / 8.0
//   65,536   7.8 / 7.4   5.1 / 4.1   9.4 / 7.4   9.1 / 7.9
// A thread of the cluster has one vector up to 32,768 tokens and two above. Where
// the two are near each other, one launch instead of two is 2 us less host time,
// which is what bounds these calls on their own.
constexpr int64_t kClusterTokens = 1 << 15;

// The same for a backward whose normaliser is given, one launch in either form
// (policy loss, us: 4,097 tokens 3.0 / 3.3, 8,192 3.0 / 2.7, 32,768 3.2 / 2.8).
constexpr int64_t kClusterGivenNorm = 1 << 12;

// Tokens up to which several sums (the value loss) run with one CTA per SM rather
// than with more CTAs than the last one adds in one round of loads (256). Value
// loss, GPU alone, one CTA per SM / as many as there are vectors for, inputs in L2:
// 350,000 tokens 9.9 / 10.4 us, 2^20 10.9 / 11.9, 2^21 14.0 / 14.0; with inputs
// from HBM about 4 million tokens are 2 us slower, hence the line. (Policy loss,
// one sum: 2^20 11.4 / 11.3.)
constexpr int64_t kNarrowTokens = 1 << 20;

// CTAs of `kernel` resident on one SM of the current device (asked once per device).
template <class K>
int resident(K kernel, int device) {
  static std::atomic<int> known[64];
  int n = device < 64 ? known[device].load(std::memory_order_relaxed) : 0;
  if (n > 0) return n;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kThreads, 0) != cudaSuccess || n < 1) n = 1;
  if (device < 64) known[device].store(n, std::memory_order_relaxed);
  return n;
}

// One call: `op` over the tokens, by one cluster or by a full wave of CTAs
// (never more than 4-token vectors, at most kMaxGrid: workspace bound).
template <class Op>
sao_status launch_tokens(const char *name, const Op &op, const uint8_t *m, int64_t N, int64_t n_norm, void *ws_body,
                         size_t body_bytes, cudaStream_t s) {
  Carver c(ws_body, body_bytes);
  long long *cnt = c.take<long long>(kMaxCountGrid);
  unsigned int *ticket = c.take<unsigned int>(1);
  double *part_s = c.take<double>(size_t(Op::kSums) * kMaxGrid);
  long long *part_c = c.take<long long>(size_t(Op::kCounts) * kMaxGrid);
  if (!c.ok()) return fail(SAO_ERR_WORKSPACE, "workspace too small for %s", name);
  // a backward whose normaliser is given is one launch either way
  if (N <= (n_norm > 0 && !Op::kReduce ? kClusterGivenNorm : kClusterTokens)) {
    int slot = launch_begin(name, s);
    pdl(token_cluster_kernel<Op>, kCluster, kClusterThreads, 0, s)(op, m, N, n_norm);
    return launch_end(slot, s);
  }
  DeviceInfo di;
  SAO_TRY(device_info(&di));
  auto kernel = token_kernel<Op>;
  int64_t grid = (N / 4 + kThreads - 1) / kThreads, cap = int64_t(di.sm_count) * resident(kernel, di.device);
  if (cap > kMaxGrid) cap = kMaxGrid;
  if (grid > cap) grid = cap;
  if (Op::kSums > 1 && N <= kNarrowTokens && grid > kThreads && grid > di.sm_count) grid = di.sm_count;
  TokenArgs a{m, N, n_norm, cnt, 0, ticket, part_s, part_c};
  if (n_norm <= 0) {  // the normaliser must be known before the token pass
    int64_t cg = (N / 64 + kThreads - 1) / kThreads;
    if (cg > 4 * di.sm_count) cg = 4 * di.sm_count;
    if (cg > kMaxCountGrid) cg = kMaxCountGrid;
    a.n_cnt = int(cg);
    int slot = launch_begin("count_mask", s);
    pdl(count_mask_kernel, unsigned(cg), kThreads, 0, s)(m, N, cnt, ticket);
    SAO_TRY(launch_end(slot, s));
  } else if (Op::kReduce) {
    SAO_TRY(clear_scratch(ticket, sizeof(unsigned int), s));
  }
  int slot = launch_begin(name, s);
  pdl(kernel, unsigned(grid), kThreads, 0, s)(op, a);
  return launch_end(slot, s);
}

}  // namespace

size_t elementwise_ws_bytes(int64_t N, int) {
  (void)N;
  return round256(sizeof(long long) * kMaxCountGrid) + round256(sizeof(unsigned int)) +
         round256(4 * sizeof(double) * kMaxGrid) + round256(6 * sizeof(long long) * kMaxGrid);
}

sao_status policy_loss_launch(const float *logp, const float *old, const float *adv, const uint8_t *m,
                              int64_t N, float eps_low, float eps_high, int64_t n_norm, float *loss,
                              float *coef, uint8_t *flags, int64_t *counts, const float *grad_loss,
                              void *ws_body, size_t body_bytes, cudaStream_t s) {
  const float lo = 1.0f - eps_low, hi = 1.0f + eps_high;
  if (grad_loss)
    return launch_tokens("policy_loss_bwd", Policy<true>{logp, old, adv, lo, hi, coef, flags, grad_loss, loss, counts},
                         m, N, n_norm, ws_body, body_bytes, s);
  return launch_tokens("policy_loss_fwd", Policy<false>{logp, old, adv, lo, hi, coef, flags, nullptr, loss, counts}, m,
                       N, n_norm, ws_body, body_bytes, s);
}

sao_status decoupled_loss_launch(const float *logp, const float *prox, const float *roll, const float *adv,
                                 const uint8_t *m, int64_t N, float eps_low, float eps_high, float w_low,
                                 float w_high, int64_t n_norm, float *loss, float *coef, uint8_t *flags,
                                 int64_t *counts, const float *grad_loss, void *ws_body, size_t body_bytes,
                                 cudaStream_t s) {
  const DLBounds b{1.0f - eps_low, 1.0f + eps_high, w_low, w_high};
  if (grad_loss)
    return launch_tokens("decoupled_loss_bwd",
                         Decoupled<true>{logp, prox, roll, adv, b, coef, flags, grad_loss, loss, counts}, m, N, n_norm,
                         ws_body, body_bytes, s);
  return launch_tokens("decoupled_loss_fwd",
                       Decoupled<false>{logp, prox, roll, adv, b, coef, flags, nullptr, loss, counts}, m, N, n_norm,
                       ws_body, body_bytes, s);
}

sao_status value_loss_launch(const float *v, const float *ret, const uint8_t *m, int64_t N, int64_t n_norm,
                             float *loss, float *grad, double *ev, void *ws_body, size_t body_bytes,
                             cudaStream_t s) {
  return launch_tokens("value_loss", Value{v, ret, grad, loss, ev}, m, N, n_norm, ws_body, body_bytes, s);
}

}  // namespace sao
