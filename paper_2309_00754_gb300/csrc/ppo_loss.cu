// Update side of PPO over the scored batch (§2 "Stage 3: PPO"; Algorithms 1 and 2 optimise
// the surrogate after scoring). Per valid token t < len_s of an [S, L] batch:
//
//   r_t   = exp(logp_new_t - logp_old_t)                   probability ratio r(theta)
//   A_t   = adv_t, or (adv_t - mean) / sqrt(M2 / n + 1e-8)   with advantage whitening
//   s_t   = min(r_t A_t, clip(r_t, 1 - eps, 1 + eps) A_t)   clipped surrogate term
//   loss_clip  = -(1/n) sum s_t,   d/d logp_new_t = -r_t A_t / n where r_t A_t <= clip term
//   loss_value =  (1/n) sum (V_t - R_t)^2,   d/d V_t = 2 (V_t - R_t) / n
//
// Batches of up to kSmallTokens tokens run in one launch: a thread-block cluster that takes the
// moments, meets over distributed shared memory, runs the loss pass, meets again and writes the
// statistics. (Four chained launches cost 10 us of device time for 2048 tokens and their
// enqueueing more; the one launch 4-5 us.)
//
// Larger ones take two launches, the second a programmatic dependent launch:
//   moments:  per block, the valid count n and (with whitening) the sums of a - c and
//             (a - c)^2 over the valid advantages, c = adv[0] a common shift;
//             The caller's moments, if given, take the place of this pass: one thread turns
//             them into (mean, 1 / std, 1 / n);
//   loss:     every block merges those partials into (mean, 1 / std, 1 / n), all in the same
//             order, while its first loads are in flight; streams float4 chunks of the flattened [S, L] batch; chunks without a
//             valid token are written as zero gradients without reading the inputs; per-block
//             sums go to the workspace, and the block that finishes last merges them, in a
//             fixed order, into the statistics. (A launch of its own for either merge cost
//             2.2 and 3.1 us of the 34 us that 16384 x 400 tokens took.)
// Every grid is one wave (SMs x resident blocks), so no block waits for a second wave.
// A chunk is four consecutive tokens of the flattened batch and may straddle two rows, so row
// lengths that are not multiples of four take the same 16-byte loads.
// Per-thread sums are compensated (Kahan) fp32, block and cross-block trees fp32: GB300
// executes fp64 at a small fraction of its fp32 rate, so fp64 appears only in a few scalar
// operations of the output.
// HBM-bound: the loss pass reads 20 B per valid token and writes 8 B per token of the
// [S, L] gradient arrays; the moments pass reads 4 B per valid token with whitening.
#include <float.h>

#include "common.cuh"
#include "kernels.h"

namespace hydra {
namespace {

constexpr int kPpoThreads = 256;
constexpr int kPpoWarps = kPpoThreads / 32;
constexpr int kLossSums = 5;  // sum s, sum (V-R)^2, sum kl, sum a, sum a^2 (+ clipped count)

// Workspace layout: moments partials, loss partials, then the merged moments.
struct MomPart {
  int n;
  float s1, s2, pad;  // sums of (a - c) and (a - c)^2
};
struct LossPart {
  int nclip;
  float s[kLossSums];
  float pad[2];
};

// Partials written by the previous launch are read through L2 (ld.global.cg).
__device__ __forceinline__ MomPart load_part(const MomPart* p) {
  const int4 q = __ldcg(reinterpret_cast<const int4*>(p));
  return MomPart{q.x, __int_as_float(q.y), __int_as_float(q.z), 0.f};
}
__device__ __forceinline__ LossPart load_part(const LossPart* p) {
  const int4 a = __ldcg(reinterpret_cast<const int4*>(p));
  const int4 b = __ldcg(reinterpret_cast<const int4*>(p) + 1);
  return LossPart{a.x, {__int_as_float(a.y), __int_as_float(a.z), __int_as_float(a.w),
                        __int_as_float(b.x), __int_as_float(b.y)}, {0.f, 0.f}};
}

struct Kahan {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Fixed-shape block sums of N floats and one int; results valid in every thread.
template <int N>
__device__ __forceinline__ void block_sums(float (&v)[N], int& k, float (*sh)[kPpoWarps],
                                           int* shk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = warp_sum(v[i]);
  k = warp_sum_i(k);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) sh[i][warp] = v[i];
    shk[warp] = k;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kPpoWarps; ++w) t += sh[i][w];
    v[i] = t;
  }
  int t = 0;
#pragma unroll
  for (int w = 0; w < kPpoWarps; ++w) t += shk[w];
  k = t;
  __syncthreads();
}

__device__ __forceinline__ int clamp_length(int n, int L, int* err) {
  if (n < 0 || n > L) {
    record_error(err, kDevBadLength);
    n = n < 0 ? 0 : L;
  }
  return n;
}

__device__ __forceinline__ int row_length(const int32_t* lengths, int s, int L, int* err) {
  return clamp_length(lengths ? __ldg(lengths + s) : L, L, err);
}

// A thread's position in the flattened batch: token e = s L + t of row s, and that row's length,
// fetched one chunk ahead so that its latency overlaps the previous chunk's data loads. Advancing
// by a fixed number of tokens steps rows and columns without a division.
struct Cursor {
  int s, t, len;
};

__device__ __forceinline__ int fetch_length(const int32_t* lengths, int s, int S, int L) {
  return s < S ? (lengths ? __ldg(lengths + s) : L) : 0;
}

__device__ __forceinline__ Cursor cursor_at(unsigned e, int L, const int32_t* lengths, int S) {
  const int s = static_cast<int>(e / static_cast<unsigned>(L));
  return Cursor{s, static_cast<int>(e - static_cast<unsigned>(s) * L), fetch_length(lengths, s, S, L)};
}

// ds, dt: rows and columns of the step
__device__ __forceinline__ void cursor_advance(Cursor& c, int ds, int dt, const int32_t* lengths, int S,
                                               int L) {
  c.t += dt;
  c.s += ds;
  if (c.t >= L) {
    c.t -= L;
    ++c.s;
  }
  c.len = fetch_length(lengths, c.s, S, L);
}

// Valid tokens of the VEC-token chunk at the cursor, one bit each (VEC <= L: at most two rows).
// ODD: rows are not whole chunks, so a chunk may straddle two rows or the end of the batch
// (16384 x 400 tokens: the loss pass 26.3 us without that code, 27.1 with it).
template <int VEC, bool ODD>
__device__ __forceinline__ int chunk_mask(const Cursor& c, const int32_t* lengths, int S, int L, int* err) {
  const int len = clamp_length(c.len, L, err);
  const int k = min(max(len - c.t, 0), VEC);
  int m = (1 << k) - 1;
  const int in_row = L - c.t;  // tokens of the chunk in this row
  if (ODD && in_row < VEC && c.s + 1 < S) {
    const int len2 = row_length(lengths, c.s + 1, L, err);
    m |= ((1 << min(len2, VEC - in_row)) - 1) << in_row;
  }
  return m;
}

template <int VEC>
struct Vec;
template <>
struct Vec<4> {
  static __device__ __forceinline__ void get(const float* p, float* v) {
    const float4 q = __ldcs(reinterpret_cast<const float4*>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
  static __device__ __forceinline__ void put(float* p, const float* v) {
    __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
  }
};
template <>
struct Vec<1> {
  static __device__ __forceinline__ void get(const float* p, float* v) { v[0] = __ldcs(p); }
  static __device__ __forceinline__ void put(float* p, const float* v) { __stcs(p, v[0]); }
};

// Chunk at element offset `off`; `n` < VEC elements at the end of the batch are moved one by one.
template <int VEC, bool ODD>
__device__ __forceinline__ void chunk_get(const float* p, unsigned off, int n, float* v) {
  if (!ODD || n >= VEC) {
    Vec<VEC>::get(p + off, v);
  } else {
#pragma unroll
    for (int j = 0; j < VEC; ++j) v[j] = j < n ? __ldcs(p + off + j) : 0.f;
  }
}
template <int VEC, bool ODD>
__device__ __forceinline__ void chunk_put(float* p, unsigned off, int n, const float* v) {
  if (!ODD || n >= VEC) {
    Vec<VEC>::put(p + off, v);
  } else {
#pragma unroll
    for (int j = 0; j < VEC; ++j)
      if (j < n) __stcs(p + off + j, v[j]);
  }
}

// Loads that keep their lines in L2 (normal eviction priority): the moments pass reads the
// advantages this way, so that the loss pass, which reads them again with the rest of its
// inputs streaming (evict-first), finds them there when the batch fits in L2.
template <int VEC>
__device__ __forceinline__ void get_keep(const float* p, float* v) {
  if constexpr (VEC == 4) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    v[0] = __ldg(p);
  }
}

// Shifted advantage sums and valid count of the chunks e = VEC (first + i step), i = 0, 1, ..., in
// batches of kMomBatch chunks whose loads are issued together.
constexpr int kMomBatch = 4;

template <int VEC, bool ODD>
__device__ __forceinline__ void moments_walk(const float* __restrict__ adv, const int32_t* lengths, int S,
                                             int L, unsigned first, unsigned nthr, float c, int& n,
                                             Kahan& s1, Kahan& s2, int* err) {
  const unsigned E = static_cast<unsigned>(S) * static_cast<unsigned>(L);
  const unsigned step = kMomBatch * nthr * VEC;  // tokens per batch over the grid
  const int ds = static_cast<int>(step / L), dt = static_cast<int>(step % L);
  Cursor cur[kMomBatch];
#pragma unroll
  for (int b = 0; b < kMomBatch; ++b) cur[b] = cursor_at((first + b * nthr) * VEC, L, lengths, S);
  while (cur[0].s < S) {
    float v[kMomBatch][VEC];
    int m[kMomBatch];
#pragma unroll
    for (int b = 0; b < kMomBatch; ++b) {
      m[b] = 0;
      if (cur[b].s < S) {
        m[b] = chunk_mask<VEC, ODD>(cur[b], lengths, S, L, err);
        const unsigned off = static_cast<unsigned>(cur[b].s) * static_cast<unsigned>(L) + cur[b].t;
        if (m[b] != 0) {
          if (!ODD || E - off >= VEC) get_keep<VEC>(adv + off, v[b]);
          else chunk_get<VEC, ODD>(adv, off, static_cast<int>(E - off), v[b]);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < kMomBatch; ++b) cursor_advance(cur[b], ds, dt, lengths, S, L);
    float b1 = 0.f, b2 = 0.f;  // this batch's sums, then one compensated add each
#pragma unroll
    for (int b = 0; b < kMomBatch; ++b)
#pragma unroll
      for (int j = 0; j < VEC; ++j) {
        const float d = (m[b] >> j) & 1 ? v[b][j] - c : 0.f;
        b1 += d;
        b2 += d * d;
      }
#pragma unroll
    for (int b = 0; b < kMomBatch; ++b) n += __popc(m[b]);
    s1.add(b1);
    s2.add(b2);
  }
}

// Pass 1: valid count and shifted advantage sums per block. `ticket` (the loss pass's block
// counter) is cleared for the launch that follows.
template <int VEC, bool ODD>
__global__ void __launch_bounds__(kPpoThreads, 3)
    ppo_moments_kernel(const float* __restrict__ adv, const int32_t* __restrict__ lengths, int S,
                       int L, int with_adv, MomPart* __restrict__ part, unsigned* ticket, int* err) {
  __shared__ float sh[2][kPpoWarps];
  __shared__ int shk[kPpoWarps];
  pdl_wait();
  const unsigned tid = blockIdx.x * kPpoThreads + threadIdx.x;
  const unsigned nthr = gridDim.x * kPpoThreads;
  if (tid == 0 && ticket != nullptr) *ticket = 0;
  int n = 0;
  Kahan s1, s2;
  if (!with_adv) {
    for (unsigned s = tid; s < static_cast<unsigned>(S); s += nthr)
      n += row_length(lengths, static_cast<int>(s), L, err);
  } else if (L >= VEC) {
    moments_walk<VEC, ODD>(adv, lengths, S, L, tid, nthr, S > 0 ? __ldg(adv) : 0.f, n, s1, s2, err);
  }
  float v[2] = {s1.s, s2.s};
  block_sums<2>(v, n, sh, shk);
  if (threadIdx.x == 0) part[blockIdx.x] = MomPart{n, v[0], v[1], 0.f};
  pdl_launch_dependents();
}

// Pass 1, float4 rows (L % 4 == 0, aligned): one warp per row, two rows in flight per warp;
// lane l loads tokens [4 l + 128 k, + 4) of a row's valid prefix, k < 4 at a time, and the
// next pair's lengths are fetched before the current pair is added. A row's tokens past its
// length are never read.
__global__ void __launch_bounds__(kPpoThreads)
    ppo_moments_rows_kernel(const float* __restrict__ adv, const int32_t* __restrict__ lengths,
                            int S, int L, MomPart* __restrict__ part, unsigned* ticket, int* err) {
  __shared__ float sh[2][kPpoWarps];
  __shared__ int shk[kPpoWarps];
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0 && ticket != nullptr) *ticket = 0;
  const int lane = threadIdx.x & 31;
  const int gw = blockIdx.x * kPpoWarps + (threadIdx.x >> 5);
  const int nw = gridDim.x * kPpoWarps;
  const float c = S > 0 ? __ldg(adv) : 0.f;
  int n = 0;
  Kahan s1, s2;
  auto len_of = [&](int s) { return s < S ? (lengths ? __ldg(lengths + s) : L) : 0; };
  int nlA = len_of(gw), nlB = len_of(gw + nw);
  for (int s0 = gw; s0 < S; s0 += 2 * nw) {
    const int sA = s0, sB = s0 + nw;
    const int lenA = clamp_length(nlA, L, lane == 0 ? err : nullptr);
    const int lenB = sB < S ? clamp_length(nlB, L, lane == 0 ? err : nullptr) : 0;
    nlA = len_of(s0 + 2 * nw);
    nlB = len_of(s0 + 3 * nw);
    const float* ra = adv + static_cast<size_t>(sA) * L;
    const float* rb = adv + static_cast<size_t>(sB < S ? sB : sA) * L;
    const int lmax = max(lenA, lenB);
    for (int base = 0; base < lmax; base += 512) {
      float va[4][4], vb[4][4];
      int ka[4], kb[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int t0 = base + 128 * k + 4 * lane;
        ka[k] = min(max(lenA - t0, 0), 4);
        kb[k] = min(max(lenB - t0, 0), 4);
        if (ka[k] > 0) get_keep<4>(ra + t0, va[k]);
        if (kb[k] > 0) get_keep<4>(rb + t0, vb[k]);
      }
      float b1 = 0.f, b2 = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float da = j < ka[k] ? va[k][j] - c : 0.f;
          const float db = j < kb[k] ? vb[k][j] - c : 0.f;
          b1 += da + db;
          b2 += da * da + db * db;
        }
#pragma unroll
      for (int k = 0; k < 4; ++k) n += ka[k] + kb[k];
      s1.add(b1);
      s2.add(b2);
    }
  }
  float v[2] = {s1.s, s2.s};
  block_sums<2>(v, n, sh, shk);
  if (threadIdx.x == 0) part[blockIdx.x] = MomPart{n, v[0], v[1], 0.f};
  pdl_launch_dependents();
}

// (n, mean, M2) and the coefficients of the loss pass
struct Moments {
  double n, mean, m2;
  float c_mean, inv_std, inv_n;
};
static_assert(sizeof(Moments) <= sizeof(MomPart) * kPpoMaxMomentBlocks, "ppo_ext_kernel writes it there");

__device__ __forceinline__ Moments load_moments(const Moments* p) {
  return Moments{__ldcg(&p->n),      __ldcg(&p->mean),    __ldcg(&p->m2),
                 __ldcg(&p->c_mean), __ldcg(&p->inv_std), __ldcg(&p->inv_n)};
}

__device__ __forceinline__ Moments moments_from_ext(const double* ext) {
  Moments m;
  m.n = __ldcg(ext);
  m.mean = __ldcg(ext + 1);
  m.m2 = __ldcg(ext + 2);
  const double var = m.n > 0.0 ? m.m2 / m.n : 0.0;
  m.c_mean = static_cast<float>(m.mean);
  m.inv_std = static_cast<float>(1.0 / sqrt(var + 1e-8));
  m.inv_n = m.n > 0.0 ? static_cast<float>(1.0 / m.n) : 0.f;
  return m;
}

// from the sums of a - c and (a - c)^2 over n tokens
__device__ __forceinline__ Moments moments_from_sums(int n, float s1, float s2, float c) {
  Moments m;
  float mean = 0.f, m2 = 0.f;
  if (n > 0) {
    const float d1 = s1 / static_cast<float>(n);
    mean = c + d1;
    m2 = fmaxf(s2 - d1 * s1, 0.f);
  }
  const float var = n > 0 ? m2 / static_cast<float>(n) : 0.f;
  m.n = static_cast<double>(n);
  m.mean = static_cast<double>(mean);
  m.m2 = static_cast<double>(m2);
  m.c_mean = mean;
  m.inv_std = rsqrtf(var + 1e-8f);
  m.inv_n = n > 0 ? 1.f / static_cast<float>(n) : 0.f;
  return m;
}

// Merge the G moments partials: every thread loads its few at once (compensated fp32), then a
// fixed block tree. The result is valid in every thread.
constexpr int kMaxPartsPerThread = (kPpoMaxLossBlocks + kPpoThreads - 1) / kPpoThreads;

__device__ __forceinline__ Moments merge_moments(const MomPart* part, int G, float c,
                                                 float (*sh)[kPpoWarps], int* shk) {
  MomPart p[kMaxPartsPerThread];
#pragma unroll
  for (int i = 0; i < kMaxPartsPerThread; ++i) {
    const int j = threadIdx.x + i * kPpoThreads;
    p[i] = j < G ? load_part(part + j) : MomPart{0, 0.f, 0.f, 0.f};
  }
  int n = 0;
  Kahan k1, k2;
#pragma unroll
  for (int i = 0; i < kMaxPartsPerThread; ++i) {
    n += p[i].n;
    k1.add(p[i].s1);
    k2.add(p[i].s2);
  }
  float v[2] = {k1.s, k2.s};
  block_sums<2>(v, n, sh, shk);
  return moments_from_sums(n, v[0], v[1], c);
}

// The moments alone (hydra_ppo_adv_moments): one block.
__global__ void __launch_bounds__(kPpoThreads)
    ppo_merge_kernel(const float* __restrict__ adv, int S, int L, const MomPart* __restrict__ part, int G,
                     double* __restrict__ moments) {
  __shared__ float sh[2][kPpoWarps];
  __shared__ int shk[kPpoWarps];
  pdl_wait();
  const Moments m = merge_moments(part, G, G > 0 && S > 0 && L > 0 ? __ldg(adv) : 0.f, sh, shk);
  if (threadIdx.x == 0) {
    moments[0] = m.n;
    moments[1] = m.mean;
    moments[2] = m.m2;
  }
  pdl_launch_dependents();
}

// Pass 2: per-token terms and gradients. Each thread holds two chunks: the next chunk's
// five loads are issued before the current chunk is computed and stored.
template <int VEC>
struct LossChunk {
  float ln[VEC], lo[VEC], a[VEC], R[VEC], V[VEC];
  int mask;      // valid tokens
  int left;      // tokens of the batch from the chunk's first on, at most VEC; 0: past its end
  unsigned off;  // element offset (S * L < 2^31)
};

struct LossAcc {
  Kahan s, v, kl, a, aa;
  int nclip = 0;
};

template <int VEC, bool ODD>
__device__ __forceinline__ void loss_load(LossChunk<VEC>& x, Cursor& cur, const float* logp_new,
                                          const float* logp_old, const float* adv,
                                          const float* ret, const float* val, int S, int L,
                                          int ds, int dt, const int32_t* lengths, int* err) {
  x.mask = 0;
  x.left = 0;
  x.off = 0;
  if (cur.s < S) {
    x.mask = chunk_mask<VEC, ODD>(cur, lengths, S, L, err);
    x.off = static_cast<unsigned>(cur.s) * static_cast<unsigned>(L) + cur.t;
    x.left = VEC;
    if (ODD) x.left = static_cast<int>(min(static_cast<unsigned>(S) * static_cast<unsigned>(L) - x.off,
                                           static_cast<unsigned>(VEC)));
    if (x.mask != 0) {
      chunk_get<VEC, ODD>(logp_new, x.off, x.left, x.ln);
      chunk_get<VEC, ODD>(logp_old, x.off, x.left, x.lo);
      chunk_get<VEC, ODD>(adv, x.off, x.left, x.a);
      chunk_get<VEC, ODD>(ret, x.off, x.left, x.R);
      chunk_get<VEC, ODD>(val, x.off, x.left, x.V);
    }
  }
  cursor_advance(cur, ds, dt, lengths, S, L);
}

template <int VEC, bool ODD, bool WHITEN>
__device__ __forceinline__ void loss_compute(const LossChunk<VEC>& x, float mean, float inv_std,
                                             float inv_n, float eps, LossAcc& acc,
                                             float* grad_logp, float* grad_val) {
  if (x.left == 0) return;
  const float lo_clip = 1.f - eps, hi_clip = 1.f + eps;
  float gl[VEC], gv[VEC];
  float bs = 0.f, bv = 0.f, bkl = 0.f, ba = 0.f, baa = 0.f;  // this chunk's sums
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    gl[j] = gv[j] = 0.f;
    if ((x.mask >> j) & 1) {
      const float d = x.ln[j] - x.lo[j];
      const float r = expf(d);
      const float A = WHITEN ? (x.a[j] - mean) * inv_std : x.a[j];
      const float rc = fminf(fmaxf(r, lo_clip), hi_clip);
      const float u = r * A, c = rc * A;
      const float dv = x.V[j] - x.R[j];
      bs += fminf(u, c);
      bv += dv * dv;
      bkl -= d;
      ba += x.a[j];
      baa += x.a[j] * x.a[j];
      acc.nclip += fabsf(r - 1.f) > eps ? 1 : 0;
      gl[j] = u <= c ? -u * inv_n : 0.f;
      gv[j] = 2.f * dv * inv_n;
    }
  }
  chunk_put<VEC, ODD>(grad_logp, x.off, x.left, gl);
  chunk_put<VEC, ODD>(grad_val, x.off, x.left, gv);
  if (x.mask != 0) {
    acc.s.add(bs);
    acc.v.add(bv);
    acc.kl.add(bkl);
    acc.a.add(ba);
    acc.aa.add(baa);
  }
}

// The moments among the statistics.
__device__ __forceinline__ void write_moment_stats(double* stats, const Moments& m) {
  stats[4] = m.mean;
  stats[5] = m.n > 0.0 ? sqrt(m.m2 / m.n) : 0.0;
  stats[6] = m.n;
}

// The statistics of a batch from its loss sums (moments_done: all but the moments).
__device__ __forceinline__ void write_stats(double* stats, const float (&v)[kLossSums], int nclip,
                                            const Moments& m, bool report_moments, bool moments_done = false) {
  const double n = m.n, inv = n > 0.0 ? 1.0 / n : 0.0;
  stats[0] = -static_cast<double>(v[0]) * inv;
  stats[1] = static_cast<double>(v[1]) * inv;
  stats[2] = static_cast<double>(nclip) * inv;
  stats[3] = static_cast<double>(v[2]) * inv;
  if (moments_done) return;
  if (report_moments) {
    stats[4] = m.mean;
    stats[5] = n > 0.0 ? sqrt(m.m2 * inv) : 0.0;
  } else {
    const double a = static_cast<double>(v[3]) * inv;
    stats[4] = a;
    stats[5] = n > 0.0 ? sqrt(fmax(static_cast<double>(v[4]) * inv - a * a, 0.0)) : 0.0;
  }
  stats[6] = n;
}

// The caller's moments for the loss pass, in the place of the moments partials, and among the
// statistics. One thread of a warp for each: the fp64 root and quotients are slow (in every thread
// of the loss pass 16384 x 400 tokens took 27.3 us, with every thread reading one thread's
// results 26.1, with one thread of each block 22.1; 700 x 1500 tokens unwhitened 10.0 with the
// statistics at the loss pass's end, 9.55 so).
__global__ void ppo_ext_kernel(const double* __restrict__ ext, Moments* __restrict__ out, unsigned* ticket,
                               double* __restrict__ stats) {
  pdl_wait();
  if (threadIdx.x == 0) {
    *out = moments_from_ext(ext);
    *ticket = 0;
  } else if (threadIdx.x == 32) {
    Moments m;
    m.n = __ldcg(ext);
    m.mean = __ldcg(ext + 1);
    m.m2 = __ldcg(ext + 2);
    write_moment_stats(stats, m);
  }
  pdl_launch_dependents();
}

// Pass 2 over the grid, and the statistics by the block that finishes last.
template <int VEC, bool ODD, bool WHITEN>
__global__ void __launch_bounds__(kPpoThreads, 3)
    ppo_loss_kernel(const float* __restrict__ logp_new, const float* __restrict__ logp_old,
                    const float* __restrict__ adv, const float* __restrict__ ret,
                    const float* __restrict__ val, const int32_t* __restrict__ lengths, int S,
                    int L, float eps, const MomPart* __restrict__ mpart, int Gm,
                    const Moments* __restrict__ ext, int report_moments, LossPart* __restrict__ lpart,
                    unsigned* ticket, float* __restrict__ grad_logp, float* __restrict__ grad_val,
                    double* __restrict__ stats, int* err) {
  __shared__ float sh[kLossSums][kPpoWarps];
  __shared__ int shk[kPpoWarps];
  __shared__ bool last;
  pdl_wait();
  const unsigned tid = blockIdx.x * kPpoThreads + threadIdx.x;
  const unsigned nthr = gridDim.x * kPpoThreads;
  // L >= VEC here: the host launches this pass only for S * L > 0
  const unsigned step = nthr * VEC;
  const int ds = static_cast<int>(step / L), dt = static_cast<int>(step % L);
  Cursor cur = cursor_at(tid * VEC, L, lengths, S);
  LossAcc acc;
  LossChunk<VEC> x, y;
  loss_load<VEC, ODD>(x, cur, logp_new, logp_old, adv, ret, val, S, L, ds, dt, lengths, err);
  Moments mom;
  if (ext != nullptr) {  // one thread: every thread of the grid at the same line took 2 us
    __shared__ Moments given;
    if (threadIdx.x == 0) given = load_moments(ext);
    __syncthreads();
    mom = given;
  } else {
    mom = merge_moments(mpart, Gm, WHITEN ? __ldg(adv) : 0.f, sh, shk);
  }
  const float mean = mom.c_mean, inv_std = mom.inv_std, inv_n = mom.inv_n;
  if (WHITEN && ext == nullptr && tid == 0) write_moment_stats(stats, mom);  // the fp64 root off the end of the launch
  while (true) {
    if (cur.s >= S) {
      loss_compute<VEC, ODD, WHITEN>(x, mean, inv_std, inv_n, eps, acc, grad_logp, grad_val);
      break;
    }
    loss_load<VEC, ODD>(y, cur, logp_new, logp_old, adv, ret, val, S, L, ds, dt, lengths, err);
    loss_compute<VEC, ODD, WHITEN>(x, mean, inv_std, inv_n, eps, acc, grad_logp, grad_val);
    if (cur.s >= S) {
      loss_compute<VEC, ODD, WHITEN>(y, mean, inv_std, inv_n, eps, acc, grad_logp, grad_val);
      break;
    }
    loss_load<VEC, ODD>(x, cur, logp_new, logp_old, adv, ret, val, S, L, ds, dt, lengths, err);
    loss_compute<VEC, ODD, WHITEN>(y, mean, inv_std, inv_n, eps, acc, grad_logp, grad_val);
  }
  float v[kLossSums] = {acc.s.s, acc.v.s, acc.kl.s, acc.a.s, acc.aa.s};
  int nclip = acc.nclip;
  block_sums<kLossSums>(v, nclip, sh, shk);
  if (threadIdx.x == 0) {
    LossPart p;
    p.nclip = nclip;
#pragma unroll
    for (int i = 0; i < kLossSums; ++i) p.s[i] = v[i];
    p.pad[0] = p.pad[1] = 0.f;
    lpart[blockIdx.x] = p;
    __threadfence();  // the partial is visible before the ticket
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    const int G = static_cast<int>(gridDim.x);
    Kahan k[kLossSums];
    nclip = 0;
#pragma unroll
    for (int i = 0; i < kMaxPartsPerThread; ++i) {
      const int j = threadIdx.x + i * kPpoThreads;
      if (j < G) {
        const LossPart p = load_part(lpart + j);
        nclip += p.nclip;
#pragma unroll
        for (int q = 0; q < kLossSums; ++q) k[q].add(p.s[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kLossSums; ++q) v[q] = k[q].s;
    block_sums<kLossSums>(v, nclip, sh, shk);
    if (threadIdx.x == 0) write_stats(stats, v, nclip, mom, report_moments != 0, WHITEN || ext != nullptr);
  }
  pdl_launch_dependents();
}

// The statistics of an empty batch (the caller's moments, or none).
__global__ void ppo_empty_kernel(const double* __restrict__ ext, int report_moments, double* __restrict__ stats) {
  pdl_wait();
  const float v[kLossSums] = {0.f, 0.f, 0.f, 0.f, 0.f};
  write_stats(stats, v, 0, ext != nullptr ? moments_from_ext(ext) : moments_from_sums(0, 0.f, 0.f, 0.f),
              report_moments != 0);
}

// ---------------------------------------------------------------- one launch for small batches

// A sum of a few partial sums with its rounding errors collected (Knuth, "The Art of Computer
// Programming", vol. 2, 4.2.2); an infinite sum collects none.
struct ExactSum {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x, b = t - s;
    const float r = (s - (t - b)) + (x - b);
    e += fabsf(t) <= FLT_MAX ? r : 0.f;
    s = t;
  }
  __device__ __forceinline__ float value() const { return s + e; }
};

// A cluster of up to kMaxCluster CTAs covers the batch; each CTA's sums go to the CTAs that need
// them with stores to distributed shared memory and are added in rank order. (Added plainly, the
// value loss of 31 x 400 tokens was 5.8e-8 from 64 bits, rms of 400 batches, where the block-wise
// launches had 4.2e-8; so 3.4e-8.)
constexpr int kMaxCluster = 8;
constexpr long long kSmallTokens = 16384;

__device__ __forceinline__ void st_cluster_u32(const void* local, uint32_t rank, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_to_rank(smem_u32(local), rank)), "r"(v) : "memory");
}

template <int VEC, bool ODD, bool WHITEN>
__global__ void __launch_bounds__(kPpoThreads)
    ppo_small_kernel(const float* __restrict__ logp_new, const float* __restrict__ logp_old,
                     const float* __restrict__ adv, const float* __restrict__ ret,
                     const float* __restrict__ val, const int32_t* __restrict__ lengths, int S,
                     int L, float eps, const double* __restrict__ ext, int report_moments,
                     float* __restrict__ grad_logp, float* __restrict__ grad_val,
                     double* __restrict__ stats, int* err) {
  __shared__ float sh[kLossSums][kPpoWarps];
  __shared__ int shk[kPpoWarps];
  __shared__ uint32_t mrecv[kMaxCluster][3], lrecv[kMaxCluster][kLossSums + 1];
  const int c = static_cast<int>(gridDim.x);
  const uint32_t rank = blockIdx.x;  // one cluster
  // first half of a cluster barrier: every CTA has started before the first push
  if (c > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait();
  pdl_launch_dependents();
  const unsigned tid = rank * kPpoThreads + threadIdx.x;
  const unsigned nthr = c * kPpoThreads;
  const unsigned step = nthr * VEC;
  const int ds = static_cast<int>(step / L), dt = static_cast<int>(step % L);
  Cursor cur = cursor_at(tid * VEC, L, lengths, S);
  LossChunk<VEC> x, y;
  loss_load<VEC, ODD>(x, cur, logp_new, logp_old, adv, ret, val, S, L, ds, dt, lengths, err);
  Moments mom;
  if (ext != nullptr) {
    __shared__ Moments given;
    if (threadIdx.x == 0) given = moments_from_ext(ext);
    __syncthreads();
    mom = given;
    if (c > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  } else {
    int n = 0;
    Kahan s1, s2;
    const float shift = WHITEN ? __ldg(adv) : 0.f;
    if (WHITEN) {
      moments_walk<VEC, ODD>(adv, lengths, S, L, tid, nthr, shift, n, s1, s2, err);
    } else {
      for (unsigned s = tid; s < static_cast<unsigned>(S); s += nthr)
        n += row_length(lengths, static_cast<int>(s), L, err);
    }
    float v[2] = {s1.s, s2.s};
    block_sums<2>(v, n, sh, shk);
    if (c > 1) {
      asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
      if (threadIdx.x < static_cast<unsigned>(c)) {
        st_cluster_u32(&mrecv[rank][0], threadIdx.x, static_cast<uint32_t>(n));
        st_cluster_u32(&mrecv[rank][1], threadIdx.x, __float_as_uint(v[0]));
        st_cluster_u32(&mrecv[rank][2], threadIdx.x, __float_as_uint(v[1]));
      }
      cluster_sync_all();
      n = 0;
      ExactSum k1, k2;
#pragma unroll
      for (int q = 0; q < kMaxCluster; ++q) {
        n += q < c ? static_cast<int>(mrecv[q][0]) : 0;
        k1.add(q < c ? __uint_as_float(mrecv[q][1]) : 0.f);
        k2.add(q < c ? __uint_as_float(mrecv[q][2]) : 0.f);
      }
      v[0] = k1.value();
      v[1] = k2.value();
    }
    mom = moments_from_sums(n, v[0], v[1], shift);
  }
  LossAcc acc;
  while (true) {
    const bool more = cur.s < S;
    if (more) loss_load<VEC, ODD>(y, cur, logp_new, logp_old, adv, ret, val, S, L, ds, dt, lengths, err);
    loss_compute<VEC, ODD, WHITEN>(x, mom.c_mean, mom.inv_std, mom.inv_n, eps, acc, grad_logp, grad_val);
    if (!more) break;
    x = y;
  }
  float v[kLossSums] = {acc.s.s, acc.v.s, acc.kl.s, acc.a.s, acc.aa.s};
  int nclip = acc.nclip;
  block_sums<kLossSums>(v, nclip, sh, shk);
  if (c > 1) {
    if (threadIdx.x == 0) {
      st_cluster_u32(&lrecv[rank][kLossSums], 0, static_cast<uint32_t>(nclip));
#pragma unroll
      for (int q = 0; q < kLossSums; ++q) st_cluster_u32(&lrecv[rank][q], 0, __float_as_uint(v[q]));
    }
    cluster_sync_all();
    if (rank == 0 && threadIdx.x < 32) {  // lane q adds sum q, the lane after them the clipped counts
      const int q = min(static_cast<int>(threadIdx.x), kLossSums);
      ExactSum k;
      nclip = 0;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r) {
        const uint32_t w = r < c ? lrecv[r][q] : 0u;
        nclip += static_cast<int>(w);
        k.add(__uint_as_float(w));
      }
      const float sum = k.value();
#pragma unroll
      for (int i = 0; i < kLossSums; ++i) v[i] = __shfl_sync(0xffffffffu, sum, i);
      nclip = __shfl_sync(0xffffffffu, nclip, kLossSums);
    }
  }
  if (rank == 0 && threadIdx.x == 0) write_stats(stats, v, nclip, mom, report_moments != 0);
}

int num_sms() {
  static int nsm = 0;
  if (nsm == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      nsm = 148;
  }
  return nsm;
}

// One wave: SMs x resident blocks per SM (capped by the work and the workspace slots).
template <typename K>
int one_wave(K kernel, long long work_items, int cap) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPpoThreads, 0) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const long long want = (work_items + kPpoThreads - 1) / kPpoThreads;
  long long g = static_cast<long long>(num_sms()) * per_sm;
  if (want < g) g = want;
  if (g > cap) g = cap;
  return g < 1 ? 1 : static_cast<int>(g);
}

struct WsLayout {
  MomPart* mom;
  LossPart* loss;
  unsigned* ticket;
};

WsLayout layout(void* ws) {
  char* p = static_cast<char*>(ws);
  WsLayout w;
  w.mom = reinterpret_cast<MomPart*>(p);
  p += sizeof(MomPart) * kPpoMaxMomentBlocks;
  w.loss = reinterpret_cast<LossPart*>(p);
  p += sizeof(LossPart) * kPpoMaxLossBlocks;
  w.ticket = reinterpret_cast<unsigned*>(p);
  return w;
}

// 16-byte chunks of four tokens: rows of at least four tokens, aligned arrays
bool vec4_ok(int64_t L, std::initializer_list<const void*> ptrs) {
  if (L < 4) return false;
  for (const void* p : ptrs)
    if (reinterpret_cast<uintptr_t>(p) % 16 != 0) return false;
  return true;
}

// Pass 1 into w.mom; returns its number of blocks, or a negative code. Clears the ticket.
int launch_moments(const float* adv, const int32_t* lengths, int S, int L, bool with_adv,
                   const WsLayout& w, int* err, cudaStream_t st) {
  const bool v4 = vec4_ok(L, {adv});
  const long long tokens = static_cast<long long>(S) * L;
  int G = 0;
  cudaError_t e;
  if (v4 && with_adv && L % 4 == 0) {
    // a warp per row pair: S / 2 warps of work
    G = one_wave(ppo_moments_rows_kernel, (static_cast<long long>(S) + 1) / 2 * 32,
                 kPpoMaxMomentBlocks);
    e = launch_pdl(ppo_moments_rows_kernel, dim3(G), dim3(kPpoThreads), 0, st, adv, lengths, S,
                   L, w.mom, w.ticket, err);
  } else if (v4) {
    G = one_wave(ppo_moments_kernel<4, true>, with_adv ? (tokens + 3) / 4 : S, kPpoMaxMomentBlocks);
    e = launch_pdl(ppo_moments_kernel<4, true>, dim3(G), dim3(kPpoThreads), 0, st, adv, lengths, S,
                   L, with_adv ? 1 : 0, w.mom, w.ticket, err);
  } else {
    G = one_wave(ppo_moments_kernel<1, false>, with_adv ? tokens : S, kPpoMaxMomentBlocks);
    e = launch_pdl(ppo_moments_kernel<1, false>, dim3(G), dim3(kPpoThreads), 0, st, adv, lengths, S,
                   L, with_adv ? 1 : 0, w.mom, w.ticket, err);
  }
  return e == cudaSuccess ? G : -3;
}

}  // namespace

size_t ppo_loss_workspace_bytes() {
  return sizeof(MomPart) * kPpoMaxMomentBlocks + sizeof(LossPart) * kPpoMaxLossBlocks +
         4 * sizeof(double) + 4 * sizeof(float);
}

int launch_ppo_adv_moments(const float* adv, const int32_t* lengths, int64_t S, int64_t L,
                           double* out, void* ws, int* err, cudaStream_t st) {
  const int Si = static_cast<int>(S), Li = static_cast<int>(L);
  const WsLayout w = layout(ws);
  int G = 0;
  if (S * L > 0) {
    G = launch_moments(adv, lengths, Si, Li, true, w, err, st);
    if (G < 0) return G;
  }
  return launch_pdl(ppo_merge_kernel, dim3(1), dim3(kPpoThreads), 0, st, adv, Si, Li,
                    static_cast<const MomPart*>(w.mom), G, out) == cudaSuccess
             ? 0
             : -3;
}

int launch_ppo_loss(const float* logp_new, const float* logp_old, const float* adv,
                    const float* ret, const float* val, const int32_t* lengths, int64_t S,
                    int64_t L, float eps, bool whiten, const double* ext_moments,
                    float* grad_logp, float* grad_val, double* stats, void* ws, int* err,
                    cudaStream_t st) {
  const int Si = static_cast<int>(S), Li = static_cast<int>(L);
  const int report = (whiten || ext_moments != nullptr) ? 1 : 0;
  cudaError_t e;
  if (S * L == 0) {
    e = launch_pdl(ppo_empty_kernel, dim3(1), dim3(1), 0, st, ext_moments, report, stats);
    return e == cudaSuccess ? 0 : -3;
  }
  const bool v4 = vec4_ok(L, {logp_new, logp_old, adv, ret, val, grad_logp, grad_val});
  const long long items = v4 ? (S * L + 3) / 4 : S * L;
  if (S * L <= kSmallTokens) {
    // CTAs until every thread has one chunk, at most a cluster
    const long long want = (items + kPpoThreads - 1) / kPpoThreads;
    const int c = want >= kMaxCluster ? kMaxCluster : (want > 4 ? kMaxCluster : (want > 2 ? 4 : static_cast<int>(want)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(c));
    cfg.blockDim = dim3(kPpoThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = static_cast<unsigned>(c);
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = c > 1 ? 2 : 1;
    auto go = [&](auto kernel) {
      return cudaLaunchKernelEx(&cfg, kernel, logp_new, logp_old, adv, ret, val, lengths, Si, Li, eps,
                                ext_moments, report, grad_logp, grad_val, stats, err);
    };
    // (one form for whole and odd rows: at this size the straddling code costs nothing)
    if (v4) e = whiten ? go(ppo_small_kernel<4, true, true>) : go(ppo_small_kernel<4, true, false>);
    else e = whiten ? go(ppo_small_kernel<1, false, true>) : go(ppo_small_kernel<1, false, false>);
    return e == cudaSuccess ? 0 : -3;
  }
  const WsLayout w = layout(ws);
  Moments* ext = nullptr;
  int Gm = 0;
  if (ext_moments != nullptr) {
    ext = reinterpret_cast<Moments*>(w.mom);
    if (launch_pdl(ppo_ext_kernel, dim3(1), dim3(64), 0, st, ext_moments, ext, w.ticket, stats) != cudaSuccess) return -3;
  } else {
    Gm = launch_moments(adv, lengths, Si, Li, whiten, w, err, st);
    if (Gm < 0) return Gm;
  }
  auto go = [&](auto kernel) {
    const int G = one_wave(kernel, items, kPpoMaxLossBlocks);
    return launch_pdl(kernel, dim3(G), dim3(kPpoThreads), 0, st, logp_new, logp_old, adv, ret, val,
                      lengths, Si, Li, eps, static_cast<const MomPart*>(w.mom), Gm, static_cast<const Moments*>(ext),
                      report, w.loss, w.ticket, grad_logp, grad_val, stats, err);
  };
  if (v4 && L % 4 == 0) e = whiten ? go(ppo_loss_kernel<4, false, true>) : go(ppo_loss_kernel<4, false, false>);
  else if (v4) e = whiten ? go(ppo_loss_kernel<4, true, true>) : go(ppo_loss_kernel<4, true, false>);
  else e = whiten ? go(ppo_loss_kernel<1, false, true>) : go(ppo_loss_kernel<1, false, false>);
  return e == cudaSuccess ? 0 : -3;
}

}  // namespace hydra
