// Reverse GAE scan, one warp per sequence (§2: GAE builds the advantage estimates from
// V(x, y); the critic is trained on the returns. Appendix B: gamma = 1.0, lambda = 0.95).
//
//   delta_t = r_t + gamma V_{t+1} [t + 1 < len] - V_t
//   A_t     = delta_t + gamma lambda A_{t+1},   A_len = 0
//   R_t     = A_t + V_t;   A_t = R_t = 0 for t >= len
//
// Rows of whole float4 groups up to 512 tokens: the sequence lives in the warp's registers
// (gae_scan_reg_kernel). 16384 x 400 tokens, ragged: 26.3 us through shared memory, 15.1 so.
// Other lengths: the warp loads its sequence into shared memory with coalesced loads.
// Lane j owns the contiguous chunk [j c, j c + c). Each lane runs the recursion over its chunk with a zero
// carry, which gives an affine map A_start = b + m A_next (m = (gamma lambda)^count). A
// warp-shuffle suffix scan composes the 32 maps, every lane then adds its carry-in times
// the matching power of gamma lambda, and the results leave through coalesced stores.
#include "common.cuh"
#include "kernels.h"

namespace hydra {
namespace {

__global__ void gae_scan_kernel(const float* __restrict__ rew, const float* __restrict__ val,
                                const int32_t* __restrict__ lengths, int S, int L, int chunk,
                                int stride, int warps_per_block, float gamma, float lam,
                                float* __restrict__ adv, float* __restrict__ ret, int* err) {
  extern __shared__ float sm[];
  pdl_wait();
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int s = blockIdx.x * warps_per_block + warp;
  if (s >= S) return;
  float* rb = sm + static_cast<size_t>(warp) * 2 * 32 * stride;
  float* vb = rb + 32 * stride;

  int n = lengths ? lengths[s] : L;
  if (n < 0 || n > L) {
    if (lane == 0) record_error(err, kDevBadLength);
    n = n < 0 ? 0 : L;
  }
  const float* rr = rew + static_cast<size_t>(s) * L;
  const float* vv = val + static_cast<size_t>(s) * L;
  // token t sits at chunk t / chunk, slot t % chunk; both step with t (a division per token cost
  // more than its loads)
  const int dj = 32 / chunk, dk = 32 - dj * chunk;
  const int j0 = lane / chunk, k0 = lane - j0 * chunk;
  {
    int j = j0, k = k0;
#pragma unroll 4
    for (int t = lane; t < n; t += 32) {
      const int o = j * stride + k;
      rb[o] = __ldcs(rr + t);
      vb[o] = __ldcs(vv + t);
      j += dj;
      k += dk;
      if (k >= chunk) {
        k -= chunk;
        ++j;
      }
    }
  }
  __syncwarp();

  const float c = gamma * lam;
  const int lo = lane * chunk;
  const int he = min(min(L, lo + chunk), n);  // end of this lane's valid range
  float* rl = rb + lane * stride;
  float* vl = vb + lane * stride;

  // value following the chunk: first element of the next chunk when it is still valid
  float v_next = (he < n) ? vb[(lane + 1) * stride] : 0.f;
  float a = 0.f;
  float m = 1.f;
  for (int t = he - 1; t >= lo; --t) {
    const float vt = vl[t - lo];
    const float delta = rl[t - lo] + gamma * v_next - vt;
    a = delta + c * a;
    rl[t - lo] = a;  // local advantage with a zero carry
    m *= c;
    v_next = vt;
  }
  float b = (he > lo) ? a : 0.f;

  // inclusive suffix scan of the maps X_j = b_j + m_j X_{j+1}
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float b2 = __shfl_down_sync(0xffffffffu, b, off);
    const float m2 = __shfl_down_sync(0xffffffffu, m, off);
    if (lane + off < 32) {
      b = fmaf(m, b2, b);
      m *= m2;
    }
  }
  float carry = __shfl_down_sync(0xffffffffu, b, 1);
  if (lane == 31) carry = 0.f;

  float p = c;
  for (int t = he - 1; t >= lo; --t) {
    const float at = fmaf(p, carry, rl[t - lo]);
    rl[t - lo] = at;
    vl[t - lo] = at + vl[t - lo];
    p *= c;
  }
  __syncwarp();

  float* ao = adv + static_cast<size_t>(s) * L;
  float* ro = ret + static_cast<size_t>(s) * L;
  int j = j0, k = k0;
#pragma unroll 4
  for (int t = lane; t < L; t += 32) {
    float av = 0.f, rv = 0.f;
    if (t < n) {
      const int o = j * stride + k;
      av = rb[o];
      rv = vb[o];
    }
    __stcs(ao + t, av);
    __stcs(ro + t, rv);
    j += dj;
    k += dk;
    if (k >= chunk) {
      k -= chunk;
      ++j;
    }
  }
}

// Register-only variant for L % 4 == 0, L <= 128 R (R at most 4): the row goes by rounds of 128
// tokens, in each of which lane l owns the float4 group l, so that every load and store of the warp
// is whole lines. The rounds' suffix scans are independent; their first lanes' maps then chain the
// carries from the last round to the first. Groups at or beyond the sequence length are neither
// read nor computed, groups beyond L not written.
// Bound by HBM (8 B per valid token read, 8 B per token written). With 16 consecutive tokens per
// lane, every access touched half of 32 sectors: 16384 x 400 ragged tokens 18.0 us, now 15.1 (5.4
// TB/s); 65536 x 512 75.4, 63.6. The warp skips the rounds past its sequence's length (without
// that the rounds' shuffles cost more than the lines gain: 20.7 and 84.9 us); a single round has
// none to skip.
template <int R>
__global__ void __launch_bounds__(256)
    gae_scan_reg_kernel(const float* __restrict__ rew, const float* __restrict__ val,
                        const int32_t* __restrict__ lengths, int S, int L, float gamma, float lam,
                        float* __restrict__ adv, float* __restrict__ ret, int* err) {
  pdl_wait();
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int s = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (s >= S) return;
  int n = lengths ? lengths[s] : L;
  if (n < 0 || n > L) {
    if (lane == 0) record_error(err, kDevBadLength);
    n = n < 0 ? 0 : L;
  }
  const float4* rr = reinterpret_cast<const float4*>(rew + static_cast<size_t>(s) * L) + lane;
  const float4* vv = reinterpret_cast<const float4*>(val + static_cast<size_t>(s) * L) + lane;
  float r[R][4], v[R][4];  // r becomes the advantages
#pragma unroll
  for (int q = 0; q < R; ++q) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (128 * q + 4 * lane < n) {
      a = __ldcs(rr + 32 * q);
      b = __ldcs(vv + 32 * q);
    }
    r[q][0] = a.x; r[q][1] = a.y; r[q][2] = a.z; r[q][3] = a.w;
    v[q][0] = b.x; v[q][1] = b.y; v[q][2] = b.z; v[q][3] = b.w;
  }
  const float c = gamma * lam;
  float b[R], m[R];  // the affine map of the lane's group, then of the groups from it to the round's end
#pragma unroll
  for (int q = 0; q < R; ++q) {
    b[q] = 0.f;
    m[q] = 1.f;
    if (R > 1 && 128 * q >= n) continue;  // the whole warp
    // value following the group: the next lane's first, the next round's for the last lane
    float after = __shfl_down_sync(0xffffffffu, v[q][0], 1);
    if (q + 1 < R) {
      const float next = __shfl_sync(0xffffffffu, v[q + 1 < R ? q + 1 : q][0], 0);
      if (lane == 31) after = next;
    }
    const int lo = 128 * q + 4 * lane;
#pragma unroll
    for (int i = 3; i >= 0; --i) {
      const int t = lo + i;
      if (t < n) {
        const float vn = t + 1 < n ? (i == 3 ? after : v[q][i < 3 ? i + 1 : 3]) : 0.f;
        b[q] = (r[q][i] + gamma * vn - v[q][i]) + c * b[q];
        r[q][i] = b[q];
        m[q] *= c;
      }
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float b2 = __shfl_down_sync(0xffffffffu, b[q], off);
      const float m2 = __shfl_down_sync(0xffffffffu, m[q], off);
      if (lane + off < 32) {
        b[q] = fmaf(m[q], b2, b[q]);
        m[q] *= m2;
      }
    }
  }
  float4* ao = reinterpret_cast<float4*>(adv + static_cast<size_t>(s) * L) + lane;
  float4* ro = reinterpret_cast<float4*>(ret + static_cast<size_t>(s) * L) + lane;
  float from_next = 0.f;  // the advantage at the first token of the next round
#pragma unroll
  for (int q = R - 1; q >= 0; --q) {
    if (R > 1 && 128 * q >= n) {  // the whole warp
      if (128 * q + 4 * lane < L) {
        __stcs(ao + 32 * q, make_float4(0.f, 0.f, 0.f, 0.f));
        __stcs(ro + 32 * q, make_float4(0.f, 0.f, 0.f, 0.f));
      }
      continue;
    }
    const float start = fmaf(m[q], from_next, b[q]);  // at the group's first token
    float carry = __shfl_down_sync(0xffffffffu, start, 1);
    if (lane == 31) carry = from_next;
    from_next = __shfl_sync(0xffffffffu, start, 0);
    const int lo = 128 * q + 4 * lane;
    float e[4], f[4], p = c;
#pragma unroll
    for (int i = 3; i >= 0; --i) {
      const bool ok = lo + i < n;
      e[i] = ok ? fmaf(p, carry, r[q][i]) : 0.f;
      f[i] = ok ? e[i] + v[q][i] : 0.f;
      if (ok) p *= c;
    }
    if (lo < L) {
      __stcs(ao + 32 * q, make_float4(e[0], e[1], e[2], e[3]));
      __stcs(ro + 32 * q, make_float4(f[0], f[1], f[2], f[3]));
    }
  }
}

}  // namespace

int launch_gae(const float* r, const float* v, const int32_t* lengths, int64_t S, int64_t L,
               float gamma, float lam, float* adv, float* ret, int* err, cudaStream_t stream) {
  if (S == 0 || L == 0) return 0;
  const bool aligned = (reinterpret_cast<uintptr_t>(r) % 16 == 0) &&
                       (reinterpret_cast<uintptr_t>(v) % 16 == 0) &&
                       (reinterpret_cast<uintptr_t>(adv) % 16 == 0) &&
                       (reinterpret_cast<uintptr_t>(ret) % 16 == 0);
  if (aligned && L % 4 == 0 && L <= 512) {
    const unsigned grid = static_cast<unsigned>((S + 7) / 8);
    auto go = [&](auto kernel) {
      return launch_pdl(kernel, dim3(grid), dim3(256), 0, stream, r, v, lengths, static_cast<int>(S),
                        static_cast<int>(L), gamma, lam, adv, ret, err) == cudaSuccess
                 ? 0
                 : -3;
    };
    if (L <= 128) return go(gae_scan_reg_kernel<1>);
    if (L <= 256) return go(gae_scan_reg_kernel<2>);
    if (L <= 384) return go(gae_scan_reg_kernel<3>);
    return go(gae_scan_reg_kernel<4>);
  }
  const int chunk = static_cast<int>((L + 31) / 32);
  const int stride = (chunk & 1) ? chunk : chunk + 1;  // odd stride: conflict-free lanes
  const size_t per_warp = static_cast<size_t>(2) * 32 * stride * sizeof(float);
  int wpb = static_cast<int>((96 * 1024) / per_warp);
  wpb = wpb < 1 ? 1 : (wpb > 8 ? 8 : wpb);
  const size_t smem = per_warp * wpb;
  static size_t attr_bytes = 0;
  if (smem > 48 * 1024 && smem > attr_bytes) {
    if (cudaFuncSetAttribute(gae_scan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem)) != cudaSuccess)
      return -1;
    attr_bytes = smem;
  }
  const unsigned grid = static_cast<unsigned>((S + wpb - 1) / wpb);
  return launch_pdl(gae_scan_kernel, dim3(grid), dim3(32 * wpb), smem, stream, r, v, lengths,
                    static_cast<int>(S), static_cast<int>(L), chunk, stride, wpb, gamma, lam, adv, ret,
                    err) == cudaSuccess
             ? 0
             : -3;
}

}  // namespace hydra
