// The dual-output LoRA linear (see lora_gemm_tc.cu for the mathematics) for up to 512 token rows
// per stream: one short sequence, a prompt, a decode batch. The work there is reading W once, and
// the tile kernel of lora_gemm_tc.cu leaves most of the chip idle: 97 rows of two streams by 4096
// columns are 32 tiles of 128 x 256, each with the whole of K, on 152 SMs.
//
// A CTA pair (tcgen05 cta_group::2) computes a tile of two row segments by bn columns:
//  * Row segments. Every stream's rows are cut into equal segments of at most 128 rows, and the
//    segments of all streams, in order, are taken two by two: segment 2 i is the first CTA's 128
//    accumulator rows, 2 i + 1 the second's. Up to 128 rows, a pair holds the off and the on
//    stream of the same rows, so one pass over a W tile serves both; three segments per stream
//    make three pairs, not four.
//  * Columns and K. bn (a multiple of 32 from 64 to 256) and the split of K over ks pairs of a cluster
//    (1 or 2) are chosen so that the pairs fill the SMs. With one slice the sums are the tile kernel's,
//    in its order, so that the faster kernel may serve each call. With two they are not, and M, K and N
//    alone decide (few_rows_halves): shared, stacked and three-stream calls and every epilogue
//    agree bit for bit. (Four slices measured slower: only 15 clusters of eight CTAs fit on the chip,
//    36 of four.)
//  * Ring items are two k-blocks of 64, and x and W have a TMA warp each. What a warp executes
//    per item is the limit at these sizes: one warp and 64-wide items took 570 clocks each, more
//    than the products of a tile (97 x 4096 x 12288: 44.8 us, then 26).
//  * LoRA. The k-blocks of u B^T follow x W^T into the accumulator of y_on. The rows of a CTA without
//    LoRA are masked out of those products, so that B, whatever it holds, never meets an off row. One
//    input with both outputs: y_off's sums are copied in TMEM first and drained beside the LoRA
//    products. Two K slices: the last one accumulates u B^T apart, and y_on's partial sum there is
//    main + lora.
//  * Reduction and epilogue. Each of two K slices finishes half of the tile's columns: it takes
//    the other slice's fp32 sums of those columns, pushed into its drained ring through
//    distributed shared memory. Once the products are done all twelve warps drain, three per
//    TMEM lane quarter, a chunk of 32 columns each (paired tiles: 16 of each half) through small
//    swizzled buffers into whole-line stores (the residual add as one fp32 reduction per element
//    in L2).
//  * Dependent launch. W is frozen: the first ring of W boxes moves into L2 before the wait on the
//    preceding kernel. Where that kernel is this call's own lora_down (which waits for its
//    predecessors before it lets this kernel start), x and W are final already and the whole main
//    loop overlaps it; only u is waited for.
//
// What bounds it: HBM for W, and an SM's fill from L2 (64 B per clock: a k-block of 64 costs
// 2 (seg + bn / 2) clocks of fill for 2 bn clocks of products), which is why the x boxes are as
// high as the segment and not 128 rows. 97 rows x 4096 x 12288 (two streams): the main loop runs
// at 6.6 TB/s of W; about 6 us of the 26 are set-up, first loads, drain and stores.
#include <float.h>

#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace hydra {
namespace smallm {

constexpr int BK = 128;  // a ring item: two k-blocks of 64 (128-byte swizzle each)
// warp 0: TMA of W; 1: TMEM and MMA; 2: TMA of x; 3: barriers, L2 prefetch; all of them: drain
constexpr int NUM_THREADS = 384;
constexpr int kMaxStages = 12;
constexpr int kSmemMax = 232448;  // dynamic shared memory of one CTA (227 KiB)
constexpr int kBarBytes = (2 * kMaxStages + 2) * 8 + 16;

// Epilogues. The kernel is compiled for each: a launch then fetches about 40 KB of code and not its
// parts of 82 KB (a 3-layer scoring pass of 97 rows 500 -> 495 us).
enum { EPI_STORE = 0, EPI_SWIGLU = 1, EPI_RESIDUAL = 2, EPI_ROPE = 3, EPI_LOGSOFTMAX = 4, EPI_STORE_F32 = 5 };
constexpr bool paired_epi(int epi) { return epi == EPI_SWIGLU || epi == EPI_ROPE; }
// columns a drain warp takes at a time; of a paired tile, as many of each half
constexpr int chunk_of(int epi) { return paired_epi(epi) ? 16 : 32; }
constexpr int kMaxBoxes = 5;  // W boxes of a CTA and k-block

struct Maps {
  CUtensorMap x[3];
  CUtensorMap w;
  CUtensorMap u[2];
  CUtensorMap b[2];
};

struct Params {
  int M, N;
  int streams, nseg, seg, row_tiles;  // nseg segments of seg rows per stream
  int kb_main, kb_lora, r;
  int bn, ks, stages;
  int shared_x, both;   // both: shared input with LoRA and both outputs wanted
  int has_on, has_crit;
  int b_box;     // rows of a W / B box
  int x_settled; // x is final before the preceding kernel of the stream ends
  int lcol;      // TMEM column of a second accumulator, 0: none. Two K slices: the LoRA sums; one, with
                 // `both`: a copy of the sums, for y_on
  uint32_t tmem_cols;
  int stg_off;   // byte offset of the drain warps' staging buffers (over the drained ring)
  int lora_first;  // `both`, one K slice: the buffers overlap the LoRA items
  int bar_off;
  void* y[3];
  int rope_P, rope_cols;
  const float2* rope_table;
  float* lsm_target;
  const int32_t* lsm_ids;
  int lsm_L, lsm_ids_ld, lsm_ids_off, lsm_tiles;
  int* err;
};

__device__ __forceinline__ void commit_pair_mask(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}
__device__ __forceinline__ void st_cluster_f4(uint32_t cluster_addr, const uint32_t* v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3])
               : "memory");
}
// bring the box at (x, y) of a tensor map into L2
__device__ __forceinline__ void prefetch_box(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y)
               : "memory");
}
// tc_mma2_bf16 that leaves the accumulator lanes of a CTA alone whose `skip` is all ones (0: not)
__device__ __forceinline__ void tc_mma2_bf16_masked(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                    uint32_t accumulate, uint32_t skip0, uint32_t skip1) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %6, %6, %6, %6}, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(skip0), "r"(skip1)
      : "memory");
}
__device__ __forceinline__ float bf16_round(float v) {
  return __bfloat162float(__float2bfloat16_rn(v));
}

// W row of the tile's B row j of CTA half `half`. In the paired layouts tile columns [0, bn/2) and
// [bn/2, bn) are partners: SwiGLU gate / up blocks of 128 rows, rotary halves of 64 rows of a head.
template <int kEpi>
__device__ __forceinline__ int b_row(const Params& p, int n0, int half, int j) {
  if (!paired_epi(kEpi)) return n0 + half * (p.bn / 2) + j;
  const int q = n0 / 2 + j;
  return kEpi == EPI_SWIGLU ? (q >> 7) * 256 + half * 128 + (q & 127)
                             : (q >> 6) * 128 + half * 64 + (q & 63);
}

__device__ __forceinline__ uint4 pack8(const float* v) {
  return make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                    pack_bf16x2(v[6], v[7]));
}

__device__ __forceinline__ void ld_cols(uint32_t taddr, uint32_t (&v)[32]) { tc_ld_32x32b_x32(taddr, v); }
__device__ __forceinline__ void ld_cols(uint32_t taddr, uint32_t (&v)[16]) { tc_ld_32x32b_x16(taddr, v); }

// An epilogue thread's accumulator row: its sums, a chunk of tile columns at a time.
struct RowSums {
  uint32_t taddr;  // TMEM address of the thread's lane, column 0 of the main accumulator
  int on_col;      // columns from there to the sums of y_on, if they are apart (one K slice)
  int lcol;        // columns from there to the LoRA sums, to be added to y_on's (two slices)
  bool own_lora;   // this CTA holds LoRA sums
  const float4* recv;  // the other K slice's sums of this CTA's columns (ks == 2), else NULL
  int lplane;      // float4 from there to the LoRA sums sent along (shared input, slice 0), or 0
  int row;         // row of the tile (TMEM lane)

  // v = the sums of columns [c, c + n), the LoRA term included or not; pos: index of the chunk
  // among those this CTA finishes. LoRA joins the last slice's sum before the slices are added.
  template <int n>
  __device__ __forceinline__ void get(int c, int pos, bool lora, float (&v)[n]) const {
    uint32_t a[n];
    ld_cols(taddr + c + (lora ? on_col : 0), a);
    if (lora && own_lora) {
      uint32_t l[n];
      ld_cols(taddr + lcol + c, l);
      tc_wait_ld();
#pragma unroll
      for (int i = 0; i < n; ++i) v[i] = __uint_as_float(a[i]) + __uint_as_float(l[i]);
    } else {
      tc_wait_ld();
#pragma unroll
      for (int i = 0; i < n; ++i) v[i] = __uint_as_float(a[i]);
    }
    if (recv == nullptr) return;
    const float4* s = recv + pos * (n / 4) * 128 + row;
#pragma unroll
    for (int j = 0; j < n / 4; ++j) {
      float4 t = s[j * 128];
      if (lora && lplane != 0) {
        const float4 l = s[lplane + j * 128];
        t.x += l.x; t.y += l.y; t.z += l.z; t.w += l.w;
      }
      v[4 * j] += t.x; v[4 * j + 1] += t.y; v[4 * j + 2] += t.z; v[4 * j + 3] += t.w;
    }
  }
};

// A drain warp's staging buffer: 32 rows of up to eight 16-byte pieces (piece index XOR row, so
// neither side conflicts). A thread writes the pieces of its own accumulator row; flush() stores
// them so that neighbouring lanes cover one row's line (a thread storing its own row touches 32
// lines per instruction, which cost 2 us of a 20 us launch).
struct Staging {
  uint4* buf;
  int lane, rows;  // rows: valid rows of the warp

  __device__ __forceinline__ void put(int piece, uint4 v) const { buf[lane * 8 + (piece ^ (lane & 7))] = v; }
  // kPieces pieces per row to base + row * ld (bytes); `keep` of them lie inside the output
  template <int kPieces, bool kAdd>
  __device__ __forceinline__ void flush(uint8_t* base, size_t ld, int keep) const {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
      const int e = i * 32 + lane, r = e / kPieces, c = e % kPieces;
      if (r < rows && c < keep) {
        const uint4 v = buf[r * 8 + (c ^ (r & 7))];
        uint8_t* d = base + r * ld + c * 16;
        if (kAdd)  // one addend per element and call: the sum does not depend on any order
          asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(d), "f"(__uint_as_float(v.x)),
                       "f"(__uint_as_float(v.y)), "f"(__uint_as_float(v.z)), "f"(__uint_as_float(v.w))
                       : "memory");
        else
          *reinterpret_cast<uint4*>(d) = v;
      }
    }
    __syncwarp();
  }
};

// Store 32 sums of the thread's row at output columns [n, n + 32) (N % 8 == 0). `y` is the row of
// the warp's lane 0.
template <int kEpi>
__device__ __forceinline__ void store32(const Params& p, const Staging& st, void* y, int n,
                                        const float (&v)[32]) {
  const int left = p.N - n;
  if constexpr (kEpi == EPI_RESIDUAL || kEpi == EPI_STORE_F32) {
    constexpr bool add = kEpi == EPI_RESIDUAL;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float* w = v + 4 * j;
      st.put(j, add ? make_uint4(__float_as_uint(bf16_round(w[0])), __float_as_uint(bf16_round(w[1])),
                                 __float_as_uint(bf16_round(w[2])), __float_as_uint(bf16_round(w[3])))
                    : make_uint4(__float_as_uint(w[0]), __float_as_uint(w[1]), __float_as_uint(w[2]),
                                 __float_as_uint(w[3])));
    }
    uint8_t* d = reinterpret_cast<uint8_t*>(static_cast<float*>(y) + n);
    const size_t ld = static_cast<size_t>(p.N) * 4;
    st.flush<8, add>(d, ld, left / 4);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) st.put(j, pack8(v + 8 * j));
    st.flush<4, false>(reinterpret_cast<uint8_t*>(static_cast<__nv_bfloat16*>(y) + n),
                       static_cast<size_t>(p.N) * 2, left / 8);
  }
}

__device__ __forceinline__ void swiglu2(uint32_t& g, uint32_t u) {
  const float2 a = unpack_bf16x2(g), b = unpack_bf16x2(u);
  g = pack_bf16x2(silu(a.x) * b.x, silu(a.y) * b.y);
}

// 16 partner columns of a paired tile: q is the first one's pair index, v / z the sums of the
// first and the second half; row: the thread's row, y: the output's first element
template <int kEpi>
__device__ __forceinline__ void store_pair16(const Params& p, const Staging& st, void* y, int row,
                                             int q, float (&v)[16], float (&z)[16]) {
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(y);
  const size_t row0 = static_cast<size_t>(row - st.lane);
  if constexpr (kEpi == EPI_SWIGLU) {
    if (q >= p.N / 2) return;  // N % 256 == 0: 16 pairs are all in or all out
    // the bf16 gates and ups through the staging buffer, and a short loop from there, eight
    // features a lane: unrolled over the registers, the quotients are 30 KB of code that every
    // launch fetches anew, and with the division operator they follow one another (13000 clocks
    // of drain per tile, now 5800; 97 rows x 4096 x 22016: 53.3 -> 47.8 us by this loop and
    // silu(), 45.3 by three drain warps per quarter in place of two, 43.9 by 160-column tiles)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      st.put(j, pack8(v + 8 * j));
      st.put(2 + j, pack8(z + 8 * j));
    }
    __syncwarp();
    const int c = st.lane & 1;
#pragma unroll 1
    for (int r = st.lane >> 1; r < 32; r += 16) {
      if (r >= st.rows) break;
      uint4 g = st.buf[r * 8 + (c ^ (r & 7))];
      const uint4 u = st.buf[r * 8 + ((2 + c) ^ (r & 7))];
      swiglu2(g.x, u.x);
      swiglu2(g.y, u.y);
      swiglu2(g.z, u.z);
      swiglu2(g.w, u.w);
      *reinterpret_cast<uint4*>(out + (row0 + r) * (p.N / 2) + q + 8 * c) = g;
    }
    __syncwarp();
  } else {
    // rotary: the roundings of hydra_rope on the bf16-rounded sums
    const int i0 = q & 63, na = (q >> 6) * 128 + i0;
    if (na < p.rope_cols) {  // whole heads: rope_cols % 128 == 0
      const float4* cs = reinterpret_cast<const float4*>(p.rope_table + (row % p.rope_P) * 64 + i0);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 t = __ldg(cs + i);
        const float a0 = bf16_round(v[2 * i]), a1 = bf16_round(v[2 * i + 1]);
        const float b0 = bf16_round(z[2 * i]), b1 = bf16_round(z[2 * i + 1]);
        v[2 * i] = __fsub_rn(__fmul_rn(a0, t.x), __fmul_rn(b0, t.y));
        v[2 * i + 1] = __fsub_rn(__fmul_rn(a1, t.z), __fmul_rn(b1, t.w));
        z[2 * i] = __fadd_rn(__fmul_rn(a0, t.y), __fmul_rn(b0, t.x));
        z[2 * i + 1] = __fadd_rn(__fmul_rn(a1, t.w), __fmul_rn(b1, t.z));
      }
    }
    uint8_t* o = reinterpret_cast<uint8_t*>(out + row0 * p.N + na);
    const size_t ld = static_cast<size_t>(p.N) * 2;
#pragma unroll
    for (int j = 0; j < 2; ++j) st.put(j, pack8(v + 8 * j));
    st.flush<2, false>(o, ld, (p.N - na) / 8);
#pragma unroll
    for (int j = 0; j < 2; ++j) st.put(j, pack8(z + 8 * j));
    st.flush<2, false>(o + 128, ld, (p.N - na - 64) / 8);
  }
}

// Log-softmax partials of the thread's row over a tile of 256 columns: the online (max, sum of
// exp) pair of every third chunk in each of the row's three warps, merged through `others` (64
// pairs of this quarter), and, where it lies, the sampled token's logit (an arithmetic select keeps the
// row in registers).
__device__ __forceinline__ void emit_lsm(const Params& p, const RowSums& r, int row, bool live, int n0,
                                         float2* part, float* target, bool lora, int par, int q,
                                         float2* others) {
  int id = -1;
  if (live) {
    const int sq = row / p.lsm_L;
    id = p.lsm_ids[static_cast<int64_t>(sq) * p.lsm_ids_ld + p.lsm_ids_off + row - sq * p.lsm_L];
  }
  float m = -FLT_MAX, sum = 0.f;
  for (int c = 32 * par; c < 256; c += 96) {
    const int nv = p.N - (n0 + c);
    if (nv <= 0) break;  // uniform over the warp
    float v[32];
    r.get(c, 0, lora, v);
    float mx = -FLT_MAX;
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < nv) mx = fmaxf(mx, v[j]);
    if (mx > m) {
      sum *= __expf(m - mx);
      m = mx;
    }
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < nv) sum += __expf(v[j] - m);
    const int k = id - (n0 + c);
    if (k >= 0 && k < min(nv, 32)) {
      float z = 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) z += (k == j) ? v[j] : 0.f;
      target[row] = z;
    }
  }
  const int lane = threadIdx.x & 31;
  if (par > 0) others[(par - 1) * 32 + lane] = make_float2(m, sum);
  asm volatile("bar.sync %0, 96;" ::"r"(1 + q) : "memory");
  if (par == 0 && live) {
    const float2 a = others[lane], b = others[32 + lane];
    const float t = fmaxf(m, fmaxf(a.x, b.x));
    part[static_cast<int64_t>(row) * p.lsm_tiles + n0 / 256] =
        make_float2(t, sum * __expf(m - t) + a.y * __expf(a.x - t) + b.y * __expf(b.x - t));
  }
  asm volatile("bar.sync %0, 96;" ::"r"(1 + q) : "memory");  // the buffer serves the next output
}

// kCopy: one input with LoRA and both outputs wanted, one K slice (see `both`). In a kernel of its own:
// as a run-time flag it cost the others 0.3 us a launch.
template <int kEpi, bool kCopy>
__global__ void __launch_bounds__(NUM_THREADS)
    lora_gemm_small_kernel(const __grid_constant__ Maps mp, const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.bar_off);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t smem_base = smem_u32(smem);
  auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
  auto empty_bar = [&](int s) { return smem_u32(&bars[kMaxStages + s]); };
  const uint32_t acc_full = smem_u32(&bars[2 * kMaxStages]);
  const uint32_t copied = smem_u32(&bars[2 * kMaxStages + 1]);
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  } else if (warp == 3) {
    if (lane < p.stages) {
      mbar_init(full_bar(lane), 1);
      mbar_init(empty_bar(lane), 1);
    }
    if (lane == 0) {
      mbar_init(acc_full, 1);
      mbar_init(copied, 2 * (NUM_THREADS / 32));
      *abort_flag = 0;
    }
    __syncwarp();
    fence_mbar_init();
  }
  tc_fence_before();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

  // (grid: x = the cluster's CTAs, y = row tile, z = column tile)
  const int rank = static_cast<int>(cluster_rank());
  const int half = rank & 1;        // which CTA of the pair
  const int slice = rank >> 1;      // which K slice
  const bool leader = half == 0;
  const uint32_t lead_rank = static_cast<uint32_t>(rank & ~1);
  const uint16_t pair_mask = static_cast<uint16_t>(3u << lead_rank);
  const int n0 = static_cast<int>(blockIdx.z) * p.bn;

  // the pair's two segments: stream and index within it (no divisions: at most three streams)
  auto stream_of = [&](int g) { return (g >= p.nseg ? 1 : 0) + (g >= 2 * p.nseg ? 1 : 0); };
  auto rows_of = [&](int g) {  // valid rows of segment g
    if (g >= p.streams * p.nseg) return 0;
    return max(0, min(p.seg, p.M - (g - stream_of(g) * p.nseg) * p.seg));
  };
  const int g0 = 2 * static_cast<int>(blockIdx.y), g1 = g0 + 1, gm = g0 + half;
  const int nrow = rows_of(gm);
  const int stream = nrow > 0 ? stream_of(gm) : 0;
  const int m0 = nrow > 0 ? (gm - stream * p.nseg) * p.seg : 0;
  const bool full1 = rows_of(g1) > 0;  // the second CTA has rows (the first always has)
  auto lora_of = [&](int g) {
    if (p.kb_lora == 0 || rows_of(g) == 0) return false;
    if (p.shared_x) return p.has_on != 0;
    const int s = stream_of(g);
    return s == 1 ? p.has_on != 0 : (s == 2 ? p.has_crit != 0 : false);
  };
  const bool lora0 = lora_of(g0), lora1 = lora_of(g1), lora_me = half ? lora1 : lora0;
  const int lset = !p.shared_x && stream_of(lora1 ? g1 : g0) == 2 ? 1 : 0;

  const int kb0 = slice * p.kb_main / p.ks;
  const int kb1 = (slice + 1) * p.kb_main / p.ks;
  const int n_main = kb1 - kb0;
  const int items = n_main + (slice == p.ks - 1 && (lora0 || lora1) ? p.kb_lora : 0);
  const uint32_t a_bytes = static_cast<uint32_t>(p.seg) * 128;  // one k-block of this CTA's rows
  const uint32_t b_bytes = static_cast<uint32_t>(p.bn) * 64;    // and of its half of the columns
  const uint32_t stage_bytes = 2 * (a_bytes + b_bytes);         // [x, x, W, W]
  // bytes of an item with `kbs` k-blocks landing on the pair's barrier
  auto tx_bytes = [&](bool lora, uint32_t kbs) {
    const uint32_t ctas = lora ? (lora0 ? 1u : 0u) + (lora1 ? 1u : 0u) : (full1 ? 2u : 1u);
    return kbs * (ctas * a_bytes + 2 * b_bytes);
  };
  // k-blocks of 64 of LoRA item i (the second may be absent)
  auto lora_kbs = [&](int i) { return p.r - i * BK > 64 ? 2 : 1; };

  // before the barrier ends: descriptors, and this CTA's first W boxes into L2 (W is frozen)
  const int nbox = p.bn / 2 / p.b_box;
  int brow[kMaxBoxes];                          // W rows of the boxes
#pragma unroll
  for (int j = 0; j < kMaxBoxes; ++j) brow[j] = b_row<kEpi>(p, n0, half, j * p.b_box);
  if (warp == 0 && elect_one()) {
    tma_prefetch_desc(&mp.w);
    if (lora0 || lora1) tma_prefetch_desc(&mp.b[lset]);
  }
  if (warp == 2 && elect_one()) {
    tma_prefetch_desc(&mp.x[stream]);
    if (lora0 || lora1) tma_prefetch_desc(&mp.u[lset]);
  }
  if (warp == 3 && elect_one()) {
    for (int i = 0; i < min(n_main, p.stages); ++i)
#pragma unroll
      for (int j = 0; j < kMaxBoxes; ++j)
        if (j < nbox) {
          prefetch_box(&mp.w, (kb0 + i) * BK, brow[j]);
          prefetch_box(&mp.w, (kb0 + i) * BK + 64, brow[j]);
        }
  }
  __syncwarp();
  // every CTA of the cluster has started, its barriers initialised
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem_acc = *tmem_slot;

  // The dependent kernel may start once every CTA has said so. After a plain linear that is the next
  // call's lora_down: let in at once, it waits on the SMs that this grid leaves free, and the SMs
  // of this grid are the next linear's (let in after the products, it spread over them and held
  // that linear up in most runs: 300 rows, shared, 22.6 us a call, now 17.9). After the fused
  // epilogues of a pass come row kernels, whose early CTAs take what the last tiles need (a
  // 97-row scoring pass 457 us, let in at once 465).
  constexpr bool kEarly = kEpi == EPI_STORE || kEpi == EPI_STORE_F32;
  if (kEarly) pdl_launch_dependents();
  int loaded = 0;  // items that a producer has asked for
  // products of LoRA item i, from stage s. With one K slice they go on in y_on's accumulator, past the
  // lanes of a CTA whose rows have none; with two they have their own.
  auto lora_products = [&](int i, int s) {
    const uint32_t st = smem_base + s * stage_bytes;
    const int nsub = min(BK / 16, (p.r - i * BK + 15) / 16);
    const bool one = p.ks == 1;
#pragma unroll 1
    for (int k = 0; k < nsub; ++k) {
      const uint32_t at = static_cast<uint32_t>(k & 3) * 32;
      tc_mma2_bf16_masked(tmem_acc + p.lcol, smem_desc_sw128(st + (k < 4 ? 0 : a_bytes) + at),
                          smem_desc_sw128(st + 2 * a_bytes + (k < 4 ? 0 : b_bytes) + at), idesc_bf16_f32(256, p.bn),
                          one || i > 0 || k > 0 ? 1u : 0u, one && !lora0 ? ~0u : 0u, one && !lora1 ? ~0u : 0u);
    }
    commit_pair_mask(empty_bar(s), pair_mask);
  };
  if (warp == 0 || warp == 2) {
    // ------------------------------------------------------------------ TMA producers: warp 0
    // moves W (and B), warp 2 x (and u). Everything an item needs is a running value, an item is
    // two k-blocks and the two operands have a warp each: one warp with 64-wide items took about
    // 570 clocks per item (a wait alone is 140), more than the pair's products.
    const uint32_t lead_full0 = map_to_rank(full_bar(0), lead_rank);
    const CUtensorMap* tm_main = warp == 0 ? &mp.w : &mp.x[stream];
    const CUtensorMap* tm_lora = warp == 0 ? &mp.b[lset] : &mp.u[lset];
    const uint32_t box_bytes = static_cast<uint32_t>(p.b_box) * 128;
    auto load_b = [&](uint32_t stage, uint32_t fbar, uint32_t bar, bool lora, int i, int kbs) {
      if (leader) mbar_arrive_expect_tx(fbar, tx_bytes(lora, kbs));
      const CUtensorMap* m = lora ? tm_lora : tm_main;
      const int k = i * BK;
      uint32_t dst = stage + 2 * a_bytes;
#pragma unroll
      for (int j = 0; j < kMaxBoxes; ++j)
        if (j < nbox) tma_load_2d_pair(dst + j * box_bytes, m, k, brow[j], bar);
      if (kbs == 2) {
        dst += b_bytes;
#pragma unroll
        for (int j = 0; j < kMaxBoxes; ++j)
          if (j < nbox) tma_load_2d_pair(dst + j * box_bytes, m, k + 64, brow[j], bar);
      }
    };
    const int pre = min(items, p.stages);
    int it = 0, s = 0;
    uint32_t ph = 0;  // parity of the next wait on stage s: its previous use is done
    if (warp == 0) {
      // W and B are frozen, but a caller may have written them just before this call: they are in
      // L2 by now, and read once everything before the call is final
      if (!p.x_settled) pdl_wait();
      for (; it < items; ++it) {
        if (it >= pre && !warp_wait_bounded(empty_bar(s), ph, abort_flag, p.err, kDevTimeoutProducer))
          break;
        if (elect_one()) {
          const bool lora = it >= n_main;
          load_b(smem_base + s * stage_bytes, full_bar(s), lead_full0 + s * 8, lora,
                 lora ? it - n_main : kb0 + it, lora ? lora_kbs(it - n_main) : 2);
        }
        __syncwarp();
        if (++s == p.stages) {
          s = 0;
          if (it >= pre) ph ^= 1;  // the first ring waits for nothing
        }
      }
    } else {
      if (!p.x_settled) pdl_wait();  // x is written by the preceding kernel
      for (; it < items; ++it) {
        const bool lora = it >= n_main;
        if (it == n_main && p.x_settled) pdl_wait();  // u is written by the preceding kernel
        if (it >= pre && !warp_wait_bounded(empty_bar(s), ph, abort_flag, p.err, kDevTimeoutProducer))
          break;
        if ((lora ? lora_me : nrow > 0) && elect_one()) {
          const uint32_t dst = smem_base + s * stage_bytes, bar = lead_full0 + s * 8;
          const CUtensorMap* m = lora ? tm_lora : tm_main;
          const int k = (lora ? it - n_main : kb0 + it) * BK;
          tma_load_2d_pair(dst, m, k, m0, bar);
          if (!lora || lora_kbs(it - n_main) == 2) tma_load_2d_pair(dst + a_bytes, m, k + 64, m0, bar);
        }
        __syncwarp();
        if (++s == p.stages) {
          s = 0;
          if (it >= pre) ph ^= 1;
        }
      }
    }
    loaded = it;
    // copies in flight land before shared memory is reused: a stage's empty barrier is
    // committed after the products that read it
    for (int k = (it > p.stages ? it - p.stages : 0); k < (kCopy ? min(it, n_main) : it); ++k) {
      volatile int no_abort = 0;
      warp_wait_bounded(empty_bar(k % p.stages), (k / p.stages) & 1, &no_abort, p.err, kDevTimeoutDrain);
    }
  } else if (warp == 1) {
    if (leader) {
      // ---------------------------------------------------------------- MMA issuer
      const uint32_t idesc = idesc_bf16_f32(256, p.bn);
      int s = 0;
      uint32_t ph = 0;
      for (int it = 0; it < (kCopy ? n_main : items); ++it) {
        if (!warp_wait_bounded(full_bar(s), ph, abort_flag, p.err, kDevTimeoutMma)) break;
        tc_fence_after();
        if (elect_one()) {
          if (it < n_main) {
            const uint32_t st = smem_base + s * stage_bytes;
            const uint64_t a0 = smem_desc_sw128(st), a1 = smem_desc_sw128(st + a_bytes);
            const uint64_t b0 = smem_desc_sw128(st + 2 * a_bytes);
            const uint64_t b1 = smem_desc_sw128(st + 2 * a_bytes + b_bytes);
#pragma unroll
            for (int k = 0; k < 4; ++k)  // + 32 bytes per k-step: 2 in the address field
              tc_mma2_bf16(tmem_acc, a0 + 2 * k, b0 + 2 * k, idesc, (it > 0 || k > 0) ? 1u : 0u);
#pragma unroll
            for (int k = 0; k < 4; ++k) tc_mma2_bf16(tmem_acc, a1 + 2 * k, b1 + 2 * k, idesc, 1u);
            commit_pair_mask(empty_bar(s), pair_mask);
          } else {
            lora_products(it - n_main, s);
          }
        }
        __syncwarp();
        if (++s == p.stages) {
          s = 0;
          ph ^= 1;
        }
      }
      // arrives in both CTAs once every product issued above is done (after an abort too)
      if (elect_one()) commit_pair_mask(acc_full, pair_mask);
      __syncwarp();
    }
    volatile int no_abort = 0;
    warp_wait_bounded(acc_full, 0, &no_abort, p.err, kDevTimeoutDrain);
  }
  // (waited for once: with kCopy the barrier may have completed again by the next look)
  bool epi_ok = mbar_wait_bounded(acc_full, 0, abort_flag, p.err, kDevTimeoutEpilogue);
  if constexpr (kCopy) {
    // y_on's sums go on from y_off's, which stay: every warp copies its part (three per quarter of
    // the TMEM lanes), then the LoRA products accumulate on the copy while y_off is drained
    tc_fence_after();
    if (__all_sync(0xffffffffu, epi_ok) && (warp & 3) * 32 < nrow) {
      const uint32_t from = tmem_acc + (static_cast<uint32_t>((warp & 3) * 32) << 16);
#pragma unroll 1
      for (int c = 16 * (warp >> 2); c < p.bn; c += 48) {
        uint32_t v[16];
        tc_ld_32x32b_x16(from + c, v);
        tc_wait_ld();
        tc_st_32x32b_x16(from + p.lcol + c, v);
      }
      tc_wait_st();
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(map_to_rank(copied, lead_rank));
    if (warp == 1 && leader) {
      const bool all = warp_wait_cluster_bounded(copied, 0, abort_flag, p.err, kDevTimeoutMma);
      tc_fence_after();
      for (int it = n_main; all && it < items; ++it) {
        const int s = it % p.stages;
        if (!warp_wait_bounded(full_bar(s), (it / p.stages) & 1, abort_flag, p.err, kDevTimeoutMma)) break;
        tc_fence_after();
        if (elect_one()) lora_products(it - n_main, s);
        __syncwarp();
      }
      if (elect_one()) commit_pair_mask(acc_full, pair_mask);
      __syncwarp();
    }
  }
  // ---------------------------------------------------------------------- drain: every warp,
  // three per quarter of the TMEM lanes
  constexpr int kDrainers = 3;
  epi_ok = __all_sync(0xffffffffu, epi_ok) && *abort_flag == 0;
  if (kEpi == EPI_LOGSOFTMAX) epi_ok = __syncthreads_and(epi_ok);  // a quarter's warps meet again
  tc_fence_after();
  if (!kEarly) pdl_launch_dependents();

  const int q = warp & 3;             // TMEM lanes 32 q .. of a drain warp
  const int trow = q * 32 + lane;     // row of the segment
  // which of the warps of its lanes; the first ones, which have had the main loop, take the fewer chunks
  const int par = kDrainers - 1 - (warp >> 2);
  const bool drain = epi_ok && q * 32 < nrow;
  const bool last = slice == p.ks - 1;
  constexpr int kChunk = chunk_of(kEpi);
  const int nch = p.bn / kChunk;      // column chunks of the tile
  // the slice that finishes chunk i (two slices: halves of the columns, or of the pairs), and
  // the chunk's index among those it finishes
  auto owner = [&](int i) {
    return p.ks == 1 ? 0 : (paired_epi(kEpi) ? (i % (nch / 2)) / (nch / 4) : i / (nch / 2));
  };
  auto pos_of = [&](int i) {
    return p.ks == 1 ? 0 : (paired_epi(kEpi) ? i % (nch / 4) + (i / (nch / 2)) * (nch / 4) : i % (nch / 2));
  };
  RowSums rs;
  rs.taddr = tmem_acc + (static_cast<uint32_t>(q * 32) << 16);
  rs.on_col = kCopy ? p.lcol : 0;
  rs.lcol = p.lcol;
  rs.own_lora = p.ks == 2 && last && lora_me;
  rs.row = trow;
  rs.recv = nullptr;
  rs.lplane = 0;
  if (p.ks == 2) {
    const int plane = p.bn / 2 / 4 * 128;  // float4 of one slice's sums
    float4* xch = reinterpret_cast<float4*>(smem);
    cluster_sync_all();  // both slices' products are done: the rings are free
    if (drain) {
      const uint32_t dst0 = map_to_rank(smem_u32(xch + trow), static_cast<uint32_t>(2 * (1 - slice) + half));
      for (int i = par; i < nch; i += kDrainers) {
        if (owner(i) == slice) continue;
        uint32_t v[kChunk], l[kChunk];
        ld_cols(rs.taddr + kChunk * i, v);
        if (rs.own_lora) ld_cols(rs.taddr + p.lcol + kChunk * i, l);
        tc_wait_ld();
        if (rs.own_lora && !p.both) {
#pragma unroll
          for (int j = 0; j < kChunk; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(l[j]));
        }
        const uint32_t dst = dst0 + pos_of(i) * (kChunk / 4 * 128 * 16);
        if (trow < nrow) {
#pragma unroll
          for (int j = 0; j < kChunk / 4; ++j) st_cluster_f4(dst + j * 2048, v + 4 * j);
          if (rs.own_lora && p.both) {
#pragma unroll
            for (int j = 0; j < kChunk / 4; ++j) st_cluster_f4(dst + plane * 16 + j * 2048, l + 4 * j);
          }
        }
      }
    }
    rs.recv = xch;
    rs.lplane = p.both && slice == 0 ? plane : 0;
    tc_fence_before();
    cluster_sync_all();  // the other slice's sums have landed
    tc_fence_after();
  }
  if (drain) {
    pdl_wait();  // outputs are written only after the preceding kernel
    const bool live = trow < nrow;
    const int row = m0 + trow;
    const Staging st{reinterpret_cast<uint4*>(smem + p.stg_off) + warp * 256, lane, nrow - q * 32};
    const size_t warp_row = static_cast<size_t>(m0 + q * 32);
    constexpr size_t elem = kEpi == EPI_STORE_F32 || kEpi == EPI_RESIDUAL ? 4 : 2;
    for (int o = 0; o < 2; ++o) {
      void* y;
      bool lora;
      if (p.shared_x) {
        y = p.y[o];
        lora = o == 1;
      } else {
        y = o == 0 ? p.y[stream] : nullptr;
        lora = true;
      }
      if (y == nullptr) continue;
      if (kCopy && (o == 1 || p.lora_first)) {  // the LoRA products are done
        if (!warp_wait_bounded(acc_full, 1, abort_flag, p.err, kDevTimeoutEpilogue)) break;
        tc_fence_after();
      }
      if constexpr (kEpi == EPI_LOGSOFTMAX) {
        emit_lsm(p, rs, row, live, n0, static_cast<float2*>(y),
                 p.lsm_target + ((p.shared_x ? o : stream) == 0 ? 0 : p.M), lora, par, q,
                 reinterpret_cast<float2*>(smem + p.stg_off) + q * 64);
      } else if constexpr (!paired_epi(kEpi)) {
        for (int i = par; i < nch; i += kDrainers) {
          if (owner(i) != slice || n0 + 32 * i >= p.N) continue;
          float v[32];
          rs.get(32 * i, pos_of(i), lora, v);
          store32<kEpi>(p, st, static_cast<uint8_t*>(y) + warp_row * p.N * elem, n0 + 32 * i, v);
        }
      } else {
        for (int i = par; i < nch / 2; i += kDrainers) {
          if (owner(i) != slice) continue;
          float v[kChunk], z[kChunk];
          rs.get(kChunk * i, pos_of(i), lora, v);
          rs.get(kChunk * (i + nch / 2), pos_of(i + nch / 2), lora, z);
          store_pair16<kEpi>(p, st, y, row, n0 / 2 + kChunk * i, v, z);
        }
      }
    }
  }
  if (kCopy && warp < 3) {  // the LoRA items, as above
    volatile int no_abort = 0;
    if (warp == 1) warp_wait_bounded(acc_full, 1, &no_abort, p.err, kDevTimeoutDrain);
    for (int k = n_main; warp != 1 && k < loaded; ++k)
      warp_wait_bounded(empty_bar(k % p.stages), (k / p.stages) & 1, &no_abort, p.err, kDevTimeoutDrain);
  }
  tc_fence_before();
  // no CTA leaves while a peer may touch its barriers or shared memory. Relaxed: nothing is
  // published here, and a releasing arrive would wait for the outputs to reach memory (2 us)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  __syncwarp();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc),
                 "r"(p.tmem_cols)
                 : "memory");
  }
}

}  // namespace smallm
// ------------------------------------------------------------------ host side

namespace {

using smallm::kBarBytes;
using smallm::kMaxStages;
using smallm::kSmemMax;

int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }
int pow2_at_least(int v) {
  int p = 32;
  while (p < v) p *= 2;
  return p;
}

struct Shape {  // what the launch needs besides the arguments
  int streams, nseg, seg, row_tiles, ks;
  bool lora, both, paired;
};

struct Config {
  int bn, stages;
  int stg_off, bar_off, smem;
};

// Shared-memory layout for a tile width; false if it does not fit with 3 stages.
bool lay_out(const Shape& s, int bn, Config* c) {
  const int stage = 2 * (s.seg * 128 + bn * 64);
  const int xch = s.ks == 2 ? bn / 2 * 128 * 4 * (s.both ? 2 : 1) : 0;
  int st = (kSmemMax - 1024 - kBarBytes) / stage;
  if (st > kMaxStages) st = kMaxStages;
  if (st < 3) return false;
  // the products read 128 rows of an x box, whatever its height: the last one stays inside
  int ring = st * stage;
  const int last = (st - 1) * stage + s.seg * 128 + 16384;
  if (last > ring) ring = last;
  const int over = xch + smallm::NUM_THREADS / 32 * 4096;  // exchange buffer and the drain warps' staging, over the ring
  const int end = ((ring > over ? ring : over) + 15) / 16 * 16;
  if (end + 1024 + kBarBytes > kSmemMax) return false;
  c->bn = bn;
  c->stages = st;
  c->stg_off = xch;
  c->bar_off = end;
  c->smem = end + 1024 + kBarBytes;
  return true;
}

using Kernel = void (*)(smallm::Maps, smallm::Params);
template <bool kCopy>
Kernel kernel_of(int epi) {
  switch (epi) {
    case smallm::EPI_SWIGLU: return smallm::lora_gemm_small_kernel<smallm::EPI_SWIGLU, kCopy>;
    case smallm::EPI_RESIDUAL: return smallm::lora_gemm_small_kernel<smallm::EPI_RESIDUAL, kCopy>;
    case smallm::EPI_ROPE: return smallm::lora_gemm_small_kernel<smallm::EPI_ROPE, kCopy>;
    case smallm::EPI_LOGSOFTMAX: return smallm::lora_gemm_small_kernel<smallm::EPI_LOGSOFTMAX, false>;
    case smallm::EPI_STORE_F32: return smallm::lora_gemm_small_kernel<smallm::EPI_STORE_F32, kCopy>;
    default: return smallm::lora_gemm_small_kernel<smallm::EPI_STORE, kCopy>;
  }
}

// Lets every kernel have kSmemMax of shared memory (needed before the occupancy query, too).
bool allow_smem(int dev) {
  static bool done[64] = {false};
  if (dev < 0 || dev >= 64) return false;
  if (done[dev]) return true;
  for (int e = smallm::EPI_STORE; e <= smallm::EPI_STORE_F32; ++e)
    for (Kernel k : {kernel_of<false>(e), kernel_of<true>(e)})
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) return false;
  return done[dev] = true;
}

// Clusters of 2 ks CTAs that the device holds at once (0: none, or it does not say, which is not kept).
// Every layout takes more than half of an SM's shared memory (131 KB and more), so an SM holds
// one CTA whatever the width and the epilogue: 76 and 36 on GB300 from 116 KB up.
int resident_clusters(int dev, int ks) {
  static std::atomic<int> known[64][2];  // the answer + 1; dev < 64: allow_smem
  int n = known[dev][ks - 1].load(std::memory_order_relaxed) - 1;
  if (n >= 0) return n;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * ks * 128));
  cfg.blockDim = dim3(smallm::NUM_THREADS);
  cfg.dynamicSmemBytes = kSmemMax;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(2 * ks);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, smallm::lora_gemm_small_kernel<smallm::EPI_STORE, false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  known[dev][ks - 1].store(n + 1, std::memory_order_relaxed);
  return n;
}

// Split of K between the two pairs of a cluster (36 of these fit on the chip) where 256-column
// tiles of two streams leave most pairs idle and half of K is worth the exchange of the sums,
// about 3 us. Measured, one slice against two, us, two streams: 4 to 12 tiles, 20 x 1024 x 776
// -4 % to 200 x 1024 x 1536 +18 %, 200 x 2048 x 1536 +4 %, 97 x 3200 x 3000 -5 %; 16 tiles,
// 128 x 2048 x 4096 +6 %, 97 x 4096 x 4096 -9 %; 24 tiles, 449 x 3200 x 1536 +26 %,
// 200 x 6000 x 3000 -1 %; 32 tiles, 200 x 4096 x 4096 +21 %, 200 x 11008 x 4096 +8 %.
int k_slices(int64_t M, int64_t K, int64_t N) {
  const int64_t kb = (K + smallm::BK - 1) / smallm::BK;
  const int64_t tiles = (M + 127) / 128 * ((N + 255) / 256);
  const int64_t kb_min = tiles <= 12 ? 16 : (tiles <= 18 ? 20 : 40);
  return tiles <= 24 && kb >= kb_min ? 2 : 1;
}

Shape shape_of(int64_t M, int streams, int epi, int ks) {
  Shape s{};
  s.streams = streams;
  s.nseg = static_cast<int>((M + 127) / 128);
  s.ks = ks;
  if (s.streams == 1 && (s.nseg & 1)) ++s.nseg;
  s.seg = static_cast<int>(((M + s.nseg - 1) / s.nseg + 7) / 8 * 8);
  s.row_tiles = (s.streams * s.nseg + 1) / 2;
  s.paired = smallm::paired_epi(epi);
  return s;
}

int64_t tiles_of(const Shape& s, int64_t N, int epi, int bn) {
  const int64_t npair = epi == smallm::EPI_SWIGLU ? N / 2 : (N + 127) / 128 * 64;
  return s.row_tiles * (s.paired ? (npair + bn / 2 - 1) / (bn / 2) : (N + bn - 1) / bn);
}
// partner rows of W that are neighbours
int box_of(int epi) { return epi == smallm::EPI_SWIGLU ? 128 : 64; }

// Tile width: the fewest clocks over the waves (returned; `best` keeps bn = 0 if none fits). A
// k-block of 64 costs the pair its products (2 bn) or a CTA's fill from L2 at 64 B per clock
// (2 (seg + bn / 2)), and a wave `per_wave` clocks of set-up, first loads and drain.
double choose_width(const Shape& s, int64_t K, int64_t N, int epi, int dev, double per_wave, Config* best) {
  const int64_t kb = (K + smallm::BK - 1) / smallm::BK;
  const int fit = resident_clusters(dev, s.ks);
  double best_t = 1e30;
  if (fit < 1) return best_t;
  for (int bn : {256, 224, 192, 160, 128, 96, 64}) {
    if (s.ks == 2 && bn % (s.paired ? 128 : 64) != 0) continue;  // whole chunks for each slice
    if (s.paired && bn / 2 / gcd(bn / 2, box_of(epi)) > smallm::kMaxBoxes) continue;
    if (epi == smallm::EPI_LOGSOFTMAX && bn != 256) continue;
    Config c{};
    if (!lay_out(s, bn, &c)) continue;
    const int fill = 2 * (s.seg + bn / 2), mma = 2 * bn;
    const double item = 2.0 * (fill > mma ? fill : mma);
    const int64_t waves = (tiles_of(s, N, epi, bn) + fit - 1) / fit;
    const double t = waves * (static_cast<double>((kb + s.ks - 1) / s.ks) * item + per_wave);
    if (t < best_t) {
      best_t = t;
      *best = c;
    }
  }
  return best_t;
}

}  // namespace

bool few_rows_halves(int64_t M, int64_t K, int64_t N) {
  if (M < 1 || M > 512 || (M > 448 && K > 4096) || K >= (1LL << 28) || k_slices(M, K, N) != 2) return false;
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && allow_smem(dev) && resident_clusters(dev, 2) > 0;
}

// Measured over 8 to 512 rows, K 256 to 11008 and N 1024 to 65536 (GB300, us in a graph with the call's
// lora_down of rank 16, this kernel / the tile kernel of lora_gemm_tc.cu, two streams unless said):
//  * up to 128 rows that kernel's 128 x 256 tiles leave most SMs idle until the columns fill them:
//    97 x 4096 x 4096 13.7 / 31.2, x 12288 26.4 / 35.0, x 16384 32.1 / 37.4; but 40 x 256 x 22016 13.0 /
//    10.3, x 65536 28.5 / 17.5. A long K is worth a second wave: 97 x 1024 x 22016 20.7 / 22.7,
//    97 x 2048 x 32000 38.0 / 38.8, 97 x 4096 x 65536 116 / 120. One stream has one of that kernel's
//    tiles where two have one of these: 40 x 1024 x 22016 19.0 / 19.1, 97 x 2048 x 32000 36.4 / 33.2;
//  * up to 256, where a stream is one 256-row tile there: 200 x 512 x 9216 11.1 / 11.5, x 11008 15.0 /
//    13.5, 200 x 2048 x 11008 26.0 / 27.4, 200 x 4096 x 12288 42.0 / 43.9;
//  * up to 384, where it is two and the second half empty: 300 x 1024 x 6144 13.8 / 17.4, x 8192 19.3 /
//    19.0, x 12288 24.0 / 24.6, x 14336 30.1 / 25.4, 300 x 4096 x 16384 69.9 / 78.2;
//  * up to 512: 448 x 1024 x 4096 13.7 / 14.2, x 5120 17.8 / 17.2, 448 x 4096 x 5120 37.1 / 43.3.
// Three streams leave a row segment over in a pair, or a wave, more often (97 x 4096 x 12288 45.5 /
// 40.2, 300 x 512 x 12288 35.7 / 25.0, but 97 x 4096 x 4096 23.7 / 34.9): the clocks of both are
// estimated, with shares per wave and a margin that choose within 0.4 % of the better kernel over 875
// sizes, 7 of them slower by more than 3 %.
bool few_rows_kernel_wins(int64_t M, int64_t K, int64_t N, int streams) {
  if (M < 1 || M > 512 || K >= (1LL << 28) || N > 64 * 65535) return false;
  const bool up_to_5k = N <= 5632 && (M <= 448 || K <= 4096);
  bool wanted;
  if (streams == 1)
    wanted = M <= 128   ? N <= 16384 || (K >= 4096 && N <= 24000)
             : M <= 256 ? N <= 14336
             : M <= 384 ? N <= 11264 || (K >= 4096 && N <= 13824)
                        : up_to_5k;
  else if (streams == 2)
    wanted = M <= 128   ? N <= 16384 || K >= 4096 || (K >= 2048 && N <= 40000) || (K >= 1024 && N <= 24000)
             : M <= 256 ? N <= 9600 || (K >= 2048 && N <= 11264) || (K >= 4096 && N <= 13824)
             : M <= 384 ? N <= 7168 || (N > 10240 && N <= 12800) || (K >= 2048 && N <= 12800) || (K >= 4096 && N <= 16384)
                        : up_to_5k && (N <= 4608 || K >= 2048);
  else
    wanted = M <= 128   ? true
             : M <= 256 ? N <= 11264 || (K >= 2048 && N <= 14336)
             : M <= 384 ? N <= 16384
                        : N <= 5120 && (M <= 448 || K <= 4096);
  int dev = 0;
  if (!wanted || cudaGetDevice(&dev) != cudaSuccess || !allow_smem(dev) || resident_clusters(dev, 1) < 1) return false;
  if (streams < 3) return true;
  Config c{};
  const double here = choose_width(shape_of(M, streams, smallm::EPI_STORE, 1), K, N, smallm::EPI_STORE, dev, 10000.0, &c);
  const int64_t kb = (K + 63) / 64, cols = (N + 255) / 256;
  // that kernel: 128-row tiles, 704 clocks of fill per k-block, on the SMs; 256-row tiles, 512 of
  // products, on pairs of them
  const int64_t nsm = sm_count(), units = M <= 128 ? nsm : nsm / 2;
  if (units < 1) return false;
  const int64_t tiles = streams * cols * (M <= 128 ? 1 : (M + 255) / 256);
  const int64_t waves = (tiles + units - 1) / units;
  const double there = static_cast<double>(waves * kb) * (M <= 128 ? 704 : 512) + 12000.0 + 1000.0 * (waves - 1);
  return c.bn != 0 && 1.1 * here < there;
}

int launch_dual_lora_gemm_small(const GemmArgs& a, cudaStream_t stream) {
  using namespace smallm;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || !allow_smem(dev)) return -1;
  const bool tri = a.x_crit != nullptr && !a.shared_x;
  const int M = static_cast<int>(a.M), N = static_cast<int>(a.N);
  const int kb = static_cast<int>((a.K + BK - 1) / BK);
  const bool lora_on = a.r > 0 && a.u != nullptr && a.B != nullptr && a.y_on != nullptr;
  // Up to 128 rows of one input with LoRA go as two streams: a CTA has one output to drain, and the
  // sums of y_on need no copy (40 x 1024 x 4096 8.9 us as one stream, 8.0 as two; 97 x 4096 x 12288
  // 26.3, 25.9).
  const int ks = a.epi != EPI_LOGSOFTMAX && few_rows_halves(a.M, a.K, a.N) ? 2 : 1;
  const bool shared = a.shared_x && !(a.M <= 128 && lora_on && a.y_off != nullptr && ks == 1);
  const bool lora_crit = tri && a.r > 0 && a.u_crit != nullptr && a.B_crit != nullptr && a.y_crit != nullptr;
  Shape s = shape_of(a.M, shared ? 1 : (tri ? 3 : 2), a.epi, ks);
  s.lora = lora_on || lora_crit;
  s.both = shared && lora_on && a.y_off != nullptr;
  Config best{};
  choose_width(s, a.K, a.N, a.epi, dev, 6000.0, &best);
  if (best.bn == 0) return -4;
  const int bn = best.bn;

  Params p{};
  p.b_box = s.paired ? gcd(bn / 2, box_of(a.epi)) : bn / 2;
  Maps mp;
  const void* xs[3] = {a.x_off, a.shared_x ? a.x_off : a.x_on, a.x_crit};
  for (int i = 0; i < 3; ++i) {
    if (i >= s.streams) mp.x[i] = mp.x[0];
    else if (!make_tma_map(&mp.x[i], xs[i], a.M, a.K, a.K, s.seg, false)) return -2;
  }
  if (!make_tma_map(&mp.w, a.W, a.N, a.K, a.K, p.b_box, false)) return -2;
  for (int i = 0; i < 2; ++i) {
    if (i == 0 ? lora_on : lora_crit) {
      if (!make_tma_map(&mp.u[i], i == 0 ? a.u : a.u_crit, a.M, a.r, a.r, s.seg, false)) return -2;
      if (!make_tma_map(&mp.b[i], i == 0 ? a.B : a.B_crit, a.N, a.r, a.r, p.b_box, false)) return -2;
    } else {  // never read
      mp.u[i] = mp.x[0];
      mp.b[i] = mp.w;
    }
  }
  p.M = M;
  p.N = N;
  p.streams = s.streams;
  p.nseg = s.nseg;
  p.seg = s.seg;
  p.row_tiles = s.row_tiles;
  p.kb_main = kb;
  p.kb_lora = s.lora ? static_cast<int>((a.r + BK - 1) / BK) : 0;
  p.r = static_cast<int>(a.r);
  p.bn = bn;
  p.ks = s.ks;
  p.stages = best.stages;
  p.shared_x = shared ? 1 : 0;
  p.both = s.both ? 1 : 0;
  p.has_on = lora_on ? 1 : 0;
  p.has_crit = lora_crit ? 1 : 0;
  p.x_settled = a.x_settled ? 1 : 0;
  const bool second = s.ks == 2 ? s.lora : s.both;
  p.lcol = second ? pow2_at_least(bn) : 0;
  p.tmem_cols = static_cast<uint32_t>(pow2_at_least(bn) * (second ? 2 : 1));
  p.stg_off = best.stg_off;
  if (s.both && s.ks == 1) {
    // y_off is drained while the LoRA items are still read: through the stages before or after them
    const int stage = 2 * (s.seg * 128 + bn * 64), first = kb % best.stages;
    const int staging = NUM_THREADS / 32 * 4096, wrapped = first + p.kb_lora > best.stages ? stage : 0;
    p.stg_off = first * stage - wrapped >= staging ? wrapped : (first + p.kb_lora) * stage;
    if (p.stg_off + staging > best.stages * stage) {  // two items in the middle of a short ring
      p.stg_off = best.stg_off;
      p.lora_first = 1;
    }
  }
  p.bar_off = best.bar_off;
  p.y[0] = a.y_off;
  p.y[1] = a.y_on;
  p.y[2] = tri ? a.y_crit : nullptr;
  p.rope_P = static_cast<int>(a.rope_P < 1 ? 1 : a.rope_P);
  p.rope_cols = static_cast<int>(a.rope_cols);
  p.rope_table = static_cast<const float2*>(a.rope_table);
  p.lsm_target = a.lsm_target;
  p.lsm_ids = a.lsm_ids;
  p.lsm_L = static_cast<int>(a.lsm_L < 1 ? 1 : a.lsm_L);
  p.lsm_ids_ld = static_cast<int>(a.lsm_ids_ld);
  p.lsm_ids_off = static_cast<int>(a.lsm_ids_off);
  p.lsm_tiles = (N + 255) / 256;
  p.err = a.err;
  const int64_t tiles = tiles_of(s, a.N, a.epi, bn);

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * s.ks), static_cast<unsigned>(s.row_tiles),
                     static_cast<unsigned>(tiles / s.row_tiles));
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = static_cast<size_t>(best.smem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(2 * s.ks);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const int epi = a.epi == EPI_STORE && a.out_f32 ? EPI_STORE_F32 : a.epi;
  return cudaLaunchKernelEx(&cfg, s.both && s.ks == 1 ? kernel_of<true>(epi) : kernel_of<false>(epi), mp, p) == cudaSuccess ? 0 : -3;
}

}  // namespace hydra
