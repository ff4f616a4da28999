// One decode step of a SMALL batch (at most 64 samples, at d = 1024 at most 32: as many as leave room for the weights of a
// layer beside their activations in shared memory) as a single persistent kernel.
//
// With a handful of rows the step is bound by reading the weights once (the mid model: 334 MB, 50 us at HBM speed)
// and by the latency of its dependent phases, not by arithmetic. The whole step -- embedding, L x (token-mixer cache
// update [Eq. 2, Eq. 3], feed-forward up and down), final norm, LM head, greedy selection -- runs in ONE cooperative
// kernel of 128 CTAs, 32 clusters of four (the largest clusters that fit on that many SMs: 33 of four, 15 of eight). Two grid-wide barriers per layer remain, after the up projection (a
// down slab reads all of its part of H) and after the down projection (a row needs all of x):
//   - row phase: every cluster computes every row (embedding or x, LN1, cache update, residual, LN2), rank r the rows
//     r, r + 4, ..., two warps per row, and sends the activation row to the shared memory of its four CTAs, so the
//     rows need no grid barrier of their own; up to kAloneRows rows every CTA computes all of them for itself. The new
//     cache row is kept in shared memory and written by one CTA of the grid after the next grid barrier, when nobody
//     reads the old one any more;
//   - up projection: every CTA computes F / 128 columns of H = gelu(a W1^T + b1) and stores them;
//   - down projection: cluster c computes d / 32 columns of x, rank r over the r-th quarter of K; the four partial
//     products meet in shared memory (each rank receives those of its quarter of the cluster's columns) and are added
//     in rank order, so x is written once, complete.
// W1 and W2 slabs have a region of shared memory each, refilled for the next layer by bulk copies as
// soon as they have been used: the weight stream runs a whole layer ahead of the barriers. The small parameter
// vectors and cache rows of the next layer are prefetched into L2 meanwhile. The contractions run on mma.sync (m16n8k16, bf16 in, fp32 accumulate): the kernel is bound by
// latency and HBM, and a tcgen05 tile would be mostly padding. K of a tile is cut into up to eight ranges that
// different warps take, fewer with more row tiles (batches of 1 to 16, 17 to 32, 33 to 64 rows add in different orders).
//
// Every wait (grid barrier, mbarrier) is bounded: on a time-out the CTA raises kStatusWaitTimeout and runs through
// the remaining phases without waiting, so the kernel always ends.
#pragma once

#include "common.cuh"
#include "gemm_tc.cuh"      // mbarrier helpers, gelu_fast
#include "mixer.cuh"        // row_stats_full
#include "mixer_stream.cuh" // bulk_g2s
#include "prefill_chunk.cuh" // ld_acquire_u32
#include "select.cuh"       // SelectOut, write_token

namespace srm {
namespace sb {

constexpr int kThreads = 512, kWarps = 16;
constexpr int kCluster = 4, kClusters = 32, kGrid = kCluster * kClusters;
constexpr int kMaxRows = 64;                 // samples per launch
constexpr int kAloneRows = 4;                // up to this many rows every CTA computes all rows for itself
constexpr int kPadBytes = 16;                // row padding in shared memory: ldmatrix rows land in distinct banks
constexpr int kLmChunkCols = 16;             // LM-head weight rows per pipeline stage
constexpr int kLmMaxStages = 6;
constexpr int kHeadBytes = 128 + 256;        // mbarriers and flags, row-phase sums
constexpr int kRowParamVecs = 5;              // parameter vectors of the row phase kept in shared memory
constexpr int kMaxGroups = 8;                // ranges that K of a tile is cut into
constexpr int kSmemBytes = 227 * 1024;
constexpr long long kBarrierLimitCycles = 1ll << 27;

struct LayerW {
  const float *ln1_g, *ln1_b, *ln2_g, *ln2_b, *alpha, *beta, *lam, *b1, *b2;
  const bf16 *W1, *W2;
};

struct Params {
  int B, d, F, V, h, n_ctx, L, t;
  float eps;
  const int32_t* tok_in;       // [B]
  const bf16* E;               // [V, d]
  const bf16* W_lm;            // [V, d]
  const float *lnf_g, *lnf_b;
  LayerW layer0;               // tensors of layer 0; layer l lies layer_bytes further on (all layers have one layout)
  int64_t layer_bytes;
  void* S;                     // cache of layer 0; layer l at S + l * layer_stride (bytes)
  int64_t layer_stride;
  float* x;                    // [B, d] residual stream
  bf16* H;                     // [B, F]
  float* logits;               // [B, V] or nullptr (then only the greedy selection leaves the kernel)
  unsigned long long* best;    // [B] (sortable logit, ~column) maxima, zero on entry
  uint32_t* bar;               // [kGrid] words of the grid barrier, then the count of CTAs done with the LM head; zero on entry
  uint32_t* status;
  const int32_t* ctr;          // device-side step counters or nullptr
  const int32_t* pos;          // [B] per-row positions or nullptr
  int greedy;                  // select inside the kernel
  SelectOut out;
  // shared-memory plan (host): byte offsets
  int off_w1, off_w2, off_part, off_recv, off_xo, off_s;
  int lm_stages;               // stages of LM-head rows from off_w1 on
  int lm_stages_w1;            // ... of which lie inside the W1 region
};

// Sizes of the slabs a CTA works on.
__host__ __device__ inline int up_cols(int F) { return F / kGrid; }
__host__ __device__ inline int dn_cols(int d) { return d / kClusters; }
__host__ __device__ inline int dn_klen(int F) { return F / kCluster; }

// The shared-memory plan for B rows; false when it does not fit. Fills the off_* / lm_* fields of p.
inline bool smem_plan(int B, int d, int F, int state_elem, Params* p, size_t* bytes) {
  const int mp = (B + 15) / 16 * 16, ld_d = 2 * d + kPadBytes, ld_k = 2 * dn_klen(F) + kPadBytes;
  const int act = mp * (ld_d > ld_k ? ld_d : ld_k);
  const int w1 = (up_cols(F) + 15) / 16 * 16 * ld_d, w2 = (dn_cols(d) + 15) / 16 * 16 * ld_k, stage = kLmChunkCols * ld_d;
  int recv = kCluster * mp * (dn_cols(d) / kCluster) * 4;
  const int part = kWarps * 1024, xo = mp * (dn_cols(d) / kCluster) * 4;
  const int srow = d * state_elem;
  if (part + recv < kRowParamVecs * d * 4) recv = kRowParamVecs * d * 4 - part;      // the row phase's parameters lie there
  int w = w1 + w2;
  if (w < 2 * stage) w = 2 * stage;
  const int fixed = kHeadBytes + act + part + recv + (xo + 15) / 16 * 16 + srow;
  if (fixed + w > kSmemBytes) return false;
  while (w + stage <= kLmMaxStages * stage && fixed + w + stage <= kSmemBytes) w += stage;       // a deeper LM-head ring
  p->off_w1 = kHeadBytes + act;
  p->off_w2 = p->off_w1 + w1;
  p->lm_stages = w / stage < kLmMaxStages ? w / stage : kLmMaxStages;
  p->lm_stages_w1 = w1 / stage;
  p->off_part = p->off_w1 + w;
  p->off_recv = p->off_part + part;
  p->off_xo = p->off_recv + recv;
  p->off_s = p->off_xo + (xo + 15) / 16 * 16;
  *bytes = (size_t)(fixed + w);
  return true;
}

template <typename P>
__device__ __forceinline__ LayerW layer_w(const P& p, int l) {
  const int64_t o = (int64_t)l * p.layer_bytes;
  auto f = [o](const float* q) { return reinterpret_cast<const float*>(reinterpret_cast<const uint8_t*>(q) + o); };
  auto b = [o](const bf16* q) { return reinterpret_cast<const bf16*>(reinterpret_cast<const uint8_t*>(q) + o); };
  const LayerW& w = p.layer0;
  return LayerW{f(w.ln1_g), f(w.ln1_b), f(w.ln2_g), f(w.ln2_b), f(w.alpha), f(w.beta), f(w.lam), f(w.b1), f(w.b2), b(w.W1), b(w.W2)};
}

__device__ __forceinline__ void red_release_inc(uint32_t* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
// eight bytes into the shared memory of a CTA of the cluster, counted on a barrier over there
__device__ __forceinline__ void st_async_v2(uint32_t addr, float a, float b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
               ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}
// shared memory of this CTA -> shared memory of a CTA of the cluster, bytes counted on a barrier over there
__device__ __forceinline__ void bulk_s2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(tc::smem_u32(src)), "r"(bytes), "r"(bar) : "memory");
}

// ---- grid-wide barrier ------------------------------------------------------------------------
// Arrive / wait on a monotonically increasing counter: barrier number n (1, 2, ...) is passed when the counter
// has reached n * gridDim.x. All CTAs are resident (cooperative launch), so the wait ends; it is bounded anyway.
// One thread polls, with relaxed loads and one acquire at the end (an acquiring poll drops the L1 cache every time; a
// word per CTA polled by 128 threads that way took 4 us instead of 1.2). `between` runs in all threads between arriving
// and waiting.
struct GridBarrier {
  uint32_t* ctr;
  uint32_t n;          // barriers passed so far
  bool dead;           // a wait timed out: stop waiting (the same value in every thread of the CTA)
  uint32_t* status;
  template <typename F>
  __device__ __forceinline__ void sync(F&& between) {
    __syncthreads();
    ++n;
    if (threadIdx.x == 0) red_release_inc(ctr);
    between();
    bool late = false;
    if (threadIdx.x == 0 && !dead) {
      const uint32_t want = n * gridDim.x;
      const long long t0 = clock64();
      while (ld_relaxed_u32(ctr) < want) {
        if (clock64() - t0 > kBarrierLimitCycles) { late = true; raise_status(status, kStatusWaitTimeout); break; }
      }
      ld_acquire_u32(ctr);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");      // what `between` has fetched
    dead = __syncthreads_or(late || dead) != 0;
  }
};

// ---- mma.sync m16n8k16 (bf16 x bf16 -> fp32) and its shared-memory fragment loads ----------------
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[8], int o, const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[o]), "+f"(c[o + 1]), "+f"(c[o + 2]), "+f"(c[o + 3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One 16 x 16 output tile over a part of K (klen, a multiple of 32): rows m0.. of A (row-major, lda bytes per row) times
// rows n0 .. n0 + 15 of W (row-major [n][k], ldw bytes per row), both in shared memory from the part's first column on.
// Fragment layout of c: lane l holds c[0], c[1] = (row m0 + l / 4, columns n0 + 2 (l % 4), + 1), c[2], c[3] = the same
// columns of row + 8, c[4..7] = the same eight columns further. Even and odd k-steps accumulate separately (four
// independent chains of dependent mma instructions: with a few rows the tile is latency-bound) and are added at the end.
__device__ __forceinline__ void tile_part(float (&c)[8], uint32_t a_addr, uint32_t b_addr, int klen) {
  float o[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) { c[i] = 0.f; o[i] = 0.f; }
#pragma unroll 4
  for (int k = 0; k < klen; k += 32) {
    uint32_t a[4], b[4], a2[4], b2[4];
    ldsm_x4(a, a_addr + k * 2);
    ldsm_x4(b, b_addr + k * 2);
    ldsm_x4(a2, a_addr + k * 2 + 32);
    ldsm_x4(b2, b_addr + k * 2 + 32);
    mma_bf16(c, 0, a, b[0], b[1]);
    mma_bf16(c, 4, a, b[2], b[3]);
    mma_bf16(o, 0, a2, b2[0], b2[1]);
    mma_bf16(o, 4, a2, b2[2], b2[3]);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) c[i] += o[i];
}

// How the tiles of a product are shared out between the warps: `groups` warps take a tile, a range of klen columns of K
// each.
struct Share { int tiles, groups, klen; };
__device__ __forceinline__ Share share_of(int tiles, int K) {
  int groups = kMaxGroups;
  while (groups > 1 && (groups * tiles > kWarps || groups * 32 > K)) groups >>= 1;
  return Share{tiles, groups, K / groups};
}
// Range g of tile (mt, nt).
__device__ __forceinline__ void tile_group(float (&c)[8], const Share& sh, int g, const uint8_t* A, int lda, int mt, const uint8_t* W,
                                           int ldw, int nt, int lane) {
  // A: matrices (rows 0-7, k 0-7), (rows 8-15, k 0-7), (rows 0-7, k 8-15), (rows 8-15, k 8-15): lane l points at
  // row (l % 16), k offset 8 (l / 16). W: (n 0-7, k 0-7), (n 0-7, k 8-15), (n 8-15, k 0-7), (n 8-15, k 8-15): lane l
  // points at row (l % 8) + 8 (l / 16), k offset 8 ((l / 8) % 2).
  const uint32_t k0 = (uint32_t)(g * sh.klen) * 2;
  const uint32_t a_addr = tc::smem_u32(A + (size_t)(mt * 16 + (lane & 15)) * lda + (lane >> 4) * 16) + k0;
  const uint32_t b_addr = tc::smem_u32(W + (size_t)(nt * 16 + (lane & 7) + ((lane >> 4) << 3)) * ldw + ((lane >> 3) & 1) * 16) + k0;
  tile_part(c, a_addr, b_addr, sh.klen);
}
// Partial sums of the groups: element e = 32 j + lane of (group g, tile) at ((g * tiles + tile) * 256 + e).
__device__ __forceinline__ void put_part(float* part, const Share& sh, int g, int tile, int lane, const float (&c)[8]) {
  float* o = part + (g * sh.tiles + tile) * 256 + lane;
#pragma unroll
  for (int j = 0; j < 8; ++j) o[32 * j] = c[j];
}
__device__ __forceinline__ float sum_groups(const float* q, int stride, int groups) {
  if (groups == 1) return q[0];
  if (groups == 2) return q[0] + q[stride];
  if (groups == 4) return (q[0] + q[stride]) + (q[2 * stride] + q[3 * stride]);
  return ((q[0] + q[stride]) + (q[2 * stride] + q[3 * stride])) + ((q[4 * stride] + q[5 * stride]) + (q[6 * stride] + q[7 * stride]));
}
// Item i (0 .. 128 tiles - 1) of a reduced product: the pair of adjacent columns (row, col), (row, col + 1) of a tile.
struct Pair { int row, col; float a, b; };
__device__ __forceinline__ Pair take_pair(const float* part, const Share& sh, int i, int m_tiles) {
  const int tile = i >> 7, q = (i >> 5) & 3, l = i & 31;
  const float* e = part + tile * 256 + q * 64 + l;           // j = 2 q: columns 8 (q / 2) .., rows 8 (q % 2) ..
  return Pair{(tile % m_tiles) * 16 + (l >> 2) + (q & 1) * 8, (tile / m_tiles) * 16 + (q >> 1) * 8 + 2 * (l & 3),
              sum_groups(e, sh.tiles * 256, sh.groups), sum_groups(e + 32, sh.tiles * 256, sh.groups)};
}

// ---- shared-memory staging --------------------------------------------------------------------
// `rows` rows of `row_bytes` bytes (a multiple of 16), `src_stride` bytes apart in global memory, to rows
// `row_bytes + kPadBytes` apart in shared memory; completion is counted on `bar`. All threads of the CTA call it: one
// announces the bytes, and the bulk copies, one per row, are spread over the warps (a warp issues its lanes' copies one
// after the other: 32 of them from one warp took 0.8 us).
__device__ __forceinline__ void stage_rows(uint8_t* dst, const void* src, int rows, int row_bytes, int64_t src_stride, uint64_t* bar) {
  const int r = (threadIdx.x & 31) * kWarps + (threadIdx.x >> 5);
  if (r < rows) {
    tc::fence_async_smem();        // earlier reads of the region (ordered by a barrier) come before the copies into it
    if (r == 0) tc::mbar_expect_tx(bar, (uint32_t)rows * (uint32_t)row_bytes);
    bulk_g2s(dst + (size_t)r * (row_bytes + kPadBytes), static_cast<const uint8_t*>(src) + (int64_t)r * src_stride, (uint32_t)row_bytes, bar);
  }
}

// Bounded wait on a phase of `bar`; all threads of the CTA call it. False after a time-out.
__device__ __forceinline__ bool wait_stage(uint64_t* bar, uint32_t parity, uint32_t* status, bool dead) {
  if (dead) return false;
  return tc::mbar_wait(bar, parity, status);
}

__device__ __forceinline__ unsigned long long pack_best(float v, int col) {
  return ((unsigned long long)order_key(v) << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)col);
}

// ---- row phase: two warps per row ---------------------------------------------------------------
// (one warp per row spills, and takes 12 us per layer at d = 1024; four warps do a row in the same time as two, but with
// 64 rows the CTA then needs four rounds instead of two, 6.8 us instead of 3.6)
constexpr int kGroups = kWarps / 2;

// LayerNorm statistics of the row that the two warps of a group hold, 4 NT channels per thread: mean and sum of squared
// deviations per thread, merged pairwise (Chan et al.; all counts are equal) over lanes and warps in one pass of shuffles
// and one barrier. `slot`: four floats that this group uses for these statistics only.
template <int d, int NT>
__device__ __forceinline__ void group_stats(const float4 (&v)[NT], float eps, float* slot, int group, float& mean, float& rstd) {
  float m = 0.f, q = 0.f, half_n = 2.f * NT;
#pragma unroll
  for (int i = 0; i < NT; ++i) m += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  m *= 1.0f / (4.f * NT);
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const float a = v[i].x - m, b = v[i].y - m, c = v[i].z - m, e = v[i].w - m;
    q += (a * a + b * b) + (c * c + e * e);
  }
  auto merge = [&half_n](float& m, float& q, float m2, float q2) {
    const float dm = m2 - m;
    q += fmaf(dm * dm, half_n, q2);
    m = 0.5f * (m + m2);
    half_n += half_n;
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), q2 = __shfl_xor_sync(0xffffffffu, q, o);
    merge(m, q, m2, q2);
  }
  if ((threadIdx.x & 31) == 0) {                         // (the lanes may differ in the last bit: lane 0's values count)
    const int w = (threadIdx.x >> 5) & 1;
    slot[w] = m;
    slot[2 + w] = q;
  }
  asm volatile("bar.sync %0, 64;" ::"r"(group + 1) : "memory");
  m = slot[0];
  q = slot[2];
  merge(m, q, slot[1], slot[3]);
  mean = m;
  rstd = rsqrtf(q * (1.0f / (float)d) + eps);
}

// The parameters of a layer's row phase (l == L: of the final norm) in shared memory: ln1_g | ln1_b | beta_t | ln2_g |
// ln2_b, fetched while the CTA waits at the grid barrier before the row phase (kRowParamVecs * d floats in the place of the
// partial sums and the exchange buffer, which are free then).
template <int d>
__device__ __forceinline__ void fetch_row_params(const Params& p, int l, int t, float* dst) {
  const bool last = l == p.L;
  const LayerW w = layer_w(p, last ? 0 : l);
  for (int i = threadIdx.x; i < kRowParamVecs * d / 4; i += kThreads) {
    const int k = i / (d / 4), c = i % (d / 4) * 4;
    const float* q = k == 0 ? w.ln1_g : k == 1 ? w.ln1_b : k == 2 ? w.beta + (int64_t)t * d : k == 3 ? (last ? p.lnf_g : w.ln2_g)
                                                                                                    : (last ? p.lnf_b : w.ln2_b);
    cp_async16(dst + i * 4, q + c);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// The head scalars of a thread's channels at position t: the multipliers of z before and of the sum after (one of them is
// 1), and lambda. Thread `th` of a group owns channels 4 th .. 4 th + 3 (and 256, 512, ... further) of every row.
template <int d, int NT, typename P>
__device__ __forceinline__ void head_scalars(const P& p, const LayerW& w, int t, int th, float (&a1)[NT], float (&a2)[NT], float (&lm)[NT]) {
  const int dh = d / p.h;
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int g = (th * 4 + 256 * i) / dh;
    const float al = __ldg(w.alpha + (int64_t)g * p.n_ctx + t);
    const bool is_row = g < (p.h >> 1);
    a1[i] = is_row ? al : 1.0f;
    a2[i] = is_row ? 1.0f : al;
    lm[i] = __ldg(w.lam + g);
  }
}

template <int d, typename ST>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kThreads, 1) step_small_kernel(const Params p) {
  extern __shared__ __align__(128) uint8_t sm[];
  uint64_t* bar1 = reinterpret_cast<uint64_t*>(sm);      // W1 slab
  uint64_t* bar2 = bar1 + 1;                             // W2 slab
  uint64_t* barA = bar1 + 2;                             // rows of H
  uint64_t* barR = bar1 + 3;                             // activation rows from the other CTAs of the cluster
  uint64_t* barP = bar1 + 4;                             // x + y and the partial products of the owned columns
  uint64_t* barL = bar1 + 5;                             // LM-head stages
  float* red = reinterpret_cast<float*>(sm + 128);       // row-phase sums: eight groups x 8 floats
  uint8_t* sA = sm + kHeadBytes;
  uint8_t* sW1 = sm + p.off_w1;
  uint8_t* sW2 = sm + p.off_w2;
  float* part = reinterpret_cast<float*>(sm + p.off_part);
  uint8_t* recv = sm + p.off_recv;
  uint8_t* xo = sm + p.off_xo;
  ST* sS = reinterpret_cast<ST*>(sm + p.off_s);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cta = blockIdx.x, cl = cta / kCluster, rank = (int)tc::cluster_ctarank();
  const int F = p.F, B = p.B, mp = (B + 15) / 16 * 16, m_tiles = mp / 16;
  constexpr int ld_d = 2 * d + kPadBytes, ncols = d / kClusters, gw = ncols / kCluster;
  const int klen = dn_klen(F), ld_k = 2 * klen + kPadBytes;
  const int ucols = up_cols(F), u0 = (cl * kCluster + rank) * ucols;
  const int n0 = cl * ncols, k0 = rank * klen;
  const int chunks_all = (p.V + kLmChunkCols - 1) / kLmChunkCols;
  const int lm_c0 = (int)((int64_t)cta * chunks_all / kGrid), lm_chunks = (int)((int64_t)(cta + 1) * chunks_all / kGrid) - lm_c0;
  constexpr int lm_stage = kLmChunkCols * ld_d;
  const bool alone = B <= kAloneRows;

  if (tid == 0) {
    for (int i = 0; i < 5 + kLmMaxStages; ++i) tc::mbar_init(bar1 + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::cluster_sync();                                    // every CTA of the cluster is up before anyone writes into its memory
  uint32_t par1 = 0, par2 = 0;
  GridBarrier gb{p.bar, 0u, false, p.status};
  const int t_all = p.ctr != nullptr ? p.ctr[kCtrPos] : p.t;
  auto t_of = [&](int row) { return p.pos != nullptr ? min(max(p.pos[row], 0), p.n_ctx - 1) : t_all; };

  auto stage_up = [&](int l) {            // W1 rows of this CTA's columns
    stage_rows(sW1, layer_w(p, l).W1 + (int64_t)u0 * d, ucols, 2 * d, 2 * (int64_t)d, bar1);
  };
  auto stage_dn = [&](int l) {            // W2 rows of the cluster's columns, this rank's part of K
    stage_rows(sW2, layer_w(p, l).W2 + (int64_t)n0 * F + k0, ncols, 2 * klen, 2 * (int64_t)F, bar2);
  };
  auto stage_lm = [&](int ch) {           // one chunk of LM-head rows into stage ch % lm_stages
    if (ch < lm_chunks) {
      const int r0 = (lm_c0 + ch) * kLmChunkCols, rows = min(kLmChunkCols, p.V - r0), s = ch % p.lm_stages;
      stage_rows(sW1 + s * lm_stage, p.W_lm + (int64_t)r0 * d, rows, 2 * d, 2 * (int64_t)d, barL + s);
    }
  };
  // the row this CTA writes the cache of, and the L2 prefetch of what layer l will ask for
  const int own_row = cl * kCluster + rank;
  auto prefetch_layer = [&](int l) {
    const LayerW w = layer_w(p, l);
    if (warp == 1 && own_row < B) {
      const uint8_t* r = static_cast<const uint8_t*>(p.S) + (int64_t)l * p.layer_stride + (int64_t)own_row * d * sizeof(ST);
      for (int i = lane * 128; i < d * (int)sizeof(ST); i += 32 * 128) prefetch_l2(r + i);
      if (p.pos != nullptr || own_row == 0) {
        const int t = t_of(own_row);
        const float* bt = w.beta + (int64_t)t * d;
        for (int i = lane * 32; i < d; i += 32 * 32) prefetch_l2(bt + i);
        if (lane < p.h) { prefetch_l2(w.alpha + (int64_t)lane * p.n_ctx + t); prefetch_l2(w.lam + lane); }
      }
    }
    if (warp == 2) {                      // CTA i takes one of the vectors, every CTA its part of the bias
      constexpr int lines = d * 4 / 128;
      if (cta < 4 && lane < lines) {
        const float* q = cta == 0 ? w.ln1_g : cta == 1 ? w.ln1_b : cta == 2 ? w.ln2_g : w.ln2_b;
        prefetch_l2(q + lane * 32);
      }
      if (cta == 4 && lane < lines) prefetch_l2(w.b2 + lane * 32);
      if (lane == 0) for (int i = 0; i < ucols; i += 32) prefetch_l2(w.b1 + u0 + i);
    }
  };

  constexpr int NT = d / 256;
  const int group = warp >> 1, c0 = (tid & 63) * 4;
  float a1[NT], a2[NT], lm[NT];
  float* prm = part;                                     // (with the exchange buffer behind it)
  fetch_row_params<d>(p, 0, p.pos != nullptr ? 0 : t_all, prm);
  head_scalars<d, NT>(p, layer_w(p, 0), p.pos != nullptr ? 0 : t_all, tid & 63, a1, a2, lm);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // bytes of the rows that the other CTAs of the cluster send per row phase
  const uint32_t peer_bytes = (uint32_t)(B - (B - rank + kCluster - 1) / kCluster) * (2 * d);
  const uint32_t part_bytes = (uint32_t)((kCluster + 1) * B * gw * 4);       // partial products, and x + y of the owned columns
  if (tid == 0) {
    if (!alone) tc::mbar_expect_tx(barR, peer_bytes);
    tc::mbar_expect_tx(barP, part_bytes);
  }
  stage_up(0);
  stage_dn(0);
  prefetch_layer(0);
  if (p.L > 1) prefetch_layer(1);
  const Share up = share_of(m_tiles * ((ucols + 15) / 16), d), dn = share_of(m_tiles * ((ncols + 15) / 16), klen);
  for (int l = 0;; ++l) {
    const bool last = l == p.L;
    const LayerW w = layer_w(p, last ? 0 : l);
    // ---- rows (after the last layer: the final norm). The activation row goes to its place here and in the other CTAs of
    //      the cluster, x + y of the cluster's own columns to the CTAs that will add the down projection to them ----
    {
      const ST* Sl = reinterpret_cast<const ST*>(static_cast<const uint8_t*>(p.S) + (int64_t)l * p.layer_stride) + c0;
      float* slot = red + group * 8;
      const int step = alone ? kMaxRows : kGroups * kCluster;
      for (int row = alone ? group : rank + group * kCluster; row < B; row += step) {
        float4 v[NT], s[NT];
        if (l == 0) {
          int tk = p.tok_in[row];
          if (tk < 0 || tk >= p.V) {
            if (c0 == 0) raise_status(p.status, kStatusTokenRange);
            tk = tk < 0 ? 0 : p.V - 1;
          }
#pragma unroll
          for (int i = 0; i < NT; ++i) v[i] = ldg4(p.E + (int64_t)tk * d + c0 + 256 * i);
        } else {                                         // other CTAs wrote it: not through L1
#pragma unroll
          for (int i = 0; i < NT; ++i) v[i] = __ldcg(reinterpret_cast<const float4*>(p.x + (int64_t)row * d + c0 + 256 * i));
        }
        float mean, rstd;
        if (!last) {
#pragma unroll
          for (int i = 0; i < NT; ++i) s[i] = ld4(Sl + (int64_t)row * d + 256 * i);
          const float* bt_p = prm + 2 * d + c0;
          if (p.pos != nullptr) {                        // a position per row: its own beta row and head scalars
            const int t = t_of(row);
            bt_p = w.beta + (int64_t)t * d + c0;
            head_scalars<d, NT>(p, w, t, tid & 63, a1, a2, lm);
          }
          group_stats<d, NT>(v, p.eps, slot, group, mean, rstd);
          const float nmr = -mean * rstd;
#pragma unroll
          for (int i = 0; i < NT; ++i) {
            const float4 g = ld4(prm + c0 + 256 * i), bb = ld4(prm + d + c0 + 256 * i), bt = ld4(bt_p + 256 * i);
            const float4 z = make_float4(fmaf(fmaf(v[i].x, rstd, nmr), g.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), g.y, bb.y),
                                         fmaf(fmaf(v[i].z, rstd, nmr), g.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), g.w, bb.w));
            // row-repeat head, Eq. 2: y = (a z + S) + b ; S' = l (S + a z).  column-repeat head, Eq. 3: y = a (z + S) + b ; S' = l (z + S)
            const float4 u = make_float4(fmaf(a1[i], z.x, s[i].x), fmaf(a1[i], z.y, s[i].y), fmaf(a1[i], z.z, s[i].z), fmaf(a1[i], z.w, s[i].w));
            if (row == own_row) st4(sS + c0 + 256 * i, make_float4(lm[i] * u.x, lm[i] * u.y, lm[i] * u.z, lm[i] * u.w));
            v[i] = make_float4(v[i].x + fmaf(a2[i], u.x, bt.x), v[i].y + fmaf(a2[i], u.y, bt.y), v[i].z + fmaf(a2[i], u.z, bt.z),
                               v[i].w + fmaf(a2[i], u.w, bt.w));
            const int o = c0 + 256 * i - n0;             // column inside the cluster's slab
            if (o >= 0 && o < ncols) {
#pragma unroll
              for (int k = 0; k < 4; k += 2) {           // (gw is even: two adjacent columns have one owner)
                const int q = (o + k) / gw;
                if (!alone || q == rank)
                  st_async_v2(tc::mapa(tc::smem_u32(xo) + (uint32_t)(row * gw + (o + k) % gw) * 4, (uint32_t)q), k ? v[i].z : v[i].x,
                              k ? v[i].w : v[i].y, tc::mapa(tc::smem_u32(barP), (uint32_t)q));
              }
            }
          }
        }
        group_stats<d, NT>(v, p.eps, slot + 4, group, mean, rstd);
        const float nmr2 = -mean * rstd;
        uint8_t* at = sA + (size_t)row * ld_d;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          const float4 g = ld4(prm + 3 * d + c0 + 256 * i), bb = ld4(prm + 4 * d + c0 + 256 * i);
          st4(reinterpret_cast<bf16*>(at) + c0 + 256 * i,
              make_float4(fmaf(fmaf(v[i].x, rstd, nmr2), g.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr2), g.y, bb.y),
                          fmaf(fmaf(v[i].z, rstd, nmr2), g.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr2), g.w, bb.w)));
        }
        if (!alone) {
          // (one bulk copy per peer: eight-byte stores into the peers' memory took 1.7 us per sixteen rows)
          tc::fence_async_smem();
          asm volatile("bar.sync %0, 64;" ::"r"(group + 1) : "memory");
          const int r = tid & 63;                        // threads 0, 1 of the group's first warp, 32, 33 of its second
          const int peer = (r & 31) < 2 ? (r & 31) + 2 * (r >> 5) : rank;
          if (peer != rank)
            bulk_s2s(tc::mapa(tc::smem_u32(at), (uint32_t)peer), at, 2 * d, tc::mapa(tc::smem_u32(barR), (uint32_t)peer));
        }
      }
      __syncthreads();                     // this CTA's rows
      if (!alone) {                        // the others'
        if (!wait_stage(barR, (uint32_t)l & 1u, p.status, gb.dead)) gb.dead = true;
      }
    }
    if (last) break;

    // ---- up projection: H[:, slab] = gelu(a W1[slab]^T + b1) ----
    if (!wait_stage(bar1, par1, p.status, gb.dead)) gb.dead = true;
    par1 ^= 1u;
    if (l > 0) stage_dn(l);                // (W2's place is free since the previous layer; issued while a barrier is waited
                                           //  for, the weight stream made the barrier itself slower, 1.3 -> 2.6 us)
    if (warp < up.tiles * up.groups) {
      const int tile = warp % up.tiles, g = warp / up.tiles;
      float c[8];
      tile_group(c, up, g, sA, ld_d, tile % m_tiles, sW1, ld_d, tile / m_tiles, lane);
      put_part(part, up, g, tile, lane, c);
    }
    __syncthreads();                       // partial sums are visible, the weight rows have been read
    for (int i = tid; i < up.tiles * 128; i += kThreads) {
      const Pair q = take_pair(part, up, i, m_tiles);
      if (q.row < B && q.col < ucols) {
        const float2 bb = __ldg(reinterpret_cast<const float2*>(w.b1 + u0 + q.col));
        *reinterpret_cast<__nv_bfloat162*>(p.H + (int64_t)q.row * F + u0 + q.col) =
            __floats2bfloat162_rn(tc::gelu_fast(q.a + bb.x), tc::gelu_fast(q.b + bb.y));
      }
    }
    gb.sync([] {});

    // ---- down projection: this rank's part of K for the cluster's columns ----
    asm volatile("fence.proxy.async.global;" ::: "memory");     // H was written through the generic proxy
    stage_rows(sA, p.H + k0, B, 2 * klen, 2 * (int64_t)F, barA);
    if (own_row < B) {                     // nobody reads the old cache row any more
      ST* Sg = reinterpret_cast<ST*>(static_cast<uint8_t*>(p.S) + (int64_t)l * p.layer_stride) + (int64_t)own_row * d;
      const uint4* src = reinterpret_cast<const uint4*>(sS);
      if (tid < d * (int)sizeof(ST) / 16) reinterpret_cast<uint4*>(Sg)[tid] = src[tid];
    }
    if (!wait_stage(bar2, par2, p.status, gb.dead)) gb.dead = true;
    if (!wait_stage(barA, par2, p.status, gb.dead)) gb.dead = true;
    par2 ^= 1u;
    // the next weights for W1's place (used up): while this phase asks for nothing else
    if (l + 1 < p.L) stage_up(l + 1);
    else for (int ch = 0; ch < p.lm_stages_w1; ++ch) stage_lm(ch);
    if (l + 2 < p.L) prefetch_layer(l + 2);
    auto send = [&](int row, int col, float a, float b) {      // to the rank that owns these columns (gw is even)
      if (row < B && col < ncols)
        st_async_v2(tc::mapa(tc::smem_u32(recv + ((size_t)(rank * mp + row) * gw + col % gw) * 4), (uint32_t)(col / gw)), a, b,
                    tc::mapa(tc::smem_u32(barP), (uint32_t)(col / gw)));
    };
    {
      const int tile = warp % dn.tiles, g = warp / dn.tiles;
      float c[8];
      if (warp < dn.tiles * dn.groups) tile_group(c, dn, g, sA, ld_k, tile % m_tiles, sW2, ld_k, tile / m_tiles, lane);
      if (warp < dn.tiles * dn.groups) put_part(part, dn, g, tile, lane, c);
      __syncthreads();
      for (int i = tid; i < dn.tiles * 128; i += kThreads) {
        const Pair q = take_pair(part, dn, i, m_tiles);
        send(q.row, q.col, q.a, q.b);
      }
    }
    if (!wait_stage(barP, (uint32_t)l & 1u, p.status, gb.dead)) gb.dead = true;      // the four partial products are here
    for (int i = tid; i < B * gw; i += kThreads) {
      const int row = i / gw, c = i % gw;
      const float* r = reinterpret_cast<const float*>(recv) + (size_t)row * gw + c;
      float v = reinterpret_cast<const float*>(xo)[i] + __ldg(w.b2 + n0 + rank * gw + c);
#pragma unroll
      for (int s = 0; s < kCluster; ++s) v += r[(size_t)s * mp * gw];
      p.x[(int64_t)row * d + n0 + rank * gw + c] = v;
    }
    gb.sync([&] {
      if (tid == 0) {
        if (!alone) tc::mbar_expect_tx(barR, peer_bytes);
        if (l + 1 < p.L) tc::mbar_expect_tx(barP, part_bytes);
      }
      const int t = p.pos != nullptr ? 0 : t_all;
      fetch_row_params<d>(p, l + 1, t, prm);
      if (l + 1 < p.L) head_scalars<d, NT>(p, layer_w(p, l + 1), t, tid & 63, a1, a2, lm);
    });
  }
  for (int ch = p.lm_stages_w1; ch < p.lm_stages; ++ch) stage_lm(ch);

  // ---- LM head over this CTA's vocabulary slab through the ring, two chunks at a time where it is deep enough ----
  const int cpi = p.lm_stages >= 4 && m_tiles <= 2 ? 2 : 1;      // (every thread takes one pair of columns)
  const Share hd = share_of(m_tiles * cpi, d);
  const int lm_end = min(p.V, (lm_c0 + lm_chunks) * kLmChunkCols);
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  bool bad = false;
  int my_row = kMaxRows;                                 // every thread keeps one pair of columns of one row
  for (int ch = 0; ch < lm_chunks; ch += cpi) {
    for (int c = ch; c < ch + cpi && c < lm_chunks; ++c)
      if (!wait_stage(barL + c % p.lm_stages, (uint32_t)(c / p.lm_stages) & 1u, p.status, gb.dead)) gb.dead = true;
    if (warp < hd.tiles * hd.groups) {
      const int tile = warp % hd.tiles, g = warp / hd.tiles;
      float c[8];
      tile_group(c, hd, g, sA, ld_d, tile % m_tiles, sW1 + (ch + tile / m_tiles) % p.lm_stages * lm_stage, ld_d, 0, lane);
      put_part(part, hd, g, tile, lane, c);
    }
    __syncthreads();                                     // partial sums are visible, the stages have been read
    for (int c = ch; c < ch + cpi; ++c) stage_lm(c + p.lm_stages);
    if (tid < hd.tiles * 128) {
      const Pair q = take_pair(part, hd, tid, m_tiles);
      const int col = (lm_c0 + ch) * kLmChunkCols + q.col;
      my_row = q.row;
      if (q.row < B && col < lm_end && !gb.dead) {       // (V is a multiple of 8: pairs are whole)
        if (p.logits != nullptr) *reinterpret_cast<float2*>(p.logits + (int64_t)q.row * p.V + col) = make_float2(q.a, q.b);
        bad |= !(q.a == q.a) | !(q.b == q.b);
        if (q.a > bv) { bv = q.a; bi = col; }            // ascending columns: the lowest among equals is kept
        if (q.b > bv) { bv = q.b; bi = col + 1; }
      }
    }
    __syncthreads();                                     // the partial sums have been taken
  }
  tc::cluster_sync();                      // the copies out of this CTA's shared memory have arrived
  if (gb.dead) {
    // a copy or a CTA never came: give whatever is still in flight time to land before shared memory goes away
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 21)) { }
  }
  if (!p.greedy) return;                   // the caller selects from the logits
  if (bad) raise_status(p.status, kStatusNonFinite);
  unsigned long long* best_s = reinterpret_cast<unsigned long long*>(part);
  if (tid < kMaxRows) best_s[tid] = 0ull;
  __syncthreads();
  if (my_row < B && bi != 0x7fffffff) atomicMax(best_s + my_row, pack_best(bv, bi));
  __syncthreads();
  if (tid < B && best_s[tid] != 0ull) atomicMax(p.best + tid, best_s[tid]);
  // ---- the CTA that comes last writes the tokens ----
  __threadfence();
  __syncthreads();
  uint32_t* am_last = reinterpret_cast<uint32_t*>(sm + 116);
  if (tid == 0) {
    *am_last = atomicAdd(p.bar + kGrid, 1u) + 1u == gridDim.x ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  if (*am_last != 0u && tid < B) {
    const unsigned long long best = __ldcg(p.best + tid);
    int tok = best == 0ull ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(best & 0xFFFFFFFFull));
    if (tok < 0 || tok >= p.V) tok = 0;
    write_token(p.out, tid, tok);
  }
}

}  // namespace sb
}  // namespace srm
