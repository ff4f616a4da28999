// All layers of a decode pass of up to 16 rows, weights split between clusters of 16 CTAs, ONE meeting of the grid per layer.
//
// With so few rows a layer is its chain of dependent steps; the weights of a CTA fit in a ring that runs ahead of it. What
// counts is how often all CTAs have to meet, and what a meeting costs. Here every cluster computes every row's token mixer
// itself and a part of the hidden layer only:
//   rows:  rank r of EVERY cluster owns row r: x + b2 + the clusters' partial products, LN1, cache update, residual, LN2; the
//          activation row goes to the 16 CTAs of the cluster through distributed shared memory. A single row is computed by
//          every CTA for itself (ALONE): its words are 56 KB, read in 700 clocks, sending it takes 1560;
//   up:    a cluster computes F / clusters columns of H (in groups of 16: 37 or 36 of 256 for seven clusters), a CTA four or five
//          8-column tiles of them; GELU; the columns go to all CTAs of the cluster;
//   down:  K = the cluster's columns of H, a CTA d / 16 output features: the cluster's partial product, written to a plane of
//          its own in global memory;
//   meeting: an owner adds the planes of its rows in cluster order.
// Every word of a plane travels with the number of its layer (eight bytes, stored and loaded whole: fp32 value, tag), so
// nobody waits for stores to be acknowledged, raises a flag and loads afterwards: a reader loads the words until all tags are
// the layer's. The planes alternate between two buffers; a CTA clears its words at the start, and the grid counts itself past
// that point before the first reader looks. A word is overwritten two layers later: its writer has by then used activations that
// were computed from planes of the layer in between, which every cluster wrote after reading the first ones.
//
// What a layer takes (device clock, 1 / 16 rows): words of the planes 2100 / 2200 after they were stored by the slowest (57 KB per row
// at 64 bytes per clock and SM), row phase 1900 / 2000, activations to the other CTAs - / 1200, up products 1800 / 1500, sums, GELU and
// H 2500 / 3700, down products 2000, sums and stores 600: 11900 / 14300 = 6.2 / 7.4 us (the single-kernel step with two grid
// barriers per layer: 10.3 / 11.6); W1 and W2 from HBM take 4900.
//
// Eight warps do the rows, eight the contractions, on mma.sync m16n8k16 (bf16 in, fp32 accumulate; a tcgen05 instruction takes 39
// clocks however few rows, and a CTA's tile would need 64 of them in a row): a warp takes two k-blocks of all the CTA's columns
// (up) or every fourth pair of 16-deep steps of half its features (down), weight fragments in registers before the
// activations have come; the partial sums meet in shared memory. A CTA's weights of a whole layer have places of their own in
// shared memory, each filled for the next layer as soon as it has been used. Buffers need no "free" signals, as in
// layers_cluster.cuh: whatever overwrites one was computed from what its last reader sent afterwards.
//
// The LM head and the greedy selection follow in the same kernel (but for selections that have an LM head of their own): every CTA
// takes its 112th of the vocabulary in chunks of 40 rows through the two places of the weights, as an up projection, writes the
// logits where they are wanted and keeps the best one of every row; the CTA that comes last writes the tokens. A step of one row takes 140 us so, 150 with kernels of their own.
//
// 512 threads leave 128 registers each: 92 (ALONE) and 124 bytes per thread are spilled around the products.
//
// All CTAs must be resident (cooperative launch). Every wait is bounded: a waiter that gives up raises kStatusWaitTimeout and
// goes on without waiting.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "layers_cluster.cuh"   // st_async_16
#include "prefill_chunk.cuh"    // ld_acquire_u32
#include "select.cuh"           // SelectOut, write_token
#include "step_small.cuh"       // LayerW, layer_w, ldsm_x4, ld_relaxed_u32, red_release_inc, pack_best

namespace srm {
namespace sp {

constexpr int kCluster = 16, kClusters = 7;    // as many as 148 SMs hold
constexpr int kWarps = 16, kThreads = kWarps * 32, kMaxRows = 16;
constexpr int kRowWarps = 8, kMmaWarps = 8, kRowThreads = kRowWarps * 32;
constexpr int kDnSplits = 4;                   // warps that share out K of the down projection (up: all)
constexpr int kBarrierBytes = 1024, kSumBytes = 2 * kRowWarps * 8;
constexpr int kSmemBytes = 227 * 1024;
constexpr long long kWaitLimitCycles = 1ll << 28;

struct Params {
  int R, V, h, n_ctx, L, t;
  float eps;
  const int32_t* tok_in;         // [R]
  const bf16* E;
  sb::LayerW layer0;             // as in sb::Params
  int64_t layer_bytes;
  void* S;                       // cache rows of layer 0; layer l at S + l * layer_stride (bytes)
  int64_t layer_stride;
  bf16* a;                       // [R, d]: the final norm's rows
  const float *lnf_g, *lnf_b;
  unsigned long long* planes;    // [2][clusters][R][d] words (value, tag)
  uint32_t* cnt;                 // CTAs that have cleared their words | CTAs done with the LM head; zero on entry
  int head = 0;                  // LM head here; else the final norm's rows to `a`
  int select = 0;                // ... and the greedy selection, to `out`
  float* logits = nullptr;       // ... and the logits, to here ([R, V])
  unsigned long long* best = nullptr;      // [R] (sortable logit, ~column) maxima, zero on entry
  SelectOut out = {};
  uint32_t* status;
  const int32_t* ctr;            // device-side step counters or nullptr
  const int32_t* pos;            // [R] per-row positions or nullptr
};
inline size_t plane_bytes(int64_t R, int d) { return (size_t)2 * kClusters * R * d * 8; }

// Shared memory: activations [k-block][row][128 bytes] | the cluster's columns of H [8-column tile][row][16 bytes] | k-blocks of W1 | of W2 | barriers |
// row-phase sums. The warps' partial sums lie in the place of the activations: of the up projection in the two k-blocks that the
// warp has used, of the down projection anywhere.
template <int D>
struct Shape {
  static constexpr int kGroups = (D / 4 + kClusters - 1) / kClusters;            // 16-column groups of H per cluster, at most (F = 4 d)
  static constexpr int kUpTiles = (2 * kGroups + kCluster - 1) / kCluster;       // 8-column tiles of H per CTA, at most
  static constexpr int kDnTiles = D / kCluster / 8;                              // 8-feature tiles of x per CTA
  static constexpr int kKb = D / 64, kHKb = (kGroups * 16 + 63) / 64;            // k-blocks of the projections
  static constexpr int kHPairs = (kGroups + 1) / 2;                              // pairs of 16-deep steps of the down projection
  static constexpr int kRowBytes = kMaxRows * 128;                               // one k-block of activations or of H
  static constexpr int kUpBytes = kUpTiles * 1024, kDnBytes = kDnTiles * 1024;   // one k-block of the weights
  static constexpr int kBarriers = (kKb + kHKb) * kRowBytes + kKb * kUpBytes + kHKb * kDnBytes;
  static constexpr size_t kSmem = kBarriers + kBarrierBytes + kSumBytes + 1024;
  static_assert(kKb == 2 * kMmaWarps && D == 4 * kRowThreads && kHKb <= 2 * kMmaWarps && kUpTiles <= kMmaWarps && kDnTiles == kMmaWarps &&
                kSmem <= kSmemBytes && kHKb * kDnBytes >= kKb * kUpBytes && kMmaWarps * kUpTiles * 512 <= kHKb * kRowBytes && kUpTiles * 512 <= 2 * kRowBytes && kDnSplits * kDnTiles * 512 <= kKb * kRowBytes, "shape");
};

__device__ __forceinline__ void tma_load_w(void* dst, const CUtensorMap* map, uint64_t* bar, int col, int row, int layer) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(tc::smem_u32(bar)), "r"(col), "r"(row), "r"(layer)
      : "memory");
}
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two words of a plane: (value, tag), (value, tag)
__device__ __forceinline__ void st_words(unsigned long long* p, float a, float b, uint32_t tag) {
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(a)), "l"(t | __float_as_uint(b)) : "memory");
}
__device__ __forceinline__ void ld_words(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ float2 ldg2(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
// Loads that stay where they are written, ahead of the waits (the compiler moves others down to their first use).
__device__ __forceinline__ float ldc1(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ldc4(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
// ... of four cache values, as stored; widened when they are used
struct alignas(16) Raw4 { uint32_t u[4]; };
template <typename T>
__device__ __forceinline__ Raw4 ld_raw4(const T* p) {
  Raw4 r;
  if constexpr (sizeof(T) == 4) asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.u[0]), "=r"(r.u[1]), "=r"(r.u[2]), "=r"(r.u[3]) : "l"(p));
  else asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(r.u[0]), "=r"(r.u[1]) : "l"(p));
  return r;
}
template <typename T>
__device__ __forceinline__ float4 widen(const Raw4& r) { return ld4(reinterpret_cast<const T*>(r.u)); }
__device__ __forceinline__ void rows_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory"); }
__device__ __forceinline__ void mma_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kMmaWarps * 32) : "memory"); }

// LayerNorm statistics of a row, four channels per thread of the row warps: mean and sum of squares about it, merged pairwise over
// the warp, then by every warp over the warps. slot: kRowWarps pairs of floats.
__device__ __forceinline__ void row_stats(const float4& x, float eps, float2* slot, float& mean, float& rstd) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float m = 0.25f * ((x.x + x.y) + (x.z + x.w)), half_n = 2.f;
  const float a = x.x - m, b = x.y - m, c = x.z - m, e = x.w - m;
  float q = (a * a + b * b) + (c * c + e * e);
  auto merge = [&](int o) {               // with lane ^ o: two sets of 2 half_n values each
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), q2 = __shfl_xor_sync(0xffffffffu, q, o), dm = m2 - m;
    q += fmaf(dm * dm, half_n, q2);
    m = 0.5f * (m + m2);
    half_n += half_n;
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) merge(o);
  if (lane == 0) slot[warp] = make_float2(m, q);         // (the lanes may differ in the last bit: lane 0's values count)
  rows_sync();
  const float2 v = slot[lane & (kRowWarps - 1)];
  m = v.x;
  q = v.y;
#pragma unroll
  for (int o = 1; o < kRowWarps; o <<= 1) merge(o);
  mean = __shfl_sync(0xffffffffu, m, 0);
  rstd = rsqrtf(__shfl_sync(0xffffffffu, q, 0) * (0.5f / half_n) + eps);
}

// ALONE: the one row there is, computed by every CTA.
template <int D, bool ALONE, typename ST>
__global__ void __launch_bounds__(kThreads, 1)
layers_kernel(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmLm,
              const Params p) {
  pdl_trigger();
  using C = Shape<D>;
  constexpr int kRowBytes = C::kRowBytes, kKb = C::kKb;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sH = sA + kKb * kRowBytes;
  uint8_t* sU = sH + C::kHKb * kRowBytes;
  uint8_t* sD = sU + kKb * C::kUpBytes;
  uint64_t* full_up = reinterpret_cast<uint64_t*>(smem + C::kBarriers);  // [kKb]
  uint64_t* full_dn = full_up + kKb;                                     // [kHKb]
  uint64_t* act_full = full_dn + C::kHKb;                                // by quarters of the channels
  uint64_t* h_full = act_full + 4;
  uint64_t* stored = h_full + 1;                                         // this CTA's words of a layer are on their way: time to look for the others'
  uint64_t* full_lm = stored + 1;                                        // [2][kKb] k-blocks of the LM head's chunks, in the places of W1 and of W2
  unsigned long long* best = reinterpret_cast<unsigned long long*>(full_lm + 2 * kKb);      // [kMaxRows] of this CTA
  uint32_t* am_last = reinterpret_cast<uint32_t*>(best + kMaxRows);
  float2* sums = reinterpret_cast<float2*>(smem + C::kBarriers + kBarrierBytes);
  static_assert((kKb + C::kHKb + 6 + 2 * kKb + kMaxRows + 1) * 8 <= kBarrierBytes, "barriers");

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int rank = (int)tc::cluster_ctarank(), cluster = (int)(blockIdx.x / kCluster);
  // this cluster's columns of H and this CTA's 8-column tiles of them
  constexpr int kAll = D / 4;                                            // 16-column groups
  const int h0 = cluster * kAll / kClusters * 16, hc = (cluster + 1) * kAll / kClusters * 16 - h0;
  const int tile0 = rank * (hc / 8) / kCluster, tiles = (rank + 1) * (hc / 8) / kCluster - tile0;
  const int h_kb = (hc + 63) / 64;
  if (tid == 0) {
    for (int i = 0; i < kKb + C::kHKb; ++i) tc::mbar_init(&full_up[i], 1);
    for (int i = 0; i < 4; ++i) tc::mbar_init(&act_full[i], ALONE ? kRowWarps / 4 : 1);
    tc::mbar_init(h_full, 1);
    tc::mbar_init(stored, kMmaWarps);
    for (int i = 0; i < 2 * kKb; ++i) tc::mbar_init(&full_lm[i], 1);
    for (int i = 0; i < kMaxRows; ++i) best[i] = 0ull;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  tc::cluster_sync();                                                    // (every CTA's barriers are set before a byte is sent to it)
  bool ok = true;                                                        // no wait has given up in this thread

  // ---- weights: constant data. One thread calls ----
  auto load_up = [&](int l, int kb) {
    if (l >= p.L) return;
    tc::mbar_expect_tx(&full_up[kb], C::kUpBytes);
    tma_load_w(sU + kb * C::kUpBytes, &tmW1, &full_up[kb], kb * 64, h0 + tile0 * 8, l);
  };
  auto load_dn = [&](int l, int kb) {
    if (l >= p.L) return;
    tc::mbar_expect_tx(&full_dn[kb], C::kDnBytes);
    tma_load_w(sD + kb * C::kDnBytes, &tmW2, &full_dn[kb], h0 + kb * 64, rank * (D / kCluster), l);
  };
  // the LM head: chunk i of this CTA's 8-row tiles of the vocabulary, into the place of W1 (even) or of W2 (odd)
  const int lm_all = (p.V + 7) / 8, lm0 = (int)((int64_t)blockIdx.x * lm_all / gridDim.x), lm_tiles = (int)((int64_t)(blockIdx.x + 1) * lm_all / gridDim.x) - lm0;
  const int lm_chunks = p.head ? (lm_tiles + C::kUpTiles - 1) / C::kUpTiles : 0;
  auto load_lm = [&](int i, int kb) {
    if (i >= lm_chunks) return;
    uint64_t* bar = &full_lm[(i & 1) * kKb + kb];
    tc::mbar_expect_tx(bar, C::kUpBytes);
    tma_load_w((i & 1 ? sD : sU) + kb * C::kUpBytes, &tmLm, bar, kb * 64, (lm0 + i * C::kUpTiles) * 8, 0);
  };
  if (tc::elect_one()) {
    load_up(0, warp);
    if (warp < h_kb) load_dn(0, warp);
  }
  __syncwarp();
  pdl_wait();
  // ---- this CTA's words of the planes: cleared, both buffers ----
  constexpr int kMine = D / kCluster;                                    // output features of this CTA
  for (int i = tid; i < 2 * p.R * (kMine / 2); i += kThreads) {
    const int f = i % (kMine / 2) * 2, r = i / (kMine / 2) % p.R, b = i / (kMine / 2) / p.R;
    st_words(p.planes + (((int64_t)b * kClusters + cluster) * p.R + r) * D + rank * kMine + f, 0.f, 0.f, 0u);
  }
  __syncthreads();
  if (tid == 0) {
    sb::red_release_inc(p.cnt);
    if (!ALONE)
      for (int i = 0; i < 4; ++i) tc::mbar_expect_tx(&act_full[i], (uint32_t)(p.R * D / 2));
    tc::mbar_expect_tx(h_full, (uint32_t)(p.R * hc * 2));
  }

  if (warp < kRowWarps) {
    // ---------------- rows ----------------
    const int t_all = p.ctr != nullptr ? p.ctr[kCtrPos] : p.t;
    const int row = ALONE ? 0 : rank, c0 = 4 * tid;                      // this thread's four channels
    const bool writes = cluster == 0 && (!ALONE || rank == 0);           // the cache, and the final norm's rows
    const int t = row < p.R && p.pos != nullptr ? min(max(p.pos[row], 0), p.n_ctx - 1) : t_all;
    const int head = c0 / (D / p.h);
    const bool is_row = head < (p.h >> 1);
    // where the 16 bytes of an activation row that this thread and its neighbour hold go
    const uint32_t act_addr = tc::smem_u32(sA) + (uint32_t)((c0 >> 6) * kRowBytes + row * 128) + (uint32_t)(((c0 >> 3 & 7) ^ (row & 7)) << 4);
    const int qd = c0 / (D / 4);                                         // this warp's quarter of the channels
    const uint32_t act_bar = tc::smem_u32(&act_full[qd]);
    const unsigned long long* plane = p.planes + (int64_t)row * D + c0;
    const int64_t plane_step = (int64_t)p.R * D;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f), keep = v;
    for (int l = 0; row < p.R; ++l) {
      const bool last = l == p.L, send = !last || p.head != 0;           // (to the LM head: the final norm's rows)
      // parameters: constant data, and this thread's part of the cache row, on their way while the projections run
      const sb::LayerW w = sb::layer_w(p, last ? 0 : l);
      auto cache_row = [&](int l) { return reinterpret_cast<ST*>(static_cast<uint8_t*>(p.S) + (int64_t)l * p.layer_stride) + (int64_t)row * D + c0; };
      float4 g1, h1, bt, bias2;
      Raw4 old;
      float al = 0.f, lam = 0.f;
      if (l > 0) bias2 = ldc4(sb::layer_w(p, l - 1).b2 + c0);
      if (!last) {
        old = ld_raw4(const_cast<const ST*>(cache_row(l)));
        g1 = ldc4(w.ln1_g + c0);
        h1 = ldc4(w.ln1_b + c0);
        bt = ldc4(w.beta + (int64_t)t * D + c0);
        al = ldc1(w.alpha + (int64_t)head * p.n_ctx + t);
        lam = ldc1(w.lam + head);
      }
      const float4 g2 = ldc4((last ? p.lnf_g : w.ln2_g) + c0), h2 = ldc4((last ? p.lnf_b : w.ln2_b) + c0);
      if (l == 0) {
        int tk = p.tok_in[row];
        if (tk < 0 || tk >= p.V) {
          if (tid == 0) raise_status(p.status, kStatusTokenRange);
          tk = tk < 0 ? 0 : p.V - 1;
        }
        v = ldg4(p.E + (int64_t)tk * D + c0);
      } else {                            // x + b2 + the clusters' partial products
        if (ok) ok = tc::mbar_wait(stored, (uint32_t)(l - 1) & 1u, p.status);
        unsigned long long w[kClusters][4];
        const unsigned long long* from = plane + (int64_t)((l - 1) & 1) * kClusters * plane_step;
        const long long t0 = clock64();
        for (uint32_t missing = (1u << kClusters) - 1;;) {               // (planes that were there are not loaded again)
#pragma unroll
          for (int c = 0; c < kClusters; ++c)
            if (missing >> c & 1) {
              ld_words(from + c * plane_step, w[c][0], w[c][1]);
              ld_words(from + c * plane_step + 2, w[c][2], w[c][3]);
            }
#pragma unroll
          for (int c = 0; c < kClusters; ++c) {
            bool all = true;
#pragma unroll
            for (int i = 0; i < 4; ++i) all &= (uint32_t)(w[c][i] >> 32) == (uint32_t)l;
            if (all) missing &= ~(1u << c);
          }
          if (missing == 0 || !ok) break;
          if (clock64() - t0 > kWaitLimitCycles) { ok = false; raise_status(p.status, kStatusWaitTimeout); }
        }
        __syncwarp();
        v = make_float4(v.x + bias2.x, v.y + bias2.y, v.z + bias2.z, v.w + bias2.w);
#pragma unroll
        for (int c = 0; c < kClusters; ++c)
          v = make_float4(v.x + __uint_as_float((uint32_t)w[c][0]), v.y + __uint_as_float((uint32_t)w[c][1]),
                          v.z + __uint_as_float((uint32_t)w[c][2]), v.w + __uint_as_float((uint32_t)w[c][3]));
      }
      const float4 kept = keep;           // the cache row of the layer before
      float mean, rstd;
      if (!last) {
        row_stats(v, p.eps, sums, mean, rstd);
        const float nmr = -mean * rstd;
        const float4 z = make_float4(fmaf(fmaf(v.x, rstd, nmr), g1.x, h1.x), fmaf(fmaf(v.y, rstd, nmr), g1.y, h1.y),
                                     fmaf(fmaf(v.z, rstd, nmr), g1.z, h1.z), fmaf(fmaf(v.w, rstd, nmr), g1.w, h1.w));
        // row-repeat head, Eq. 2: y = (a z + S) + b ; S' = l (S + a z).  column-repeat head, Eq. 3: y = a (z + S) + b ; S' = l (z + S)
        const float a1 = is_row ? al : 1.0f, a2 = is_row ? 1.0f : al;
        const float4 s = widen<ST>(old);
        const float4 u = make_float4(fmaf(a1, z.x, s.x), fmaf(a1, z.y, s.y), fmaf(a1, z.z, s.z), fmaf(a1, z.w, s.w));
        keep = make_float4(lam * u.x, lam * u.y, lam * u.z, lam * u.w);
        v = make_float4(v.x + fmaf(a2, u.x, bt.x), v.y + fmaf(a2, u.y, bt.y), v.z + fmaf(a2, u.z, bt.z), v.w + fmaf(a2, u.w, bt.w));
      }
      row_stats(v, p.eps, sums + kRowWarps, mean, rstd);
      const float nmr2 = -mean * rstd;
      const float4 o = make_float4(fmaf(fmaf(v.x, rstd, nmr2), g2.x, h2.x), fmaf(fmaf(v.y, rstd, nmr2), g2.y, h2.y),
                                   fmaf(fmaf(v.z, rstd, nmr2), g2.z, h2.z), fmaf(fmaf(v.w, rstd, nmr2), g2.w, h2.w));
      if (!send) {
        if (writes) st4(p.a + (int64_t)row * D + c0, o);
      } else if (ALONE) {                 // (row 0 of this CTA's activations: it has no swizzle)
        st4(reinterpret_cast<bf16*>(sA + (c0 >> 6) * kRowBytes) + (c0 & 63), o);
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&act_full[qd]);
      } else {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(o.x, o.y), hi = __floats2bfloat162_rn(o.z, o.w);
        const uint32_t q0 = *reinterpret_cast<const uint32_t*>(&lo), q1 = *reinterpret_cast<const uint32_t*>(&hi);
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, q0, 1), r1 = __shfl_xor_sync(0xffffffffu, q1, 1);
        const int odd = lane & 1;
        const uint4 w = odd ? make_uint4(r0, r1, q0, q1) : make_uint4(q0, q1, r0, r1);
        // One quarter of the channels after the other, so that the first k-blocks are there early (layers_cluster.cuh)
        if (qd > 0) asm volatile("bar.sync %0, %1;" ::"r"(9 + qd), "n"(kRowThreads / 2) : "memory");
#pragma unroll
        for (int j = 0; j < kCluster / 2; ++j) {         // even lanes: eight of the ranks, odd lanes: the other eight
          const uint32_t to = (uint32_t)(rank + 8 * odd + j) % kCluster;
          cl::st_async_16(tc::mapa(act_addr, to), w, tc::mapa(act_bar, to));
        }
        if (qd < 3) asm volatile("bar.arrive %0, %1;" ::"r"(10 + qd), "n"(kRowThreads / 2) : "memory");
      }
      if (l > 0 && writes) st4(cache_row(l - 1), kept);                  // (every cluster has used the old row)
      if (last) break;
    }
  } else {
    // ---------------- projections ----------------
    const int m = warp - kRowWarps, leader = kRowThreads;                // this warp of eight; the thread that speaks for all
    // Fragments: rows g, g + 8 of the batch, columns 2 q, 2 q + 1 of a tile. ldmatrix: A takes row (lane % 16), half (lane / 16) of 16
    // columns; W takes row (lane % 8), quarter (lane / 8) of 32 columns.
    const int g = lane >> 2, q = lane & 3;
    const uint32_t a_row = (uint32_t)((lane & 15) * 128), a_sw = lane & 7, a_c = lane >> 4, w_row = (uint32_t)((lane & 7) * 128), w_c = lane >> 3;
    for (int l = 0; l < p.L; ++l) {
      // ---- up: k-blocks 2 m and 2 m + 1 ----
      {
        float2 bias1 = make_float2(0.f, 0.f);
        if (m < tiles) bias1 = ldg2(sb::layer_w(p, l).b1 + h0 + (tile0 + m) * 8 + 2 * q);
        uint32_t b[2][C::kUpTiles][2][4], a[4][4];
        float c[C::kUpTiles][4] = {};
        auto weights = [&](int i) {                                      // (kUpTiles tiles are there, whether they are this CTA's or not)
          if (ok) ok = tc::mbar_wait(&full_up[2 * m + i], (uint32_t)(l & 1), p.status);
          __syncwarp();
          const uint32_t w0 = tc::smem_u32(sU) + (2 * m + i) * C::kUpBytes + w_row;
#pragma unroll
          for (int j = 0; j < C::kUpTiles; ++j)
#pragma unroll
            for (int k = 0; k < 2; ++k) sb::ldsm_x4(b[i][j][k], w0 + (uint32_t)(j * 1024) + (((4 * k + w_c) ^ (lane & 7)) << 4));
        };
        auto products = [&](int i) {
          const uint32_t a0 = tc::smem_u32(sA) + (2 * m + i) * kRowBytes + a_row;
#pragma unroll
          for (int k = 0; k < 4; ++k) sb::ldsm_x4(a[k], a0 + (((2 * k + a_c) ^ a_sw) << 4));
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < C::kUpTiles; ++j) mma(c[j], a[k], b[i][j][k >> 1][2 * (k & 1)], b[i][j][k >> 1][2 * (k & 1) + 1]);
        };
        weights(0);
        if (ok) ok = tc::mbar_wait(&act_full[m / 2], (uint32_t)(l & 1), p.status);
        __syncwarp();
        // W2 for this layer (used up since the last one): not while the words of the planes are on their way, which took 3000
        // clocks behind it instead of 1100
        if (l > 0 && tc::elect_one()) {
          load_dn(l, m);
          if (m + kMmaWarps < h_kb) load_dn(l, m + kMmaWarps);
        }
        __syncwarp();
        products(0);
        weights(1);
        products(1);
        __syncwarp();                                                    // (only this warp uses these k-blocks of the activations and of W1)
        float4* part = reinterpret_cast<float4*>(sA) + lane;
        constexpr int kStep = 2 * kRowBytes / 16;                        // from warp to warp
#pragma unroll
        for (int j = 0; j < C::kUpTiles; ++j) part[m * kStep + j * 32] = make_float4(c[j][0], c[j][1], c[j][2], c[j][3]);
        mma_sync();
        if (m < tiles) {
          float4 e = part[m * 32];
#pragma unroll
          for (int k = 1; k < kMmaWarps; ++k) {
            const float4 f = part[k * kStep + m * 32];
            e = make_float4(e.x + f.x, e.y + f.y, e.z + f.z, e.w + f.w);
          }
          const __nv_bfloat162 lo = __floats2bfloat162_rn(tc::gelu_fast(e.x + bias1.x), tc::gelu_fast(e.y + bias1.y));
          const __nv_bfloat162 hi = __floats2bfloat162_rn(tc::gelu_fast(e.z + bias1.x), tc::gelu_fast(e.w + bias1.y));
          uint32_t u[4], d[4];            // the 16 bytes of rows g and g + 8
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            u[i] = __shfl_sync(0xffffffffu, *reinterpret_cast<const uint32_t*>(&lo), (lane & ~3) + i);
            d[i] = __shfl_sync(0xffffffffu, *reinterpret_cast<const uint32_t*>(&hi), (lane & ~3) + i);
          }
          // The tile is 256 bytes in one piece over there: 16 lanes per rank (16 bytes to each of 16 rows, 128 bytes apart, took
          // 3400 clocks for 16 rows).
          const int r = g + 8 * (q & 1);
          const uint4 w = q & 1 ? make_uint4(d[0], d[1], d[2], d[3]) : make_uint4(u[0], u[1], u[2], u[3]);
          const uint32_t at = tc::smem_u32(sH) + (uint32_t)((tile0 + m) * (kMaxRows * 16) + r * 16), bar = tc::smem_u32(h_full);
#pragma unroll
          for (int j = 0; j < kCluster / 2; ++j) {
            const uint32_t to = (uint32_t)(rank + 8 * (q >> 1) + j) % kCluster;
            if (r < p.R) cl::st_async_16(tc::mapa(at, to), w, tc::mapa(bar, to));
          }
        }
        __syncwarp();
        if (tc::elect_one()) {
          for (int i = 2 * m; i < 2 * m + 2; ++i) {
            if (l + 1 < p.L) load_up(l + 1, i);
            else load_lm(0, i);
          }
        }
        if (!ALONE && tid == leader && (l + 1 < p.L || p.head))          // (every phase of this layer has been waited for)
          for (int i = 0; i < 4; ++i) tc::mbar_expect_tx(&act_full[i], (uint32_t)(p.R * D / 2));
        __syncwarp();
      }
      // ---- down: pairs m % 4, + 4, .. of 16-deep steps of half the features ----
      {
        constexpr int kT = C::kDnTiles / 2, kPairs = (C::kHPairs + kDnSplits - 1) / kDnSplits, kAhead = kPairs < 3 ? kPairs : 3;
        const int ks = m % kDnSplits, f0 = m / kDnSplits * kT;
        uint32_t b[kPairs][kT][4];
        float c[kT][4] = {};
        auto weights = [&](int j) {
          const int pr = ks + j * kDnSplits;
          if (pr * 32 < hc) {
            if (ok) ok = tc::mbar_wait(&full_dn[pr >> 1], (uint32_t)(l & 1), p.status);
            __syncwarp();
            const uint32_t w0 = tc::smem_u32(sD) + (pr >> 1) * C::kDnBytes + w_row;
#pragma unroll
            for (int i = 0; i < kT; ++i) sb::ldsm_x4(b[j][i], w0 + (uint32_t)((f0 + i) * 1024) + (((4 * (pr & 1) + w_c) ^ (lane & 7)) << 4));
          }
        };
#pragma unroll
        for (int j = 0; j < kAhead; ++j) weights(j);
        if (ok) ok = tc::mbar_wait(h_full, (uint32_t)(l & 1), p.status);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kPairs; ++j) {
          const int pr = ks + j * kDnSplits;
          if (j + kAhead < kPairs) weights(j + kAhead);
          if (pr * 32 < hc) {
            const uint32_t a0 = tc::smem_u32(sH) + (pr * 4 + a_c) * (kMaxRows * 16) + (lane & 15) * 16;
            uint32_t a[2][4];
#pragma unroll
            for (int k = 0; k < 2; ++k) sb::ldsm_x4(a[k], a0 + k * 2 * (kMaxRows * 16));
            const bool both = pr * 32 + 16 < hc;                         // (the cluster's last step may stand alone)
#pragma unroll
            for (int i = 0; i < kT; ++i) {
              mma(c[i], a[0], b[j][i][0], b[j][i][1]);
              if (both) mma(c[i], a[1], b[j][i][2], b[j][i][3]);
            }
          }
        }
        float4* part = reinterpret_cast<float4*>(sA) + lane;
#pragma unroll
        for (int i = 0; i < kT; ++i) part[(ks * C::kDnTiles + f0 + i) * 32] = make_float4(c[i][0], c[i][1], c[i][2], c[i][3]);
        if (l == 0 && tid == leader && ok) {     // all CTAs have cleared their words, before anyone here looks at one
          const long long t0 = clock64();
          while (sb::ld_relaxed_u32(p.cnt) < gridDim.x) {
            if (clock64() - t0 > kWaitLimitCycles) { ok = false; raise_status(p.status, kStatusWaitTimeout); break; }
          }
          ld_acquire_u32(p.cnt);
        }
        mma_sync();
        float4 e = part[m * 32];
#pragma unroll
        for (int k = 1; k < kDnSplits; ++k) {
          const float4 f = part[(k * C::kDnTiles + m) * 32];
          e = make_float4(e.x + f.x, e.y + f.y, e.z + f.z, e.w + f.w);
        }
        unsigned long long* to = p.planes + (((int64_t)(l & 1) * kClusters + cluster) * p.R + g) * D + rank * kMine + m * 8 + 2 * q;
        if (g < p.R) st_words(to, e.x, e.y, (uint32_t)(l + 1));
        if (g + 8 < p.R) st_words(to + 8 * D, e.z, e.w, (uint32_t)(l + 1));
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(stored);
        if (tid == leader && l + 1 < p.L) tc::mbar_expect_tx(h_full, (uint32_t)(p.R * hc * 2));
        __syncwarp();
      }
    }
    if (p.head) {
      // ---- LM head ----
      if (tc::elect_one())
        for (int i = 2 * m; i < 2 * m + 2; ++i) load_lm(1, i);           // (all warps have used W2)
      __syncwarp();
      float bv[2] = {-INFINITY, -INFINITY};                              // rows g and g + 8
      int bi[2] = {-1, -1};
      bool bad = false;
      if (ok) ok = tc::mbar_wait(&act_full[m / 2], (uint32_t)(p.L & 1), p.status);
      __syncwarp();
      uint32_t a[2][4][4];                                               // this warp's two k-blocks of the rows, for all chunks
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) sb::ldsm_x4(a[i][k], tc::smem_u32(sA) + (2 * m + i) * kRowBytes + a_row + (((2 * k + a_c) ^ a_sw) << 4));
      float4* part = reinterpret_cast<float4*>(sH) + lane;
      for (int ch = 0; ch < lm_chunks; ++ch) {
        float c[C::kUpTiles][4] = {};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int kb = 2 * m + i;
          if (ok) ok = tc::mbar_wait(&full_lm[(ch & 1) * kKb + kb], (uint32_t)(ch >> 1) & 1u, p.status);
          __syncwarp();
          const uint32_t w0 = tc::smem_u32(ch & 1 ? sD : sU) + kb * C::kUpBytes + w_row;
#pragma unroll
          for (int j = 0; j < C::kUpTiles; ++j) {
            uint32_t b[2][4];
#pragma unroll
            for (int k = 0; k < 2; ++k) sb::ldsm_x4(b[k], w0 + (uint32_t)(j * 1024) + (((4 * k + w_c) ^ (lane & 7)) << 4));
#pragma unroll
            for (int k = 0; k < 4; ++k) mma(c[j], a[i][k], b[k >> 1][2 * (k & 1)], b[k >> 1][2 * (k & 1) + 1]);
          }
        }
        mma_sync();                                                      // the partial sums of the chunk before have been taken
#pragma unroll
        for (int j = 0; j < C::kUpTiles; ++j) part[(m * C::kUpTiles + j) * 32] = make_float4(c[j][0], c[j][1], c[j][2], c[j][3]);
        __syncwarp();                                                    // (only this warp uses these k-blocks)
        if (tc::elect_one())
          for (int i = 2 * m; i < 2 * m + 2; ++i) load_lm(ch + 2, i);
        mma_sync();
        const int tile = ch * C::kUpTiles + m;
        if (m < C::kUpTiles && tile < lm_tiles && ok) {
          float4 e = part[m * 32];
#pragma unroll
          for (int k = 1; k < kMmaWarps; ++k) {
            const float4 f = part[(k * C::kUpTiles + m) * 32];
            e = make_float4(e.x + f.x, e.y + f.y, e.z + f.z, e.w + f.w);
          }
          const int col = (lm0 + tile) * 8 + 2 * q;                      // (V is a multiple of 8; ascending: the lowest among equals is kept)
          if (p.logits != nullptr) {
            float* to = p.logits + (int64_t)g * p.V + col;
            if (g < p.R) *reinterpret_cast<float2*>(to) = make_float2(e.x, e.y);
            if (g + 8 < p.R) *reinterpret_cast<float2*>(to + (int64_t)8 * p.V) = make_float2(e.z, e.w);
          }
          if (g < p.R) {
            bad |= !(e.x == e.x) | !(e.y == e.y);
            if (e.x > bv[0]) { bv[0] = e.x; bi[0] = col; }
            if (e.y > bv[0]) { bv[0] = e.y; bi[0] = col + 1; }
          }
          if (g + 8 < p.R) {
            bad |= !(e.z == e.z) | !(e.w == e.w);
            if (e.z > bv[1]) { bv[1] = e.z; bi[1] = col; }
            if (e.w > bv[1]) { bv[1] = e.w; bi[1] = col + 1; }
          }
        }
      }
      if (p.select) {
        if (bad) raise_status(p.status, kStatusNonFinite);
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (bi[i] >= 0) atomicMax(&best[g + 8 * i], sb::pack_best(bv[i] + 0.0f, bi[i]));      // (minus zero equals zero)
        mma_sync();
        const int r = tid - leader;
        if (r < p.R && best[r] != 0ull) atomicMax(p.best + r, best[r]);
        // ---- the CTA that comes last writes the tokens ----
        __threadfence();
        mma_sync();
        if (r == 0) {
          *am_last = atomicAdd(p.cnt + 1, 1u) + 1u == gridDim.x ? 1u : 0u;
          __threadfence();
        }
        mma_sync();
        if (*am_last != 0u && r < p.R) {
          const unsigned long long k = __ldcg(p.best + r);
          int tok = k == 0ull ? 0 : (int)(0xFFFFFFFFu - (uint32_t)k);      // (no finite logit: 0)
          if (tok < 0 || tok >= p.V) tok = 0;
          write_token(p.out, r, tok);
        }
      }
    }
  }

  if (!ok) {      // copies of this CTA, or into it, may still be on their way
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 21)) { }
  }
  __syncwarp();
  tc::cluster_sync();                                                    // the CTAs of a cluster write one another's shared memory
}

}  // namespace sp
}  // namespace srm
