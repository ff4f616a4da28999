// All layers of a small decode pass, every row inside ONE cluster of 16 CTAs from the embedding to the final norm.
//
// The rows of a pass are independent of one another. A kernel that shares a layer's weights out over the whole device has to
// bring the rows together across the grid three times per layer (activations, hidden activations, partial sums), and with a
// few hundred rows those meetings, through L2 and counters in global memory, are all the time there is. Here a cluster takes
// up to 8, 16, 32, 48 or 64 rows (RC) and streams ALL weights of a layer, a sixteenth per CTA; its CTAs meet in distributed
// shared memory only, by stores and copies whose bytes are counted on the receiver's mbarrier. Clusters know nothing of one
// another, so the launch needs no co-residency. The price is that every cluster reads every weight through L2: 1 MB per CTA
// and layer at d = 1024, at 65 to 83 bytes per clock and SM; that stream, which runs ahead of everything, is the bound there.
//
// What a layer takes (device clock, 16 rows per cluster unless said otherwise): d = 512, 9000 clocks = 4.7 us (the layers kernel over
// the whole grid 11 us): activations -> up products 2150, GELU and copies 900, down products 2300, partial products out 600
// and in 900, row phase 1600, activations out 500. With 37 rows per cluster 14200: distributed shared memory takes 21 bytes
// per clock out of an SM and 32 into it. d = 1024, 8 rows: 19500 = 10.1 us, of which the weight stream needs 12600. (Taken when partial
// products were staged in shared memory and copied; from registers, as now, whole calls take the same within half a percent.)
//
// Rank r of the cluster is (K-group kg = r / 4, column ng = r % 4) of a 4 x 4 arrangement:
//   rows:  rank r owns rows r, r + 16, .. of the cluster, whole warps per row, a float4 of the residual stream per thread, in
//          registers for all layers: x + b2 + four partial products, LN1, cache update, residual, LN2; the activation row goes
//          to all 16 CTAs;
//   up:    H columns [kg F / 4 + ng F / 16, + F / 16) for all rows of the cluster (D^T = W1 a^T: weights are the 128-row operand
//          of tcgen05.mma, rows of the batch its N columns, so a few rows waste no tensor time); GELU; each finished tile is
//          copied to the three ranks of the same K-group;
//   down:  output features [ng d / 4, + d / 4) over K = the K-group's quarter of H; the partial product's rows go from
//          registers to the ranks that own them, which add the four K-groups' in rank order.
// A row's bits depend on neither its place in the pass nor the number of rows: every output is one fixed sequence of
// 16-deep tensor steps, and N columns of an instruction do not mix.
//
// At d = 512 the LM head and the greedy selection may follow in the same kernel: 128 vocabulary rows per tile, every 16th tile per
// rank, the logits to global memory where they are wanted, the best logit of a row from every rank to its owner. A kernel of
// its own for each takes longer to start than to run, up to a size of the vocabulary: every cluster reads all of it.
//
// No buffer needs a "free" signal of its own: an owner sends the next layer's activations after it has received every CTA's
// partial products for its rows, a CTA sends those after the products that they come from, and everything else a CTA sends
// in a layer is sent after the activations of ALL owners have come. So, when bytes of layer l + 1 are written,
//   activations: the products that read layer l's have completed (the last partial products come after all of them);
//   H: every owner has all its partial products, so every CTA's products that read H have completed, and with them the copies of
//      hidden columns that these products waited for;
//   partial products received: their owner has added up layer l's, or its activations would not have come.
// Nothing else may leave from shared memory: a copy is counted where it arrives, and that tells one receiver, nobody else, that its
// source has been read (partial products staged over the activations could meet another owner's activations of the next layer).
// For the same reason no byte of a layer can be counted in the phase of the layer before.
// Every wait is bounded: a waiter that gives up raises kStatusWaitTimeout and goes on without waiting; all CTAs meet at the
// final cluster barrier.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "select.cuh"       // SelectOut, write_token
#include "step_small.cuh"   // LayerW, layer_w, bulk_s2s, st_async_v2, pack_best

namespace srm {
namespace cl {

constexpr int kCluster = 16, kGroups = 4, kCols = 4;
constexpr int kIssuers = 2;                                       // MMA warps
constexpr int kWorker0 = 1 + kIssuers, kWorkerWarps = 16;         // warp 0: weight stream, 1 and 2: MMA, then rows and epilogues
constexpr int kWorkers = kWorkerWarps * 32, kThreads = kWorker0 * 32 + kWorkers;
constexpr int kTile = 128;                                        // weight rows per tile
constexpr int kSlotBytes = kTile * 128;                           // one k-block (64 columns) of a weight tile
constexpr int kMaxSlots = 12;
constexpr int kBarrierBytes = 512, kSumBytes = 2 * 16 * 8;
constexpr int kSmemBytes = 227 * 1024;
constexpr long long kWaitLimitCycles = 1ll << 28;

struct Params {
  int R, V, h, n_ctx, L, t;
  float eps;
  int rows;                      // rows per cluster, at most RC
  const int32_t* tok_in;         // [R]
  const bf16* E;
  sb::LayerW layer0;             // as in sb::Params
  int64_t layer_bytes;
  void* S;                       // cache rows of layer 0; layer l at S + l * layer_stride (bytes)
  int64_t layer_stride;
  bf16* a;                       // [R, d]: the final norm's rows
  const float *lnf_g, *lnf_b;
  uint32_t* status;
  const int32_t* ctr;            // device-side step counters or nullptr
  const int32_t* pos;            // [R] per-row positions or nullptr
  int head = 0;                  // D = 512: LM head here; else the final norm's rows to `a`
  int select = 0;                // ... and the greedy selection, to `out`
  float* logits = nullptr;       // ... and the logits, to here ([R, V])
  SelectOut out = {};
};
__host__ __device__ constexpr bool has_head(int d) { return d == 512; }

// Shared memory: activations [k-block][row][128 bytes] | H of the K-group, the same | partial products received
// [K-group][column][tile][own row][128] | weight ring | barriers | row-phase sums.
template <int D, int RC>
struct Shape {
  static constexpr int kUpTiles = D / 512, kDnTiles = D / 512;   // 128-wide tiles per CTA: F / 16, d / 4 with F = 4 d
  static constexpr int kKb = D / 64;                             // k-blocks of either product
  static constexpr int kN = RC < 16 ? 16 : RC;                   // columns of an instruction (RC = 8: the other eight are what follows the rows)
  static constexpr int kOwn = kN / 16, kRowWarps = D / 128;      // rows per CTA, warps per row
  static constexpr int kActBytes = RC * D * 2, kHBytes = RC * D * 2, kRecvBytes = kGroups * kOwn * D * 4;
  static constexpr int kFixed = kActBytes + kHBytes + kRecvBytes + kBarrierBytes + kSumBytes + 1024;
  static constexpr int kSlots = (kSmemBytes - kFixed) / kSlotBytes < kMaxSlots ? (kSmemBytes - kFixed) / kSlotBytes : kMaxSlots;
  static constexpr size_t kSmem = kFixed + (size_t)kSlots * kSlotBytes;
  static constexpr int kAccCols = kIssuers * (kUpTiles + kDnTiles) * kN;
  static constexpr int kTmemCols = kAccCols <= 64 ? 64 : kAccCols <= 128 ? 128 : kAccCols <= 256 ? 256 : 512;
  static_assert(kOwn * kRowWarps <= kWorkerWarps && kSlots >= 4 && kAccCols <= 512 && kKb % kIssuers == 0, "rows of a cluster");
};

__device__ __forceinline__ void tma_load_w(void* dst, const CUtensorMap* map, uint64_t* bar, int row, int kb, int layer) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(tc::smem_u32(bar)), "r"(0), "r"(row), "r"(kb), "r"(layer)
      : "memory");
}
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// 16 bytes into the shared memory of a CTA of the cluster, counted on a barrier over there
__device__ __forceinline__ void st_async_16(uint32_t addr, const uint4& v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
// Four fp32 columns of this thread's TMEM lane (complete after tmem_ld_wait)
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
// Columns 16 g .. 16 g + 3 from `taddr` on of a tile, g < OWN: the sum of the issuers' accumulators, `stride` columns apart.
template <int OWN>
__device__ __forceinline__ void take_tile(uint32_t taddr, int stride, float (&v)[OWN][4]) {
  uint32_t acc[kIssuers][OWN][4];
#pragma unroll
  for (int i = 0; i < kIssuers; ++i)
#pragma unroll
    for (int g = 0; g < OWN; ++g) tmem_ld4(taddr + i * stride + 16 * g, acc[i][g]);
  tc::tmem_ld_wait();
#pragma unroll
  for (int g = 0; g < OWN; ++g)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[g][j] = __uint_as_float(acc[0][g][j]);
#pragma unroll
      for (int i = 1; i < kIssuers; ++i) v[g][j] += __uint_as_float(acc[i][g][j]);
    }
}
// Four values of each of four neighbouring lanes, transposed: lane i of the four gets value i of all four.
__device__ __forceinline__ uint4 transpose4(const float (&v)[4], int lane) {
  const bool odd = lane & 1, high = lane & 2;
  const float a = __shfl_xor_sync(0xffffffffu, odd ? v[0] : v[1], 1), b = __shfl_xor_sync(0xffffffffu, odd ? v[2] : v[3], 1);
  const float w0 = odd ? a : v[0], w1 = odd ? v[1] : a, w2 = odd ? b : v[2], w3 = odd ? v[3] : b;
  const float c = __shfl_xor_sync(0xffffffffu, high ? w0 : w2, 2), e = __shfl_xor_sync(0xffffffffu, high ? w1 : w3, 2);
  return make_uint4(__float_as_uint(high ? c : w0), __float_as_uint(high ? e : w1), __float_as_uint(high ? w2 : c), __float_as_uint(high ? w3 : e));
}
// The i-th k-block of the down projection: the first tile of each rank of the K-group, the own one in front, then the second
// tiles (they come later).
template <int UP, int KB>
__device__ __forceinline__ int down_kb(int i, int ng) {
  constexpr int kPer = KB / UP;
  const int w = i % kPer;
  return ((ng + (w >> 1)) % kCols * UP + i / kPer) * 2 + (w & 1);
}
__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 9, %0;" ::"n"(kWorkers) : "memory"); }

// LayerNorm statistics of a row that WPR warps hold, four channels per thread: mean and sum of squares about it, merged
// pairwise over the warp, then over the warps in order. slot: 2 WPR floats of the group.
template <int WPR>
__device__ __forceinline__ void row_stats(const float4& v, float eps, float* slot, int group, float& mean, float& rstd) {
  float m = ((v.x + v.y) + (v.z + v.w)) * 0.25f;
  const float a = v.x - m, b = v.y - m, c = v.z - m, e = v.w - m;
  float q = (a * a + b * b) + (c * c + e * e), half_n = 2.f;
  auto merge = [](float& m, float& q, float half_n, float m2, float q2) {        // of two sets of 2 half_n values each
    const float dm = m2 - m;
    q += fmaf(dm * dm, half_n, q2);
    m = 0.5f * (m + m2);
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), q2 = __shfl_xor_sync(0xffffffffu, q, o);
    merge(m, q, half_n, m2, q2);
    half_n += half_n;
  }
  if ((threadIdx.x & 31) == 0) {                         // (the lanes may differ in the last bit: lane 0's values count)
    const int w = ((threadIdx.x >> 5) - kWorker0) % WPR;
    slot[w] = m;
    slot[WPR + w] = q;
  }
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(WPR * 32) : "memory");
  float mm[WPR], qq[WPR];
#pragma unroll
  for (int w = 0; w < WPR; ++w) { mm[w] = slot[w]; qq[w] = slot[WPR + w]; }
#pragma unroll
  for (int s = 1; s < WPR; s += s) {
#pragma unroll
    for (int w = 0; w < WPR; w += 2 * s) merge(mm[w], qq[w], half_n, mm[w + s], qq[w + s]);
    half_n += half_n;
  }
  mean = mm[0];
  rstd = rsqrtf(qq[0] * (0.5f / half_n) + eps);
}

template <int D, int RC, typename ST>
__global__ void __launch_bounds__(kThreads, 1)
layers_kernel(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmLm,
              const Params p) {
  pdl_trigger();
  using C = Shape<D, RC>;
  constexpr int kUp = C::kUpTiles, kDn = C::kDnTiles, kKb = C::kKb, kOwn = C::kOwn, kRowWarps = C::kRowWarps;
  constexpr int kRowBytes = RC * 128;                                    // one k-block of activations or of H
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sH = sA + C::kActBytes;
  float* recv = reinterpret_cast<float*>(sH + C::kHBytes);
  uint8_t* sW = sH + C::kHBytes + C::kRecvBytes;
  uint64_t* fullW = reinterpret_cast<uint64_t*>(sW + C::kSlots * kSlotBytes);
  uint64_t* emptyW = fullW + kMaxSlots;
  uint64_t* act_full = emptyW + kMaxSlots;
  uint64_t* recv_full = act_full + 4;                                    // act_full: by quarters of the channels
  uint64_t* up_done = recv_full + 1;                                     // [kUp] accumulators
  uint64_t* dn_done = up_done + kUp;                                     // [kDn]
  uint64_t* h_full = dn_done + kDn;                                      // [column of the K-group][tile]
  uint64_t* head_empty = h_full + kCols * kUp;                           // [2] accumulators of the LM head drained
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(head_empty + 2);
  float* sums = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(fullW) + kBarrierBytes);
  static_assert((2 * kMaxSlots + 7 + kUp + kDn + kCols * kUp) * 8 + 4 <= kBarrierBytes, "barriers");

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = (int)tc::cluster_ctarank();
  const int kg = rank / kCols, ng = rank % kCols;
  const int row_base = (int)(blockIdx.x / kCluster) * p.rows;            // first row of this cluster
  const int rows = min(p.rows, p.R - row_base);                          // its rows; rank r owns rows r, r + 16, ...
  auto rows_of = [rows](int r) { return (rows - r + kCluster - 1) / kCluster; };
  if (threadIdx.x == 0) {
    for (int i = 0; i < kMaxSlots; ++i) { tc::mbar_init(&fullW[i], 1); tc::mbar_init(&emptyW[i], 1); }
    for (int i = 0; i < 4; ++i) tc::mbar_init(&act_full[i], 1);
    tc::mbar_init(recv_full, 1);
    for (int i = 0; i < kUp; ++i) tc::mbar_init(&up_done[i], kIssuers);
    for (int i = 0; i < kDn; ++i) tc::mbar_init(&dn_done[i], kIssuers);
    for (int i = 0; i < kCols * kUp; ++i) tc::mbar_init(&h_full[i], 1);
    for (int i = 0; i < 2; ++i) tc::mbar_init(&head_empty[i], kWorkerWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc::tc_fence_before();
  tc::cluster_sync();                                                    // (every CTA's barriers are set before a byte is sent to it)
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;                                      // up tiles, then down tiles, an accumulator per issuer each
  bool ok = true;                                                        // no wait has given up in this thread
  const bool head_here = has_head(D) && p.head != 0;
  const int head_tiles = head_here ? (p.V + kTile - 1) / kTile : 0;      // tiles rank, rank + 16, ... are this CTA's

  if (warp == 0) {
    // ---------------- weight stream: constant data, it waits for nothing but its ring ----------------
    if (tc::elect_one()) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmW1)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmW2)) : "memory");
      int slot = 0;
      uint32_t phase = 0;
      for (int l = 0; ok && l < p.L; ++l) {
        for (int i = 0; i < (kUp + kDn) * kKb; ++i) {
          const int tile = i / kKb, kb = i % kKb;
          const bool dn = tile >= kUp;
          if (!tc::mbar_wait(&emptyW[slot], phase ^ 1u, p.status)) { ok = false; break; }
          tc::mbar_expect_tx(&fullW[slot], kSlotBytes);
          tma_load_w(sW + slot * kSlotBytes, dn ? &tmW2 : &tmW1, &fullW[slot],
                     dn ? (ng * kDn + tile - kUp) * kTile : ((kg * kCols + ng) * kUp + tile) * kTile,
                     dn ? kg * kKb + down_kb<kUp, kKb>(kb, ng) : kb, l);
          if (++slot == C::kSlots) { slot = 0; phase ^= 1u; }
        }
      }
      if constexpr (has_head(D)) {
        for (int tile = rank; ok && tile < head_tiles; tile += kCluster) {
          for (int kb = 0; kb < kKb; ++kb) {
            if (!tc::mbar_wait(&emptyW[slot], phase ^ 1u, p.status)) { ok = false; break; }
            tc::mbar_expect_tx(&fullW[slot], kSlotBytes);
            tma_load_w(sW + slot * kSlotBytes, &tmLm, &fullW[slot], tile * kTile, kb, 0);
            if (++slot == C::kSlots) { slot = 0; phase ^= 1u; }
          }
        }
      }
    }
  } else if (warp < kWorker0) {
    // ---------------- MMA issuers: each takes every other k-block, into an accumulator of its own ----------------
    // (waits, descriptors and commit of a k-block keep one thread busy for 350 to 400 cycles, its four instructions the tensor
    // pipe for 156 to 192; two issuers reach the latter)
    if (tc::elect_one()) {
      // fp32 accumulate, bf16 operands, both K-major, M = 128 weight rows, N = rows of the batch
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(C::kN >> 3) << 17) | (uint32_t(kTile >> 4) << 24);
      const int mine = warp - 1;
      int slot = mine;
      uint32_t phase = 0;
      auto k_block = [&](uint32_t acc, const uint8_t* b, bool first) {
        if (!tc::mbar_wait(&fullW[slot], phase, p.status)) { ok = false; return; }
        tc::tc_fence_after();
        const uint64_t da = tc::make_smem_desc(tc::smem_u32(sW + slot * kSlotBytes)), db = tc::make_smem_desc(tc::smem_u32(b));
#pragma unroll
        for (int k = 0; k < 4; ++k) umma(acc, da + 2u * k, db + 2u * k, idesc, (first && k == 0) ? 0u : 1u);
        umma_commit(&emptyW[slot]);
        slot += kIssuers;
        if (slot >= C::kSlots) { slot -= C::kSlots; phase ^= 1u; }
      };
      for (int l = 0; ok && l < p.L; ++l) {
        if (mine == 0) {
          for (int i = 0; i < 4; ++i) tc::mbar_expect_tx(&act_full[i], (uint32_t)(rows * D / 2));
          for (int i = 0; i < kCols * kUp; ++i)
            if (i / kUp != ng) tc::mbar_expect_tx(&h_full[i], 2 * kRowBytes);
        }
        for (int m = 0; ok && m < kUp; ++m) {
          const uint32_t acc = tmem + (m * kIssuers + mine) * C::kN;
          for (int kb = mine; ok && kb < kKb; kb += kIssuers) {
            if (m == 0 && kb % (kKb / 4) == mine) {
              ok = tc::mbar_wait(&act_full[kb / (kKb / 4)], (uint32_t)(l & 1), p.status);
              tc::fence_async_smem();                                    // the rows came by ordinary stores of other CTAs
            }
            if (ok) k_block(acc, sA + kb * kRowBytes, kb == mine);
          }
          if (ok) umma_commit(&up_done[m]);
        }
        for (int m = 0; ok && m < kDn; ++m) {
          const uint32_t acc = tmem + ((kUp + m) * kIssuers + mine) * C::kN;
          for (int i = mine; ok && i < kKb; i += kIssuers) {
            const int kb = down_kb<kUp, kKb>(i, ng);
            if (m == 0) {                                                // a tile of H is two k-blocks
              ok = tc::mbar_wait(&h_full[kb >> 1], (uint32_t)(l & 1), p.status);
              tc::fence_async_smem();
            }
            if (ok) k_block(acc, sH + kb * kRowBytes, i == mine);
          }
          if (ok) umma_commit(&dn_done[m]);
        }
      }
      if constexpr (has_head(D)) {
        if (head_here && ok) {
          if (mine == 0)
            for (int i = 0; i < 4; ++i) tc::mbar_expect_tx(&act_full[i], (uint32_t)(rows * D / 2));
          for (int i = 0; ok && i < 4; ++i) ok = tc::mbar_wait(&act_full[i], (uint32_t)(p.L & 1), p.status);
          tc::fence_async_smem();
          int n = 0;
          for (int tile = rank; ok && tile < head_tiles; tile += kCluster, ++n) {
            if (n >= 2) ok = tc::mbar_wait(&head_empty[n & 1], (uint32_t)((n >> 1) - 1) & 1u, p.status);
            tc::tc_fence_after();
            const uint32_t acc = tmem + ((n & 1) * kIssuers + mine) * C::kN;
            for (int kb = mine; ok && kb < kKb; kb += kIssuers) k_block(acc, sA + kb * kRowBytes, kb == mine);
            if (ok) umma_commit(n & 1 ? &dn_done[0] : &up_done[0]);
          }
        }
      }
    }
  } else {
    // ---------------- rows and epilogues ----------------
    const int wid = threadIdx.x - kWorker0 * 32, ww = wid >> 5;
    const int group = ww / kRowWarps, th = wid % (kRowWarps * 32), c0 = th * 4;
    const int quad = warp & 3, cgrp = ww >> 2;                           // TMEM lanes this warp may read; its quarter of the columns
    const bool cols = cgrp * 4 < RC;                                     // rows 4 cgrp .. 4 cgrp + 3, and 16, 32, 48 further
    pdl_wait();
    const int t_all = p.ctr != nullptr ? p.ctr[kCtrPos] : p.t;
    const int local = group * kCluster + rank, row = row_base + local;   // the row of this thread's warps
    const bool mine = group < kOwn && local < rows;
    const int own = rows_of(rank);                                       // rows of this CTA
    const int t = mine && p.pos != nullptr ? min(max(p.pos[row], 0), p.n_ctx - 1) : t_all;
    const int head = c0 / (D / p.h);
    const bool is_row = head < (p.h >> 1);
    float* slot = sums + group * (2 * kRowWarps);                        // (a second set of sums lies 2 * kWorkerWarps floats on)
    const float* part = recv + ((c0 / (D / 4) * kDn + c0 % (D / 4) / kTile) * kOwn + group) * kTile + c0 % kTile;
    const uint32_t recv_bytes = (uint32_t)(kGroups * own * D * 4);
    // where this thread's pair of lanes puts its 16 bytes of an activation row
    const uint32_t act_addr = tc::smem_u32(sA) + (uint32_t)((c0 >> 6) * kRowBytes + local * 128) +
                              (uint32_t)(((c0 >> 3 & 7) ^ (local & 7)) << 4);
    const int qd = c0 / (D / 4);                                         // this warp's quarter of the channels
    const uint32_t act_bar = tc::smem_u32(&act_full[qd]);

    // Parameters of a row phase, fetched a layer ahead: constant data, and this thread's part of the cache row.
    float4 g1, h1, bt, g2, h2, bias2, s, v;
    float al = 0.f, lam = 0.f, bias1[kUp];
    auto fetch = [&](int l) {
      const bool last = l == p.L;
      const sb::LayerW w = sb::layer_w(p, last ? 0 : l);
      if (mine) {
        g2 = ldg4((last ? p.lnf_g : w.ln2_g) + c0);
        h2 = ldg4((last ? p.lnf_b : w.ln2_b) + c0);
        if (l > 0) bias2 = ldg4(sb::layer_w(p, l - 1).b2 + c0);
        if (!last) {
          g1 = ldg4(w.ln1_g + c0);
          h1 = ldg4(w.ln1_b + c0);
          bt = ldg4(w.beta + (int64_t)t * D + c0);
          al = __ldg(w.alpha + (int64_t)head * p.n_ctx + t);
          lam = __ldg(w.lam + head);
          s = ld4(reinterpret_cast<const ST*>(static_cast<const uint8_t*>(p.S) + (int64_t)l * p.layer_stride) + (int64_t)row * D + c0);
        }
      }
    };
    fetch(0);
    for (int l = 0;; ++l) {
      const bool last = l == p.L;
      if (mine) {
        if (l == 0) {
          int tk = p.tok_in[row];
          if (tk < 0 || tk >= p.V) {
            if (th == 0) raise_status(p.status, kStatusTokenRange);
            tk = tk < 0 ? 0 : p.V - 1;
          }
          v = ldg4(p.E + (int64_t)tk * D + c0);
        } else {                          // x + b2 + the K-groups' partial products
          if (ok) ok = tc::mbar_wait(recv_full, (uint32_t)(l - 1) & 1u, p.status, kWaitLimitCycles);
          v = make_float4(v.x + bias2.x, v.y + bias2.y, v.z + bias2.z, v.w + bias2.w);
#pragma unroll
          for (int k = 0; k < kGroups; ++k) {
            const float4 e = ld4(part + k * (kOwn * D));
            v = make_float4(v.x + e.x, v.y + e.y, v.z + e.z, v.w + e.w);
          }
        }
        float mean, rstd;
        if (!last) {
          row_stats<kRowWarps>(v, p.eps, slot, group, mean, rstd);
          const float nmr = -mean * rstd;
          const float4 z = make_float4(fmaf(fmaf(v.x, rstd, nmr), g1.x, h1.x), fmaf(fmaf(v.y, rstd, nmr), g1.y, h1.y),
                                       fmaf(fmaf(v.z, rstd, nmr), g1.z, h1.z), fmaf(fmaf(v.w, rstd, nmr), g1.w, h1.w));
          // row-repeat head, Eq. 2: y = (a z + S) + b ; S' = l (S + a z).  column-repeat head, Eq. 3: y = a (z + S) + b ; S' = l (z + S)
          const float a1 = is_row ? al : 1.0f, a2 = is_row ? 1.0f : al;
          const float4 u = make_float4(fmaf(a1, z.x, s.x), fmaf(a1, z.y, s.y), fmaf(a1, z.z, s.z), fmaf(a1, z.w, s.w));
          st4(reinterpret_cast<ST*>(static_cast<uint8_t*>(p.S) + (int64_t)l * p.layer_stride) + (int64_t)row * D + c0,
              make_float4(lam * u.x, lam * u.y, lam * u.z, lam * u.w));
          v = make_float4(v.x + fmaf(a2, u.x, bt.x), v.y + fmaf(a2, u.y, bt.y), v.z + fmaf(a2, u.z, bt.z), v.w + fmaf(a2, u.w, bt.w));
        }
        row_stats<kRowWarps>(v, p.eps, slot + 2 * kWorkerWarps, group, mean, rstd);
        const float nmr2 = -mean * rstd;
        const float4 o = make_float4(fmaf(fmaf(v.x, rstd, nmr2), g2.x, h2.x), fmaf(fmaf(v.y, rstd, nmr2), g2.y, h2.y),
                                     fmaf(fmaf(v.z, rstd, nmr2), g2.z, h2.z), fmaf(fmaf(v.w, rstd, nmr2), g2.w, h2.w));
        if (last && !head_here) {
          st4(p.a + (int64_t)row * D + c0, o);
        } else {
          const __nv_bfloat162 lo = __floats2bfloat162_rn(o.x, o.y), hi = __floats2bfloat162_rn(o.z, o.w);
          const uint32_t q0 = *reinterpret_cast<const uint32_t*>(&lo), q1 = *reinterpret_cast<const uint32_t*>(&hi);
          const uint32_t r0 = __shfl_xor_sync(0xffffffffu, q0, 1), r1 = __shfl_xor_sync(0xffffffffu, q1, 1);
          const int odd = lane & 1;
          const uint4 w = odd ? make_uint4(r0, r1, q0, q1) : make_uint4(q0, q1, r0, r1);
          // One quarter of the channels after the other, so that the first k-blocks are there early: distributed shared memory
          // takes 21 bytes per clock from an SM, a row of 1024 channels to 16 CTAs 1560 clocks.
          const uint32_t turn = (uint32_t)own * (kRowWarps / 4) * 64;
          if (qd > 0) asm volatile("bar.sync %0, %1;" ::"r"(9 + qd), "r"(turn) : "memory");
#pragma unroll
          for (int j = 0; j < kCluster / 2; ++j) {       // even lanes: eight of the ranks, odd lanes: the other eight
            const uint32_t to = (uint32_t)(rank + 8 * odd + j) % kCluster;
            st_async_16(tc::mapa(act_addr, to), w, tc::mapa(act_bar, to));
          }
          if (qd < 3) asm volatile("bar.arrive %0, %1;" ::"r"(10 + qd), "r"(turn) : "memory");
        }
      }
      if (last) break;
      if (wid == 0 && own > 0) tc::mbar_expect_tx(recv_full, recv_bytes);      // (this thread has waited for the phase before)
      {
        const sb::LayerW w = sb::layer_w(p, l);
#pragma unroll
        for (int m = 0; m < kUp; ++m) bias1[m] = __ldg(w.b1 + ((kg * kCols + ng) * kUp + m) * kTile + quad * 32 + lane);
      }
      fetch(l + 1);

      // ---- up: lane = feature, columns = rows. GELU, bf16, into H of the K-group in the 128-byte swizzle ----
#pragma unroll
      for (int m = 0; m < kUp; ++m) {
        if (ok) ok = tc::mbar_wait(&up_done[m], (uint32_t)(l & 1), p.status);
        tc::tc_fence_after();
        if (cols) {
          float acc[kOwn][4];
          take_tile<kOwn>(tmem + (static_cast<uint32_t>(quad * 32) << 16) + (uint32_t)(m * kIssuers * C::kN + cgrp * 4), C::kN, acc);
          const int f = (ng * kUp + m) * kTile + quad * 32 + lane;       // column of the K-group's quarter of H
          uint8_t* col = sH + (f >> 6) * kRowBytes + (f & 7) * 2 + cgrp * 4 * 128;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint8_t* at = col + j * 128 + (((f >> 3 & 7) ^ ((cgrp & 1) * 4 + j)) << 4);
#pragma unroll
            for (int g = 0; g < kOwn; ++g)
              *reinterpret_cast<bf16*>(at + g * 16 * 128) = __float2bfloat16_rn(tc::gelu_fast(acc[g][j] + bias1[m]));
          }
        }
        tc::tc_fence_before();
        tc::fence_async_smem();
        workers_sync();
        if (wid < kCols) {                                               // one copy per rank of the K-group, this CTA's own: a count
          const int i = ng * kUp + m;
          if (wid == ng) tc::mbar_arrive(&h_full[i]);
          else sb::bulk_s2s(tc::mapa(tc::smem_u32(sH + i * 2 * kRowBytes), (uint32_t)(kg * kCols + wid)), sH + i * 2 * kRowBytes, 2 * kRowBytes,
                            tc::mapa(tc::smem_u32(&h_full[i]), (uint32_t)(kg * kCols + wid)));
        }
      }
      // ---- down: partial products of this CTA's features, by rows, to the ranks that own them ----
#pragma unroll
      for (int m = 0; m < kDn; ++m) {
        if (ok) ok = tc::mbar_wait(&dn_done[m], (uint32_t)(l & 1), p.status);
        tc::tc_fence_after();
        // (a warp whose rows do not exist reads what nobody uses; with a test of `rows` instead, the same for the whole warp, a step of 8 layers
        // with 10 or 16 rows per cluster at d = 512 took 52.4 and 54.3 us instead of 50.8 and 52.9)
        if (cols) {
          float acc[kOwn][4];
          take_tile<kOwn>(tmem + (static_cast<uint32_t>(quad * 32) << 16) + (uint32_t)((kUp + m) * kIssuers * C::kN + cgrp * 4), C::kN, acc);
          const int to = cgrp * 4 + (lane & 3);                          // four features of one row per lane, 128 bytes per row and warp
          const uint32_t at = tc::mapa(tc::smem_u32(recv + ((kg * kCols + ng) * kDn + m) * kOwn * kTile + quad * 32 + (lane & ~3)), (uint32_t)to);
          const uint32_t bar = tc::mapa(tc::smem_u32(recv_full), (uint32_t)to);
#pragma unroll
          for (int g = 0; g < kOwn; ++g) {
            const uint4 e = transpose4(acc[g], lane);
            if (to + kCluster * g < rows) st_async_16(at + g * kTile * 4, e, bar);
          }
        }
        tc::tc_fence_before();
      }
    }
  }

  if constexpr (has_head(D)) {
    if (head_here && warp >= kWorker0) {
      // ---- LM head: the largest logit of each row (lowest column among equals), in a thread over its columns, then over the lanes,
      //      the warps, and by the row's owner over the ranks ----
      const int wid = threadIdx.x - kWorker0 * 32, ww = wid >> 5, quad = warp & 3, cgrp = ww >> 2;
      unsigned long long* best = reinterpret_cast<unsigned long long*>(recv);                     // [RC]
      unsigned long long* slots = best + 64;                                                      // [own row][rank]
      const int own = rows_of(rank);
      // The final norm's rows have come from every owner: each has added up its partial products, and the phase that counted them is over.
      // Without this a rank that has no tile of the vocabulary, and so waits for no product, could send its logits into that phase.
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (ok) ok = tc::mbar_wait(&act_full[i], (uint32_t)(p.L & 1), p.status);
      if (p.select && wid == 0 && own > 0) tc::mbar_expect_tx(recv_full, (uint32_t)(own * kCluster * 8));
      float bv[kOwn][4];
      int bi[kOwn][4];
      bool bad = false;
#pragma unroll
      for (int g = 0; g < kOwn; ++g)
#pragma unroll
        for (int j = 0; j < 4; ++j) { bv[g][j] = -INFINITY; bi[g][j] = -1; }
      int n = 0;
      for (int tile = rank; tile < head_tiles; tile += kCluster, ++n) {
        if (ok) ok = tc::mbar_wait(n & 1 ? &dn_done[0] : &up_done[0], (uint32_t)(p.L + (n >> 1)) & 1u, p.status);
        tc::tc_fence_after();
        if (cgrp * 4 < RC) {
          float acc[kOwn][4];
          take_tile<kOwn>(tmem + (static_cast<uint32_t>(quad * 32) << 16) + (uint32_t)((n & 1) * kIssuers * C::kN + cgrp * 4), C::kN, acc);
          const int col = tile * kTile + quad * 32 + lane;
          if (p.logits != nullptr && col < p.V) {
#pragma unroll
            for (int g = 0; g < kOwn; ++g)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int r = g * kCluster + cgrp * 4 + j;
                if (r < rows) p.logits[(int64_t)(row_base + r) * p.V + col] = acc[g][j];
              }
          }
          if (col < p.V && ok) {
#pragma unroll
            for (int g = 0; g < kOwn; ++g)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                bad |= g * kCluster + cgrp * 4 + j < rows && !(acc[g][j] == acc[g][j]);
                if (acc[g][j] > bv[g][j]) { bv[g][j] = acc[g][j]; bi[g][j] = col; }              // (ascending columns)
              }
          }
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&head_empty[n & 1]);
      }
      if (p.select) {
        if (bad) raise_status(p.status, kStatusNonFinite);
        workers_sync();                                                    // (the partial products that lay here have been read)
        for (int i = wid; i < RC; i += kWorkers) best[i] = 0ull;
        workers_sync();
        if (cgrp * 4 < RC) {
#pragma unroll
          for (int g = 0; g < kOwn; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              unsigned long long k = bi[g][j] < 0 ? 0ull : sb::pack_best(bv[g][j] + 0.0f, bi[g][j]);      // (minus zero equals zero)
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, k, o);
                k = k2 > k ? k2 : k;
              }
              if (lane == 0 && k != 0ull) atomicMax(&best[g * kCluster + cgrp * 4 + j], k);
            }
        }
        workers_sync();
        if (wid < rows) {                                                  // row wid: to its owner
          const uint32_t to = (uint32_t)(wid % kCluster);
          const unsigned long long k = best[wid];
          sb::st_async_v2(tc::mapa(tc::smem_u32(slots + (wid / kCluster) * kCluster + rank), to), __uint_as_float((uint32_t)k),
                          __uint_as_float((uint32_t)(k >> 32)), tc::mapa(tc::smem_u32(recv_full), to));
        }
        if (wid < own) {
          if (ok) ok = tc::mbar_wait(recv_full, (uint32_t)(p.L & 1), p.status, kWaitLimitCycles);
          unsigned long long k = 0ull;
          for (int r = 0; r < kCluster; ++r) {
            const unsigned long long k2 = slots[wid * kCluster + r];
            k = k2 > k ? k2 : k;
          }
          int tok = k == 0ull ? 0 : (int)(0xFFFFFFFFu - (uint32_t)k);      // (no finite logit: 0)
          if (tok < 0 || tok >= p.V) tok = 0;
          write_token(p.out, row_base + wid * kCluster + rank, tok);
        }
      }
    }
  }

  if (!ok) {      // copies of this CTA, or into it, may still be on their way
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 21)) { }
  }
  // All CTAs stay until the cluster is done: they write one another's shared memory.
  tc::tc_fence_before();
  __syncwarp();
  tc::cluster_sync();
  if (warp == 1) {
    tc::tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
  }
}

}  // namespace cl
}  // namespace srm
