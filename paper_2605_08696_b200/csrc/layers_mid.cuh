// All layers of a decode pass of up to about a thousand rows as ONE persistent kernel.
//
// With so few rows a layer is a chain of three short kernels (token mixer, up projection, down projection over ranges of
// K), and launch, ramp, first loads and drain of each cost more than its work: 25 us per layer at 256 rows of the mid
// model, of which the operands need 5. Here one CTA pair per SM pair stays for the whole pass:
//   - weights are constant, so a producer thread of their own streams every CTA's W1 and W2 tiles through a ring that
//     runs ahead of everything else: a projection finds its first k-blocks in shared memory when its input is ready;
//   - a pair computes at most one 256 x N tile of the up projection and one of the down projection per layer (the down
//     projection's K cut into ranges), N 64 or 128, the smaller with which the tiles fit on the pairs;
//   - row phases (x + partial products of the previous down projection, LN1, cache update, residual, LN2) are done by four
//     warps per row (two where there are more rows than that serves at once), the rows dealt to all CTAs. With four all
//     loads of a row are in flight at once: 2.9 -> 1.5 us per layer at 256 rows of the mid model (two warps per row spill 76 to
//     88 bytes at d = 1536 and with combined heads at d = 1024);
//   - the phases are ordered by counters in global memory, one per 256-row block (and range of K): rows done -> up tiles
//     of the block start; up tiles of a range done -> down tiles of that range start; down tiles done -> rows of the
//     block start. Nothing waits for a block it does not read.
// Combined heads and kernels of size k (MIX) differ in the row phase only: their cache planes and scalars, and for kernels a
// barrier of the row's warps per filter.
// Mixed-head models of other widths than 512, 1024 and 1536 (kMixedAny, up to 64 rows): threads beyond the last channel hold
// nothing, the last column tile may be partly filled, and what a stage holds beyond the last k-block is zeros.
// Projections run as in gemm_tc_kernel: TMA loads (128-byte swizzle), tcgen05.mma.cta_group::2 issued by one thread of
// the leader CTA, accumulator in tensor memory, 16 epilogue warps.
//
// Every piece of work waits for pieces of an earlier phase only, all CTAs are resident (the grid is the number of pairs
// the device holds), and every wait is bounded: a waiter that gives up raises kStatusWaitTimeout and leaves its loops;
// the others time out in turn, both CTAs of a pair meet at the final cluster barrier and the kernel ends.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "gemm_tc_splitk.cuh"   // fence_async_global
#include "prefill_chunk.cuh"    // ld_acquire_u32
#include "step_small.cuh"       // LayerW, group_stats, head_scalars, cp_async16, ld_relaxed_u32

namespace srm {
namespace mid {

constexpr int kEpiWarp0 = 3;                                      // warp 0: A producer, 1: MMA, 2: W producer
constexpr int kThreads = (kEpiWarp0 + tc::kEpiWarps) * 32;
constexpr int kWorkers = tc::kEpiWarps * 32;                      // threads of the epilogue / row warps
constexpr int kMaxGroups = tc::kEpiWarps / 2;                     // rows a CTA works on at a time, at most
constexpr int kStep = 2;                                          // k-blocks (of 64) per stage: the waits and commits of a stage take as long as a k-block's MMAs
constexpr int kMaxWSlots = 8, kMaxASlots = 4;
constexpr int kABytes = kStep * tc::kRowsPerCta * tc::BK * 2;     // one stage of A per CTA
constexpr int kTmemCols = 128;
constexpr int kBarrierBytes = 512;
constexpr int kMaxRowBlocks = 8, kMaxKSlices = 4;
constexpr int kSmemBytes = 227 * 1024;
constexpr long long kWaitLimitCycles = 1ll << 28;

struct Params {
  int R, d, F, V, h, n_ctx, L, t;
  float eps;
  int rb, n, cu, cd, ks;         // row blocks, tile width, column tiles of the up / down projection, ranges of K
  int slice_tiles;               // column tiles of H per range of K (the last range may have fewer)
  int w_slots, a_slots;
  int box;                       // rows of an activation box: 128, or the rows there are (a multiple of 8); rows of zeros that the copy
                                 // unit fills in for rows beyond the last cost it more than rows it reads (45 rows: 2.7 against 1.2 us per tile)
  const int32_t* tok_in;         // [R]
  const bf16* E;
  sb::LayerW layer0;             // as in sb::Params
  int64_t layer_bytes;
  void* S;                       // cache rows of layer 0; layer l at S + l * layer_stride (bytes)
  int64_t layer_stride;
  float* x;                      // [R, d]
  bf16* a;                       // [R, d]: activations of the up projection, at the end of the final norm
  const float *lnf_g, *lnf_b;
  bf16* H;                       // [R, F]
  float* part;                   // [ks] planes of plane_rows x d 
  int64_t plane;                 // elements per plane
  int plane_rows;                // rows per plane
  uint32_t* cnt;                 // rows done [8] | up pieces done [8][4] | down pieces done [8]; zero on entry
  uint32_t* status;
  const int32_t* ctr;            // device-side step counters or nullptr
  const int32_t* pos;            // [R] per-row positions or nullptr (mixed heads only)
  // the further mixers: cache planes `s_plane` elements apart, parameters of layer 0 (as in VariantParams)
  int k = 1;
  int64_t s_plane = 0;
  const float *alpha_col = nullptr, *lam_col = nullptr, *w_comb = nullptr;
};
// Row-phase parameters in shared memory: ln1_g | ln1_b | beta_t | ln2_g | ln2_b | b2 of the previous layer, then this CTA's
// part of b1 (first touched in the epilogue it came from HBM there: 0.7 us).
constexpr int kVecs = 6;
// Token mixers: mixed heads; combined heads; kernels of size k; mixed heads of any width (d a multiple of 64, at most
// NT * kStride: threads beyond the last channel hold nothing).
constexpr int kMixed = 0, kCombined = 1, kKernel = 2, kMixedAny = 3;
__host__ __device__ constexpr bool mixed_heads(int mix) { return mix == kMixed || mix == kMixedAny; }
constexpr int kMixScalars = 64;      // of a layer at the pass's position: combined 6 h <= 48 floats, kernel 2 k <= 32
constexpr int kCntWords = kMaxRowBlocks * (2 + kMaxKSlices);
__global__ void __launch_bounds__(64) zero_counters_kernel(uint32_t* __restrict__ cnt) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x < kCntWords) cnt[threadIdx.x] = 0;
}
static_assert(kCntWords <= 64, "one thread per counter");

// Shared memory: W ring | A ring (both 1024-byte aligned) | row-phase parameters | row-phase sums | barriers | for the
// further mixers their scalars and, for kernels, the channels a warp's last lanes read of the next warp.
__host__ __device__ inline size_t smem_bytes(int d, int n, int w_slots, int a_slots, int mix) {
  return 1024 + (mixed_heads(mix) ? 0 : kMixScalars * 4 + (mix == kKernel ? (size_t)kMaxGroups * d : 0)) + (size_t)w_slots * kStep * (n / 2) * 128 + (size_t)a_slots * kABytes + ((size_t)kVecs * d + n) * 4 + kMaxGroups * 32 + kBarrierBytes;
}

// Tile widths and ranges of K (at most most_ks: kMaxKSlices, twice that for kMixedAny, whose single row block uses the counters
// of a second for the further ranges) for R rows of a model (d, F) on `pairs` CTA pairs; false: the pieces do not fit. (256-wide
// tiles, which would take mid passes of 513 to 1024 rows, measured slower than a kernel per operation: 0.59 against
// 0.54 ms per step.)
inline bool plan(int64_t R, int d, int F, int pairs, int mix, int most_ks, Params* p) {
  const int rb = (int)((R + tc::BM - 1) / tc::BM);
  if (rb < 1 || rb > (mix == kMixedAny ? 1 : kMaxRowBlocks)) return false;
  for (int n = 64; n <= 128; n *= 2) {
    const int cu = (F + n - 1) / n, cd = (d + n - 1) / n;            // (the last tile of a row block may be partly filled)
    if (n > d || rb * cu > pairs || rb * cd > pairs) continue;
    // ranges of whole column tiles of H and of whole stages; what a stage holds beyond the last k-block is zeros
    const int grain = kStep * 64 / n;
    int ks = most_ks;
    auto per = [&] { return ((cu + ks - 1) / ks + grain - 1) / grain * grain; };
    while (ks > 1 && (rb * cd * ks > pairs || (ks - 1) * per() >= cu)) ks >>= 1;
    p->slice_tiles = per();
    p->box = R < tc::kRowsPerCta ? (int)(R + 7) / 8 * 8 : tc::kRowsPerCta;
    p->rb = rb; p->n = n; p->cu = cu; p->cd = cd; p->ks = ks;
    // the weight ring runs a phase ahead; the activation ring hides the latency of L2 and holds the output tile of an
    // epilogue (128 rows of n fp32 columns)
    p->w_slots = n == 64 ? 8 : 6;
    p->a_slots = n == 64 ? 4 : 3;
    while (smem_bytes(d, n, p->w_slots, p->a_slots, mix) > (size_t)kSmemBytes)
      if (--p->w_slots < 2) return false;
    return true;
  }
  return false;
}

// One stage: kStep k-blocks of 64 columns, each a tile of its own (128-byte rows, swizzled). a: {64, rows, K / 64};
// W: {64, rows, K / 64, layer}.
__device__ __forceinline__ void tma_load_a(void* dst, const CUtensorMap* map, uint32_t bar_cluster_addr, int row, int kb) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster_addr), "r"(0), "r"(row), "r"(kb)
      : "memory");
}
__device__ __forceinline__ void tma_load_w(void* dst, const CUtensorMap* map, uint32_t bar_cluster_addr, int row, int kb, int layer) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster_addr), "r"(0), "r"(row), "r"(kb), "r"(layer)
      : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(tc::smem_u32(src)), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void red_release_add(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// One thread waits until the counter has reached `want`.
__device__ __forceinline__ bool count_wait(const uint32_t* p, uint32_t want, uint32_t* status) {
  if (sb::ld_relaxed_u32(p) < want) {
    const long long t0 = clock64();
    while (sb::ld_relaxed_u32(p) < want) {
      if (clock64() - t0 > kWaitLimitCycles) { raise_status(status, kStatusWaitTimeout); return false; }
    }
  }
  ld_acquire_u32(p);
  return true;
}
__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 9, %0;" ::"n"(kWorkers) : "memory"); }

// LayerNorm statistics of a row held by WPG warps (thread th of them: float4s 32 WPG apart): every thread's mean and sum of
// squares about it are merged over the warp, then over the warps in order. slot: 2 WPG floats of the group.
template <int NT, int WPG>
__device__ __forceinline__ void group_stats(const float4 (&v)[NT], float eps, float* slot, int group, float& mean, float& rstd) {
  float m = 0.f, q = 0.f, cnt = 4.f * NT;
#pragma unroll
  for (int i = 0; i < NT; ++i) m += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  m *= 1.0f / (4.f * NT);
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const float a = v[i].x - m, b = v[i].y - m, c = v[i].z - m, e = v[i].w - m;
    q += (a * a + b * b) + (c * c + e * e);
  }
  auto merge = [](float& m, float& q, float cnt, float m2, float q2) {        // of two sets of cnt values each
    const float dm = m2 - m;
    q += fmaf(dm * dm, 0.5f * cnt, q2);
    m = 0.5f * (m + m2);
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), q2 = __shfl_xor_sync(0xffffffffu, q, o);
    merge(m, q, cnt, m2, q2);
    cnt += cnt;
  }
  if ((threadIdx.x & 31) == 0) {                         // (the lanes may differ in the last bit: lane 0's values count)
    const int w = ((threadIdx.x >> 5) - kEpiWarp0) % WPG;
    slot[w] = m;
    slot[WPG + w] = q;
  }
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(WPG * 32) : "memory");
  float mm[WPG], qq[WPG];
#pragma unroll
  for (int w = 0; w < WPG; ++w) { mm[w] = slot[w]; qq[w] = slot[WPG + w]; }
#pragma unroll
  for (int s = 1; s < WPG; s += s) {
#pragma unroll
    for (int w = 0; w < WPG; w += 2 * s) merge(mm[w], qq[w], cnt, mm[w + s], qq[w + s]);
    cnt += cnt;
  }
  mean = mm[0];
  rstd = rsqrtf(qq[0] / cnt + eps);
}

// The same for a row of d channels, of which this thread holds the first `mine` of its float4s (the others are zero).
template <int NT, int WPG>
__device__ __forceinline__ void group_stats_any(const float4 (&v)[NT], int mine, int d, float eps, float* slot, int group, float& mean, float& rstd) {
  auto sum = [&](float x, float* part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) part[((threadIdx.x >> 5) - kEpiWarp0) % WPG] = x;
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(WPG * 32) : "memory");
    float all = part[0];
#pragma unroll
    for (int w = 1; w < WPG; ++w) all += part[w];
    return all;
  };
  float m = 0.f, q = 0.f;
#pragma unroll
  for (int i = 0; i < NT; ++i) m += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  const float inv_d = 1.0f / (float)d;
  mean = sum(m, slot) * inv_d;
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const float a = v[i].x - mean, b = v[i].y - mean, c = v[i].z - mean, e = v[i].w - mean;
    if (i < mine) q += (a * a + b * b) + (c * c + e * e);
  }
  rstd = rsqrtf(sum(q, slot + WPG) * inv_d + eps);
}

// Combined heads and kernels of size k on the row of a group of WPG warps (thread th: channels 4 th .. 4 th + 3 and 128 WPG,
// 256 WPG, ... further), as in mixer_variant_step_kernel: v = x in, x + y out; z = LN1(x); f = plane 0 of the cache.
// hs: the mixer's scalars, edge: see smem_bytes.
template <int NT, int WPG, int MIX, typename ST>
__device__ __forceinline__ void mix_row(const Params& p, float4 (&v)[NT], const float4 (&z)[NT], float4 (&f)[NT], const float4 (&f1)[NT],
                                        const float* bt_p, ST* Sr, const float* hs, float4* edge, int group, int th) {
  if (MIX == kCombined) {
    const int dh = NT * WPG * 128 / p.h;
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const float* q = hs + 6 * ((th * 4 + 128 * WPG * i) / dh);
      const float ar = q[0], ac = q[1], lr = q[2], lc = q[3], wr = q[4], wc = q[5];
      const float4 bt = ld4(bt_p + 128 * WPG * i), sr = f[i], sc = f1[i];
      const float4 u = make_float4(ar * z[i].x, ar * z[i].y, ar * z[i].z, ar * z[i].w);
      const float4 w = make_float4(z[i].x + sc.x, z[i].y + sc.y, z[i].z + sc.z, z[i].w + sc.w);
      v[i] = make_float4(v[i].x + (wr * (u.x + sr.x) + wc * (ac * w.x) + bt.x), v[i].y + (wr * (u.y + sr.y) + wc * (ac * w.y) + bt.y),
                         v[i].z + (wr * (u.z + sr.z) + wc * (ac * w.z) + bt.z), v[i].w + (wr * (u.w + sr.w) + wc * (ac * w.w) + bt.w));
      st4(Sr + 128 * WPG * i, make_float4(lr * (sr.x + u.x), lr * (sr.y + u.y), lr * (sr.z + u.z), lr * (sr.w + u.w)));
      st4(Sr + p.s_plane + 128 * WPG * i, make_float4(lc * w.x, lc * w.y, lc * w.z, lc * w.w));
    }
  } else {
    // v_i = z + P_i ;  y[c] = beta_t[c] + sum_i alpha_i[t] v_i[c + i] ;  P_i <- lam_i v_i. A shifted read reaches at most four
    // lanes ahead: by shuffle inside the warp, the warp's last lanes from what the next 128 channels' first lanes left in
    // `edge` (two buffers, filters in turn: one barrier of the group per filter).
    const int lane = threadIdx.x & 31, wi = th >> 5;
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const float4 bt = ld4(bt_p + 128 * WPG * i);
      v[i] = make_float4(v[i].x + bt.x, v[i].y + bt.y, v[i].z + bt.z, v[i].w + bt.w);
    }
    for (int fi = 0; fi < p.k; ++fi) {
      const float al = hs[2 * fi], lm = hs[2 * fi + 1];
      ST* Pf = Sr + (int64_t)fi * p.s_plane;
      float4 nx[NT];
#pragma unroll
      for (int i = 0; i < NT; ++i) nx[i] = fi + 1 < p.k ? ld4(Pf + p.s_plane + 128 * WPG * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < NT; ++i) {
        const float4 w = make_float4(z[i].x + f[i].x, z[i].y + f[i].y, z[i].z + f[i].z, z[i].w + f[i].w);
        st4(Pf + 128 * WPG * i, make_float4(lm * w.x, lm * w.y, lm * w.z, lm * w.w));
        f[i] = make_float4(al * w.x, al * w.y, al * w.z, al * w.w);
      }
      if (fi > 0) {
        float4* e = edge + (fi & 1) * (NT * WPG * 4);          // [128-channel vector][4 lanes]
        if (lane < 4) {
#pragma unroll
          for (int i = 0; i < NT; ++i) e[(WPG * i + wi) * 4 + lane] = f[i];
        }
        asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(WPG * 32) : "memory");
        auto ahead = [&](int i, int delta) {                // the float4 `delta` lanes ahead, 0 <= delta <= 4
          const int src = lane + delta;
          float4 r = make_float4(__shfl_sync(0xffffffffu, f[i].x, src & 31), __shfl_sync(0xffffffffu, f[i].y, src & 31),
                                 __shfl_sync(0xffffffffu, f[i].z, src & 31), __shfl_sync(0xffffffffu, f[i].w, src & 31));
          if (src >= 32) {
            const int next = WPG * i + wi + 1;
            r = next < WPG * NT ? e[next * 4 + src - 32] : make_float4(0.f, 0.f, 0.f, 0.f);
          }
          return r;
        };
        const int q = fi >> 2, s = fi & 3;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          const float4 A = q == 0 ? f[i] : ahead(i, q);
          float4 r = A;
          if (s != 0) {
            const float4 B = ahead(i, q + 1);
            r = s == 1 ? make_float4(A.y, A.z, A.w, B.x) : s == 2 ? make_float4(A.z, A.w, B.x, B.y) : make_float4(A.w, B.x, B.y, B.z);
          }
          v[i] = make_float4(v[i].x + r.x, v[i].y + r.y, v[i].z + r.z, v[i].w + r.w);
        }
      } else {
#pragma unroll
        for (int i = 0; i < NT; ++i) v[i] = make_float4(v[i].x + f[i].x, v[i].y + f[i].y, v[i].z + f[i].z, v[i].w + f[i].w);
      }
#pragma unroll
      for (int i = 0; i < NT; ++i) f[i] = nx[i];
    }
  }
}

// WPG: warps per row; NT: float4s of a row per thread.
template <int NT, int WPG, typename ST, int MIX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
layers_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmW1,
              const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmHs, const __grid_constant__ CUtensorMap tmP,
              const Params p) {
  pdl_trigger();
  constexpr int kRowThreads = WPG * 32, kStride = kRowThreads * 4;
  const int d = MIX == kMixedAny ? p.d : NT * kStride;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int n = p.n, w_rows = n >> 1, w_bytes = kStep * w_rows * 128;
  uint8_t* sW = smem;
  uint8_t* sA = sW + p.w_slots * w_bytes;
  float* prm = reinterpret_cast<float*>(sA + p.a_slots * kABytes);
  float* b1_s = prm + kVecs * d;
  float* red = b1_s + n;
  uint64_t* fullW = reinterpret_cast<uint64_t*>(red + kMaxGroups * 8);      // used in the leader CTA
  uint64_t* emptyW = fullW + kMaxWSlots;
  uint64_t* fullA = emptyW + kMaxWSlots;                                 // used in the leader CTA
  uint64_t* emptyA = fullA + kMaxASlots;
  uint64_t* tfull = emptyA + kMaxASlots;
  uint64_t* tempty = tfull + 1;                                          // leader: accumulator drained by both CTAs
  uint64_t* ring = tempty + 1;                                           // the epilogue has left the activation ring
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ring + 1);
  float* hs = red + kMaxGroups * 8 + kBarrierBytes / 4;                  // not for mixed heads
  float4* edge = reinterpret_cast<float4*>(hs + kMixScalars);            // MIX == kKernel: d bytes per group

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_ctarank();
  const int pair = blockIdx.x >> 1;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kMaxWSlots; ++i) { tc::mbar_init(&fullW[i], 2); tc::mbar_init(&emptyW[i], 1); }
    for (int i = 0; i < kMaxASlots; ++i) { tc::mbar_init(&fullA[i], 2); tc::mbar_init(&emptyA[i], 1); }
    tc::mbar_init(tfull, 1);
    tc::mbar_init(tempty, 2 * tc::kEpiWarps);
    tc::mbar_init(ring, tc::kEpiWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tc::tmem_alloc(tmem_slot, kTmemCols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  tc::cluster_sync();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // this pair's pieces
  const int up_rb = pair % p.rb, up_col = pair / p.rb;
  const bool up_on = up_col < p.cu;
  const int dn_rb = up_rb, dn_col = up_col % p.cd, dn_slice = up_col / p.cd;
  const bool dn_on = dn_slice < p.ks;
  const int slice_kb = p.slice_tiles * (n / tc::BK);
  const int kb_up = d / tc::BK, kb_dn = min(slice_kb, p.F / tc::BK - dn_slice * slice_kb);      // k-blocks per piece
  const int up_boxes = n / 64, dn_boxes = n / 32;                        // boxes of 128 bytes per row that an output tile consists of
  const int up_slice = up_col / p.slice_tiles;                           // range of K that this pair's column tile of H belongs to
  const int slice_up = min(p.slice_tiles, p.cu - dn_slice * p.slice_tiles);      // column tiles of H that the down piece reads
  uint32_t* cnt_rows = p.cnt;
  uint32_t* cnt_up = p.cnt + kMaxRowBlocks;
  uint32_t* cnt_dn = cnt_up + kMaxRowBlocks * kMaxKSlices;

  if (warp == 2) {
    // ---------------- weight stream (both CTAs): constant data, it waits for nothing but its ring ----------------
    if (tc::elect_one()) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmW1)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmW2)) : "memory");
      int slot = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int l = 0; ok && l < p.L; ++l) {
        for (int ph = 0; ok && ph < 2; ++ph) {
          if (!(ph ? dn_on : up_on)) continue;
          const CUtensorMap* map = ph ? &tmW2 : &tmW1;
          const int kbs = ph ? kb_dn : kb_up, kb0 = ph ? dn_slice * slice_kb : 0;
          const int row = (ph ? dn_col : up_col) * n + (int)rank * w_rows;
          for (int kb = 0; kb < kbs; kb += kStep) {
            if (!tc::mbar_wait(&emptyW[slot], phase ^ 1u, p.status)) { ok = false; break; }
            const uint32_t full = tc::mapa(tc::smem_u32(&fullW[slot]), 0);
            tc::mbar_expect_tx_cluster(full, (uint32_t)w_bytes);
            tma_load_w(sW + slot * w_bytes, map, full, row, kb0 + kb, l);
            if (++slot == p.w_slots) { slot = 0; phase ^= 1u; }
          }
        }
      }
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < (1ll << 21)) { }
      }
    }
  } else if (warp == 0) {
    // ---------------- activations (both CTAs) ----------------
    if (tc::elect_one()) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmH)) : "memory");
      pdl_wait();
      int slot = 0, piece = 0;
      uint32_t phase = 0;
      bool ok = true;
      const int block_rows = min(tc::BM, p.R - up_rb * tc::BM);
      for (int l = 0; ok && l < p.L; ++l) {
        for (int ph = 0; ok && ph < 2; ++ph) {
          if (!(ph ? dn_on : up_on)) continue;
          // rows of the block done / the up tiles of this range of K done
          if (!(ph ? count_wait(cnt_up + dn_rb * kMaxKSlices + dn_slice, (uint32_t)(l + 1) * (uint32_t)(slice_up * up_boxes) * 8u, p.status)
                   : count_wait(cnt_rows + up_rb, (uint32_t)(l + 1) * (uint32_t)block_rows, p.status))) { ok = false; break; }
          if (piece > 0 && !tc::mbar_wait(ring, (uint32_t)(piece & 1) ^ 1u, p.status)) { ok = false; break; }
          ++piece;
          tc::fence_async_global();
          const CUtensorMap* map = ph ? &tmH : &tmA;
          const int kbs = ph ? kb_dn : kb_up, kb0 = ph ? dn_slice * slice_kb : 0;
          const int row = up_rb * tc::BM + (int)rank * tc::kRowsPerCta;
          for (int kb = 0; kb < kbs; kb += kStep) {
            if (!tc::mbar_wait(&emptyA[slot], phase ^ 1u, p.status)) { ok = false; break; }
            const uint32_t full = tc::mapa(tc::smem_u32(&fullA[slot]), 0);
            // (a CTA without rows arrives and loads nothing: its half of the accumulator is not stored)
            tc::mbar_expect_tx_cluster(full, row < p.R ? (uint32_t)(kStep * p.box * 128) : 0u);
            if (row < p.R) tma_load_a(sA + slot * kABytes, map, full, row, kb0 + kb);
            if (++slot == p.a_slots) { slot = 0; phase ^= 1u; }
          }
        }
      }
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < (1ll << 21)) { }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA only) ----------------
    if (rank == 0 && tc::elect_one()) {
      const uint32_t idesc = tc::instr_desc(n);
      int sw = 0, sa = 0, piece = 0;
      uint32_t pw = 0, pa = 0;
      bool ok = true;
      for (int l = 0; ok && l < p.L; ++l) {
        for (int ph = 0; ok && ph < 2; ++ph) {
          if (!(ph ? dn_on : up_on)) continue;
          if (!tc::mbar_wait(tempty, (uint32_t)(piece & 1) ^ 1u, p.status)) { ok = false; break; }
          tc::tc_fence_after();
          const int kbs = ph ? kb_dn : kb_up;
          for (int kb = 0; kb < kbs; kb += kStep) {
            if (!tc::mbar_wait(&fullW[sw], pw, p.status) || !tc::mbar_wait(&fullA[sa], pa, p.status)) { ok = false; break; }
            tc::tc_fence_after();
            const uint64_t da = tc::make_smem_desc(tc::smem_u32(sA + sa * kABytes));
            const uint64_t db = tc::make_smem_desc(tc::smem_u32(sW + sw * w_bytes));
#pragma unroll
            for (int q = 0; q < kStep; ++q) {               // (descriptor addresses count 16 bytes)
#pragma unroll
              for (int k = 0; k < tc::BK / 16; ++k)
                tc::umma_bf16(tmem, da + (uint32_t)(q * p.box * 8) + 2u * k, db + (uint32_t)(q * w_rows * 8) + 2u * k, idesc,
                              (kb | q | k) != 0 ? 1u : 0u);
            }
            tc::umma_commit_pair(&emptyW[sw]);
            tc::umma_commit_pair(&emptyA[sa]);
            if (++sw == p.w_slots) { sw = 0; pw ^= 1u; }
            if (++sa == p.a_slots) { sa = 0; pa ^= 1u; }
          }
          if (ok) tc::umma_commit_pair(tfull);
          ++piece;
        }
      }
    }
  } else {
    // ---------------- rows and epilogues (both CTAs) ----------------
    const int wid = threadIdx.x - kEpiWarp0 * 32;                // 0 .. kWorkers - 1
    const int group = wid / kRowThreads, th = wid % kRowThreads, c0 = th * 4;
    const int quad = warp & 3, cgrp = (warp - kEpiWarp0) >> 2;
    const int cols = n >> 2;                                     // accumulator columns per warp: 16, 32 or 64
    pdl_wait();
    const int t_all = p.ctr != nullptr ? p.ctr[kCtrPos] : p.t;
    float* slot = red + group * (2 * WPG);               // (a second set of sums lies kMaxGroups * 4 floats on)
    int piece = 0;
    bool ok = true;
    for (int l = 0;; ++l) {
      const bool last = l == p.L;         // after the last layer: the final norm
      const sb::LayerW w = sb::layer_w(p, last ? 0 : l);
      // ---- rows: row blockIdx.x + grid * group. Parameters first (constant data), then the wait ----
      workers_sync();                     // the previous layer's parameters have been read
      for (int i = wid; i < (kVecs * d + n) / 4; i += kWorkers) {
        const int k = i / (d / 4), c = i % (d / 4) * 4;
        const float* q = k == 0 ? w.ln1_g : k == 1 ? w.ln1_b : k == 2 ? w.beta + (int64_t)t_all * d : k == 3 ? (last ? p.lnf_g : w.ln2_g)
                         : k == 4 ? (last ? p.lnf_b : w.ln2_b) : k == 5 ? sb::layer_w(p, l > 0 ? l - 1 : 0).b2 : w.b1 + (up_on ? up_col : 0) * n;
        if (MIX != kMixedAny || k < kVecs || !up_on || up_col * n + c < p.F) sb::cp_async16(prm + i * 4, q + c);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const int row = (int)blockIdx.x + (int)gridDim.x * group;
      const bool mine = row < p.R;
      auto on = [&](int i) { return MIX != kMixedAny || c0 + kStride * i < d; };      // float4 i lies inside the row
      const int t = mine && p.pos != nullptr ? min(max(p.pos[row], 0), p.n_ctx - 1) : t_all;
      float a1[NT], a2[NT], lm[NT];                  // (mixed heads)
      float4 s[NT], s1[NT], v[NT];                   // (s1: combined heads)
      ST* Sr = reinterpret_cast<ST*>(static_cast<uint8_t*>(p.S) + (int64_t)l * p.layer_stride) + (int64_t)row * d + c0;
      if (mine) {
        if (!last) {
          if (mixed_heads(MIX)) {         // the multipliers of z before and of the sum after (one of them is 1), and lambda
#pragma unroll
            for (int i = 0; i < NT; ++i) {
              if (!on(i)) continue;
              const int g = (c0 + kStride * i) / (d / p.h);
              const float al = __ldg(w.alpha + (int64_t)g * p.n_ctx + t);
              const bool is_row = g < (p.h >> 1);
              a1[i] = is_row ? al : 1.0f;
              a2[i] = is_row ? 1.0f : al;
              lm[i] = __ldg(w.lam + g);
            }
          }
#pragma unroll
          for (int i = 0; i < NT; ++i)
            if (on(i)) s[i] = ld4(Sr + kStride * i);
          if (p.pos != nullptr) {
#pragma unroll
            for (int i = 0; i < NT; ++i)
              if (on(i)) asm volatile("prefetch.global.L2 [%0];" ::"l"(w.beta + (int64_t)t * d + c0 + kStride * i));
          }
          if (MIX == kCombined) {
#pragma unroll
            for (int i = 0; i < NT; ++i) s1[i] = ld4(Sr + p.s_plane + kStride * i);
          }
        }
        if (l > 0) {                      // (this thread's part of x, from the previous layer: not through L1)
#pragma unroll
          for (int i = 0; i < NT; ++i)
            v[i] = on(i) ? __ldcg(reinterpret_cast<const float4*>(p.x + (int64_t)row * d + c0 + kStride * i)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (l > 0 && th == 0 && ok)               // the down tiles of the row's block
          ok = count_wait(cnt_dn + row / tc::BM, (uint32_t)l * (uint32_t)(p.cd * p.ks * dn_boxes) * 8u, p.status);
      }
      if (!mixed_heads(MIX) && !last) {     // scalar wid of the layer
        const int64_t o = (int64_t)l * p.layer_bytes;
        auto at = [o](const float* q, int64_t i) { return __ldg(reinterpret_cast<const float*>(reinterpret_cast<const uint8_t*>(q) + o) + i); };
        if (MIX == kCombined && wid < 6 * p.h) {
          const int g = wid / 6, q = wid % 6;
          const int64_t ia = (int64_t)g * p.n_ctx + t_all;
          hs[wid] = q == 0 ? __ldg(w.alpha + ia) : q == 1 ? at(p.alpha_col, ia) : q == 2 ? __ldg(w.lam + g) : q == 3 ? at(p.lam_col, g)
                                                                                          : at(p.w_comb, 2 * g + q - 4);
        }
        if (MIX == kKernel && wid < 2 * p.k) hs[wid] = wid & 1 ? __ldg(w.lam + (wid >> 1)) : __ldg(w.alpha + (int64_t)(wid >> 1) * p.n_ctx + t_all);
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      workers_sync();
      if (mine) {
        if (l == 0) {
          int tk = p.tok_in[row];
          if (tk < 0 || tk >= p.V) {
            if (th == 0) raise_status(p.status, kStatusTokenRange);
            tk = tk < 0 ? 0 : p.V - 1;
          }
#pragma unroll
          for (int i = 0; i < NT; ++i) v[i] = on(i) ? ldg4(p.E + (int64_t)tk * d + c0 + kStride * i) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {                          // x + b2 + plane 0 + plane 1 + ... (other CTAs wrote the planes: not through L1)
#pragma unroll
          for (int i = 0; i < NT; ++i) {
            if (!on(i)) continue;
            const float4 bb = ld4(prm + 5 * d + c0 + kStride * i);
            v[i] = make_float4(v[i].x + bb.x, v[i].y + bb.y, v[i].z + bb.z, v[i].w + bb.w);
          }
          const float* part = p.part + (int64_t)row * d + c0;
          auto add = [&](auto planes) {   // all planes' loads in flight, of four at most
            constexpr int K = decltype(planes)::value;
            float4 e[K][NT];
#pragma unroll
            for (int k = 0; k < K; ++k)
#pragma unroll
              for (int i = 0; i < NT; ++i)
                e[k][i] = on(i) ? __ldcg(reinterpret_cast<const float4*>(part + k * p.plane + kStride * i)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k)
#pragma unroll
              for (int i = 0; i < NT; ++i) v[i] = make_float4(v[i].x + e[k][i].x, v[i].y + e[k][i].y, v[i].z + e[k][i].z, v[i].w + e[k][i].w);
          };
          if (MIX == kMixedAny && p.ks == 8) {
            add(std::integral_constant<int, 4>());
            part += 4 * p.plane;
          }
          if (p.ks >= 4) add(std::integral_constant<int, 4>());
          else if (p.ks == 2) add(std::integral_constant<int, 2>());
          else add(std::integral_constant<int, 1>());
        }
        float mean, rstd;
        auto stats = [&](float* sums) {
          if constexpr (MIX == kMixedAny) group_stats_any<NT, WPG>(v, c0 < d ? (d - c0 + kStride - 1) / kStride : 0, d, p.eps, sums, group, mean, rstd);
          else group_stats<NT, WPG>(v, p.eps, sums, group, mean, rstd);
        };
        if (!last) {
          const float* bt_p = p.pos != nullptr ? w.beta + (int64_t)t * d + c0 : prm + 2 * d + c0;
          stats(slot);
          const float nmr = -mean * rstd;
          if constexpr (!mixed_heads(MIX)) {
            float4 z[NT];
#pragma unroll
            for (int i = 0; i < NT; ++i) {
              const float4 g = ld4(prm + c0 + kStride * i), bb = ld4(prm + d + c0 + kStride * i);
              z[i] = make_float4(fmaf(fmaf(v[i].x, rstd, nmr), g.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), g.y, bb.y),
                                 fmaf(fmaf(v[i].z, rstd, nmr), g.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), g.w, bb.w));
            }
            mix_row<NT, WPG, MIX>(p, v, z, s, s1, bt_p, Sr, hs, edge + group * (d / 16), group, th);
#pragma unroll
            for (int i = 0; i < NT; ++i) st4(p.x + (int64_t)row * d + c0 + kStride * i, v[i]);
          }
#pragma unroll
          for (int i = 0; mixed_heads(MIX) && i < NT; ++i) {
            if (!on(i)) continue;
            const float4 g = ld4(prm + c0 + kStride * i), bb = ld4(prm + d + c0 + kStride * i), bt = ld4(bt_p + kStride * i);
            const float4 z = make_float4(fmaf(fmaf(v[i].x, rstd, nmr), g.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), g.y, bb.y),
                                         fmaf(fmaf(v[i].z, rstd, nmr), g.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), g.w, bb.w));
            // row-repeat head, Eq. 2: y = (a z + S) + b ; S' = l (S + a z).  column-repeat head, Eq. 3: y = a (z + S) + b ; S' = l (z + S)
            const float4 u = make_float4(fmaf(a1[i], z.x, s[i].x), fmaf(a1[i], z.y, s[i].y), fmaf(a1[i], z.z, s[i].z), fmaf(a1[i], z.w, s[i].w));
            st4(Sr + kStride * i, make_float4(lm[i] * u.x, lm[i] * u.y, lm[i] * u.z, lm[i] * u.w));
            v[i] = make_float4(v[i].x + fmaf(a2[i], u.x, bt.x), v[i].y + fmaf(a2[i], u.y, bt.y), v[i].z + fmaf(a2[i], u.z, bt.z),
                               v[i].w + fmaf(a2[i], u.w, bt.w));
            st4(p.x + (int64_t)row * d + c0 + kStride * i, v[i]);
          }
        }
        stats(slot + kMaxGroups * 4);
        const float nmr2 = -mean * rstd;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          if (!on(i)) continue;
          const float4 g = ld4(prm + 3 * d + c0 + kStride * i), bb = ld4(prm + 4 * d + c0 + kStride * i);
          st4(p.a + (int64_t)row * d + c0 + kStride * i,
              make_float4(fmaf(fmaf(v[i].x, rstd, nmr2), g.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr2), g.y, bb.y),
                          fmaf(fmaf(v[i].z, rstd, nmr2), g.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr2), g.w, bb.w)));
        }
        tc::fence_async_global();         // read by bulk tensor copies of other CTAs
        asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kRowThreads) : "memory");
        if (th == 0) red_release_add(cnt_rows + row / tc::BM, 1u);
      }
      if (last) break;

      // ---- epilogues ----
      for (int ph = 0; ph < 2; ++ph) {
        if (!(ph ? dn_on : up_on)) continue;
        if (ok && !tc::mbar_wait(tfull, (uint32_t)(piece & 1), p.status)) ok = false;
        ++piece;
        tc::tc_fence_after();
        const int boxes = ph ? dn_boxes : up_boxes;
        const int row0 = up_rb * tc::BM + (int)rank * tc::kRowsPerCta + quad * 32;
        const int col0 = (ph ? dn_col : up_col) * n;
        const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(cgrp * cols);
        // The tile goes out as bulk tensor stores (every thread storing its own row took 1.1 to 6.2 us per tile): the
        // four warps of a row quarter fill boxes of 32 rows x 128 bytes in the activation ring, which is idle between
        // the last MMA of this piece and the loads of the next, in the 128-byte swizzle of the output's tensor map.
        uint8_t* stage = sA + quad * boxes * tc::kOutBoxBytes + lane * 128;
        for (int c = 0; c < cols; c += 16) {
          uint32_t acc[16];
          tc::tmem_ld16(taddr + c, acc);
          tc::tmem_ld_wait();
          const int byte = (cgrp * cols + c) * (ph ? 4 : 2);               // of the tile's row
          uint8_t* box = stage + (byte >> 7) * tc::kOutBoxBytes;
          const int chunk = (byte & 127) >> 4;
          if (ph == 0) {
            uint32_t o[8];
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
              const float4 b = ld4(b1_s + cgrp * cols + c + j);
              const __nv_bfloat162 lo = __floats2bfloat162_rn(tc::gelu_fast(__uint_as_float(acc[j]) + b.x), tc::gelu_fast(__uint_as_float(acc[j + 1]) + b.y));
              const __nv_bfloat162 hi = __floats2bfloat162_rn(tc::gelu_fast(__uint_as_float(acc[j + 2]) + b.z), tc::gelu_fast(__uint_as_float(acc[j + 3]) + b.w));
              o[j / 2] = *reinterpret_cast<const uint32_t*>(&lo);
              o[j / 2 + 1] = *reinterpret_cast<const uint32_t*>(&hi);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
              *reinterpret_cast<uint4*>(box + (((chunk + j) ^ (lane & 7)) << 4)) = make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              *reinterpret_cast<uint4*>(box + (((chunk + j) ^ (lane & 7)) << 4)) = make_uint4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
          }
        }
        tc::tc_fence_before();
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive_cluster(tc::mapa(tc::smem_u32(tempty), 0));
        asm volatile("bar.sync %0, 128;" ::"r"(quad + 10) : "memory");      // the four warps of this row quarter
        if (cgrp < boxes && tc::elect_one()) {
          const uint8_t* src = sA + (quad * boxes + cgrp) * tc::kOutBoxBytes;
          if (row0 < p.R && (MIX != kMixedAny || (ph ? col0 + cgrp * 32 < d : col0 + cgrp * 64 < p.F))) {
            if (ph == 0) tc::tma_store_2d(&tmHs, src, col0 + cgrp * 64, row0);
            else if (MIX == kMixedAny) tma_store_3d(&tmP, src, col0 + cgrp * 32, row0, dn_slice);
            else tc::tma_store_2d(&tmP, src, col0 + cgrp * 32, dn_slice * p.plane_rows + row0);
            tc::bulk_commit();
            tc::bulk_wait_all();
          }
          tc::fence_async_global();
          red_release_add(ph ? cnt_dn + dn_rb : cnt_up + up_rb * kMaxKSlices + up_slice, 1u);
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(ring);
      }
    }
  }

  // Both CTAs stay until the pair is done (see gemm_tc_kernel)
  tc::tc_fence_before();
  __syncwarp();
  tc::cluster_sync();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace mid
}  // namespace srm
