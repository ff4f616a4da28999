// Token mixing over many prompts (Method/Architecture, Eq. 1 and Eq. 3, applied through their recurrence): one CTA owns a
// prompt and walks it in chunks of eight positions, the cache in registers.
//
// Per chunk: the rows of the residual stream are in shared memory (a bulk copy issued while the previous chunk was worked
// on); LN1 statistics, one warp per row; one thread per four channels runs the recurrence over the chunk, adding y to the
// rows in place; LN2, one warp per row, writes x and the activation. Three block barriers per eight positions.
//
// What bounds it: the latency of its three phases; 524288 rows of 1024 channels take 1.43 ms, 3.7 TB/s of the 10 bytes per
// element it moves (LN2's parameters fetched through L1 instead of kept in shared memory: 1.60 ms). One warp per prompt (the design before) walks a chain of 14000 cycles
// per position, and with 14 prompts per SM that was the limit: 1.83 ms.
// T = 8, two slots: 72 KB per CTA at d = 1024, three CTAs per SM, 24 rows in work and 24 in flight. Eight positions of beta per
// thread do not quite fit beside the rest at 80 registers: 52 to 56 bytes are spilled at d = 1024, 120 at d = 1536 (fp32
// activations 156 and 220).
// Needs d = 128 NV (a thread per four channels, a warp per 128). The waits are bounded (status bit).
#pragma once

#include "common.cuh"
#include "gemm_tc.cuh"        // mbarrier helpers, elect_one
#include "mixer.cuh"          // row_stats_full
#include "mixer_stream.cuh"   // bulk_g2s
#include "prefill.cuh"        // PrefillParams

namespace srm {

constexpr int kWalkRows = 8, kWalkSlots = 2;
inline size_t prefill_walk_smem(int d) { return (size_t)(kWalkSlots * kWalkRows + 2) * d * 4 + 2 * kWalkRows * 4 + kWalkSlots * 8; }

template <int NV, typename WT, typename ST>
__global__ void __launch_bounds__(NV * 32, NV <= 4 ? 6 : NV <= 8 ? 3 : NV <= 12 ? 2 : 1) prefill_walk_kernel(const PrefillParams p) {
  pdl_trigger();
  constexpr int T = kWalkRows, d = NV * 128, kThreads = NV * 32;
  extern __shared__ __align__(128) uint8_t sm[];
  float* xs = reinterpret_cast<float*>(sm);                          // [slots][T][d]
  float* ln2 = xs + kWalkSlots * T * d;                              // ln2_g | ln2_b (from L1, which is small here, every row waited for them)
  float* rs = ln2 + 2 * d;                                           // rstd of the rows
  float* nm = rs + T;                                                // -mean * rstd
  uint64_t* bar = reinterpret_cast<uint64_t*>(nm + T);

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int64_t b = blockIdx.x;
  const int c = tid * 4;
  const int g = c / (d / p.h);
  const bool is_row = g < (p.h >> 1);
  const float4 g1 = ldg4(p.ln1_g + c), b1 = ldg4(p.ln1_b + c);       // constant data, fetched ahead of the dependency wait
  const float lam = __ldg(p.lam + g);
  st4(ln2 + c, ldg4(p.ln2_g + c));
  st4(ln2 + d + c, ldg4(p.ln2_b + c));
  if (tid < kWalkSlots) tc::mbar_init(bar + tid, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  pdl_wait();

  int n = p.n;                                         // positions of this prompt
  if (p.len != nullptr) {
    n = p.len[b];
    if (n < 1 || n > p.n) {
      if (tid == 0) raise_status(p.status, kStatusTokenRange);
      n = n < 1 ? 1 : p.n;
    }
  }
  const int64_t row0 = p.row_start != nullptr ? (int64_t)p.row_start[b] : b * p.n;
  const int chunks = (n + T - 1) / T;
  auto issue = [&](int ch) {                           // warp 0: the rows of chunk ch into slot ch % 2
    if (p.tok == nullptr && ch < chunks && tc::elect_one()) {
      const int rows = min(T, n - ch * T), s = ch % kWalkSlots;
      tc::mbar_expect_tx(bar + s, (uint32_t)(rows * d * 4));
      bulk_g2s(xs + s * T * d, p.x + (row0 + ch * T) * d, (uint32_t)(rows * d * 4), bar + s);
    }
  };
  if (warp == 0) { issue(0); issue(1); }

  constexpr float inv_d = 1.0f / (float)d;
  const float* alpha = p.alpha + (int64_t)g * p.n_ctx;
  float4 S = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int ch = 0; ch < chunks; ++ch) {
    const int s = ch % kWalkSlots, j0 = ch * T, rows = min(T, n - j0);
    float* xc = xs + s * T * d;
    // what the recurrence asks of the parameters: from L2, while the statistics are taken
    float4 bt[T];
    float al[T];
#pragma unroll
    for (int j = 0; j < T; ++j) {
      bt[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      al[j] = 0.f;
      if (j < rows) {
        bt[j] = ldg4(p.beta + (int64_t)(j0 + j) * d + c);
        al[j] = __ldg(alpha + j0 + j);
      }
    }
    if (p.tok == nullptr) tc::mbar_wait(bar + s, (uint32_t)(ch / kWalkSlots) & 1u, p.status);
    // ---- LN1 statistics ----
    for (int r = warp; r < rows; r += NV) {
      float4 v[NV];
      if (p.tok != nullptr) {
        int tk = p.tok[b * p.n + j0 + r];
        if (tk < 0 || tk >= p.vocab) {
          if (lane == 0) raise_status(p.status, kStatusTokenRange);
          tk = tk < 0 ? 0 : p.vocab - 1;
        }
        const WT* e = reinterpret_cast<const WT*>(p.E) + (int64_t)tk * d + lane * 4;
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = ldg4(e + i * 128);
#pragma unroll
        for (int i = 0; i < NV; ++i) st4(xc + r * d + lane * 4 + i * 128, v[i]);
      } else {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = ld4(xc + r * d + lane * 4 + i * 128);
      }
      float mean, rstd;
      row_stats_full<NV>(v, inv_d, p.eps, mean, rstd);
      if (lane == 0) { rs[r] = rstd; nm[r] = -mean * rstd; }
    }
    __syncthreads();
    // ---- y_j and the residual, in place ----
#pragma unroll
    for (int j = 0; j < T; ++j) {
      if (j < rows) {
        const float4 v = ld4(xc + j * d + c);
        const float r = rs[j], m = nm[j];
        const float4 z = make_float4(fmaf(fmaf(v.x, r, m), g1.x, b1.x), fmaf(fmaf(v.y, r, m), g1.y, b1.y),
                                     fmaf(fmaf(v.z, r, m), g1.z, b1.z), fmaf(fmaf(v.w, r, m), g1.w, b1.w));
        // row-repeat head, Eq. 2: y = (a z + S) + b ; S' = l (S + a z).  column-repeat head, Eq. 3: y = a (z + S) + b ; S' = l (z + S)
        const float a1 = is_row ? al[j] : 1.0f, a2 = is_row ? 1.0f : al[j];
        const float4 u = make_float4(fmaf(a1, z.x, S.x), fmaf(a1, z.y, S.y), fmaf(a1, z.z, S.z), fmaf(a1, z.w, S.w));
        S = make_float4(lam * u.x, lam * u.y, lam * u.z, lam * u.w);
        st4(xc + j * d + c, make_float4(v.x + fmaf(a2, u.x, bt[j].x), v.y + fmaf(a2, u.y, bt[j].y), v.z + fmaf(a2, u.z, bt[j].z),
                                        v.w + fmaf(a2, u.w, bt[j].w)));
      }
    }
    __syncthreads();
    // ---- LN2 and write-back ----
    for (int r = warp; r < rows; r += NV) {
      float4 v[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ld4(xc + r * d + lane * 4 + i * 128);
      float mean, rstd;
      row_stats_full<NV>(v, inv_d, p.eps, mean, rstd);
      const float nmr = -mean * rstd;
      float* xo = p.x + (row0 + j0 + r) * d + lane * 4;
      WT* ao = reinterpret_cast<WT*>(p.a) + (row0 + j0 + r) * d + lane * 4;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        st4(xo + i * 128, v[i]);
        const float4 gg = ld4(ln2 + lane * 4 + i * 128), bb = ld4(ln2 + d + lane * 4 + i * 128);
        st4(ao + i * 128, make_float4(fmaf(fmaf(v[i].x, rstd, nmr), gg.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), gg.y, bb.y),
                                      fmaf(fmaf(v[i].z, rstd, nmr), gg.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), gg.w, bb.w)));
      }
    }
    tc::fence_async_smem();               // the slot has been read and written by this thread before the next copy into it
    __syncthreads();
    if (warp == 0) issue(ch + kWalkSlots);
  }
  st4(reinterpret_cast<ST*>(p.S) + b * d + c, S);      // the cache the recurrent form continues from
  if (p.row_start != nullptr) return;
  // positions beyond the prompt: defined values for the GEMMs that follow (their results are not used)
  for (int64_t i = (int64_t)n * d + c; i < (int64_t)p.n * d; i += kThreads * 4) {
    st4(p.x + row0 * d + i, make_float4(0.f, 0.f, 0.f, 0.f));
    st4(reinterpret_cast<WT*>(p.a) + row0 * d + i, make_float4(0.f, 0.f, 0.f, 0.f));
  }
}

}  // namespace srm
