// Token mixing over prompts in chunks of positions (Method/Architecture, Eq. 1 and Eq. 3; the scan the paper names as
// an open option, in parallel over the positions of a prompt).
//
// The sum term of Eq. 2 / Eq. 3 is linear in its start value: over a chunk of T positions it goes from S to
// lambda^T S + E, where E is what the chunk leaves when it starts from zero. One CTA owns one chunk of one prompt:
//   - its T rows of the residual stream come into shared memory with one bulk copy;
//   - LN1 statistics, one warp per row;
//   - one thread per four channels runs the recurrence over the chunk from zero and publishes E (a d-vector in
//     scratch memory, then a flag);
//   - the thread reads the E of all earlier chunks of the prompt, folds them in position order (a fixed order: the
//     result does not depend on timing, nor on how many prompts share the launch) into the chunk's true start value,
//     and runs the recurrence again, now forming y and x + y;
//   - LN2, one warp per row, writes x and the activation.
// Each row is read once and written once. A chunk waits only for chunks of its own prompt with a smaller block index,
// and a block publishes before it waits, so the waits end whatever the number of resident blocks; they are bounded
// all the same (status bit).
//
// What bounds it: with few prompts the chain load -> statistics -> E -> flags -> rows of one chunk (about 11 us per launch
// for one prompt of 777 positions at d = 1024, where one CTA walking the prompt took 2061 us; 33.4 -> 0.74 ms for the
// whole prefill of the mid model; 16.4 us while the second pass waited for beta and LN2 for its parameters), with many the
// latency of its loads (131072 rows: 383 us, 3.5 TB/s of the 10 bytes per element it moves). T = 16: the rows of a chunk
// (64 KB at d = 1024) and LN2's parameters leave room for three CTAs per SM.
// Needs d = 128 NV (a thread per four channels, a warp per 128).
#pragma once

#include "common.cuh"
#include "gemm_tc.cuh"        // mbarrier helpers
#include "mixer.cuh"          // row_stats_full
#include "mixer_stream.cuh"   // bulk_g2s
#include "prefill.cuh"        // PrefillParams

namespace srm {

constexpr int kChunkRows = 16;
constexpr long long kChunkWaitLimitCycles = 1ll << 30;

// Scratch of a launch: E of every chunk but a prompt's last [Bp * (chunks - 1), d] fp32 (times the sum terms per
// channel of the mixer) and one flag per chunk. A flag counts the launches that
// have published into it (epoch 1, 2, ... of a zeroed array), so the array is cleared once for all layers of a pass.
struct ChunkScratch {
  float* E = nullptr;
  uint32_t* flags = nullptr;
  uint32_t epoch = 0;
};

inline int64_t prefill_chunks(int n) { return (n + kChunkRows - 1) / kChunkRows; }
inline size_t prefill_chunk_smem(int d) { return (size_t)(kChunkRows + 2) * d * 4 + 2 * kChunkRows * 4 + 16; }

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Rows of a parameter on their way into L2 (bytes: a multiple of 16).
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void st_release_u32(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <int NV, typename WT, typename ST>
__global__ void __launch_bounds__(NV * 32, NV <= 8 ? 3 : NV <= 12 ? 2 : 1)
prefill_chunk_kernel(const PrefillParams p, const ChunkScratch cs, int chunks) {
  pdl_trigger();
  constexpr int T = kChunkRows, d = NV * 128, kThreads = NV * 32;
  extern __shared__ __align__(128) uint8_t sm[];
  float* xs = reinterpret_cast<float*>(sm);                          // [T][d]
  float* ln2 = xs + T * d;                                           // ln2_g | ln2_b (every row of a warp waited for them otherwise)
  float* rs = ln2 + 2 * d;                                           // rstd of the rows
  float* nm = rs + T;                                                // -mean * rstd
  uint64_t* bar = reinterpret_cast<uint64_t*>(nm + T);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t b = blockIdx.x / (unsigned)chunks;
  const int ch = (int)(blockIdx.x - (unsigned)b * (unsigned)chunks);
  const int j0 = ch * T;
  const int64_t tok0 = b * p.n + j0;
  int64_t row0 = tok0;
  const int c = tid * 4;
  const int g = c / (d / p.h);
  const bool is_row = g < (p.h >> 1);
  // parameters: constant data, fetched ahead of the dependency wait
  const float4 g1 = ldg4(p.ln1_g + c), b1 = ldg4(p.ln1_b + c);
  const float lam = __ldg(p.lam + g);
  st4(ln2 + c, ldg4(p.ln2_g + c));
  st4(ln2 + d + c, ldg4(p.ln2_b + c));
  if (tid == 0) {
    bulk_prefetch_l2(p.beta + (int64_t)j0 * d, (uint32_t)(min(T, p.n - j0) * d * 4));
    tc::mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
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
  const int rows = max(0, min(T, n - j0));             // rows of the prompt in this chunk
  if (p.row_start != nullptr) row0 = (int64_t)p.row_start[b] + j0;
  const int rows_all = p.row_start != nullptr ? rows : min(T, p.n - j0);      // ... and of the padded prompt
  // positions beyond the prompt: defined values for the GEMMs that follow (their results are not used)
  for (int i = rows * d + c; i < rows_all * d; i += kThreads * 4) {
    st4(p.x + row0 * d + i, make_float4(0.f, 0.f, 0.f, 0.f));
    st4(reinterpret_cast<WT*>(p.a) + row0 * d + i, make_float4(0.f, 0.f, 0.f, 0.f));
  }
  if (rows == 0) return;

  // ---- the chunk's rows (embedding rows for the first layer) and their LN1 statistics ----
  if (p.tok == nullptr) {
    if (tid == 0) {
      const uint32_t bytes = (uint32_t)(rows * d * 4);
      tc::mbar_expect_tx(bar, bytes);
      bulk_g2s(xs, p.x + row0 * d, bytes, bar);
    }
    tc::mbar_wait(bar, 0u, p.status);
  }
  constexpr float inv_d = 1.0f / (float)d;
  for (int r = warp; r < rows; r += NV) {
    float4 v[NV];
    if (p.tok != nullptr) {
      int tk = p.tok[tok0 + r];
      if (tk < 0 || tk >= p.vocab) {
        if (lane == 0) raise_status(p.status, kStatusTokenRange);
        tk = tk < 0 ? 0 : p.vocab - 1;
      }
      const WT* e = reinterpret_cast<const WT*>(p.E) + (int64_t)tk * d + lane * 4;
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ldg4(e + i * 128);
#pragma unroll
      for (int i = 0; i < NV; ++i) st4(xs + r * d + lane * 4 + i * 128, v[i]);
    } else {
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ld4(xs + r * d + lane * 4 + i * 128);
    }
    float mean, rstd;
    row_stats_full<NV>(v, inv_d, p.eps, mean, rstd);
    if (lane == 0) { rs[r] = rstd; nm[r] = -mean * rstd; }
  }
  __syncthreads();

  const float* alpha = p.alpha + (int64_t)g * p.n_ctx + j0;
  auto z_of = [&](const float4& v, int j) {
    const float r = rs[j], m = nm[j];
    return make_float4(fmaf(fmaf(v.x, r, m), g1.x, b1.x), fmaf(fmaf(v.y, r, m), g1.y, b1.y),
                       fmaf(fmaf(v.z, r, m), g1.z, b1.z), fmaf(fmaf(v.w, r, m), g1.w, b1.w));
  };
  float4 S = make_float4(0.f, 0.f, 0.f, 0.f);
  if (j0 + T < n) {
    // ---- what this (whole) chunk leaves when it starts from zero, for the chunks after it ----
#pragma unroll 4
    for (int j = 0; j < T; ++j) {
      const float4 z = z_of(ld4(xs + j * d + c), j);
      const float u = is_row ? __ldg(alpha + j) : 1.0f;
      S = make_float4(lam * fmaf(u, z.x, S.x), lam * fmaf(u, z.y, S.y), lam * fmaf(u, z.z, S.z), lam * fmaf(u, z.w, S.w));
    }
    __stcg(reinterpret_cast<float4*>(cs.E + (b * (chunks - 1) + ch) * d + c), S);
    __syncthreads();
    if (tid == 0) st_release_u32(cs.flags + b * chunks + ch, cs.epoch);
  }
  // beta and alpha of the second pass over the chunk, four positions ahead
  const float* beta = p.beta + (int64_t)j0 * d + c;
  float4 bt[4];
  float al[4];
  auto fetch = [&](int j0b) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (j0b + k < rows) {
        bt[k] = ldg4(beta + (int64_t)(j0b + k) * d);
        al[k] = __ldg(alpha + j0b + k);
      }
    }
  };
  fetch(0);
  S = make_float4(0.f, 0.f, 0.f, 0.f);
  if (ch > 0) {
    // ---- the start value: S <- lambda^T S + E over the earlier chunks, in order ----
    for (int i = tid; i < ch; i += kThreads) {
      const uint32_t* f = cs.flags + b * chunks + i;
      const long long t0 = clock64();
      while (ld_acquire_u32(f) != cs.epoch) {
        if (clock64() - t0 > kChunkWaitLimitCycles) { raise_status(p.status, kStatusWaitTimeout); break; }
      }
    }
    __syncthreads();
    float lT = lam;                                    // lambda^T by squaring
#pragma unroll
    for (int k = 1; k < T; k <<= 1) lT *= lT;
    const float* E = cs.E + b * (chunks - 1) * d + c;
#pragma unroll 8
    for (int i = 0; i < ch; ++i) {
      const float4 e = __ldcg(reinterpret_cast<const float4*>(E + (int64_t)i * d));
      S = make_float4(fmaf(lT, S.x, e.x), fmaf(lT, S.y, e.y), fmaf(lT, S.z, e.z), fmaf(lT, S.w, e.w));
    }
  }
  // ---- y_j and the residual, in place ----
  for (int jb = 0; jb < rows; jb += 4) {
    float4 bc[4];
    float ac[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) { bc[k] = bt[k]; ac[k] = al[k]; }
    fetch(jb + 4);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = jb + k;
      if (j >= rows) break;
      const float4 v = ld4(xs + j * d + c), z = z_of(v, j), b = bc[k];
      const float a = ac[k];
      float4 y;
      if (is_row) {               // row-repeat head, Eq. 2
        const float4 u = make_float4(a * z.x, a * z.y, a * z.z, a * z.w);
        y = make_float4(u.x + b.x + S.x, u.y + b.y + S.y, u.z + b.z + S.z, u.w + b.w + S.w);
        S = make_float4(lam * (S.x + u.x), lam * (S.y + u.y), lam * (S.z + u.z), lam * (S.w + u.w));
      } else {                    // column-repeat head, Eq. 3
        const float4 w = make_float4(z.x + S.x, z.y + S.y, z.z + S.z, z.w + S.w);
        y = make_float4(a * w.x + b.x, a * w.y + b.y, a * w.z + b.z, a * w.w + b.w);
        S = make_float4(lam * w.x, lam * w.y, lam * w.z, lam * w.w);
      }
      st4(xs + j * d + c, make_float4(v.x + y.x, v.y + y.y, v.z + y.z, v.w + y.w));
    }
  }
  if (j0 + rows == n) st4(reinterpret_cast<ST*>(p.S) + b * d + c, S);      // the cache the recurrent form continues from
  __syncthreads();

  // ---- LN2 and write-back ----
  for (int r = warp; r < rows; r += NV) {
    float4 v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = ld4(xs + r * d + lane * 4 + i * 128);
    float mean, rstd;
    row_stats_full<NV>(v, inv_d, p.eps, mean, rstd);
    const float nmr = -mean * rstd;
    float* xo = p.x + (row0 + r) * d + lane * 4;
    WT* ao = reinterpret_cast<WT*>(p.a) + (row0 + r) * d + lane * 4;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      st4(xo + i * 128, v[i]);
      const float4 gg = ld4(ln2 + lane * 4 + i * 128), bb = ld4(ln2 + d + lane * 4 + i * 128);
      st4(ao + i * 128, make_float4(fmaf(fmaf(v[i].x, rstd, nmr), gg.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), gg.y, bb.y),
                                    fmaf(fmaf(v[i].z, rstd, nmr), gg.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), gg.w, bb.w)));
    }
  }
}

}  // namespace srm
