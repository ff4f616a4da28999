// Token mixing over prompts in chunks of positions for the two further mixers (linearly combined heads; kernels of
// size k, Eq. 11). Same scheme as prefill_chunk_kernel (one CTA per chunk of 16 positions of a prompt; every sum term
// is linear in its start value, so a chunk publishes what it leaves when started from zero, folds the earlier chunks'
// vectors in position order and then runs its positions), with C sum terms per channel: C = 2, or the k filters.
//
// Kernels of size k: output channel c takes channel c + i of filter i. The thread that owns output channels c .. c + 3
// keeps filter i's sum term for channels c + i .. c + i + 3 (modulo d: the wrapped ones feed no output, but are part of
// the cache), so nothing is exchanged between threads; it reads z at c .. c + 3 + k - 1 from shared memory, which
// therefore holds z = LN1(x), and takes x for the residual from global memory (L2: the same CTA has just read it).
// KM: compiled bound of k (filters k .. KM - 1 have zero weights); 0: combined heads.
//
// What bounds it: the latency of a chunk's chain of phases. mid, k = 4, 96 prompts of 120 positions: 57 us per layer
// (62 while beta and the norms' parameters were fetched where they are used); with one launch per position 120 launches of 8
// to 9 us (prefill and four tokens: 22.3 -> 6.4 ms).
#pragma once

#include "mixer_model_variants.cuh"   // VariantParams
#include "mixer_variants.cuh"         // cp_async16
#include "prefill_chunk.cuh"

namespace srm {

template <int NV, int KM>
inline size_t variant_chunk_smem() { return prefill_chunk_smem(NV * 128) + (size_t)KM * kChunkRows * 4; }

// Parameters as in VariantParams: row b * n + j of x and a, S plane 0 of the pass's prompts, planes p.plane apart.
template <int NV, typename WT, typename ST, int KM>
__global__ void __launch_bounds__(NV * 32, NV <= 4 ? 4 : KM <= 8 ? 3 : 2)
variant_chunk_kernel(const VariantParams p, const ChunkScratch cs, int n, int chunks) {
  pdl_trigger();
  constexpr int T = kChunkRows, d = NV * 128, kThreads = NV * 32;
  constexpr int C = KM > 0 ? KM : 2;                                 // sum terms per channel
  extern __shared__ __align__(128) uint8_t sm[];
  float* xs = reinterpret_cast<float*>(sm);                          // [T][d]: x, from the statistics on z (KM > 0)
  float* ln = xs + T * d;                                            // gains | shifts of LN1 (KM > 0), then of LN2
  float* rs = ln + 2 * d;                                            // rstd of the rows
  float* nm = rs + T;                                                // -mean * rstd
  float* al_s = nm + T + 4;                                          // KM > 0: alpha_i at the chunk's positions [KM][T]
  uint64_t* bar = reinterpret_cast<uint64_t*>(nm + T);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t b = blockIdx.x / (unsigned)chunks;
  const int ch = (int)(blockIdx.x - (unsigned)b * (unsigned)chunks);
  const int j0 = ch * T, rows = min(T, n - j0), planes = KM > 0 ? p.k : 2;
  const int64_t row0 = b * n + j0;
  const int c = tid * 4;
  // parameters: constant data, fetched ahead of the dependency wait
  float4 g1 = make_float4(0.f, 0.f, 0.f, 0.f), b1 = g1;
  float lam[C], w_row = 0.f, w_col = 0.f;
  const float *alpha = p.alpha, *alpha_col = nullptr;
  if (KM == 0) {
    const int g = c / (d / p.h);
    g1 = ldg4(p.ln1_g + c); b1 = ldg4(p.ln1_b + c);
    lam[0] = __ldg(p.lam + g); lam[1] = __ldg(p.lam_col + g);
    w_row = __ldg(p.w_comb + 2 * g); w_col = __ldg(p.w_comb + 2 * g + 1);
    alpha = p.alpha + (int64_t)g * p.n_ctx + j0;
    alpha_col = p.alpha_col + (int64_t)g * p.n_ctx + j0;
  } else {
    for (int i = tid; i < KM * T; i += kThreads) {
      const int f = i / T, j = i % T;
      al_s[i] = f < p.k && j < rows ? __ldg(p.alpha + (int64_t)f * p.n_ctx + j0 + j) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < C; ++i) lam[i] = i < p.k ? __ldg(p.lam + i) : 0.f;
    st4(ln + c, ldg4(p.ln1_g + c));
    st4(ln + d + c, ldg4(p.ln1_b + c));
  }
  if (tid == 0) {
    bulk_prefetch_l2(p.beta + (int64_t)j0 * d, (uint32_t)(rows * d * 4));
    tc::mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();

  // ---- the chunk's rows (embedding rows for the first layer), LN1 statistics, and z for kernels of size k ----
  auto token = [&](int r) {
    const int tk = p.tok[row0 + r];
    if (tk < 0 || tk >= p.vocab) {
      raise_status(p.status, kStatusTokenRange);
      return tk < 0 ? 0 : p.vocab - 1;
    }
    return tk;
  };
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
      const WT* e = reinterpret_cast<const WT*>(p.E) + (int64_t)token(r) * d + lane * 4;
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ldg4(e + i * 128);
    } else {
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ld4(xs + r * d + lane * 4 + i * 128);
    }
    float mean, rstd;
    row_stats_full<NV>(v, inv_d, p.eps, mean, rstd);
    const float nmr = -mean * rstd;
    if (KM > 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float4 gg = ld4(ln + lane * 4 + i * 128), bb = ld4(ln + d + lane * 4 + i * 128);
        st4(xs + r * d + lane * 4 + i * 128,
            make_float4(fmaf(fmaf(v[i].x, rstd, nmr), gg.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), gg.y, bb.y),
                        fmaf(fmaf(v[i].z, rstd, nmr), gg.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), gg.w, bb.w)));
      }
    } else {
      if (p.tok != nullptr) {
#pragma unroll
        for (int i = 0; i < NV; ++i) st4(xs + r * d + lane * 4 + i * 128, v[i]);
      }
      if (lane == 0) { rs[r] = rstd; nm[r] = nmr; }
    }
  }
  __syncthreads();
  cp_async16(ln + c, p.ln2_g + c);                                   // (waited for before LN2)
  cp_async16(ln + d + c, p.ln2_b + c);
  asm volatile("cp.async.commit_group;" ::: "memory");

  // ---- one position of this thread's sum terms; returns y without beta ----
  float4 S[C];
  auto clear = [&] {
#pragma unroll
    for (int i = 0; i < C; ++i) S[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto step = [&](int j) {
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    if (KM == 0) {
      const float4 v = ld4(xs + j * d + c);
      const float r = rs[j], m = nm[j];
      const float4 z = make_float4(fmaf(fmaf(v.x, r, m), g1.x, b1.x), fmaf(fmaf(v.y, r, m), g1.y, b1.y),
                                   fmaf(fmaf(v.z, r, m), g1.z, b1.z), fmaf(fmaf(v.w, r, m), g1.w, b1.w));
      const float ar = __ldg(alpha + j), ac = __ldg(alpha_col + j);
      const float4 u = make_float4(fmaf(ar, z.x, S[0].x), fmaf(ar, z.y, S[0].y), fmaf(ar, z.z, S[0].z), fmaf(ar, z.w, S[0].w));
      const float4 w = make_float4(z.x + S[1].x, z.y + S[1].y, z.z + S[1].z, z.w + S[1].w);
      const float q = w_col * ac;
      y = make_float4(fmaf(w_row, u.x, q * w.x), fmaf(w_row, u.y, q * w.y), fmaf(w_row, u.z, q * w.z), fmaf(w_row, u.w, q * w.w));
      S[0] = make_float4(lam[0] * u.x, lam[0] * u.y, lam[0] * u.z, lam[0] * u.w);
      S[1] = make_float4(lam[1] * w.x, lam[1] * w.y, lam[1] * w.z, lam[1] * w.w);
    } else {
      constexpr int W4 = KM > 0 ? (KM + 2) / 4 + 1 : 1;              // float4s of z that the window c .. c + 3 + KM - 1 touches
      float z[4 * W4];
#pragma unroll
      for (int q = 0; q < W4; ++q) {
        const int cc = c + 4 * q;
        const float4 f = ld4(xs + j * d + (cc < d ? cc : cc - d));
        z[4 * q] = f.x; z[4 * q + 1] = f.y; z[4 * q + 2] = f.z; z[4 * q + 3] = f.w;
      }
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const float a = al_s[i * T + j], l = lam[i];
        const float4 w = make_float4(z[i] + S[i].x, z[i + 1] + S[i].y, z[i + 2] + S[i].z, z[i + 3] + S[i].w);
        if (c + i + 3 < d) {
          y.x = fmaf(a, w.x, y.x); y.y = fmaf(a, w.y, y.y); y.z = fmaf(a, w.z, y.z); y.w = fmaf(a, w.w, y.w);
        } else {                                                     // terms past the last channel vanish
          if (c + i < d) y.x = fmaf(a, w.x, y.x);
          if (c + i + 1 < d) y.y = fmaf(a, w.y, y.y);
          if (c + i + 2 < d) y.z = fmaf(a, w.z, y.z);
        }
        S[i] = make_float4(l * w.x, l * w.y, l * w.z, l * w.w);
      }
    }
    return y;
  };

  const int64_t E0 = b * (chunks - 1) * planes * d + c;              // this thread's column of the prompt's end states
  clear();
  if (ch + 1 < chunks) {
    // ---- what this (whole) chunk leaves when it starts from zero, for the chunks after it ----
#pragma unroll 2
    for (int j = 0; j < T; ++j) step(j);
#pragma unroll
    for (int i = 0; i < C; ++i)
      if (i < planes) __stcg(reinterpret_cast<float4*>(cs.E + E0 + ((int64_t)ch * planes + i) * d), S[i]);
    __syncthreads();
    if (tid == 0) st_release_u32(cs.flags + b * chunks + ch, cs.epoch);
    clear();
  }
  if (ch > 0) {
    // ---- the start values: S <- lambda^T S + E over the earlier chunks, in order ----
    for (int i = tid; i < ch; i += kThreads) {
      const uint32_t* f = cs.flags + b * chunks + i;
      const long long t0 = clock64();
      while (ld_acquire_u32(f) != cs.epoch) {
        if (clock64() - t0 > kChunkWaitLimitCycles) { raise_status(p.status, kStatusWaitTimeout); break; }
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < C; ++i) {
      if (i < planes) {
        float lT = lam[i];                                           // lambda^T by squaring
#pragma unroll
        for (int k = 1; k < T; k <<= 1) lT *= lT;
#pragma unroll 4
        for (int q = 0; q < ch; ++q) {
          const float4 e = __ldcg(reinterpret_cast<const float4*>(cs.E + E0 + ((int64_t)q * planes + i) * d));
          S[i] = make_float4(fmaf(lT, S[i].x, e.x), fmaf(lT, S[i].y, e.y), fmaf(lT, S[i].z, e.z), fmaf(lT, S[i].w, e.w));
        }
      }
    }
  }
  // ---- y_j and the residual. z of a row is read by several threads, so with KM > 0 x + y of row j goes into the
  //      place of row j only once all threads are past it: rows are finished in groups of four ----
  const float* beta = p.beta + (int64_t)j0 * d + c;
  auto x_of = [&](int j) {
    if (KM == 0) return ld4(xs + j * d + c);
    if (p.tok != nullptr) return ldg4(reinterpret_cast<const WT*>(p.E) + (int64_t)token(j) * d + c);
    return __ldcg(reinterpret_cast<const float4*>(p.x + (row0 + j) * d + c));
  };
  if (KM == 0) {
#pragma unroll 4
    for (int j = 0; j < rows; ++j) {
      const float4 v = x_of(j), bt = ldg4(beta + (int64_t)j * d), y = step(j);
      st4(xs + j * d + c, make_float4(v.x + (y.x + bt.x), v.y + (y.y + bt.y), v.z + (y.z + bt.z), v.w + (y.w + bt.w)));
    }
  } else {
    constexpr int H = 4;                                             // rows per group
    for (int jg = 0; jg < rows; jg += H) {
      float4 o[H];
#pragma unroll
      for (int q = 0; q < H; ++q) {
        const int j = jg + q;
        if (j < rows) {
          const float4 v = x_of(j), bt = ldg4(beta + (int64_t)j * d), y = step(j);
          o[q] = make_float4(v.x + (y.x + bt.x), v.y + (y.y + bt.y), v.z + (y.z + bt.z), v.w + (y.w + bt.w));
        }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < H; ++q)
        if (jg + q < rows) st4(xs + (jg + q) * d + c, o[q]);
    }
  }
  if (ch + 1 == chunks) {                                            // the cache the recurrent form continues from
    ST* So = reinterpret_cast<ST*>(p.S) + b * d;
#pragma unroll
    for (int i = 0; i < C; ++i) {
      if (KM == 0) {
        st4(So + (int64_t)i * p.plane + c, S[i]);
      } else if (i < planes) {
        ST* Pi = So + (int64_t)i * p.plane;
        const float s4[4] = {S[i].x, S[i].y, S[i].z, S[i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int cc = c + i + e;
          Pi[cc < d ? cc : cc - d] = from_float<ST>(s4[e]);
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
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
      const float4 gg = ld4(ln + lane * 4 + i * 128), bb = ld4(ln + d + lane * 4 + i * 128);
      st4(ao + i * 128, make_float4(fmaf(fmaf(v[i].x, rstd, nmr), gg.x, bb.x), fmaf(fmaf(v[i].y, rstd, nmr), gg.y, bb.y),
                                    fmaf(fmaf(v[i].z, rstd, nmr), gg.z, bb.z), fmaf(fmaf(v[i].w, rstd, nmr), gg.w, bb.w)));
    }
  }
}

}  // namespace srm
