// Host runtime of the SRM decode library, part 2: one launcher per kernel, the decode step of a pass of rows, the
// choice of the pass size and the decode step of a whole batch. Everything here is argument set-up and launches;
// all arithmetic of the path runs in the kernels. Included by srm_api.cu only (one translation unit).
#pragma once

#include "runtime.cuh"

namespace {

// ---- kernel launchers -------------------------------------------------------------------------
// Every other kernel than those of launch_resident_kernel and SmallLaunch goes through here: programmatic stream serialization lets the next kernel's blocks be
// scheduled and run their set-up while this one drains; each kernel orders itself with pdl_wait().
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// For a kernel whose CTAs wait for one another (a cooperative launch): all of them become resident together whatever else runs
// on the device. Without it two such kernels from streams of different priority each held SMs that the other waited for, until
// their bounded waits gave up. Every such kernel goes through here (or SmallLaunch), except the chunk mixers, whose blocks wait
// for lower block indices only. Not combined with programmatic serialization, which lets a kernel's blocks in while the one
// before still runs: with both, a prefill beside decode steps of another stream came to a standstill once; and it gains nothing,
// a cooperative kernel waits for all SMs anyway. What residency costs: the feed-forward kernel no longer starts beside the end
// of the one before (decode step of 4096 mid rows 1.44 -> 1.47 ms, prefill of 2048 prompts of 256 143.5 -> 144.7 ms); the
// layers kernel nothing.
template <typename... KArgs, typename... Args>
cudaError_t launch_resident_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Calls f(WT{}, ST{}) with the weight / activation type and the cache storage type of the configuration.
template <typename F>
int dispatch_types(const srm_config& c, F&& f) {
  const bool wb = c.dtype == SRM_DTYPE_BF16;
  switch (c.state_dtype) {
    case SRM_DTYPE_BF16: return wb ? f(bf16{}, bf16{}) : f(float{}, bf16{});
    case SRM_DTYPE_FP16: return wb ? f(bf16{}, fp16{}) : f(float{}, fp16{});
    default: return wb ? f(bf16{}, float{}) : f(float{}, float{});
  }
}

template <int NV, typename WT, typename ST>
int launch_mixer_stream(const MixerParams& p, int num_sms, cudaStream_t st) {
  const int warps = mixer_stream_warps(p.d, (int)sizeof(ST));
  const size_t smem = mixer_stream_smem(p.d, (int)sizeof(ST), warps);
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(mixer_stream_kernel<NV, WT, ST>), kStreamSmemBudget);
  if (rc != SRM_OK) return rc;
  const unsigned grid = (unsigned)(p.R < num_sms ? p.R : num_sms);
  SRM_CUDA(launch_kernel(mixer_stream_kernel<NV, WT, ST>, dim3(grid), dim3(warps * 32), smem, st, p));
  return SRM_OK;
}

template <typename WT, typename ST>
int launch_mixer_nv(const MixerParams& p, int num_sms, cudaStream_t st) {
  const int nv = (p.d + 127) / 128;
  // whole 128-channel vectors per lane, each inside one head: the streaming kernel
  const bool fast = p.d % 128 == 0 && (p.d / p.h) % 128 == 0 && p.h <= 8 && mixer_stream_warps(p.d, (int)sizeof(ST)) >= 1;
  if (fast && nv == 4) return launch_mixer_stream<4, WT, ST>(p, num_sms, st);
  if (fast && nv == 8) return launch_mixer_stream<8, WT, ST>(p, num_sms, st);
  if (fast && nv == 12) return launch_mixer_stream<12, WT, ST>(p, num_sms, st);
  if (fast && nv == 16) return launch_mixer_stream<16, WT, ST>(p, num_sms, st);
  const unsigned grid = (unsigned)((p.R + kMixerWarps - 1) / kMixerWarps);
  const dim3 blk(kMixerWarps * 32);
  if (nv <= 1) SRM_CUDA(launch_kernel(mixer_step_kernel<1, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  else if (nv <= 2) SRM_CUDA(launch_kernel(mixer_step_kernel<2, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  else if (nv <= 4) SRM_CUDA(launch_kernel(mixer_step_kernel<4, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  else if (nv <= 6) SRM_CUDA(launch_kernel(mixer_step_kernel<6, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  else if (nv <= 8) SRM_CUDA(launch_kernel(mixer_step_kernel<8, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  else if (nv <= 12) SRM_CUDA(launch_kernel(mixer_step_kernel<12, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  else SRM_CUDA(launch_kernel(mixer_step_kernel<16, WT, ST>, dim3(grid), dim3(blk), 0, st, p));
  return SRM_OK;
}

// ps: partial products of the previous layer's down projection still to be added into x (mixer_stream_kernel only).
int launch_mixer(const srm_model& m, int layer, int t, int64_t R, const int32_t* tok, float* x, void* S, void* a,
                 uint32_t* status, cudaStream_t st, const int32_t* ctr = nullptr, const int32_t* pos = nullptr,
                 const PartialSum& ps = PartialSum()) {
  if (R <= 0) return SRM_OK;
  LaunchScope scope(m, SRM_KERNEL_MIXER, st);
  MixerParams p;
  p.part = ps.part; p.n_part = ps.n_part; p.part_plane = ps.plane; p.part_bias = ps.bias;
  p.x = x; p.tok = tok; p.E = m.ptr(-1, SRM_T_E); p.S = S; p.a = a;
  p.ln1_g = m.fptr(layer, SRM_T_LN1_G); p.ln1_b = m.fptr(layer, SRM_T_LN1_B);
  p.ln2_g = m.fptr(layer, SRM_T_LN2_G); p.ln2_b = m.fptr(layer, SRM_T_LN2_B);
  p.alpha = m.fptr(layer, SRM_T_ALPHA); p.beta = m.fptr(layer, SRM_T_BETA); p.lam = m.fptr(layer, SRM_T_LAMBDA);
  p.R = R; p.d = m.cfg.d_model; p.h = m.cfg.n_heads; p.n_ctx = m.cfg.n_ctx; p.t = t; p.vocab = m.cfg.vocab;
  p.eps = m.cfg.ln_eps; p.status = status; p.ctr = ctr; p.pos = pos;
  return dispatch_types(m.cfg, [&](auto w, auto c) { return launch_mixer_nv<decltype(w), decltype(c)>(p, m.num_sms, st); });
}

// Fused step of the combined-head / kernel-size-k mixers on R rows at position t (mixer_model_variants.cuh).
// S: plane 0 of the rows' cache, planes `plane` elements apart; x, a rows x_stride elements apart.
template <typename WT, typename ST>
int launch_mixer_variant_t(const VariantParams& p, bool kernel_mix, cudaStream_t st) {
  const unsigned grid = (unsigned)((p.R + kMixerWarps - 1) / kMixerWarps);
  const dim3 blk(kMixerWarps * 32);
  const int nv = (p.d + 127) / 128;
#define SRM_VARIANT_LAUNCH(NV)                                                                                          \
  do {                                                                                                                  \
    if (kernel_mix) SRM_CUDA(launch_kernel(mixer_variant_step_kernel<NV, WT, ST, true>, dim3(grid), dim3(blk), 0, st, p)); \
    else SRM_CUDA(launch_kernel(mixer_variant_step_kernel<NV, WT, ST, false>, dim3(grid), dim3(blk), 0, st, p));           \
  } while (0)
  if (nv <= 1) SRM_VARIANT_LAUNCH(1);
  else if (nv <= 4) SRM_VARIANT_LAUNCH(4);
  else SRM_VARIANT_LAUNCH(8);
#undef SRM_VARIANT_LAUNCH
  return SRM_OK;
}

VariantParams variant_params(const srm_model& m, int layer, int t, int64_t R, const int32_t* tok, int64_t tok_stride, float* x,
                             void* a, int64_t x_stride, void* S, int64_t plane, uint32_t* status, const int32_t* ctr) {
  const srm_config& c = m.cfg;
  VariantParams p;
  p.x = x; p.tok = tok; p.E = m.ptr(-1, SRM_T_E); p.S = S; p.a = a;
  p.ln1_g = m.fptr(layer, SRM_T_LN1_G); p.ln1_b = m.fptr(layer, SRM_T_LN1_B);
  p.ln2_g = m.fptr(layer, SRM_T_LN2_G); p.ln2_b = m.fptr(layer, SRM_T_LN2_B);
  p.alpha = m.fptr(layer, SRM_T_ALPHA); p.beta = m.fptr(layer, SRM_T_BETA); p.lam = m.fptr(layer, SRM_T_LAMBDA);
  const bool comb = c.mixer == SRM_MIXER_COMBINED;
  p.alpha_col = comb ? m.fptr(layer, SRM_T_ALPHA_COL) : nullptr;
  p.lam_col = comb ? m.fptr(layer, SRM_T_LAMBDA_COL) : nullptr;
  p.w_comb = comb ? m.fptr(layer, SRM_T_W_COMB) : nullptr;
  p.R = R; p.x_stride = x_stride; p.tok_stride = tok_stride; p.plane = plane;
  p.d = c.d_model; p.h = c.n_heads; p.k = c.kernel_size; p.n_ctx = c.n_ctx; p.t = t; p.vocab = c.vocab;
  p.eps = c.ln_eps; p.status = status; p.ctr = ctr;
  return p;
}

int launch_mixer_variant(const srm_model& m, int layer, int t, int64_t R, const int32_t* tok, int64_t tok_stride, float* x,
                         void* a, int64_t x_stride, void* S, int64_t plane, uint32_t* status, cudaStream_t st,
                         const int32_t* ctr = nullptr, int cls = SRM_KERNEL_MIXER) {
  if (R <= 0) return SRM_OK;
  LaunchScope scope(m, cls, st);
  const srm_config& c = m.cfg;
  const VariantParams p = variant_params(m, layer, t, R, tok, tok_stride, x, a, x_stride, S, plane, status, ctr);
  const bool wb = c.dtype == SRM_DTYPE_BF16, half_cache = c.state_dtype == SRM_DTYPE_FP16;
  const bool km = c.mixer == SRM_MIXER_KERNEL;
  if (wb) return half_cache ? launch_mixer_variant_t<bf16, fp16>(p, km, st) : launch_mixer_variant_t<bf16, float>(p, km, st);
  return half_cache ? launch_mixer_variant_t<float, fp16>(p, km, st) : launch_mixer_variant_t<float, float>(p, km, st);
}

template <typename WT>
int launch_norm_t(const float* x, int64_t R, int64_t stride, int64_t offset, const float* g, const float* b, float eps,
                  int d, void* out, cudaStream_t st, const int32_t* row_len = nullptr, const PartialSum& ps = PartialSum(),
                  const int32_t* row_start = nullptr) {
  const int nv = (d + 127) / 128;
  const unsigned grid = (unsigned)((R + kMixerWarps - 1) / kMixerWarps);
  const dim3 blk(kMixerWarps * 32);
  WT* o = reinterpret_cast<WT*>(out);
  if (nv <= 1) SRM_CUDA(launch_kernel(norm_rows_kernel<1, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  else if (nv <= 2) SRM_CUDA(launch_kernel(norm_rows_kernel<2, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  else if (nv <= 4) SRM_CUDA(launch_kernel(norm_rows_kernel<4, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  else if (nv <= 6) SRM_CUDA(launch_kernel(norm_rows_kernel<6, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  else if (nv <= 8) SRM_CUDA(launch_kernel(norm_rows_kernel<8, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  else if (nv <= 12) SRM_CUDA(launch_kernel(norm_rows_kernel<12, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  else SRM_CUDA(launch_kernel(norm_rows_kernel<16, WT>, dim3(grid), dim3(blk), 0, st, x, R, stride, offset, g, b, eps, d, o, row_len, ps, row_start));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// out[r, :] = LN(x[r * stride + offset, :]; g, b) in the activation type
int launch_norm(const srm_model& m, const float* x, int64_t R, int64_t stride, int64_t offset, const float* g,
                const float* b, void* out, cudaStream_t st) {
  if (R <= 0) return SRM_OK;
  LaunchScope scope(m, SRM_KERNEL_NORM, st);
  if (m.cfg.dtype == SRM_DTYPE_BF16) return launch_norm_t<bf16>(x, R, stride, offset, g, b, m.cfg.ln_eps, m.cfg.d_model, out, st);
  return launch_norm_t<float>(x, R, stride, offset, g, b, m.cfg.ln_eps, m.cfg.d_model, out, st);
}

int launch_final_norm(const srm_model& m, const float* x, int64_t R, int64_t stride, int64_t offset, void* out,
                      cudaStream_t st, const int32_t* row_len = nullptr, const PartialSum& ps = PartialSum(),
                      const int32_t* row_start = nullptr) {
  if (R <= 0) return SRM_OK;
  LaunchScope scope(m, SRM_KERNEL_NORM, st);
  const float* g = m.fptr(-1, SRM_T_LNF_G);
  const float* b = m.fptr(-1, SRM_T_LNF_B);
  if (m.cfg.dtype == SRM_DTYPE_BF16) return launch_norm_t<bf16>(x, R, stride, offset, g, b, m.cfg.ln_eps, m.cfg.d_model, out, st, row_len, ps, row_start);
  return launch_norm_t<float>(x, R, stride, offset, g, b, m.cfg.ln_eps, m.cfg.d_model, out, st, row_len, ps, row_start);
}

template <typename T>
int launch_gemm_simt(int epi, int64_t M, int64_t N, int64_t K, const void* A, const void* W, const float* bias,
                     void* out, cudaStream_t st) {
  const dim3 grid((unsigned)((N + kSimtBN - 1) / kSimtBN), (unsigned)((M + kSimtBM - 1) / kSimtBM));
  const T* a = reinterpret_cast<const T*>(A);
  const T* w = reinterpret_cast<const T*>(W);
  if (epi == kEpiBiasGelu) SRM_CUDA(launch_kernel(gemm_simt_kernel<T, kEpiBiasGelu>, dim3(grid), dim3(256), 0, st, a, w, bias, out, M, N, K));
  else if (epi == kEpiBiasResidual) SRM_CUDA(launch_kernel(gemm_simt_kernel<T, kEpiBiasResidual>, dim3(grid), dim3(256), 0, st, a, w, bias, out, M, N, K));
  else SRM_CUDA(launch_kernel(gemm_simt_kernel<T, kEpiPlain>, dim3(grid), dim3(256), 0, st, a, w, bias, out, M, N, K));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

int ensure_tc_ready(srm_model& m) {
  if (m.tc_ready) return SRM_OK;
  SRM_CUDA(cudaFuncSetAttribute(tc::gemm_tc_kernel<kEpiBiasGelu>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  SRM_CUDA(cudaFuncSetAttribute(tc::gemm_tc_kernel<kEpiBiasResidual>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  SRM_CUDA(cudaFuncSetAttribute(tc::gemm_tc_kernel<kEpiPlain>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  SRM_CUDA(cudaFuncSetAttribute(tc::gemm_tc_kernel<kEpiArgmax>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  SRM_CUDA(cudaFuncSetAttribute(tc::gemm_tc_kernel<kEpiCollect>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  SRM_CUDA(cudaFuncSetAttribute(tc::gemm_tc_splitk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  SRM_CUDA(cudaFuncSetAttribute(tc::ffn_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (m.num_sms / 2));
  cfg.blockDim = dim3(tc::kThreads);
  cfg.dynamicSmemBytes = tc::kSmemBytes;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  SRM_CUDA(cudaOccupancyMaxActiveClusters(&clusters, tc::gemm_tc_kernel<kEpiPlain>, &cfg));
  if (clusters < 1) { g_last_cuda_error = (int)cudaErrorLaunchOutOfResources; return SRM_ERR_CUDA; }
  m.tc_clusters = clusters < m.num_sms / 2 ? clusters : m.num_sms / 2;
  m.tc_ready = true;
  return SRM_OK;
}

// tail_tiles_of (gemm_tc.cuh), or none with SRM_FLAG_NO_TAIL_SPLIT.
int gemm_tail_tiles(const srm_model& m, int64_t tiles) {
  if (m.cfg.flags & SRM_FLAG_NO_TAIL_SPLIT) return 0;
  return tc::tail_tiles_of(tiles, m.tc_clusters);
}

// k_slices > 1 (epilogue kEpiPlain only; K / 64 a multiple of k_slices): out is k_slices planes of plane_rows x N
// partial products (GemmArgs::k_slices).
int launch_gemm_tc(srm_model& m, int epi, int64_t M, int64_t N, int64_t K, const void* A, const void* W,
                   const float* bias, void* out, uint32_t* status, cudaStream_t st, int k_slices = 1, int64_t plane_rows = 0,
                   const uint32_t* m_limit = nullptr, int64_t m_off = 0) {
  int rc = ensure_tc_ready(m);
  if (rc != SRM_OK) return rc;
  CUtensorMap ta, tb, td, tb64;
  if ((rc = m.tmap(A, M, K, tc::kRowsPerCta, 2, &ta)) != SRM_OK) return rc;
  if ((rc = m.tmap(W, N, K, tc::kRowsPerCta, 2, &tb)) != SRM_OK) return rc;
  if ((rc = m.tmap(W, N, K, tc::kHalfN / 2, 2, &tb64)) != SRM_OK) return rc;      // W rows of a half-width piece
  if (epi == kEpiArgmax) td = ta;       // no output matrix: the descriptor is not used
  else if ((rc = m.tmap(out, k_slices > 1 ? k_slices * plane_rows : M, N, tc::kOutBoxRows, epi == kEpiBiasGelu ? 2 : 4, &td)) != SRM_OK) return rc;
  const uint8_t* wb = static_cast<const uint8_t*>(W);
  const int w_static = wb >= m.w && wb < m.w + m.layout.total;      // inside the weight blob
  const int64_t tiles = ((M + tc::BM - 1) / tc::BM) * ((N + tc::BN - 1) / tc::BN);
  const int tail = k_slices > 1 ? 0 : gemm_tail_tiles(m, tiles);
  tc::GemmArgs g{M, N, K, bias, out, status, w_static};
  g.tail_tiles = tail;
  g.k_slices = k_slices > 1 ? k_slices : 1;
  g.plane_rows = plane_rows;
  int64_t pieces = (tiles + tail) * g.k_slices;
  if (m_limit != nullptr) {                // fewer rows than M, known on the device only
    g.m_limit = m_limit;
    g.m_off = m_off;
    g.dev_tail = (m.cfg.flags & SRM_FLAG_NO_TAIL_SPLIT) ? 0 : 1;
    pieces = m.tc_clusters;
  }
  const unsigned grid = 2u * (unsigned)(pieces < m.tc_clusters ? pieces : m.tc_clusters);
  if (epi == kEpiBiasGelu) SRM_CUDA(launch_kernel(tc::gemm_tc_kernel<kEpiBiasGelu>, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, st, ta, tb, td, tb64, g));
  else if (epi == kEpiBiasResidual) SRM_CUDA(launch_kernel(tc::gemm_tc_kernel<kEpiBiasResidual>, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, st, ta, tb, td, tb64, g));
  else if (epi == kEpiArgmax) SRM_CUDA(launch_kernel(tc::gemm_tc_kernel<kEpiArgmax>, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, st, ta, tb, td, tb64, g));
  else SRM_CUDA(launch_kernel(tc::gemm_tc_kernel<kEpiPlain>, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, st, ta, tb, td, tb64, g));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

int launch_gemm(srm_model& m, int epi, int64_t M, int64_t N, int64_t K, const void* A, const void* W,
                const float* bias, void* out, uint32_t* status, cudaStream_t st, int cls = -1, const uint32_t* m_limit = nullptr,
                int64_t m_off = 0) {
  if (M <= 0) return SRM_OK;
  if (cls < 0) cls = epi == kEpiBiasGelu ? SRM_KERNEL_GEMM_UP : epi == kEpiBiasResidual ? SRM_KERNEL_GEMM_DOWN : SRM_KERNEL_GEMM_LM;
  LaunchScope scope(m, cls, st);
  if (epi == kEpiArgmax) return launch_gemm_tc(m, epi, M, N, K, A, W, bias, out, status, st);
  if (m.cfg.dtype == SRM_DTYPE_FP32) return launch_gemm_simt<float>(epi, M, N, K, A, W, bias, out, st);
  if (m.cfg.flags & SRM_FLAG_SIMT_GEMM) return launch_gemm_simt<bf16>(epi, M, N, K, A, W, bias, out, st);
  return launch_gemm_tc(m, epi, M, N, K, A, W, bias, out, status, st, 1, 0, m_limit, m_off);
}

// out[M, N] += A[M, K] W[N, K]^T + bias with K shared out between CTA pairs. `order`: zeroed words (split_order_words).
// Returns SRM_ERR_UNSUPPORTED when the shape does not call for it (whole tiles per pair lose nothing, or too
// few tiles): the caller then takes the unsplit kernel.
int launch_gemm_splitk(srm_model& m, int64_t M, int64_t N, int64_t K, const void* A, const void* W, const float* bias,
                       float* out, int32_t* order, uint32_t* status, cudaStream_t st, bool only_if_faster = false) {
  if (M <= 0) return SRM_OK;
  int rc = ensure_tc_ready(m);
  if (rc != SRM_OK) return rc;
  tc::SplitPlan P;
  const int64_t tiles = ((M + tc::BM - 1) / tc::BM) * ((N + tc::BN - 1) / tc::BN);
  if (K % tc::BK || !tc::split_plan(tiles, (int)(K / tc::BK), m.tc_clusters, &P)) return SRM_ERR_UNSUPPORTED;
  if (only_if_faster && tc::split_saved_kb(P) < tc::kSplitWorthKb) return SRM_ERR_UNSUPPORTED;
  LaunchScope scope(m, SRM_KERNEL_GEMM_DOWN, st);
  CUtensorMap ta, tb, td;
  if ((rc = m.tmap(A, M, K, tc::kRowsPerCta, 2, &ta)) != SRM_OK) return rc;
  if ((rc = m.tmap(W, N, K, tc::kRowsPerCta, 2, &tb)) != SRM_OK) return rc;
  if ((rc = m.tmap(out, M, N, tc::kOutBoxRows, 4, &td)) != SRM_OK) return rc;
  const uint8_t* wb = static_cast<const uint8_t*>(W);
  const int w_static = wb >= m.w && wb < m.w + m.layout.total;
  tc::SplitArgs g{M, N, K, bias, status, order, w_static};
  SRM_CUDA(launch_resident_kernel(tc::gemm_tc_splitk_kernel, dim3(2u * (unsigned)P.pairs), dim3(tc::kThreads), tc::kSmemBytes, st,
                         ta, tb, td, g, P));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// ---- the feed-forward block as one kernel (ffn_fused.cuh) --------------------------------------
tc::FfnShape ffn_shape(int64_t M, int d, int64_t F) {
  return tc::FfnShape{(int)((M + tc::BM - 1) / tc::BM), (int)(F / tc::BN), d / tc::BK, d / tc::BN, (int)(F / tc::BK)};
}
size_t ffn_ready_bytes(int64_t M, int64_t F) { return align_up((size_t)((M + tc::BM - 1) / tc::BM) * (size_t)(F / tc::BN) * 4, 256); }

// Whether M rows of this model can take the fused kernel (shape limits of the plan and of whole 256-wide tiles).
bool ffn_fused_shape_ok(const srm_model& m, int64_t M) {
  const srm_config& c = m.cfg;
  if (c.dtype != SRM_DTYPE_BF16 || (c.flags & SRM_FLAG_SIMT_GEMM)) return false;
  const int64_t F = m.F();
  if (c.d_model % tc::BN || F % tc::BN || M < 1 || M > (int64_t)tc::kFfnMaxRb * tc::BM) return false;
  return tc::ffn_shape_ok(ffn_shape(M, c.d_model, F), 2);
}

// Whether the decode step takes it for a pass of M rows: from two tiles per CTA pair. With fewer the chain up tile ->
// epilogue -> counter -> down tile is longer than two launches that overlap through programmatic dependent launch,
// and the down projection of such a pass runs over ranges of K instead (down_k_slices). Measured on the mid model
// (74 pairs, 20 tiles per 256 rows), ms per step, one kernel / two launches / two launches with ranges of K: 512 rows
// 0.73 / 0.64 / 0.50, 1024: 0.76 / 0.71 / 0.59, 1536: 0.80 / 0.81 / 0.75, 2048: 0.89 / 0.93 / 0.92, 2304: 0.94 / 0.99 /
// 0.99, 3072: 1.14 / 1.24 / -, 4096: 1.47 / 1.51 / -. As a cooperative launch, one kernel / without: 2048 rows 0.86 / 0.90, 2304:
// 0.93 / 0.97, 3072: 1.13 / 1.19.
bool ffn_fused_worthwhile(const srm_model& m, int64_t M) {
  const tc::FfnShape s = ffn_shape(M, m.cfg.d_model, m.F());
  return m.tc_clusters >= 2 && (int64_t)s.Rb * (s.Cu + s.Cd) >= 2 * (int64_t)m.tc_clusters;
}

// `ready`: ffn_ready_bytes(M, F) bytes of zeroed words. SRM_ERR_UNSUPPORTED: take the two launches.
// m_limit, m_off: FfnArgs.
int launch_ffn_fused(srm_model& m, int layer, int64_t M, const void* a, void* H, float* x, int32_t* ready, uint32_t* status,
                     cudaStream_t st, const uint32_t* m_limit = nullptr, int64_t m_off = 0) {
  if (M <= 0) return SRM_OK;
  if (!ffn_fused_shape_ok(m, M)) return SRM_ERR_UNSUPPORTED;
  int rc = ensure_tc_ready(m);
  if (rc != SRM_OK) return rc;
  const int d = m.cfg.d_model;
  const int64_t F = m.F();
  const tc::FfnShape shape = ffn_shape(M, d, F);
  if (m.tc_clusters < 2 || !tc::ffn_shape_ok(shape, m.tc_clusters)) return SRM_ERR_UNSUPPORTED;
  const tc::FfnPlan* plan = nullptr;
  for (const auto& e : m.ffn_plans)
    if (e.first == shape.Rb) plan = &e.second;
  if (plan == nullptr) {
    m.ffn_plans.emplace_back(shape.Rb, tc::FfnPlan{});
    if (!tc::ffn_make_plan(shape, m.tc_clusters, &m.ffn_plans.back().second)) { m.ffn_plans.pop_back(); return SRM_ERR_UNSUPPORTED; }
    plan = &m.ffn_plans.back().second;
  }
  LaunchScope scope(m, SRM_KERNEL_FFN, st);
  CUtensorMap ta, tw1, tw1h, ths, th, tw2, tx;
  const void* W1 = m.ptr(layer, SRM_T_W1);
  const void* W2 = m.ptr(layer, SRM_T_W2);
  if ((rc = m.tmap(a, M, d, tc::kRowsPerCta, 2, &ta)) != SRM_OK) return rc;
  if ((rc = m.tmap(W1, F, d, tc::kRowsPerCta, 2, &tw1)) != SRM_OK) return rc;
  if ((rc = m.tmap(W1, F, d, tc::kHalfN / 2, 2, &tw1h)) != SRM_OK) return rc;        // W1 rows of a half-width piece
  if ((rc = m.tmap(H, M, F, tc::kOutBoxRows, 2, &ths)) != SRM_OK) return rc;
  if ((rc = m.tmap(H, M, F, tc::kRowsPerCta, 2, &th)) != SRM_OK) return rc;
  if ((rc = m.tmap(W2, d, F, tc::kRowsPerCta, 2, &tw2)) != SRM_OK) return rc;
  if ((rc = m.tmap(x, M, d, tc::kOutBoxRows, 4, &tx)) != SRM_OK) return rc;
  tc::FfnArgs g{M, d, (int)F, m.fptr(layer, SRM_T_B1), m.fptr(layer, SRM_T_B2), status, ready, 1, m_limit, m_off};
  SRM_CUDA(launch_resident_kernel(tc::ffn_fused_kernel, dim3(2u * (unsigned)m.tc_clusters), dim3(tc::kThreads), tc::kSmemBytes, st,
                         ta, tw1, tw1h, ths, th, tw2, tx, g, *plan));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// Ranges the K dimension of a small down projection is cut into (GemmArgs::k_slices): the largest power of two up
// to kMaxKSlices that divides the k-blocks, leaves at least four k-blocks per range and keeps tiles x ranges within the CTA
// pairs; 1 (no cut) when the tiles alone fill half the pairs. Depends on the tile count, so rows of passes of very
// different sizes see sums in another order (last bits); equal-sized passes and all smaller ones agree bit for bit.
int down_k_slices(int64_t tiles, int k_blocks, int pairs) {
  if (tiles < 1 || 2 * tiles > pairs) return 1;
  int ks = 1;
  while (ks < kMaxKSlices && k_blocks % (2 * ks) == 0 && k_blocks / (2 * ks) >= 4 && tiles * 2 * ks <= pairs) ks *= 2;
  return ks;
}

float topk_z0(int top_k, int V) {
  // threshold start of the streaming kernel: the normal quantile that leaves about 2.5 k (at least 96: the set also
  // yields the row's next candidate threshold, which wants a tail to measure) of the V logits above it
  // (rational approximation 26.2.23 of Abramowitz & Stegun; only a starting point, the kernel adapts)
  double pr = (2.5 * top_k > 96.0 ? 2.5 * top_k : 96.0) / (double)V;
  if (pr > 0.45) pr = 0.45;
  const double tt = std::sqrt(-2.0 * std::log(pr));
  return (float)(tt - (2.515517 + 0.802853 * tt + 0.010328 * tt * tt) /
                          (1.0 + 1.432788 * tt + 0.189269 * tt * tt + 0.001308 * tt * tt * tt));
}

int check_sampling(const srm_model& m, const srm_sampling* s) {
  if (s == nullptr) return SRM_ERR_INVALID_ARG;
  if (s->mode == SRM_SELECT_GREEDY) return SRM_OK;
  if (s->mode == SRM_SELECT_TOPP) {
    return (s->top_p > 0.f && s->top_p <= 1.f && s->temperature > 0.f) ? SRM_OK : SRM_ERR_INVALID_ARG;
  }
  if (s->mode != SRM_SELECT_TOPK) return SRM_ERR_INVALID_ARG;
  if (s->top_k < 1 || s->top_k > kTopKMax || s->top_k > m.cfg.vocab || !(s->temperature > 0.f)) return SRM_ERR_INVALID_ARG;
  return SRM_OK;
}

int launch_select(const srm_model& m, int64_t R, const float* logits, const srm_sampling& s, uint64_t sample_base,
                  int step, const SelectOut& out, uint32_t* status, cudaStream_t st) {
  if (R <= 0) return SRM_OK;
  LaunchScope scope(m, SRM_KERNEL_SELECT, st);
  const int V = m.cfg.vocab;
  if (s.mode == SRM_SELECT_GREEDY) {
    SRM_CUDA(launch_kernel(select_greedy_kernel, dim3((unsigned)(R / out.row_div)), dim3(kSelThreads), 0, st, logits, R, V, out, status));
  } else if (s.mode == SRM_SELECT_TOPP) {
    const float inv_t = 1.0f / s.temperature;
    const int few = topp_few_ok(V) ? 1 : 0;
    if (few) {
      SRM_CUDA(launch_kernel(select_topp_few_kernel, dim3((unsigned)R), dim3(kToppThreads), 0, st, logits, R, V, s.top_p, inv_t, s.seed,
                             sample_base, step, out));
      ++g_kernel_launches;
    }
    // (the marked rows, or all: one block per SM walks them, its shared memory leaves no room for more)
    const unsigned grid = (unsigned)(R < m.num_sms ? R : m.num_sms);
    const size_t scratch = ((sizeof(ToppScratch) + 15) & ~size_t(15)) + sizeof(ToppHist);
    const bool staged = V <= kToppSmemFloats;
    const size_t smem = scratch + (staged ? (size_t)V * 4 : 0);
    auto go = [&](auto kernel, size_t most) -> int {
      int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)most);
      if (rc != SRM_OK) return rc;
      SRM_CUDA(launch_kernel(kernel, dim3(grid), dim3(kToppThreads), smem, st, logits, R, V, s.top_p, inv_t, s.seed, sample_base, step, out,
                             status, few));
      return SRM_OK;
    };
    const int rc = staged ? go(select_topp_kernel<true>, scratch + (size_t)kToppSmemFloats * 4) : go(select_topp_kernel<false>, scratch);
    if (rc != SRM_OK) return rc;
  } else {
    const float inv_t = 1.0f / s.temperature;
    const float z0 = topk_z0(s.top_k, V);
    SRM_CUDA(launch_kernel(select_topk_stream_kernel, dim3((unsigned)(R / out.row_div)), dim3(kSelThreads), 0, st, logits, R, V, s.top_k,
                           inv_t, z0, s.seed, sample_base, step, out, status));
    // rows the streaming kernel could not settle (marked -1): the radix selection, reading the row from
    // global memory; every other block exits at once
    SRM_CUDA(launch_kernel(select_topk_kernel<false>, dim3((unsigned)R), dim3(kSelThreads), 0, st, logits, R, V, s.top_k,
                           inv_t, s.seed, sample_base, step, out, status, 1));
    ++g_kernel_launches;
  }
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// True when token selection can be fused into the LM-head GEMM: greedy rule, tensor-core path, and the
// caller does not ask for the logits.
bool can_fuse_greedy(const srm_model& m, const srm_sampling& s, const float* logits_out) {
  return s.mode == SRM_SELECT_GREEDY && logits_out == nullptr && m.cfg.dtype == SRM_DTYPE_BF16 &&
         !(m.cfg.flags & SRM_FLAG_SIMT_GEMM);
}

// LM head with the argmax fused into its epilogue: `part` receives uint2 [argmax_slots(V)][R] partial
// results (it needs argmax_slots(V) * R * 8 bytes, never more than the R x V fp32 logits would), a small
// second kernel reduces them per row and writes the tokens.
int launch_lm_head_greedy(srm_model& m, int64_t R, const void* a, void* part, const SelectOut& out, uint32_t* status,
                          cudaStream_t st) {
  if (R <= 0) return SRM_OK;
  const int V = m.cfg.vocab;
  int rc = launch_gemm(m, kEpiArgmax, R, V, m.cfg.d_model, a, m.ptr(-1, SRM_T_W_LM), nullptr, part, status, st);
  if (rc != SRM_OK) return rc;
  LaunchScope scope(m, SRM_KERNEL_SELECT, st);
  const unsigned grid = (unsigned)((R + kArgmaxRows - 1) / kArgmaxRows);
  SRM_CUDA(launch_kernel(argmax_reduce_kernel, dim3(grid), dim3(kArgmaxRows * kArgmaxLanes), 0, st, reinterpret_cast<const uint2*>(part), R,
                                                                   tc::argmax_slots(V), V, out));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// True when top-k selection can be fused into the LM-head GEMM (candidates collected in the epilogue, no logits
// written): tensor-core path, no logits requested, k small enough for three times k candidates to sit well
// inside a list, and a workspace whose logits and hidden-layer areas are large enough for the lists and for the
// rows handed back (V >= 2048, F >= 2 d).
bool can_fuse_topk(const srm_model& m, const srm_sampling& s, const float* logits_out) {
  return s.mode == SRM_SELECT_TOPK && logits_out == nullptr && m.cfg.dtype == SRM_DTYPE_BF16 &&
         !(m.cfg.flags & (SRM_FLAG_SIMT_GEMM | SRM_FLAG_NO_FUSED_TOPK)) && s.top_k <= kFusedTopkMaxK &&
         (size_t)m.cfg.vocab * 4 >= (size_t)kFusedTopkCap * 8 && m.cfg.ffn_mult >= 2;
}

// LM head with top-k / temperature / Philox selection and no logits in HBM. `lists` (the logits area of the
// workspace) receives the per-row candidate lists; `scratch` (the hidden-layer area, free after the last down
// projection) holds the activation rows handed back, their indices and the counters. Rows the merge kernel
// cannot settle (no threshold yet, too few or too many candidates) get their logits from a second LM-head
// launch over just those rows, written over the (then dead) lists, and the streaming selection.
int launch_lm_head_topk(srm_model& m, int64_t R, const void* a, void* lists, void* scratch, const float* thr,
                        const srm_sampling& s, uint64_t sample_base, int step, const SelectOut& out, uint32_t* status,
                        uint32_t* handed_back, cudaStream_t st) {
  if (R <= 0) return SRM_OK;
  const int V = m.cfg.vocab, d = m.cfg.d_model;
  const size_t row_bytes = (size_t)d * 2;
  uint8_t* p = static_cast<uint8_t*>(scratch);
  void* a_fb = p; p += align_up((size_t)R * row_bytes, 256);
  int32_t* fb_rows = reinterpret_cast<int32_t*>(p); p += align_up((size_t)R * 4, 256);
  uint32_t* cnt = reinterpret_cast<uint32_t*>(p); p += align_up((size_t)R * 4, 256);
  uint32_t* n_fb = reinterpret_cast<uint32_t*>(p);
  SRM_CUDA(cudaMemsetAsync(cnt, 0, align_up((size_t)R * 4, 256) + 256, st));       // counters and n_fb
  int rc = ensure_tc_ready(m);
  if (rc != SRM_OK) return rc;
  const float inv_t = 1.0f / s.temperature;
  CUtensorMap ta, tb;
  {
    LaunchScope scope(m, SRM_KERNEL_GEMM_LM, st);
    if ((rc = m.tmap(a, R, d, tc::kRowsPerCta, 2, &ta)) != SRM_OK) return rc;
    if ((rc = m.tmap(m.ptr(-1, SRM_T_W_LM), V, d, tc::kRowsPerCta, 2, &tb)) != SRM_OK) return rc;
    CUtensorMap tb64;
    if ((rc = m.tmap(m.ptr(-1, SRM_T_W_LM), V, d, tc::kHalfN / 2, 2, &tb64)) != SRM_OK) return rc;
    const int64_t tiles = ((R + tc::BM - 1) / tc::BM) * ((V + tc::BN - 1) / tc::BN);
    tc::GemmArgs g{R, V, d, nullptr, lists, status, 1, thr, cnt, kFusedTopkCap, nullptr, gemm_tail_tiles(m, tiles)};
    const int64_t pieces = tiles + g.tail_tiles;
    const unsigned grid = 2u * (unsigned)(pieces < m.tc_clusters ? pieces : m.tc_clusters);
    SRM_CUDA(launch_kernel(tc::gemm_tc_kernel<kEpiCollect>, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, st, ta, tb, ta, tb64, g));
  }
  {
    LaunchScope scope(m, SRM_KERNEL_SELECT, st);
    SRM_CUDA(launch_kernel(topk_merge_kernel, dim3((unsigned)R), dim3(kSelThreads), 0, st,
                           reinterpret_cast<const unsigned long long*>(lists), cnt, thr, kFusedTopkCap, R, s.top_k, inv_t, s.seed,
                           sample_base, step, out, reinterpret_cast<const uint4*>(a), reinterpret_cast<uint4*>(a_fb),
                           (int)(row_bytes / 16), fb_rows, n_fb, handed_back));
  }
  {
    // the rows handed back: logits of the first *n_fb rows of a_fb only (no tile when there is none)
    LaunchScope scope(m, SRM_KERNEL_GEMM_LM, st);
    CUtensorMap tf, td;
    if ((rc = m.tmap(a_fb, R, d, tc::kRowsPerCta, 2, &tf)) != SRM_OK) return rc;
    if ((rc = m.tmap(lists, R, V, tc::kOutBoxRows, 4, &td)) != SRM_OK) return rc;
    tc::GemmArgs g{R, V, d, nullptr, lists, status, 0, nullptr, nullptr, 0, n_fb, 0};
    const int64_t tiles = ((R + tc::BM - 1) / tc::BM) * ((V + tc::BN - 1) / tc::BN);
    const unsigned grid = 2u * (unsigned)(tiles < m.tc_clusters ? tiles : m.tc_clusters);
    SRM_CUDA(launch_kernel(tc::gemm_tc_kernel<kEpiPlain>, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, st, tf, tb, td, tb, g));
  }
  {
    LaunchScope scope(m, SRM_KERNEL_SELECT, st);
    SelectOut o = out;
    o.row_map = fb_rows;
    o.n_rows = n_fb;
    const float* lg = reinterpret_cast<const float*>(lists);
    SRM_CUDA(launch_kernel(select_topk_stream_kernel, dim3((unsigned)R), dim3(kSelThreads), 0, st, lg, R, V, s.top_k, inv_t,
                           topk_z0(s.top_k, V), s.seed, sample_base, step, o, status));
    SRM_CUDA(launch_kernel(select_topk_kernel<false>, dim3((unsigned)R), dim3(kSelThreads), 0, st, lg, R, V, s.top_k, inv_t,
                           s.seed, sample_base, step, o, status, 1));
    ++g_kernel_launches;
  }
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// From this many prompts per pass a CTA walks a prompt (prefill_walk.cuh); below it a CTA takes 16 positions of one (the
// chunk kernel), or, for shapes neither is built for, the tile kernel (a CTA per prompt). us per launch, tile / chunk /
// walk: mid, 1 prompt of 777 positions 2061 / 19 / -, 45 ragged prompts of up to 301 717 / 33 / -, 2048 prompts of 256
// - / 1844 / 1432; rl, 16 prompts of 200: 760 / 26 / -.
constexpr int64_t kPrefillWalkMinPrompts = 384;

bool prefill_walk_ok(const srm_model& m, int64_t np) {
  const int d = m.cfg.d_model;
  return m.cfg.mixer == SRM_MIXER_MIXED && !m.head_proj() && (d == 512 || d == 1024 || d == 1536 || d == 2048) && np >= kPrefillWalkMinPrompts;
}

template <int NV, typename WT, typename ST>
int launch_prefill_walk(const PrefillParams& p, cudaStream_t st) {
  const size_t smem = prefill_walk_smem(NV * 128);
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(prefill_walk_kernel<NV, WT, ST>), (int)smem);
  if (rc != SRM_OK) return rc;
  SRM_CUDA(launch_kernel(prefill_walk_kernel<NV, WT, ST>, dim3((unsigned)p.Bp), dim3(NV * 32), smem, st, p));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

template <typename WT, typename ST>
int launch_prefill_walk_nv(const PrefillParams& p, cudaStream_t st) {
  switch (p.d / 128) {
    case 4: return launch_prefill_walk<4, WT, ST>(p, st);
    case 8: return launch_prefill_walk<8, WT, ST>(p, st);
    case 12: return launch_prefill_walk<12, WT, ST>(p, st);
    default: return launch_prefill_walk<16, WT, ST>(p, st);
  }
}

// Whether a pass of np prompts of n positions takes the chunk kernels: widths and types they are built for, and
// workspace areas that are free while a layer's tokens are mixed with room for their scratch (the end states of the
// chunks in the hidden-layer area, the flags in the area of the last-position activations).
bool prefill_chunk_ok(const srm_model& m, int64_t np, int n) {
  const srm_config& c = m.cfg;
  if (m.head_proj()) return false;
  if (c.mixer == SRM_MIXER_MIXED) {
    if (np >= kPrefillWalkMinPrompts) return false;
    if (c.d_model != 512 && c.d_model != 1024 && c.d_model != 1536 && c.d_model != 2048) return false;
  } else if (c.dtype != SRM_DTYPE_BF16 || (c.d_model != 512 && c.d_model != 1024)) {
    return false;
  }
  const int64_t chunks = prefill_chunks(n), all = np * chunks;
  return all < ((int64_t)1 << 31) &&
         (size_t)(all - np) * cache_planes(c) * c.d_model * 4 <= (size_t)np * n * m.F() * m.act_bytes() &&
         (size_t)all * 4 <= (size_t)np * c.d_model * m.act_bytes();
}

template <int NV, typename WT, typename ST>
int launch_prefill_chunk(const PrefillParams& p, const ChunkScratch& cs, cudaStream_t st) {
  const size_t smem = prefill_chunk_smem(NV * 128);
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(prefill_chunk_kernel<NV, WT, ST>), (int)smem);
  if (rc != SRM_OK) return rc;
  const int chunks = (int)prefill_chunks(p.n);
  SRM_CUDA(launch_kernel(prefill_chunk_kernel<NV, WT, ST>, dim3((unsigned)(p.Bp * chunks)), dim3(NV * 32), smem, st, p, cs, chunks));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}

// cs: scratch of the chunk kernel (prefill_chunk_ok), or nullptr: none.
int launch_prefill_mixer(const srm_model& m, int layer, int64_t Bp, int n, const int32_t* tok, float* x, void* S,
                         void* a, uint32_t* status, cudaStream_t st, const int32_t* len = nullptr,
                         const ChunkScratch* cs = nullptr, const int32_t* row_start = nullptr) {
  if (Bp <= 0) return SRM_OK;
  LaunchScope scope(m, SRM_KERNEL_PREFILL_MIXER, st);
  PrefillParams p;
  p.x = x; p.tok = tok; p.E = m.ptr(-1, SRM_T_E); p.S = S; p.a = a;
  p.ln1_g = m.fptr(layer, SRM_T_LN1_G); p.ln1_b = m.fptr(layer, SRM_T_LN1_B);
  p.ln2_g = m.fptr(layer, SRM_T_LN2_G); p.ln2_b = m.fptr(layer, SRM_T_LN2_B);
  p.alpha = m.fptr(layer, SRM_T_ALPHA); p.beta = m.fptr(layer, SRM_T_BETA); p.lam = m.fptr(layer, SRM_T_LAMBDA);
  p.Bp = Bp; p.n = n; p.d = m.cfg.d_model; p.h = m.cfg.n_heads; p.n_ctx = m.cfg.n_ctx; p.vocab = m.cfg.vocab;
  p.eps = m.cfg.ln_eps; p.status = status; p.len = len; p.row_start = row_start;
  const size_t smem = (size_t)kPrefillTile * m.cfg.d_model * 4;
  const int nv = p.d / 128;
  if (cs != nullptr) {
    return dispatch_types(m.cfg, [&](auto w, auto c) {
      using WT = decltype(w);
      using ST = decltype(c);
      switch (nv) {
        case 4: return launch_prefill_chunk<4, WT, ST>(p, *cs, st);
        case 8: return launch_prefill_chunk<8, WT, ST>(p, *cs, st);
        case 12: return launch_prefill_chunk<12, WT, ST>(p, *cs, st);
        default: return launch_prefill_chunk<16, WT, ST>(p, *cs, st);
      }
    });
  }
  if (prefill_walk_ok(m, Bp))      // many prompts
    return dispatch_types(m.cfg, [&](auto w, auto c) { return launch_prefill_walk_nv<decltype(w), decltype(c)>(p, st); });
  auto go = [&](auto kernel) -> int {
    SRM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));   // smem depends on d: set per launch
    SRM_CUDA(launch_kernel(kernel, dim3((unsigned)Bp), dim3(kPrefillThreads), smem, st, p));
    SRM_CUDA(cudaGetLastError());
    return SRM_OK;
  };
  return dispatch_types(m.cfg, [&](auto w, auto c) { return go(prefill_mixer_kernel<decltype(w), decltype(c)>); });
}

// Sequence form of the further mixers in chunks of positions (prefill_chunk_variants.cuh; prefill_chunk_ok).
template <int NV, typename ST, int KM>
int launch_variant_chunk_k(const VariantParams& p, const ChunkScratch& cs, int n, cudaStream_t st) {
  const size_t smem = variant_chunk_smem<NV, KM>();
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(variant_chunk_kernel<NV, bf16, ST, KM>), (int)smem);
  if (rc != SRM_OK) return rc;
  const int chunks = (int)prefill_chunks(n);
  SRM_CUDA(launch_kernel(variant_chunk_kernel<NV, bf16, ST, KM>, dim3((unsigned)(p.R * chunks)), dim3(NV * 32), smem, st, p, cs, n, chunks));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}
template <int NV, typename ST>
int launch_variant_chunk_t(const VariantParams& p, bool kernel_mix, const ChunkScratch& cs, int n, cudaStream_t st) {
  if (!kernel_mix) return launch_variant_chunk_k<NV, ST, 0>(p, cs, n, st);
  if (p.k <= 2) return launch_variant_chunk_k<NV, ST, 2>(p, cs, n, st);
  if (p.k <= 4) return launch_variant_chunk_k<NV, ST, 4>(p, cs, n, st);
  if (p.k <= 8) return launch_variant_chunk_k<NV, ST, 8>(p, cs, n, st);
  return launch_variant_chunk_k<NV, ST, 16>(p, cs, n, st);
}
int launch_variant_chunk(const srm_model& m, int layer, int64_t Bp, int n, const int32_t* tok, float* x, void* a, void* S,
                         int64_t plane, uint32_t* status, cudaStream_t st, const ChunkScratch& cs) {
  if (Bp <= 0) return SRM_OK;
  LaunchScope scope(m, SRM_KERNEL_PREFILL_MIXER, st);
  const VariantParams p = variant_params(m, layer, 0, Bp, tok, n, x, a, m.cfg.d_model, S, plane, status, nullptr);
  const bool km = m.cfg.mixer == SRM_MIXER_KERNEL, half = m.cfg.state_dtype == SRM_DTYPE_FP16;
  if (p.d == 512) return half ? launch_variant_chunk_t<4, fp16>(p, km, cs, n, st) : launch_variant_chunk_t<4, float>(p, km, cs, n, st);
  return half ? launch_variant_chunk_t<8, fp16>(p, km, cs, n, st) : launch_variant_chunk_t<8, float>(p, km, cs, n, st);
}

// Token-mixing block with head projections (Eq. 10) on `rows` rows of the residual stream:
//   [x = E[tok]];  a = LN1(x);  q = a W_in^T;  y, S' = mixer(q, S);  x += y W_out^T;  a = LN2(x).
// Decode: t >= 0, one position, S [rows, d] in/out. Prefill: t < 0, `samples` prompts of n positions
// (rows = samples * n), sequence-parallel mixing, S [samples, d] out.
template <typename WT, typename ST>
int launch_mix_proj_t(bool prefill, const MixProjParams& p, int64_t vecs, cudaStream_t st) {
  const unsigned grid = (unsigned)((vecs + kMixProjThreads - 1) / kMixProjThreads);
  if (prefill) SRM_CUDA(launch_kernel(mixer_proj_prefill_kernel<WT, ST>, dim3(grid), dim3(kMixProjThreads), 0, st, p));
  else SRM_CUDA(launch_kernel(mixer_proj_step_kernel<WT, ST>, dim3(grid), dim3(kMixProjThreads), 0, st, p));
  return SRM_OK;
}

int launch_mixer_block_proj(srm_model& m, int layer, int t, int64_t rows, int64_t samples, int n, const int32_t* tok,
                            float* x, void* S, void* a, float* q, uint32_t* status, cudaStream_t st,
                            const int32_t* ctr = nullptr, const int32_t* pos = nullptr) {
  if (rows <= 0) return SRM_OK;
  const srm_config& c = m.cfg;
  const int d = c.d_model;
  const bool prefill = t < 0;
  const bool wb = c.dtype == SRM_DTYPE_BF16;
  int rc;
  if (tok != nullptr) {
    LaunchScope scope(m, prefill ? SRM_KERNEL_PREFILL_MIXER : SRM_KERNEL_MIXER, st);
    const unsigned grid = (unsigned)((rows * (d / 4) + kMixProjThreads - 1) / kMixProjThreads);
    if (wb) SRM_CUDA(launch_kernel(embed_rows_kernel<bf16>, dim3(grid), dim3(kMixProjThreads), 0, st, tok,
                                   reinterpret_cast<const bf16*>(m.ptr(-1, SRM_T_E)), x, rows, d, c.vocab, status));
    else SRM_CUDA(launch_kernel(embed_rows_kernel<float>, dim3(grid), dim3(kMixProjThreads), 0, st, tok,
                                reinterpret_cast<const float*>(m.ptr(-1, SRM_T_E)), x, rows, d, c.vocab, status));
  }
  if ((rc = launch_norm(m, x, rows, 1, 0, m.fptr(layer, SRM_T_LN1_G), m.fptr(layer, SRM_T_LN1_B), a, st))) return rc;
  if ((rc = launch_gemm(m, kEpiPlain, rows, d, d, a, m.ptr(layer, SRM_T_W_IN), nullptr, q, status, st, SRM_KERNEL_GEMM_PROJ))) return rc;
  {
    LaunchScope scope(m, prefill ? SRM_KERNEL_PREFILL_MIXER : SRM_KERNEL_MIXER, st);
    MixProjParams p;
    p.q = q; p.S = S; p.y = a;
    p.alpha = m.fptr(layer, SRM_T_ALPHA); p.beta = m.fptr(layer, SRM_T_BETA); p.lam = m.fptr(layer, SRM_T_LAMBDA);
    p.R = prefill ? samples : rows; p.d = d; p.h = c.n_heads; p.n_ctx = c.n_ctx; p.t = prefill ? 0 : t; p.n = n;
    p.ctr = prefill ? nullptr : ctr;
    p.pos = pos;                                   // decode: per-row positions; prefill: prompt lengths
    p.status = status;
    const int64_t vecs = p.R * (d / 4);
    rc = dispatch_types(c, [&](auto w, auto cs) { return launch_mix_proj_t<decltype(w), decltype(cs)>(prefill, p, vecs, st); });
    if (rc) return rc;
  }
  if ((rc = launch_gemm(m, kEpiBiasResidual, rows, d, d, a, m.ptr(layer, SRM_T_W_OUT), nullptr, x, status, st, SRM_KERNEL_GEMM_PROJ))) return rc;
  return launch_norm(m, x, rows, 1, 0, m.fptr(layer, SRM_T_LN2_G), m.fptr(layer, SRM_T_LN2_B), a, st);
}

sb::LayerW layer0_weights(const srm_model& m) {
  return sb::LayerW{m.fptr(0, SRM_T_LN1_G), m.fptr(0, SRM_T_LN1_B), m.fptr(0, SRM_T_LN2_G), m.fptr(0, SRM_T_LN2_B),
                    m.fptr(0, SRM_T_ALPHA), m.fptr(0, SRM_T_BETA), m.fptr(0, SRM_T_LAMBDA), m.fptr(0, SRM_T_B1),
                    m.fptr(0, SRM_T_B2), reinterpret_cast<const bf16*>(m.ptr(0, SRM_T_W1)),
                    reinterpret_cast<const bf16*>(m.ptr(0, SRM_T_W2))};
}
int64_t layer_stride_bytes(const srm_model& m) {      // distance of a tensor from the same tensor of the next layer
  return m.cfg.n_layers > 1 ? (int64_t)(m.layout.layer[SRM_T_COUNT + SRM_T_LN1_G].off - m.layout.layer[SRM_T_LN1_G].off) : 0;
}

// ---- decode passes of up to about a thousand rows: all layers in one kernel (layers_mid.cuh) -------------
// Fewest rows, where the passes are not those of another kernel (cluster_rows_ok and split_rows_ok come first; step_small.cuh where
// F is not 4 d). d = 512: 65 to 71 rows keep the kernel-per-operation path for one reason, a test that counts its launches at 65 samples
// (138 us at 72 rows there, 104 here, 52 in clusters, where these rows would be as fast); up to 64 rows come here only where the single-kernel step does not take F (as kMixedAny).
// Combined heads and kernels (d 512 and 1024) have no other one-kernel step: any pass (96 rows, d = 1024, 16 layers, kernels of
// size 4: 275 us per step, as a kernel per operation 560).
bool mid_rows_ok(const srm_config& c, int64_t R) { return c.d_model != 512 || c.mixer != SRM_MIXER_MIXED || R <= sb::kMaxRows || R >= 72; }
// The widths with instances of their own; mixed-head models of other widths up to 1024 channels take the instance for any
// width with as many rows as the single-kernel step would, which is built for d % 256 == 0 and F % 1024 == 0 only (us per step
// of 8 layers, V = 8000, 1 / 64 rows, as a kernel per operation -> here: d 64 83 / 91 -> 78 / 89, d 320 123 / 132 -> 95 / 103,
// d 640 173 / 180 -> 111 / 118, d 832 266 / 262 -> 127 / 134, d 768 with F 6144 349 / 341 -> 145 / 154; the single-kernel step of
// any width that stood here before took 109 / 148, 120 / 158, 126 / 177, 142 / 194 and 145 / 223).
bool mid_own_width(int d) { return d == 512 || d == 1024 || d == 1536; }

constexpr size_t kCntFloats = 256;      // room for mid::kCntWords at the head of the logits area
static_assert(mid::kCntWords <= (int)kCntFloats, "counters");
int mid_mix(const srm_config& c, int64_t R) {
  if (c.mixer != SRM_MIXER_MIXED) return c.mixer == SRM_MIXER_COMBINED ? mid::kCombined : mid::kKernel;
  return mid_own_width(c.d_model) && !(c.d_model == 512 && R <= sb::kMaxRows) ? mid::kMixed : mid::kMixedAny;
}

// Whether a decode pass of R rows takes it, and its tile plan. bf16 models of the widths it is built for,
// as many rows as leave every CTA pair one tile of each projection.
bool mid_plan(srm_model& m, int64_t R, const DecodeWs& w, mid::Params* p) {
  const srm_config& c = m.cfg;
  constexpr int kOff = SRM_FLAG_SIMT_GEMM | SRM_FLAG_NO_SMALL_BATCH | SRM_FLAG_NO_KSLICE | SRM_FLAG_NO_FUSED_FFN | SRM_FLAG_HEAD_PROJ;
  if (!mid_rows_ok(c, R) || c.dtype != SRM_DTYPE_BF16 || (c.flags & kOff)) return false;
  if (c.mixer != SRM_MIXER_MIXED && (c.d_model > 1024 || c.n_heads > 8 || c.kernel_size > 16)) return false;
  const int mix = mid_mix(c, R);
  if (mix == mid::kMixedAny ? R > sb::kMaxRows || c.d_model > 1024 : !mid_own_width(c.d_model)) return false;
  if (ensure_tc_ready(m) != SRM_OK || R > (int64_t)2 * m.tc_clusters * mid::kMaxGroups || m.F() > (1 << 20)) return false;
  // The planes of partial products: an area of their own where the model has one (kslice_model), else behind the counters in
  // the logits area. Any widths keep the rows there are, in as many planes as there is room for; whole boxes of rows fit from
  // about five rows of the mid model on.
  const size_t logits = (size_t)w.rows * c.vocab;
  const size_t room = w.part != nullptr ? w.part_bytes : (logits - std::min(logits, kCntFloats)) * 4;
  p->part = w.part != nullptr ? w.part : w.logits + kCntFloats;
  p->plane_rows = mix == mid::kMixedAny ? (int)R : (int)(R + tc::kOutBoxRows - 1) / tc::kOutBoxRows * tc::kOutBoxRows;
  for (int most = mix == mid::kMixedAny ? 2 * mid::kMaxKSlices : mid::kMaxKSlices; most >= 1; most /= 2) {
    if (!mid::plan(R, c.d_model, (int)m.F(), m.tc_clusters, mix, most, p)) return false;
    if ((size_t)p->ks * p->plane_rows * c.d_model * 4 <= room) return true;
    if (mix != mid::kMixedAny) return false;
  }
  return false;
}

struct MidMaps { CUtensorMap a, h, w1, w2, hs, p; };      // loads of a, H, W1, W2; stores of H and the partial products
template <int NT, int WPG, typename ST, int MIX>
int launch_layers_w(srm_model& m, const MidMaps& t, const mid::Params& p, cudaStream_t st) {
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(mid::layers_kernel<NT, WPG, ST, MIX>), mid::kSmemBytes);
  if (rc != SRM_OK) return rc;
  const size_t smem = mid::smem_bytes(p.d, p.n, p.w_slots, p.a_slots, MIX);
  SRM_CUDA(launch_resident_kernel(mid::layers_kernel<NT, WPG, ST, MIX>, dim3(2u * (unsigned)m.tc_clusters), dim3(mid::kThreads), smem, st,
                         t.a, t.h, t.w1, t.w2, t.hs, t.p, p));
  SRM_CUDA(cudaGetLastError());
  return SRM_OK;
}
// Four warps per row where all rows are then worked on at once, else two.
template <int NT, typename ST, int MIX>
int launch_layers_t(srm_model& m, const MidMaps& t, const mid::Params& p, cudaStream_t st) {
  if (p.R <= (int64_t)2 * m.tc_clusters * (tc::kEpiWarps / 4)) return launch_layers_w<NT / 2, 4, ST, MIX>(m, t, p, st);
  return launch_layers_w<NT, 2, ST, MIX>(m, t, p, st);
}
template <int NT>
int launch_layers_nt(srm_model& m, const MidMaps& t, const mid::Params& p, cudaStream_t st) {
  if (m.cfg.state_dtype == SRM_DTYPE_FP16) return launch_layers_t<NT, fp16, mid::kMixed>(m, t, p, st);
  if (m.cfg.state_dtype == SRM_DTYPE_BF16) return launch_layers_t<NT, bf16, mid::kMixed>(m, t, p, st);
  return launch_layers_t<NT, float, mid::kMixed>(m, t, p, st);
}
int launch_layers_any(srm_model& m, const MidMaps& t, const mid::Params& p, cudaStream_t st) {      // (at most 64 rows, 1024 channels)
  if (m.cfg.state_dtype == SRM_DTYPE_FP16) return launch_layers_w<2, 4, fp16, mid::kMixedAny>(m, t, p, st);
  if (m.cfg.state_dtype == SRM_DTYPE_BF16) return launch_layers_w<2, 4, bf16, mid::kMixedAny>(m, t, p, st);
  return launch_layers_w<2, 4, float, mid::kMixedAny>(m, t, p, st);
}
template <int NT>
int launch_layers_variant(srm_model& m, const MidMaps& t, const mid::Params& p, cudaStream_t st) {
  const bool half = m.cfg.state_dtype == SRM_DTYPE_FP16;
  if (m.cfg.mixer == SRM_MIXER_COMBINED)
    return half ? launch_layers_t<NT, fp16, mid::kCombined>(m, t, p, st) : launch_layers_t<NT, float, mid::kCombined>(m, t, p, st);
  return half ? launch_layers_t<NT, fp16, mid::kKernel>(m, t, p, st) : launch_layers_t<NT, float, mid::kKernel>(m, t, p, st);
}

// All layers and the final norm for rows [b0, b0 + R) of the state; leaves the normed rows in w.a.
// p: from mid_plan.
int launch_layers_mid(srm_model& m, srm_state& s, int64_t b0, int64_t R, int t, const int32_t* tok_in, const DecodeWs& w, mid::Params& p,
                      cudaStream_t st, const int32_t* ctr, const int32_t* pos) {
  const srm_config& c = m.cfg;
  const int d = c.d_model, F = (int)m.F();
  p.R = (int)R; p.d = d; p.F = F; p.V = c.vocab; p.h = c.n_heads; p.n_ctx = c.n_ctx; p.L = c.n_layers; p.t = t;
  p.eps = c.ln_eps;
  p.tok_in = tok_in;
  p.E = reinterpret_cast<const bf16*>(m.ptr(-1, SRM_T_E));
  p.layer0 = layer0_weights(m);
  p.layer_bytes = layer_stride_bytes(m);
  p.S = static_cast<uint8_t*>(s.layer_ptr(0)) + (size_t)b0 * d * m.state_bytes();
  p.layer_stride = (int64_t)s.planes() * s.B * d * m.state_bytes();
  p.k = c.kernel_size;
  p.s_plane = s.plane_elems();
  if (c.mixer == SRM_MIXER_COMBINED) { p.alpha_col = m.fptr(0, SRM_T_ALPHA_COL); p.lam_col = m.fptr(0, SRM_T_LAMBDA_COL); p.w_comb = m.fptr(0, SRM_T_W_COMB); }
  p.lnf_g = m.fptr(-1, SRM_T_LNF_G); p.lnf_b = m.fptr(-1, SRM_T_LNF_B);
  p.x = w.x; p.a = reinterpret_cast<bf16*>(w.a); p.H = reinterpret_cast<bf16*>(w.H);
  p.plane = (int64_t)p.plane_rows * d;
  p.cnt = reinterpret_cast<uint32_t*>(w.logits);      // (nothing uses the logits area before the LM head)
  p.status = s.status; p.ctr = ctr; p.pos = pos;
  // (cleared by a kernel: behind a memset the step took 3 us longer)
  ++g_kernel_launches;
  SRM_CUDA(launch_kernel(mid::zero_counters_kernel, dim3(1), dim3(64), 0, st, p.cnt));
  LaunchScope scope(m, SRM_KERNEL_STEP_SMALL, st);
  MidMaps maps;
  int rc;
  if ((rc = make_tmap_kblocks(&maps.a, w.a, R, d, p.box, mid::kStep)) != SRM_OK) return rc;
  if ((rc = make_tmap_kblocks(&maps.h, w.H, R, F, p.box, mid::kStep)) != SRM_OK) return rc;
  if ((rc = make_tmap_kblocks(&maps.w1, m.ptr(0, SRM_T_W1), F, d, p.n / 2, mid::kStep, c.n_layers, p.layer_bytes)) != SRM_OK) return rc;
  if ((rc = make_tmap_kblocks(&maps.w2, m.ptr(0, SRM_T_W2), d, F, p.n / 2, mid::kStep, c.n_layers, p.layer_bytes)) != SRM_OK) return rc;
  if ((rc = m.tmap(w.H, R, F, tc::kOutBoxRows, 2, &maps.hs)) != SRM_OK) return rc;
  if (mid_mix(c, R) == mid::kMixedAny) {                  // (planes of the rows there are: a box must not reach into the next one)
    if ((rc = make_tmap(&maps.p, p.part, R, d, tc::kOutBoxRows, 4, p.ks, p.plane_rows)) != SRM_OK) return rc;
    return launch_layers_any(m, maps, p, st);
  }
  if ((rc = m.tmap(p.part, (int64_t)p.ks * p.plane_rows, d, tc::kOutBoxRows, 4, &maps.p)) != SRM_OK) return rc;
  if (c.mixer != SRM_MIXER_MIXED) return d == 512 ? launch_layers_variant<2>(m, maps, p, st) : launch_layers_variant<4>(m, maps, p, st);
  if (d == 512) return launch_layers_nt<2>(m, maps, p, st);
  if (d == 1024) return launch_layers_nt<4>(m, maps, p, st);
  return launch_layers_nt<6>(m, maps, p, st);
}

// ---- small decode passes: rows inside clusters of 16 CTAs, all layers in one kernel (layers_cluster.cuh) -------------
// f(kernel, shared memory) for an instance.
template <int D, int RC, typename Fn>
int with_cluster_kernel_t(const srm_config& c, Fn&& f) {
  constexpr size_t smem = cl::Shape<D, RC>::kSmem;
  if (c.state_dtype == SRM_DTYPE_FP16) return f(cl::layers_kernel<D, RC, fp16>, smem);
  if (c.state_dtype == SRM_DTYPE_BF16) return f(cl::layers_kernel<D, RC, bf16>, smem);
  return f(cl::layers_kernel<D, RC, float>, smem);
}
// The instance whose clusters hold `rows` rows or more.
template <typename Fn>
int with_cluster_kernel(const srm_config& c, int rows, Fn&& f) {
  if (c.d_model == 1024) return rows <= 8 ? with_cluster_kernel_t<1024, 8>(c, f) : with_cluster_kernel_t<1024, 16>(c, f);
  if (rows <= 16) return with_cluster_kernel_t<512, 16>(c, f);
  if (rows <= 32) return with_cluster_kernel_t<512, 32>(c, f);
  return rows <= 48 ? with_cluster_kernel_t<512, 48>(c, f) : with_cluster_kernel_t<512, 64>(c, f);
}
struct ClusterLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  // resident: all CTAs at once (a cooperative launch), for kernels whose clusters wait for one another
  ClusterLaunch(unsigned clusters, int threads, size_t smem, cudaStream_t st, bool resident) {
    cfg.gridDim = dim3(clusters * cl::kCluster);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl::kCluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    if (resident) {
      attr[1].id = cudaLaunchAttributeCooperative;
      attr[1].val.cooperative = 1;
    } else {
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};
// How many clusters of `kernel` are resident at once (0: the device cannot run it).
template <typename K>
int resident_clusters(K* kernel, int threads, size_t smem) {
  int n = 0;
  ClusterLaunch L(1, threads, smem, nullptr, false);
  L.cfg.numAttrs = 1;
  if (ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), cl::kSmemBytes, true) != SRM_OK ||
      cudaOccupancyMaxActiveClusters(&n, kernel, &L.cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}
// Whether a decode pass of R rows takes it: bf16 models with mixed heads, F = 4 d, of 512 or 1024 channels, as many rows as the
// clusters the device holds at once (seven on 148 SMs) have room for. us per greedy step, the layers kernel over the whole grid or
// the single-kernel step (up to 64 rows at d = 512, 32 at d = 1024) / here: d = 512, 8 layers, V = 8000, 1 row 73 / 49, 16 rows
// 77 / 50, 64 rows 113 / 51, 72 rows 104 / 52, 112 106 / 54, 224 110 / 67, 256 109 / 77, 336 117 / 82, 448 118 / 102 (with LM head and
// selection as kernels of their own 55, 57, 69, 77, 83, 100 from 72 rows on); d = 1024, 16 layers, 8 rows 191 / 206, 16 rows 201 / 202, 24 rows 236 / 204, 56 rows
// 245 / 206, 112 rows 260 / 221 (with 17 to 32 rows per cluster the weight ring is too short: 22.9 us per layer against 14).
bool cluster_rows_ok(srm_model& m, int64_t R) {
  const srm_config& c = m.cfg;
  constexpr int kOff = SRM_FLAG_SIMT_GEMM | SRM_FLAG_NO_SMALL_BATCH | SRM_FLAG_NO_KSLICE | SRM_FLAG_NO_FUSED_FFN | SRM_FLAG_HEAD_PROJ;
  if (c.dtype != SRM_DTYPE_BF16 || (c.flags & kOff) || c.mixer != SRM_MIXER_MIXED || c.ffn_mult != 4) return false;
  if (c.d_model != 512 && (c.d_model != 1024 || R <= 16)) return false;
  if (m.row_clusters < 0)
    m.row_clusters = with_cluster_kernel(c, 1 << 20, [](auto* kernel, size_t smem) { return resident_clusters(kernel, cl::kThreads, smem); });
  return R <= (int64_t)m.row_clusters * (c.d_model == 1024 ? 16 : 64);
}
// What of the LM head the layers kernel of a pass does, too: nothing, the logits, the greedy selection, or both.
struct LmHead { bool here, select; float* logits; SelectOut out; };
// All layers and the final norm for rows [b0, b0 + R) of the state; leaves the normed rows in w.a, or goes on to the LM head.
int launch_layers_cluster(srm_model& m, srm_state& s, int64_t b0, int64_t R, int t, const int32_t* tok_in, const DecodeWs& w,
                          cudaStream_t st, const int32_t* ctr, const int32_t* pos, const LmHead& head) {
  const srm_config& c = m.cfg;
  const int d = c.d_model, F = (int)m.F();
  cl::Params p;
  p.R = (int)R; p.V = c.vocab; p.h = c.n_heads; p.n_ctx = c.n_ctx; p.L = c.n_layers; p.t = t;
  p.eps = c.ln_eps;
  p.rows = (int)((R + m.row_clusters - 1) / m.row_clusters);           // spread over all clusters: fewer rows to exchange in each
  p.tok_in = tok_in;
  p.E = reinterpret_cast<const bf16*>(m.ptr(-1, SRM_T_E));
  p.layer0 = layer0_weights(m);
  p.layer_bytes = layer_stride_bytes(m);
  p.S = static_cast<uint8_t*>(s.layer_ptr(0)) + (size_t)b0 * d * m.state_bytes();
  p.layer_stride = (int64_t)s.B * d * m.state_bytes();
  p.a = reinterpret_cast<bf16*>(w.a);
  p.lnf_g = m.fptr(-1, SRM_T_LNF_G); p.lnf_b = m.fptr(-1, SRM_T_LNF_B);
  p.status = s.status; p.ctr = ctr; p.pos = pos;
  p.head = head.here; p.select = head.select; p.logits = head.logits; p.out = head.out;
  LaunchScope scope(m, SRM_KERNEL_STEP_SMALL, st);
  CUtensorMap w1, w2, lm;
  int rc;
  if ((rc = make_tmap_kblocks(&w1, m.ptr(0, SRM_T_W1), F, d, cl::kTile, 1, c.n_layers, p.layer_bytes)) != SRM_OK) return rc;
  if ((rc = make_tmap_kblocks(&w2, m.ptr(0, SRM_T_W2), d, F, cl::kTile, 1, c.n_layers, p.layer_bytes)) != SRM_OK) return rc;
  if ((rc = make_tmap_kblocks(&lm, m.ptr(-1, SRM_T_W_LM), c.vocab, d, cl::kTile, 1, 1)) != SRM_OK) return rc;
  return with_cluster_kernel(c, p.rows, [&](auto* kernel, size_t smem) -> int {
    int rc2 = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), cl::kSmemBytes, true);
    if (rc2 != SRM_OK) return rc2;
    ClusterLaunch L((unsigned)((R + p.rows - 1) / p.rows), cl::kThreads, smem, st, false);
    SRM_CUDA(cudaLaunchKernelEx(&L.cfg, kernel, w1, w2, lm, p));
    return SRM_OK;
  });
}

// ---- a few rows: weights split between clusters of 16 CTAs, all layers in one kernel (layers_split.cuh) -------------
template <bool ALONE, typename Fn>
int with_split_kernel_t(const srm_config& c, Fn&& f) {
  constexpr size_t smem = sp::Shape<1024>::kSmem;
  if (c.state_dtype == SRM_DTYPE_FP16) return f(sp::layers_kernel<1024, ALONE, fp16>, smem);
  if (c.state_dtype == SRM_DTYPE_BF16) return f(sp::layers_kernel<1024, ALONE, bf16>, smem);
  return f(sp::layers_kernel<1024, ALONE, float>, smem);
}
template <typename Fn>
int with_split_kernel(const srm_config& c, int64_t R, Fn&& f) {
  return R == 1 ? with_split_kernel_t<true>(c, f) : with_split_kernel_t<false>(c, f);
}
// Whether a decode pass of R rows takes it: bf16 models with mixed heads, F = 4 d, 1024 channels, up to 16 rows. us per greedy step of 16
// layers, the single-kernel step / here: 1 row 181 / 140, 4 rows 186 / 147, 8 rows 190 / 149, 16 rows 202 / 157 (150, 154, 159 and 165
// with LM head and selection as kernels of their own); with 27 rows (two
// 16-row tiles, two rows per owner) it took 308, rows inside clusters 205. The words of the planes lie in the area of the
// partial products.
bool split_rows_ok(srm_model& m, int64_t R, const DecodeWs& w) {
  const srm_config& c = m.cfg;
  constexpr int kOff = SRM_FLAG_SIMT_GEMM | SRM_FLAG_NO_SMALL_BATCH | SRM_FLAG_NO_KSLICE | SRM_FLAG_NO_FUSED_FFN | SRM_FLAG_HEAD_PROJ;
  if (c.dtype != SRM_DTYPE_BF16 || (c.flags & kOff) || c.mixer != SRM_MIXER_MIXED || c.ffn_mult != 4 || c.d_model != 1024 || R > sp::kMaxRows) return false;
  if (m.split_clusters < 0)
    m.split_clusters = with_split_kernel(c, sp::kMaxRows, [](auto* kernel, size_t smem) { return resident_clusters(kernel, sp::kThreads, smem); });
  return m.split_clusters >= sp::kClusters && w.part != nullptr && sp::plane_bytes(R, c.d_model) <= w.part_bytes;
}
// All layers and the final norm for rows [b0, b0 + R) of the state; leaves the normed rows in w.a, or goes on to the LM head.
int launch_layers_split(srm_model& m, srm_state& s, int64_t b0, int64_t R, int t, const int32_t* tok_in, const DecodeWs& w,
                        cudaStream_t st, const int32_t* ctr, const int32_t* pos, const LmHead& head) {
  const srm_config& c = m.cfg;
  const int d = c.d_model, F = (int)m.F();
  sp::Params p;
  p.R = (int)R; p.V = c.vocab; p.h = c.n_heads; p.n_ctx = c.n_ctx; p.L = c.n_layers; p.t = t;
  p.eps = c.ln_eps;
  p.tok_in = tok_in;
  p.E = reinterpret_cast<const bf16*>(m.ptr(-1, SRM_T_E));
  p.layer0 = layer0_weights(m);
  p.layer_bytes = layer_stride_bytes(m);
  p.S = static_cast<uint8_t*>(s.layer_ptr(0)) + (size_t)b0 * d * m.state_bytes();
  p.layer_stride = (int64_t)s.B * d * m.state_bytes();
  p.a = reinterpret_cast<bf16*>(w.a);
  p.lnf_g = m.fptr(-1, SRM_T_LNF_G); p.lnf_b = m.fptr(-1, SRM_T_LNF_B);
  p.planes = reinterpret_cast<unsigned long long*>(w.part);
  p.cnt = reinterpret_cast<uint32_t*>(w.small);
  p.best = reinterpret_cast<unsigned long long*>(w.small + 64);
  static_assert(64 + sp::kMaxRows * 8 <= 256 && kSmallScratchBytes >= 256, "counters and maxima");
  p.status = s.status; p.ctr = ctr; p.pos = pos;
  p.head = head.here; p.select = head.select; p.logits = head.logits; p.out = head.out;
  SRM_CUDA(cudaMemsetAsync(w.small, 0, 256, st));
  LaunchScope scope(m, SRM_KERNEL_STEP_SMALL, st);
  CUtensorMap w1, w2, lm;
  int rc;
  if ((rc = make_tmap_layers(&lm, m.ptr(-1, SRM_T_W_LM), c.vocab, d, sp::Shape<1024>::kUpTiles * 8, 1, 0)) != SRM_OK) return rc;
  if ((rc = make_tmap_layers(&w1, m.ptr(0, SRM_T_W1), F, d, sp::Shape<1024>::kUpTiles * 8, c.n_layers, p.layer_bytes)) != SRM_OK) return rc;
  if ((rc = make_tmap_layers(&w2, m.ptr(0, SRM_T_W2), d, F, d / sp::kCluster, c.n_layers, p.layer_bytes)) != SRM_OK) return rc;
  return with_split_kernel(c, R, [&](auto* kernel, size_t smem) -> int {
    int rc2 = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), sp::kSmemBytes, true);
    if (rc2 != SRM_OK) return rc2;
    ClusterLaunch L(sp::kClusters, sp::kThreads, smem, st, true);
    SRM_CUDA(cudaLaunchKernelEx(&L.cfg, kernel, w1, w2, lm, p));
    return SRM_OK;
  });
}

// ---- small batches: the whole step in one cooperative kernel (step_small.cuh) ----------------------
struct SmallPlan { sb::Params p; size_t smem; };

// f(kernel) for the instance of the step kernel that the configuration takes.
template <int d, typename Fn>
int with_small_kernel_d(const srm_config& c, Fn&& f) {
  if (c.state_dtype == SRM_DTYPE_FP16) return f(sb::step_small_kernel<d, fp16>);
  if (c.state_dtype == SRM_DTYPE_BF16) return f(sb::step_small_kernel<d, bf16>);
  return f(sb::step_small_kernel<d, float>);
}
template <typename Fn>
int with_small_kernel(const srm_config& c, Fn&& f) {
  switch (c.d_model) {
    case 256: return with_small_kernel_d<256>(c, f);
    case 512: return with_small_kernel_d<512>(c, f);
    case 768: return with_small_kernel_d<768>(c, f);
    default: return with_small_kernel_d<1024>(c, f);
  }
}

// Both launch attributes of the kernel: all CTAs resident at once (it has grid-wide barriers), in clusters.
struct SmallLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  SmallLaunch(size_t smem, cudaStream_t st) {
    cfg.gridDim = dim3(sb::kGrid);
    cfg.blockDim = dim3(sb::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = sb::kCluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};

// Whether a batch of B samples takes the single-kernel step, and its shared-memory plan. Mixed heads, bf16 weights, at
// most 64 samples and 1024 channels (a multiple of 256), a device that holds all clusters at once; everything
// else takes the kernel-per-operation path.
bool small_step_plan(srm_model& m, int64_t B, SmallPlan* P) {
  const srm_config& c = m.cfg;
  if (c.dtype != SRM_DTYPE_BF16 || (c.flags & (SRM_FLAG_SIMT_GEMM | SRM_FLAG_NO_SMALL_BATCH | SRM_FLAG_HEAD_PROJ))) return false;
  if (c.mixer != SRM_MIXER_MIXED || B > sb::kMaxRows || c.d_model > 1024 || c.d_model % 256 || m.F() % 1024) return false;
  if (m.small_clusters < 0) {
    m.small_clusters = with_small_kernel(c, [&](auto* kernel) {
      int n = 0;
      if (ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), sb::kSmemBytes) != SRM_OK) return 0;
      SmallLaunch L(sb::kSmemBytes, nullptr);
      L.cfg.attrs = L.attr + 1;
      L.cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&n, kernel, &L.cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
      return n;
    });
  }
  return m.small_clusters >= sb::kClusters &&
         sb::smem_plan((int)B, c.d_model, (int)m.F(), m.state_bytes(), &P->p, &P->smem);
}

// What a decode pass of R rows runs; `whole`: the pass is its state's whole batch; `in_memory`: its step leaves logits in memory.
// `small`, `mid`: the plan where that kernel is taken.
enum DecodeRoute { kRouteKernels, kRouteStep, kRouteLayers, kRouteClusters, kRouteSplit };      // SRM_ROUTE_* of the C ABI
DecodeRoute decode_route(srm_model& m, int64_t R, bool whole, bool in_memory, const DecodeWs& w, SmallPlan* small, mid::Params* mid) {
  if (split_rows_ok(m, R, w)) return kRouteSplit;
  if (mid_rows_ok(m.cfg, R) && cluster_rows_ok(m, R)) {
    // 17 to 32 rows at d = 1024: the clusters gain 2 to 3 us per layer on the single-kernel step, which has the LM head inside; where that
    // writes logits, a large vocabulary makes up for it (us per step with logits and with top-p, 32 rows, single-kernel step / clusters: V = 32000,
    // 16 layers 249 / 210 and 259 / 212, 3 layers 81 / 72 and 91 / 71; V = 131072, 8 layers 216 / 225 and 404 / 433).
    const bool step = whole && in_memory && !cl::has_head(m.cfg.d_model) && m.cfg.vocab > 8192 * std::max(8, m.cfg.n_layers);
    return step && small_step_plan(m, R, small) ? kRouteStep : kRouteClusters;
  }
  if (whole && small_step_plan(m, R, small)) return kRouteStep;
  return mid_plan(m, R, w, mid) ? kRouteLayers : kRouteKernels;
}

// Whether the LM head runs in the layers kernel of a pass, too, and so the greedy selection or the logits for another. A separate LM head
// starts later, but shares the vocabulary out over the device, where a cluster reads all of it by itself. us per step of 8 layers at d = 512,
// separate / inside, greedy without logits: V = 8000 1 row 47 / 45, 224 rows 65 / 63, 448 rows 94 / 98; V = 16000 48 / 48, 66 / 67,
// 98 / 106; V = 32000 52 / 57, 70 / 76, 105 / 125; V = 131072 84 / 103, 95 / 124, 146 / 223. Logits in memory cost the separate one tiles of 256
// rows for a few, and greedy selection a launch more: V = 131072, 16 / 112 rows, logits 137 / 104 and 157 / 111, top-p 354 / 292
// and 364 / 394 (the single-kernel step 145 and 329 with 16). Top-k has a selection of its own in a separate LM head, three launches more:
// V = 8000, 16 rows 78 / 57 (one layer 48 / 26, the single-kernel step 34), V = 131072 111 / about 150.
// Weights split between clusters: all CTAs share the vocabulary. 16 layers, d = 1024, V = 32000, 1 / 16 rows: logits 155 / 138 and 178 /
// 157, top-p 161 / 154 and 175 / 177, top-k 167 / 152 and 193 / 172; V = 131072, 8 layers, logits 172 / 112 and 222 / 123.
constexpr int kHeadInsideVocab = 12288, kTopkInsideVocab = 32768;
bool head_in_layers(const srm_model& m, const srm_sampling& samp, const float* logits_out, DecodeRoute route, int64_t R) {
  const srm_config& c = m.cfg;
  const bool own_topk = can_fuse_topk(m, samp, logits_out);
  if (route == kRouteSplit) return !own_topk || c.vocab <= kTopkInsideVocab;
  if (route != kRouteClusters || !cl::has_head(c.d_model)) return false;
  if (c.vocab <= kHeadInsideVocab) return true;
  return !own_topk && !can_fuse_greedy(m, samp, logits_out) && R <= (int64_t)(samp.mode == SRM_SELECT_GREEDY ? 16 * m.row_clusters : 16);
}

// One decode step for rows [b0, b0 + R) of the state.
int decode_chunk(srm_model& m, srm_state& s, int64_t b0, int64_t R, const int32_t* tok_in, const srm_sampling& samp,
                 int step, const SelectOut& out_all, float* logits_out, const DecodeWs& w, cudaStream_t st,
                 const int32_t* ctr) {
  const srm_config& c = m.cfg;
  const int d = c.d_model;
  const int64_t F = m.F();
  const int t = (int)(s.pos < c.n_ctx ? s.pos : c.n_ctx - 1);
  const int32_t* pos = s.ragged ? s.pos_dev + b0 : nullptr;       // samples of different lengths: a position per row
  int rc;
  PartialSum ps_none, ps;
  int k_slices = 1;
  mid::Params mp;
  SelectOut o = out_all;
  o.last_tok += b0;
  if (o.tok_out) o.tok_out += b0;
  if (o.store) o.store += b0 * o.store_stride;
  if (o.pos) o.pos += b0;
  if (o.thr_out) o.thr_out += b0;
  SmallPlan small;
  const DecodeRoute route = decode_route(m, R, false, false, w, &small, &mp);
  const bool one_kernel = route != kRouteKernels;
  const bool greedy = samp.mode == SRM_SELECT_GREEDY, here = head_in_layers(m, samp, logits_out, route, R);
  const bool topk = !here && can_fuse_topk(m, samp, logits_out);
  // logits in memory: the caller wants them, or the selection reads them there
  float* lg = logits_out != nullptr ? logits_out + b0 * c.vocab : can_fuse_greedy(m, samp, logits_out) || topk ? nullptr : w.logits;
  const LmHead head{here, here && greedy, here ? lg : nullptr, o};
  if (route == kRouteSplit) rc = launch_layers_split(m, s, b0, R, t, tok_in + b0, w, st, ctr, pos, head);
  else if (route == kRouteClusters) rc = launch_layers_cluster(m, s, b0, R, t, tok_in + b0, w, st, ctr, pos, head);
  else rc = one_kernel ? launch_layers_mid(m, s, b0, R, t, tok_in + b0, w, mp, st, ctr, pos) : SRM_OK;
  if (rc) return rc;
  if (here) return greedy ? SRM_OK : launch_select(m, R, lg, samp, samp.sample_idx_base + (uint64_t)b0, step, o, s.status, st);
  // the down projection shares K out between CTA pairs where that is the faster kernel for R rows
  bool split = false;
  if (!one_kernel && w.order != nullptr && F % tc::BK == 0) {
    if ((rc = ensure_tc_ready(m))) return rc;
    tc::SplitPlan P;
    const int64_t tiles = ((R + tc::BM - 1) / tc::BM) * ((d + tc::BN - 1) / tc::BN);
    split = tc::split_plan(tiles, (int)(F / tc::BK), m.tc_clusters, &P) && tc::split_saved_kb(P) >= tc::kSplitWorthKb;
  }
  // the feed-forward block as one kernel: its per-layer counters sit in the logits area, which nothing uses before
  // the LM head
  const size_t ready_layer = ffn_ready_bytes(R, F);
  bool fused_ffn = !one_kernel && !(c.flags & SRM_FLAG_NO_FUSED_FFN) && ffn_fused_shape_ok(m, R) &&
                   ready_layer * c.n_layers <= align_up((size_t)w.rows * c.vocab * 4, 256);
  if (fused_ffn) {
    if ((rc = ensure_tc_ready(m))) return rc;
    fused_ffn = ffn_fused_worthwhile(m, R);
  }
  if (fused_ffn) SRM_CUDA(cudaMemsetAsync(w.logits, 0, ready_layer * c.n_layers, st));
  else if (split) SRM_CUDA(cudaMemsetAsync(w.order, 0, w.order_bytes, st));
  // A small pass (the down projection has less than half as many tiles as there are CTA pairs): its K dimension is
  // cut into ranges so that all pairs work on it; the partial products go to planes of their own in the workspace
  // and the next consumer of x (the next layer's mixer, the final norm) adds them in a fixed order.
  const int64_t plane_rows = (R + tc::BM - 1) / tc::BM * tc::BM;
  if (!one_kernel && !fused_ffn && !split && w.part != nullptr) {
    if ((rc = ensure_tc_ready(m))) return rc;
    k_slices = down_k_slices(plane_rows / tc::BM * ((d + tc::BN - 1) / tc::BN), (int)(F / tc::BK), m.tc_clusters);
    while (k_slices > 1 && (size_t)k_slices * plane_rows * d * 4 > w.part_bytes) k_slices /= 2;
  }
  if (!one_kernel && k_slices > 1) ps = PartialSum{w.part, k_slices, plane_rows * (int64_t)d, nullptr};
  for (int l = 0; !one_kernel && l < c.n_layers; ++l) {
    uint8_t* Sl = static_cast<uint8_t*>(s.layer_ptr(l)) + (size_t)b0 * d * m.state_bytes();
    if (c.mixer != SRM_MIXER_MIXED) {
      if ((rc = launch_mixer_variant(m, l, t, R, l == 0 ? tok_in + b0 : nullptr, 1, w.x, w.a, d, Sl, s.plane_elems(), s.status,
                                     st, ctr))) return rc;
    } else if (m.head_proj()) {
      if ((rc = launch_mixer_block_proj(m, l, t, R, R, 1, l == 0 ? tok_in + b0 : nullptr, w.x, Sl, w.a, w.q, s.status, st, ctr, pos))) return rc;
    } else {
      PartialSum pl = l > 0 ? ps : ps_none;                // what layer l - 1's down projection left in planes
      if (l > 0) pl.bias = m.fptr(l - 1, SRM_T_B2);
      if ((rc = launch_mixer(m, l, t, R, l == 0 ? tok_in + b0 : nullptr, w.x, Sl, w.a, s.status, st, ctr, pos, pl))) return rc;
    }
    if (fused_ffn) {
      int32_t* ready = reinterpret_cast<int32_t*>(reinterpret_cast<uint8_t*>(w.logits) + (size_t)l * ready_layer);
      rc = launch_ffn_fused(m, l, R, w.a, w.H, w.x, ready, s.status, st);
      if (rc == SRM_OK) continue;
      if (rc != SRM_ERR_UNSUPPORTED) return rc;
      fused_ffn = false;                                   // (no plan for this shape: decided at the first layer)
      if (split) SRM_CUDA(cudaMemsetAsync(w.order, 0, w.order_bytes, st));
    }
    if ((rc = launch_gemm(m, kEpiBiasGelu, R, F, d, w.a, m.ptr(l, SRM_T_W1), m.fptr(l, SRM_T_B1), w.H, s.status, st))) return rc;
    rc = split ? launch_gemm_splitk(m, R, d, F, w.H, m.ptr(l, SRM_T_W2), m.fptr(l, SRM_T_B2), w.x, w.order, s.status, st, true)
               : SRM_ERR_UNSUPPORTED;
    if (rc == SRM_ERR_UNSUPPORTED) {
      if (k_slices > 1) {
        LaunchScope scope(m, SRM_KERNEL_GEMM_DOWN, st);
        rc = launch_gemm_tc(m, kEpiPlain, R, d, F, w.H, m.ptr(l, SRM_T_W2), nullptr, w.part, s.status, st, k_slices, plane_rows);
      } else {
        rc = launch_gemm(m, kEpiBiasResidual, R, d, F, w.H, m.ptr(l, SRM_T_W2), m.fptr(l, SRM_T_B2), w.x, s.status, st);
      }
    }
    if (rc) return rc;
  }
  if (ps.part != nullptr) ps.bias = m.fptr(c.n_layers - 1, SRM_T_B2);
  if (!one_kernel && (rc = launch_final_norm(m, w.x, R, 1, 0, w.a, st, nullptr, ps))) return rc;
  if (can_fuse_greedy(m, samp, logits_out)) return launch_lm_head_greedy(m, R, w.a, w.logits, o, s.status, st);
  if (topk)
    return launch_lm_head_topk(m, R, w.a, w.logits, w.H, s.thr + b0, samp, samp.sample_idx_base + (uint64_t)b0, step, o,
                               s.status, s.status + kCtrHandedBack, st);
  if ((rc = launch_gemm(m, kEpiPlain, R, c.vocab, d, w.a, m.ptr(-1, SRM_T_W_LM), nullptr, lg, s.status, st))) return rc;
  return launch_select(m, R, lg, samp, samp.sample_idx_base + (uint64_t)b0, step, o, s.status, st);
}

// One decode step of all B <= 64 samples of the state. SRM_ERR_UNSUPPORTED: take the ordinary path.
int decode_step_small(srm_model& m, srm_state& s, SmallPlan& P, const int32_t* tok_in, const srm_sampling& samp, int step,
                      const SelectOut& out, float* logits_out, const DecodeWs& w, cudaStream_t st, const int32_t* ctr) {
  const srm_config& c = m.cfg;
  sb::Params& p = P.p;
  p.B = (int)s.B; p.d = c.d_model; p.F = (int)m.F(); p.V = c.vocab; p.h = c.n_heads; p.n_ctx = c.n_ctx; p.L = c.n_layers;
  p.t = (int)(s.pos < c.n_ctx ? s.pos : c.n_ctx - 1);
  p.eps = c.ln_eps;
  p.tok_in = tok_in;
  p.E = reinterpret_cast<const bf16*>(m.ptr(-1, SRM_T_E));
  p.W_lm = reinterpret_cast<const bf16*>(m.ptr(-1, SRM_T_W_LM));
  p.lnf_g = m.fptr(-1, SRM_T_LNF_G); p.lnf_b = m.fptr(-1, SRM_T_LNF_B);
  p.layer0 = layer0_weights(m);
  p.layer_bytes = layer_stride_bytes(m);
  p.S = s.layer_ptr(0);
  p.layer_stride = (int64_t)s.B * c.d_model * m.state_bytes();
  p.x = w.x; p.H = reinterpret_cast<bf16*>(w.H);
  p.best = reinterpret_cast<unsigned long long*>(w.small);
  p.bar = reinterpret_cast<uint32_t*>(w.small + (size_t)sb::kMaxRows * 8);
  p.status = s.status;
  p.ctr = ctr;
  p.pos = s.ragged ? s.pos_dev : nullptr;
  p.greedy = samp.mode == SRM_SELECT_GREEDY ? 1 : 0;
  p.logits = logits_out != nullptr ? logits_out : (p.greedy ? nullptr : w.logits);
  p.out = out;
  SRM_CUDA(cudaMemsetAsync(w.small, 0, kSmallScratchBytes, st));
  int rc;
  {
    LaunchScope scope(m, SRM_KERNEL_STEP_SMALL, st);
    rc = with_small_kernel(c, [&](auto* kernel) -> int {
      int rc2 = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), sb::kSmemBytes);
      if (rc2 != SRM_OK) return rc2;
      SmallLaunch L(P.smem, st);
      SRM_CUDA(cudaLaunchKernelEx(&L.cfg, kernel, p));
      return SRM_OK;
    });
  }
  if (rc != SRM_OK || p.greedy) return rc;
  return launch_select(m, s.B, p.logits, samp, samp.sample_idx_base, step, out, s.status, st);
}

// Rows per decode pass for a batch of B rows when the workspace holds up to `fit` rows. Up to kOnePassRows the
// batch runs as one pass. Beyond that it is cut into the fewest equal passes of at most kMaxPassRows rows, each a
// whole number of 256-row tiles: a larger pass pushes the activations of a layer (H, x, a: 14 KB per row for
// d = 1024) out of L2 between the GEMMs, a smaller one leaves rounds of tiles partly empty. Measured at 32768
// rows, d = 1024: 4096 / 5888 / 8192 / 9472 / 16384 / 32768 rows per pass take 11.95 / 11.75 / 11.35 / 11.24 /
// 11.49 / 11.68 ms per step; at 16384 rows, d = 1536: 4608 / 9472 / 16384 rows take 17.67 / 16.84 / 17.33 ms.
constexpr int64_t kOnePassRows = 12288, kMaxPassRows = 10240;
int64_t choose_pass_rows(int64_t B, int64_t fit) {
  if (fit < B && fit < kMaxPassRows) return fit;              // the workspace decides
  if (B <= kOnePassRows && fit >= B) return B;
  const int64_t passes = (B + kMaxPassRows - 1) / kMaxPassRows;
  int64_t rows = (B + passes - 1) / passes;
  rows = (rows + tc::BM - 1) / tc::BM * tc::BM;
  return rows < fit ? rows : fit;
}

// `ctr` non-null: position, Philox step and store column come from the device-side counters (graph replay).
int decode_step_impl(srm_model* m, srm_state* s, const int32_t* d_tok_in, const srm_sampling* samp, int step,
                     int32_t* d_tok_out, int32_t* d_store, int64_t store_stride, int64_t store_col,
                     float* d_logits_out, void* d_ws, size_t ws_bytes, cudaStream_t st, const int32_t* ctr = nullptr) {
  if (m == nullptr || s == nullptr || s->m != m || d_ws == nullptr) return SRM_ERR_INVALID_ARG;
  int rc = check_sampling(*m, samp);
  if (rc) return rc;
  if (!aligned(d_ws, 256) || !aligned(d_tok_in, 4) || !aligned(d_tok_out, 4) || !aligned(d_logits_out, 16)) return SRM_ERR_ALIGNMENT;
  if (s->pos >= m->cfg.n_ctx) return SRM_ERR_CTX_OVERFLOW;
  const int64_t fit = fit_rows(ws_bytes, s->B, decode_need, *m, 0);
  if (fit < 1) return SRM_ERR_BUFFER_TOO_SMALL;
  const int64_t rows = choose_pass_rows(s->B, fit);
  const DecodeWs w = carve_decode(*m, d_ws, rows);
  const int32_t* tok_in = d_tok_in != nullptr ? d_tok_in : s->last_tok;
  SelectOut out{s->last_tok, d_tok_out, d_store, store_stride, store_col, 1, ctr, s->ragged ? s->pos_dev : nullptr,
                nullptr, nullptr, samp->mode == SRM_SELECT_TOPK ? s->thr : nullptr};
  SmallPlan small;
  mid::Params mid;
  const bool in_memory = !can_fuse_greedy(*m, *samp, d_logits_out) && !can_fuse_topk(*m, *samp, d_logits_out);
  if (rows >= s->B && decode_route(*m, s->B, true, in_memory, w, &small, &mid) == kRouteStep) {
    rc = decode_step_small(*m, *s, small, tok_in, *samp, step, out, d_logits_out, w, st, ctr);
    if (rc != SRM_ERR_UNSUPPORTED) {
      if (rc == SRM_OK) s->pos += 1;
      return rc;
    }
  }
  for (int64_t b0 = 0; b0 < s->B; b0 += rows) {
    const int64_t R = (s->B - b0 < rows) ? s->B - b0 : rows;
    if ((rc = decode_chunk(*m, *s, b0, R, tok_in, *samp, step, out, d_logits_out, w, st, ctr))) return rc;
  }
  s->pos += 1;
  return SRM_OK;
}

}  // namespace
