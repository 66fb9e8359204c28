// fdlbm_step_f64.cu -- the FP64-storage step's launches (kernels in fdlbm_fx64.cuh).
#include "fdlbm_fx64.cuh"

namespace fdlbm {

namespace {

template <typename K, typename... A>
cudaError_t launch_dependent(K kernel, dim3 grid, int threads, int smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

dim3 tiles(const Grid& g, int tw, int th) { return dim3((g.nx + tw - 1) / tw, (g.ny + th - 1) / th); }

template <int TW, int TH, int MINB>
cudaError_t launch_fx(const void* f, void* fn, const Grid& g, const Coeffs& c, unsigned* health, cudaStream_t s) {
  constexpr int smem = sizeof(FxTile<TW, TH>);
  static std::atomic<unsigned long long> attr{0};
  const cudaError_t e = allow_dynamic_smem(k_step_fx<TW, TH, MINB>, smem, attr);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_step_fx<TW, TH, MINB>, tiles(g, TW, TH), TW * TH, smem, s, static_cast<const double*>(f),
                          static_cast<double*>(fn), g, c, health);
}
template <int TW, int TH, int PPT, int MINB>
cudaError_t launch_fx_small(const void* f, void* fn, const Grid& g, const Coeffs& c, unsigned* health,
                            cudaStream_t s) {
  using S = FxSmall<TW, TH, PPT>;
  static std::atomic<unsigned long long> attr{0};
  const cudaError_t e = allow_dynamic_smem(k_step_fx_small<TW, TH, PPT, MINB>, sizeof(S), attr);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_step_fx_small<TW, TH, PPT, MINB>, tiles(g, TW, TH), S::NT, sizeof(S), s,
                          static_cast<const double*>(f), static_cast<double*>(fn), g, c, health);
}
template <int TW, int TH, int MINB>
cudaError_t prepare_batch_t() {
  static std::atomic<unsigned long long> attr{0};
  return allow_dynamic_smem(k_step_batch_fx<TW, TH, MINB>, sizeof(FxTile<TW, TH>), attr);
}
template <int TW, int TH, int MINB>
cudaError_t launch_batch_fx(const BatchMember* mem, int nmem, long long n, unsigned long long step, const Coeffs& c,
                            cudaStream_t s) {
  const cudaError_t e = prepare_batch_t<TW, TH, MINB>();
  if (e != cudaSuccess) return e;
  k_step_batch_fx<TW, TH, MINB><<<dim3((unsigned)n), TW * TH, sizeof(FxTile<TW, TH>), s>>>(mem, nmem, step, c);
  return cudaGetLastError();
}

}  // namespace

// Five shapes serve the variants: every shape gives the same bits, and a larger tile than 32 x 8 does not
// fit its planes and powers twice per SM. On a grid of up to kF64SmallSites the large tiles leave most SMs idle
// (400 x 4: 40 us per step against 13.9 with 8 x 4 tiles; 200 x 200: 62.6 against 52.6), so it gets the 8 x 4
// tile instead; at 333 x 333 it is 121 against 94. The 32 x 8 shape at three CTAs per SM spills (2048 x 2048: 2.48 against
// 2.43 ms per step), but takes 305 to 456 tiles in one wave instead of two (500 x 200: 83 against 87 us).
cudaError_t launch_step_f64(int variant, const void* f, void* fn, const Grid& g, const Coeffs& c, unsigned* health,
                          cudaStream_t s) {
  switch (variant_kernel(FDLBM_FP64, variant, (long long)g.nx * g.ny)) {
    case V_RP8x4: return launch_fx_small<4, 4, 1, 2>(f, fn, g, c, health, s);
    case V_RP16x4: return launch_fx_small<8, 4, 2, 4>(f, fn, g, c, health, s);
    case V_T32x4: return launch_fx<32, 4, 4>(f, fn, g, c, health, s);
    case V_T32x8: return launch_fx<32, 8, 3>(f, fn, g, c, health, s);
    default: return launch_fx<32, 8, 2>(f, fn, g, c, health, s);
  }
}

cudaError_t prepare_batch_f64(int variant) {
  return batch_kernel(FDLBM_FP64, variant) == V_T32x4 ? prepare_batch_t<32, 4, 4>() : prepare_batch_t<32, 8, 2>();
}
cudaError_t launch_batch_f64(int variant, const BatchMember* mem, int nmem, long long n, unsigned long long step,
                             const Coeffs& c, cudaStream_t s) {
  return batch_kernel(FDLBM_FP64, variant) == V_T32x4 ? launch_batch_fx<32, 4, 4>(mem, nmem, n, step, c, s)
                                                      : launch_batch_fx<32, 8, 2>(mem, nmem, n, step, c, s);
}

}  // namespace fdlbm
