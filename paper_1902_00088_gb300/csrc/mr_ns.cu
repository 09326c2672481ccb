// Launchers of the Navier-Stokes kernels of Sec. 4 (the stages of both forms and the
// shock-capturing filter), 2D, Bs 17 and 33.
#include "mr_launch.cuh"
#include "mr_ns.cuh"

namespace mr {

// One stage of either form: stage s reads y, Ya, Yb, Ya and writes Ya, Yb, Ya, (Yb:
// the new state's copy for the filter).
template <int B, bool SKEW, typename TS, typename TY>
static void stage_form(const PoolView& pv, const Fields& f, int stage, const StageArgs& sa,
                       const LaunchCfg& lc, cudaStream_t st) {
  constexpr int threads = SKEW ? NssCfg<B, TY>::NT : NsCfg<B, TY>::NT;
  constexpr size_t smem = SKEW ? NssSmem<B, TY>::BYTES : NsSmem<B, TY>::BYTES;
  TY* ynext = (TY*)(stage == 1 || stage == 3 ? f.Yb : f.Ya);
  auto go = [&](auto k, auto src) {
    prep_smem(k, smem);
    launch_k(lc.pdl, k, persistent_grid(k, threads, smem, lc, lc.grid_mult), threads, smem, st, pv, src,
             (TS*)f.y, (TS*)f.acc, ynext, (TY*)f.Yn, stage, sa);
  };
  const TY* src = (const TY*)(stage == 2 ? f.Yb : f.Ya);
  if constexpr (SKEW) {
    if (stage == 0) go(k_stage_nss<B, TS, TY, TS>, (const TS*)f.y);
    else go(k_stage_nss<B, TS, TY, TY>, src);
  } else {
    if (stage == 0) go(k_stage_ns<B, TS, TY, TS>, (const TS*)f.y);
    else go(k_stage_ns<B, TS, TY, TY>, src);
  }
  count_launch();
}

template <int B, bool SKEW>
static void stage_prec_ns(const PoolView& pv, const Fields& f, int stage, const StageArgs& sa,
                          const LaunchCfg& lc, cudaStream_t st) {
  switch (pv.prec) {
    case MR_PREC_FP64: stage_form<B, SKEW, double, double>(pv, f, stage, sa, lc, st); break;
    case MR_PREC_FP32: stage_form<B, SKEW, float, float>(pv, f, stage, sa, lc, st); break;
    default: stage_form<B, SKEW, double, float>(pv, f, stage, sa, lc, st); break;
  }
}
template <int B>
void launch_stage_ns(const PoolView& pv, const Fields& f, int stage, const StageArgs& sa, const LaunchCfg& lc,
                     cudaStream_t st) {
  stage_prec_ns<B, false>(pv, f, stage, sa, lc, st);
}
template <int B>
void launch_stage_nss(const PoolView& pv, const Fields& f, int stage, const StageArgs& sa, const LaunchCfg& lc,
                      cudaStream_t st) {
  stage_prec_ns<B, true>(pv, f, stage, sa, lc, st);
}
#define MR_NS_STAGE(B)                                                                                                \
  template void launch_stage_ns<B>(const PoolView&, const Fields&, int, const StageArgs&, const LaunchCfg&,           \
                                   cudaStream_t);                                                                     \
  template void launch_stage_nss<B>(const PoolView&, const Fields&, int, const StageArgs&, const LaunchCfg&,          \
                                    cudaStream_t);
MR_NS_STAGE(17)
MR_NS_STAGE(33)

template <int B, typename TS, typename TC, int KIND>
static void filter_impl(const PoolView& pv, const Fields& f, bool copy, const LaunchCfg& lc, cudaStream_t st) {
  constexpr int threads = kFilterThreads;
  constexpr size_t smem = FilterSmem<B, TC>::BYTES;
  if (copy) {
    launch_k(lc.pdl, k_state_copy<TS, TC>, lc.num_sms * 8, 256, 0, st, pv, (const TS*)f.y, (TC*)f.Yb);
    count_launch();
  }
  auto k = k_filter<B, TS, TC, KIND>;
  prep_smem(k, smem);
  launch_k(lc.pdl, k, persistent_grid(k, threads, smem, lc, lc.grid_mult), threads, smem, st, pv,
           (const TC*)f.Yb, (TS*)f.y);
  count_launch();
}

template <int B, int KIND>
static void filter_prec(const PoolView& pv, const Fields& f, bool copy, const LaunchCfg& lc, cudaStream_t st) {
  switch (pv.prec) {
    case MR_PREC_FP64: filter_impl<B, double, double, KIND>(pv, f, copy, lc, st); break;
    case MR_PREC_FP32: filter_impl<B, float, float, KIND>(pv, f, copy, lc, st); break;
    default: filter_impl<B, double, float, KIND>(pv, f, copy, lc, st); break;
  }
}

void launch_filter(const PoolView& pv, const Fields& f, bool copy, const LaunchCfg& lc, cudaStream_t st) {
  const bool skew = pv.rhs_kind == MR_RHS_NS_SKEW;
  if (pv.Bs == 17) {
    if (skew) filter_prec<17, MR_RHS_NS_SKEW>(pv, f, copy, lc, st);
    else filter_prec<17, MR_RHS_NS>(pv, f, copy, lc, st);
  } else {
    if (skew) filter_prec<33, MR_RHS_NS_SKEW>(pv, f, copy, lc, st);
    else filter_prec<33, MR_RHS_NS>(pv, f, copy, lc, st);
  }
}

}  // namespace mr
