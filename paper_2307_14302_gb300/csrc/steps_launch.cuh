// steps_launch.cuh -- launchers of the small-mesh kernel, instantiated per precision policy by
// steps_mixed.cu and steps_fp64.cu.
#pragma once
#include "steps.cuh"

namespace dg {
template <class Pol>
struct StepsKernel {
  int p, flux, ft;
  bool (*fit)(int ctas, int wpc, int nrec);
  cudaError_t (*launch)(const StageArgs<Pol>& a, const StepsArgs& st, int ctas, int wpc, cudaStream_t s);
};
template <class Pol, int P, int FLUX, int FT>
constexpr StepsKernel<Pol> steps_entry() {
  return {P, FLUX, FT, steps_fit_one<P, FLUX, Pol, FT>, steps_launch_one<P, FLUX, Pol, FT>};
}
// as the tile form: the narrowest specialised instantiation that covers the run, else the generic
template <class Pol>
const StepsKernel<Pol>& steps_find(int p, int flux, int feat) {
  static const StepsKernel<Pol> generic[4] = {steps_entry<Pol, 1, 0, FT_ALL>(), steps_entry<Pol, 1, 1, FT_ALL>(),
                                              steps_entry<Pol, 2, 0, FT_ALL>(), steps_entry<Pol, 2, 1, FT_ALL>()};
  if constexpr (sizeof(typename Pol::T) == 4) {
#define DG_STEPS_SPEC(P, FLUX, FT) steps_entry<Pol, P, FLUX, FT>(),
    static const StepsKernel<Pol> spec[] = {DG_SPECIALISED(DG_STEPS_SPEC)};
#undef DG_STEPS_SPEC
    const int ft = tile_spec_features(p, flux, feat);
    for (const auto& k : spec)
      if (k.p == p && k.flux == flux && k.ft == ft) return k;
  }
  return generic[(p == 1 ? 0 : 2) + (flux ? 1 : 0)];
}
}  // namespace dg

#define DG_DEFINE_STEPS_LAUNCHERS(POL)                                                                       \
  template <>                                                                                                \
  bool steps_fit<POL>(int p, int flux, int feat, int ctas, int wpc, int nrec) {                              \
    return steps_find<POL>(p, flux, feat).fit(ctas, wpc, nrec);                                              \
  }                                                                                                          \
  template <>                                                                                                \
  cudaError_t launch_steps<POL>(int p, int flux, int feat, const StageArgs<POL>& a, const StepsArgs& st,     \
                                int ctas, int wpc, cudaStream_t s) {                                         \
    return steps_find<POL>(p, flux, feat).launch(a, st, ctas, wpc, s);                                       \
  }                                                                                                          \
  template <>                                                                                                \
  cudaError_t upload_steps_tables<POL>(int p, const RefTab<float>& tf, const RefTab<double>& td) {           \
    const cudaError_t e = cudaMemcpyToSymbol(c_tab_f, &tf, sizeof(RefTab<float>), p * sizeof(RefTab<float>)); \
    return e != cudaSuccess ? e : cudaMemcpyToSymbol(c_tab_d, &td, sizeof(RefTab<double>), p * sizeof(RefTab<double>)); \
  }
