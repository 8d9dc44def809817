// tile_spec.cu -- specialised instantiations of the mixed-precision tile kernel.
//
// Each instantiation compiles in only the features of its set (Feature bits): the code of
// absent boundary kinds, forcing kinds, friction laws and stage-weight kinds, and their run-time
// tests, are left out, which shortens the kernel's instruction stream and its code.  A run
// whose features a set covers is launched with the narrowest such instantiation; any other run
// uses the generic one (tile_mixed.cu).
#include <algorithm>

#include "tile_launch.cuh"

namespace dg {
namespace {

using Kernel = void (*)(const StageArgs<Mixed>);
struct Spec {
  int p, flux, ft;
  Kernel k;
  int smem;  // dynamic shared memory per warp
};
template <int P, int FLUX, int FT>
constexpr Spec spec() {
  return {P, FLUX, FT, tile_kernel<P, FLUX, Mixed, FT>, tile_smem_bytes<P, Mixed, FT>(32)};
}
#define DG_SPEC(P, FLUX, FT) spec<P, FLUX, FT>(),
const Spec kSpecs[] = {DG_SPECIALISED(DG_SPEC)};
#undef DG_SPEC

int bits(int x) {
  int n = 0;
  for (; x; x &= x - 1) ++n;
  return n;
}
// the narrowest instantiation that covers feat, or null
const Spec* find_spec(int p, int flux, int feat) {
  const Spec* best = nullptr;
  for (const Spec& sp : kSpecs)
    if (sp.p == p && sp.flux == flux && ft_covers(sp.ft, feat) && (!best || bits(sp.ft) < bits(best->ft)))
      best = &sp;
  return best;
}
int smem_bytes(const Spec& sp, int block) { return sp.smem * (block / 32); }

}  // namespace

cudaError_t launch_tile_spec(int p, int flux, int feat, const StageArgs<Mixed>& a, int grid, int block,
                             cudaStream_t s) {
  const Spec* sp = find_spec(p, flux, feat);
  if (!sp) return cudaErrorNotSupported;
  return launch_pdl(sp->k, grid, block, smem_bytes(*sp, block), s, a);
}

int tile_spec_features(int p, int flux, int feat) {
  const Spec* sp = find_spec(p, flux, feat);
  return sp ? sp->ft : -1;
}

int tile_spec_blocks_per_sm(int p, int flux, int feat, int block) {
  const Spec* sp = find_spec(p, flux, feat);
  if (!sp) return -1;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sp->k, block, smem_bytes(*sp, block)) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t upload_tile_spec_tables(int p, const RefTab<float>& tf, const RefTab<double>& td) {
  cudaError_t e = cudaMemcpyToSymbol(c_tab_f, &tf, sizeof(RefTab<float>), p * sizeof(RefTab<float>));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_tab_d, &td, sizeof(RefTab<double>), p * sizeof(RefTab<double>));
  if (e != cudaSuccess) return e;
  int dev = 0, optin = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  for (const Spec& sp : kSpecs)
    if ((e = tile_smem_limit(sp.k, optin, smem_bytes(sp, 256))) != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace dg
