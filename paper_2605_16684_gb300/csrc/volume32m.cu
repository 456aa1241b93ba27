// volume32m.cu -- the mixed-precision volume kernel without a background or
// relative to a moving one (a flow carried by the background, e.g. the channel's
// balanced jet: FP32 pairs formed as differences against the background's
// fluxes, pair32bgm).
#include "volume_impl.cuh"
#include "volume_mixed.cuh"

cudaError_t esdg_launch_volume_mixed_other(const EsdgGrid& g, const EsdgLGL& L, const EsdgPhys& P,
                                           int mode, const EsdgVolArgs& a, cudaStream_t s) {
  using namespace esdg_vol;
  return for_order(g.N, cudaErrorInvalidValue, [&](auto n) {
    if (a.bgq)
      return mode ? launch_volume32<n.value, 1, 2>(g, P, L, a, s)
                  : launch_volume32<n.value, 0, 2>(g, P, L, a, s);
    return mode ? launch_volume32<n.value, 1, 0>(g, P, L, a, s)
                : launch_volume32<n.value, 0, 0>(g, P, L, a, s);
  });
}
