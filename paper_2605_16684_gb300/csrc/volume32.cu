// volume32.cu -- mixed-precision instantiations (FP32 pairs, FP64 state and
// pressure recovery) of the flux-differencing volume kernel with a background at
// rest: single-mesh launches and the batched kernel.
#include "volume_impl.cuh"
#include "volume_mixed.cuh"

cudaError_t esdg_launch_volume_mixed(const EsdgGrid& g, const EsdgLGL& L, const EsdgPhys& P,
                                     int mode, const EsdgVolArgs& a, cudaStream_t s) {
  if (!a.bg || a.bgq) return esdg_launch_volume_mixed_other(g, L, P, mode, a, s);
  return esdg_vol::for_order(g.N, cudaErrorInvalidValue, [&](auto n) {
    return mode ? esdg_vol::launch_volume32<n.value, 1, 1>(g, P, L, a, s)
                : esdg_vol::launch_volume32<n.value, 0, 1>(g, P, L, a, s);
  });
}

// what: 0 launch (returns 0 / -1), 1 elements per tile, 2 CTAs per SM
int esdg_volume_batch_mixed(int what, int N, const EsdgMember* members,
                          const int2* tiles, const int* ntiles, int grid, const EsdgLGL& L,
                          double A, double B, cudaStream_t s) {
  return esdg_vol::for_order(N, -1, [&](auto n) {
    return esdg_vol::batch_volume32<n.value>(what, members, tiles, ntiles, grid, L, A, B, s);
  });
}
