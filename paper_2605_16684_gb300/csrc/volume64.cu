// volume64.cu -- FP64 instantiations of the flux-differencing volume kernel:
// single-mesh launches and the batched kernel.
#include "volume_fp64.cuh"
#include "volume_impl.cuh"

cudaError_t esdg_launch_volume_f64(const EsdgGrid& g, const EsdgLGL& L, const EsdgPhys& P, int mode,
                                   const EsdgVolArgs& a, cudaStream_t s) {
  return esdg_vol::for_order(g.N, cudaErrorInvalidValue, [&](auto n) {
    return mode ? esdg_vol::launch_volume64<n.value, 1>(g, P, L, a, s)
                : esdg_vol::launch_volume64<n.value, 0>(g, P, L, a, s);
  });
}

// what: 0 launch (returns 0 / -1), 1 elements per tile, 2 CTAs per SM
int esdg_volume_batch_f64(int what, int N, const EsdgMember* members,
                          const int2* tiles, const int* ntiles, int grid, const EsdgLGL& L,
                          double A, double B, cudaStream_t s) {
  return esdg_vol::for_order(N, -1, [&](auto n) {
    return esdg_vol::batch_volume64<n.value>(what, members, tiles, ntiles, grid, L, A, B, s);
  });
}
