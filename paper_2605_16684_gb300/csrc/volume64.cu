// volume64.cu -- FP64 instantiations of the flux-differencing volume kernel:
// single-mesh launches and the batched kernel.
#include "volume_impl.cuh"

int esdg_volume_f64_take_timeout() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, esdg_vol::g_esdg_vol_timeout, sizeof(int)) != cudaSuccess) return -1;
  if (v) {
    const int z = 0;
    if (cudaMemcpyToSymbol(esdg_vol::g_esdg_vol_timeout, &z, sizeof(int)) != cudaSuccess) return -1;
  }
  return v ? 1 : 0;
}

cudaError_t esdg_launch_volume_f64(const EsdgGrid& g, const EsdgLGL& L, const EsdgPhys& P, int mode,
                                   const EsdgVolArgs& a, cudaStream_t s) {
  return esdg_vol::launch_volume_t<false>(g, L, P, mode, a, s);
}

namespace {
// The batched volume kernel has one variant.
template <int NN>
int batch_variant(int what, int variant, const EsdgMember* members, const int2* tiles,
                  const int* ntiles, int grid, const EsdgLGL& L, double A, double B, cudaStream_t s) {
  if (what == 3) return 1;
  if (variant != 0) return -1;
  return esdg_vol::batch_volume64<NN>(what, members, tiles, ntiles, grid, L, A, B, s);
}

int batch_dispatch(int what, int N, int variant, const EsdgMember* members, const int2* tiles,
                   const int* ntiles, int grid, const EsdgLGL& L, double A, double B, cudaStream_t s) {
  switch (N) {
    case 1: return batch_variant<1>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    case 2: return batch_variant<2>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    case 3: return batch_variant<3>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    case 4: return batch_variant<4>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    case 5: return batch_variant<5>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    case 6: return batch_variant<6>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    case 7: return batch_variant<7>(what, variant, members, tiles, ntiles, grid, L, A, B, s);
    default: return -1;
  }
}
}  // namespace

int esdg_volume_batch_variants_f64(int N) {
  const int n = batch_dispatch(3, N, 0, nullptr, nullptr, nullptr, 0, EsdgLGL{}, 0, 0, 0);
  return n > 0 ? n : 1;
}

// what: 0 launch (returns 0 / -1), 1 elements per tile, 2 CTAs per SM
int esdg_volume_batch_f64(int what, int N, int variant, const EsdgMember* members,
                          const int2* tiles, const int* ntiles, int grid, const EsdgLGL& L,
                          double A, double B, cudaStream_t s) {
  return batch_dispatch(what, N, variant, members, tiles, ntiles, grid, L, A, B, s);
}
