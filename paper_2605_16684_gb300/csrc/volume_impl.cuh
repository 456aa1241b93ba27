// volume_impl.cuh -- flux-differencing volume kernel (Section 3, the volume term
// of Eq. (nm:semi), with the optimisations of Section 4.1).
// The arithmetic lives in volume_pairs.cuh and volume_fx.cuh, the kernels in
// volume_fp64.cuh and volume_mixed.cuh; this file dispatches on the order.
//
//   rhs_i = -(1/J_i) [ sum_d sum_l Dt^{(d)}_{il} H^d(q_i, q_l) + face lifts ] + h_i
//
// H^d is the two-point entropy-conservative flux with the metric average
// n = {{Ja^d}}_{il} plus the non-symmetric gravity term 1/2 rho_hat [[phi]] n.
//
// Layout on the GPU (one CTA = EPB elements):
//   prologue   one thread per node: primitives once per node (u = rho u/rho, p,
//              b = rho/(2p), 1/b), staged in shared memory with 1/2 Ja;
//   pair pass  one thread per pencil (element, direction d, transverse node):
//              every unordered pair (i < l) of the pencil is evaluated once and
//              added to both nodes in registers -- node i gets Dt_il H(i,l),
//              node l gets Dt_li H(l,i), where H(l,i) shares the symmetric flux
//              and takes the gravity part -G(i,l) b_i/b_l (Section 4.1).  The
//              pencil's two end nodes also receive the interface fluxes of the
//              two faces the pencil pierces;
//   epilogue   one thread per node: sum the three directions, scale by -1/J,
//              add the Coriolis source, then write rhs or apply the LSRK stage.
//
// The pencil-per-thread pair pass evaluates exactly N_q (N_q - 1)/2 pairs per
// pencil for every N (no antipodal double counting at odd N, no load
// imbalance, no shuffles or atomics); the pencil's accumulators live in
// registers and are exchanged once through shared memory.
//
// FP64: pairs in 60-bit fixed point where the element's fields fit it, else FP64
// with the artanh series for log means when u = f^2 < 1e-4 and per-node logarithms
// otherwise.  Mixed: the
// prologue recovers the pressure in FP64 and stages FP32 node data; pairs,
// sums and face lifts run in FP32; the log branch uses log1pf of the ratio;
// the geopotential is carried relative to each element's first node.
#pragma once
#include <type_traits>

#include "esdg_internal.cuh"

namespace esdg_vol {

// f(std::integral_constant<int, N>) for the order N = 1..7, or `other`
template <typename T, typename F>
T for_order(int N, T other, const F& f) {
  switch (N) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    default: return other;
  }
}

}  // namespace esdg_vol
