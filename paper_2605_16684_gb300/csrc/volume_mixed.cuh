// volume_mixed.cuh -- the mixed-precision volume kernel (FP32 pairs, FP64 state and
// pressure recovery), for every order, with no background, one at rest or a moving
// one, single meshes or batch work tables.
//
// A tile alternates between memory latency (its loads), the conversions between
// FP64 and FP32 (integer and FP64 pipes) and the FP32 pair pass.  No phase alone
// bounds it, so tiles are small (1 to 8 elements, 64 to 192 threads) and three to
// ten CTAs share an SM: phases of different tiles overlap without any pipeline
// inside a CTA.  Within a tile the loads of two nodes per thread are in flight
// together, and 1/J, which only the epilogue reads, comes by bulk copies behind the
// pair pass.  It replaced a warp-specialised kernel (N = 4 at rest), a pipelined
// kernel with one CTA per SM and a kernel without a pipeline for moving backgrounds.
// One RK stage's launch, ms, before -> with this kernel:
//   at rest       N = 1 (80^3) 0.433 -> 0.297   N = 2 (60^3) 0.533 -> 0.430
//                 N = 3 (40^3) 0.367 -> 0.293   N = 4 (32^3) 0.345 -> 0.330
//                 N = 5 (24^3) 0.321 -> 0.270   N = 6 (20^3) 0.392 -> 0.275
//                 N = 7 (16^3) 0.382 -> 0.298
//   moving        N = 3 (140x28x14) 0.691 -> 0.397   N = 4 (120x24x12) 0.801 -> 0.507
//                 N = 7 (60x12x6) 0.685 -> 0.491
// Copying q or the nine Ja rows by bulk copies as well was slower at N <= 4 (0.36 to
// 0.39 ms at 32^3): their shared memory costs a CTA, and their words are read once.
#pragma once
#include "volume_pipe.cuh"

namespace esdg_vol {

// Elements per tile and the CTAs planned per SM (MINB, which sets the registers).
// Measured alternatives (ms, sizes as above): N = 1 16/3 0.389, 8/6 0.351; N = 2 7/3
// 0.448, 4/6 0.443; N = 3 4/3 0.311, 1/12 0.312, 4/2 0.395; N = 4 2/3 0.384; N = 5
// 2/2 0.276, 1/3 0.311; N = 6 1/4 0.292, 1/2 0.366; N = 7 1/2 0.316.  A moving
// background's pairs hold more registers: N = 3 2/5 0.406; N = 4 2/4 0.539, 2/2 0.636;
// N = 6 1/2 0.678; N = 7 runs with two CTAs.
template <int N, int BG> struct MixCfg;
template <int BG> struct MixCfg<1, BG> { static constexpr int EPB = 8, MINB = BG == 2 ? 6 : 8; };
template <int BG> struct MixCfg<2, BG> { static constexpr int EPB = BG == 2 ? 4 : 2, MINB = BG == 2 ? 5 : 10; };
template <int BG> struct MixCfg<3, BG> { static constexpr int EPB = BG == 2 ? 4 : 2, MINB = BG == 2 ? 3 : 7; };
template <int BG> struct MixCfg<4, BG> { static constexpr int EPB = 2, MINB = BG == 2 ? 3 : 4; };
template <int BG> struct MixCfg<5, BG> { static constexpr int EPB = 1, MINB = 4; };
template <int BG> struct MixCfg<6, BG> { static constexpr int EPB = 1, MINB = 3; };
template <int BG> struct MixCfg<7, BG> { static constexpr int EPB = 1, MINB = BG == 2 ? 2 : 3; };
// The pencil's pairs are unrolled to N = 3 and rolled above, where the unrolled code
// outgrows the instruction cache (N = 6 0.308 unrolled, 0.275 rolled; moving, N = 4
// 0.538 and 0.507; N = 3 at rest 0.311 and 0.342).
template <int N>
constexpr bool MIX_UNROLL = N <= 3;

template <int N, int BG>
struct Mix {
  using SH = Shape<N, true, BG, MixCfg<N, BG>::EPB>;
  static constexpr int P = SH::NP * SH::EPB;                        // nodes per tile
  // floats: the node fields [el][NF][NP] (a direction's momentum sums replace its
  // Ja), the mass and energy sums [el][6][NP], 1/J [el][JS] (bulk-copy targets)
  static constexpr int X0 = SH::NF * P;
  static constexpr int JS = (SH::NP + 11) / 4 * 4;
  static constexpr int J0 = (X0 + 6 * P + 3) / 4 * 4;
  static constexpr size_t SMEM = 4 * (size_t)(J0 + SH::EPB * JS);
};

template <int N, int MODE, int BG, bool TABLE>
__global__ void __launch_bounds__(Mix<N, BG>::SH::THREADS, MixCfg<N, BG>::MINB)
    k_volume32(const __grid_constant__ EsdgMember one, const EsdgMember* __restrict__ members,
               const int2* __restrict__ tiles, const int* __restrict__ ntiles_d, int ntiles_1,
               const __grid_constant__ EsdgLGL L, double rkA, double rkB, unsigned phantom, int t1,
               int s1) {
  static_assert(!TABLE || MODE == 1, "the batched kernel applies an RK stage");
  using SH = typename Mix<N, BG>::SH;
  constexpr int Nq = SH::Nq, NP = SH::NP, NPEN = SH::NPEN, EPB = SH::EPB, NF = SH::NF;
  constexpr int T = SH::THREADS;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long bar;
  float* const sm = reinterpret_cast<float*>(smraw);
  float* const xs = sm + Mix<N, BG>::X0;
  float* const js = sm + Mix<N, BG>::J0;
  const int tid = threadIdx.x;
  if constexpr (!TABLE) esdg_wait_before();
  if (tid == 0) {
    esdg_mbar_init(&bar, 1);
    esdg_fence_mbar_init();
  }
  __syncthreads();
  unsigned parity = 0;
  const int ntiles = TABLE ? *ntiles_d : ntiles_1;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, parity ^= 1u) {
    // the descriptor stays in the constant bank (or global memory: a batch); in
    // shared memory every store there would force its fields to be read again
    const EsdgMember& M = TABLE ? members[tiles[tile].x] : one;
    const EsdgGrid& g = M.g;
    const EsdgPhys& P = M.P;
    const EsdgVolArgs& a = M.a;
    const int4 tr = pipe_tile<TABLE, EPB>(tiles, tile, t1, s1, g.E);
    const int e0 = tr.y, ne = tr.z, nodes = ne * NP;
    const double* const qin = a.q_in;
    const float* const vg = reinterpret_cast<const float*>(a.vgeo) + (size_t)e0 * ESDG_NVGEO * NP;
    const double* const vphi = a.vgeo64 + (size_t)e0 * ESDG_NVGEO * NP + 10 * NP;
    auto fields = [&](int el) { return sm + el * NF * NP; };
    // 1/J comes by bulk copies, read by the epilogue: element el's row and the up to
    // three words before it that align the copy
    auto jrow = [&](int el) {
      return (unsigned)(reinterpret_cast<unsigned long long>(vg + ((size_t)el * ESDG_NVGEO + 9) * NP) >> 2) & 3u;
    };
    if (tid == 0) {
      unsigned total = phantom;
      for (int el = 0; el < ne; el++) total += (jrow(el) + NP + 3u) / 4u * 16u;
      esdg_mbar_arrive_tx(&bar, total);
      esdg_fence_proxy_async();
      for (int el = 0; el < ne; el++)
        esdg_bulk_g2s(js + el * Mix<N, BG>::JS,
                      vg + ((size_t)el * ESDG_NVGEO + 9) * NP - jrow(el), (jrow(el) + NP + 3u) / 4u * 16u, &bar);
      phantom = 0;
    }

    // ---- prologue: primitives once per node ------------------------------------
    struct In {
      double q[5], phi, b[5];  // b: rho_bg, E_bg, or the moving background's state
      float phh, bp[4], bu[3], nh[9];
    };
    auto fetch = [&](int idx) {
      const int el = idx / NP, n = idx - el * NP;
      const size_t e = e0 + el;
      In x;
#pragma unroll
      for (int v = 0; v < 5; v++) x.q[v] = qin[(e * 5 + v) * NP + n];
      x.phi = vphi[(size_t)el * ESDG_NVGEO * NP + n];
      const float* ge = vg + (size_t)el * ESDG_NVGEO * NP + n;
      x.phh = ge[10 * NP];
      if constexpr (BG == 2) {
#pragma unroll
        for (int v = 0; v < 5; v++) x.b[v] = a.bgq[(e * 5 + v) * NP + n];
#pragma unroll
        for (int k = 0; k < 3; k++) x.bu[k] = a.bgu[(e * 3 + k) * NP + n];
      } else if constexpr (BG) {
        x.b[0] = a.bg[e * 3 * NP + n];
        x.b[1] = a.bg[e * 3 * NP + NP + n];
      }
      if constexpr (BG) {
#pragma unroll
        for (int k = 0; k < 4; k++) x.bp[k] = a.bgp[(e * 4 + k) * NP + n];
      }
#pragma unroll
      for (int k = 0; k < 9; k++) x.nh[k] = ge[k * NP];
      return x;
    };
    const double gm1 = P.gamma - 1.0;
    const float gm1f = esdg_d2f(gm1);
    auto convert = [&](int idx, const In& x) {
      const int el = idx / NP, n = idx - el * NP;
      float* S = fields(el);
      if constexpr (BG == 2) {
        const Prim32m o = prims32bgm(x.q[0], x.q[1], x.q[2], x.q[3], x.q[4], x.phi, x.phh, gm1f,
                                     x.b[0], x.b[1], x.b[2], x.b[3], x.b[4], x.bp[0], x.bp[1],
                                     x.bp[2], x.bp[3], x.bu[0], x.bu[1], x.bu[2]);
#pragma unroll
        for (int k = 0; k < 7; k++) {
          S[k * NP + n] = o.s[k];
          S[(SH::F_BG + k) * NP + n] = o.bgf[k];
        }
#pragma unroll
        for (int k = 0; k < 3; k++) S[(SH::F_BG + 7 + k) * NP + n] = o.up[k];
      } else if constexpr (BG) {
        const Prim32 o = prims32bg(x.q[0], x.q[1], x.q[2], x.q[3], x.q[4], x.phi, x.phh, gm1f,
                                   x.b[0], x.b[1], x.bp[0], x.bp[1], x.bp[2], x.bp[3]);
#pragma unroll
        for (int k = 0; k < 7; k++) {
          S[k * NP + n] = o.s[k];
          S[(SH::F_BG + k) * NP + n] = o.bgf[k];
        }
      } else {
        prims32<NP>(x.q[0], x.q[1], x.q[2], x.q[3], x.q[4], x.phi, x.phh, gm1, S, n);
      }
#pragma unroll
      for (int k = 0; k < 9; k++) S[(SH::F_NH + k) * NP + n] = x.nh[k];
    };
    for (int i0 = tid; i0 < nodes; i0 += 2 * T) {
      const int i1 = i0 + T;
      const In x0 = fetch(i0), x1 = fetch(i1 < nodes ? i1 : i0);
      convert(i0, x0);
      if (i1 < nodes) convert(i1, x1);
    }
    __syncthreads();
    int need_logs = 0;
    for (int idx = tid; idx < nodes; idx += T) {
      const int el = idx / NP, n = idx - el * NP;
      const float* S = fields(el);
      const float r0 = S[0], rn = S[n], b0 = S[NP], bn = S[NP + n];
      // |f| < 0.14 keeps u < ESDG_LOG_EPS32 for every pair
      if (fabsf(rn - r0) > 0.13f * r0 || fabsf(bn - b0) > 0.13f * b0) need_logs = 1;
    }
    need_logs = __syncthreads_or(need_logs);

    // ---- pair pass: one pencil per thread -----------------------------------------
    const int el = tid / (3 * NPEN);
    const bool active = tid < SH::PENCILS && el < ne;
    const int rr = tid - el * 3 * NPEN;
    const int d = rr / NPEN;
    const int pen = rr - d * NPEN;
    const int s = pen % Nq, t = pen / Nq;
    const int stride = (d == 0) ? 1 : ((d == 1) ? Nq : Nq * Nq);
    const int base = (d == 0) ? Nq * (s + Nq * t) : ((d == 1) ? (s + Nq * Nq * t) : (s + Nq * t));
    if (active) {
      // the face terms and the element's reference geopotential are fetched ahead
      // of the pair pass and applied as the nodes complete
      const FaceTerms<float> ft = face_fetch<N, float>(g, a, e0 + el, d, s + Nq * t);
      const float phi0 = esdg_d2f(vphi[(size_t)el * ESDG_NVGEO * NP]);
      float* const S = fields(el);
      float* const om = S + (SH::F_NH + 3 * d) * NP + base;
      float* const ox = xs + ((size_t)el * 6 + 2 * d) * NP + base;
      const float ce = esdg_d2f(0.5 * P.igm1);
      float acc[Nq][5];
#pragma unroll
      for (int i = 0; i < Nq; i++)
#pragma unroll
        for (int v = 0; v < 5; v++) acc[i][v] = 0.0f;
      const auto done = [&](int i, const float* r) {
        // restore the element's reference geopotential in the energy flux
        float o[5] = {r[0], r[1], r[2], r[3], fmaf(phi0, r[0], r[4])};
        if (i == 0) {
#pragma unroll
          for (int v = 0; v < 5; v++) o[v] -= ft.m[v];
        }
        if (i == N) {
#pragma unroll
          for (int v = 0; v < 5; v++) o[v] += ft.p[v];
        }
        const int n = i * stride;
        ox[n] = o[0];
        ox[NP + n] = o[4];
        om[n] = o[1];
        om[NP + n] = o[2];
        om[2 * NP + n] = o[3];
      };
      auto pass = [&](auto logs) {
        constexpr bool LOGS = decltype(logs)::value;
        const auto load = [&](int i) {
          return load_node<float, LOGS, SH::F_NH, NP, BG>(S, base + i * stride, d);
        };
        const auto pair = [&](const Node<float>& A, const Node<float>& B, int i, int l, float* ai,
                              float* al) {
          if constexpr (BG == 2) pair32bgm<LOGS>(A, B, L.Dtf[i][l], L.Dtf[l][i], ce, ai, al);
          else if constexpr (BG) pair32bg<LOGS>(A, B, L.Dtf[i][l], L.Dtf[l][i], ce, ai, al);
          else pair32<LOGS>(A, B, L.Dtf[i][l], L.Dtf[l][i], ce, ai, al);
        };
        if constexpr (MIX_UNROLL<N>) pencil_unrolled<N>(acc, load, pair, done);
        else pencil_rolled<N>(acc, load, pair, done);
      };
      if (need_logs) pass(std::true_type{});
      else pass(std::false_type{});
    }
    const bool landed = tile_wait(&bar, parity, a.timeout);
    if (__syncthreads_or(!landed)) {  // also: every sum written
      if (tid == 0) atomicExch(a.timeout, 1);
      return;
    }

    // ---- epilogue: one thread per node, two nodes' loads in flight together ----------
    const bool rotating = (P.f0 != 0.0) || (P.beta != 0.0);
    constexpr int NRB = BG == 2 ? 5 : 3;
    struct Old {
      double q[5], qb[3], y;
      float d[5], rb[5];
    };
    auto old = [&](int idx) {
      const int el2 = idx / NP, n = idx - el2 * NP;
      const size_t e2 = e0 + el2, qv = e2 * 5 * NP + n;
      Old o;
#pragma unroll
      for (int v = 0; v < 5; v++)
        if (MODE != 0 || (rotating && (v == 1 || v == 2))) o.q[v] = qin[qv + v * NP];
      if (MODE != 0 && rkA != 0.0) {
#pragma unroll
        for (int v = 0; v < 5; v++) o.d[v] = reinterpret_cast<const float*>(a.dq)[qv + v * NP];
      }
      if constexpr (BG) {
        const float* rb = BG == 2 ? a.rhs_bgm + qv : a.rhs_bg + e2 * 3 * NP + n;
#pragma unroll
        for (int k = 0; k < NRB; k++) o.rb[k] = rb[k * NP];
      }
      if (rotating) {
        o.y = a.x[(e2 * 3 + 1) * NP + n];
        if constexpr (BG == 2) {
          o.qb[1] = a.bgq[qv + NP];
          o.qb[2] = a.bgq[qv + 2 * NP];
        }
      }
      return o;
    };
    bool bad = false;
    auto update = [&](int idx, const Old& o) {
      const int el2 = idx / NP, n = idx - el2 * NP;
      const float* S = fields(el2) + SH::F_NH * NP + n;
      const float* X = xs + (size_t)el2 * 6 * NP + n;
      const size_t qb = (size_t)(e0 + el2) * 5 * NP + n;
      const float iJ = js[el2 * Mix<N, BG>::JS + jrow(el2) + n];
      float r32[5];
#pragma unroll
      for (int v = 0; v < 5; v++)
        r32[v] = v >= 1 && v <= 3
                     ? -iJ * (S[(v - 1) * NP] + S[(v + 2) * NP] + S[(v + 5) * NP])
                     : -iJ * (X[(v / 4) * NP] + X[(2 + v / 4) * NP] + X[(4 + v / 4) * NP]);
      if constexpr (MODE != 0) {
        bad |= stage32<NP, BG, 1>(r32, o.rb, P, rotating ? o.y : 0.0, o.q, o.d,
                                  reinterpret_cast<float*>(a.dq) + qb, a.q_io + qb, rkA, rkB, a.dt,
                                  o.qb);
      } else {  // right-hand side in FP64
        double r[5];
#pragma unroll
        for (int v = 0; v < 5; v++) {
          // plus the background's own right-hand side (at rest: momentum only)
          r[v] = esdg_f2d(r32[v]);
          if (BG == 1 && v >= 1 && v <= 3) r[v] += o.rb[v - 1];
          if (BG == 2) r[v] += o.rb[v];
        }
        if (rotating) {
          const double f = P.f0 + P.beta * (o.y - P.y0);
          // with a moving background its Coriolis force is part of its rhs
          r[1] = fma(f, BG == 2 ? o.q[2] - o.qb[2] : o.q[2], r[1]);
          r[2] = fma(-f, BG == 2 ? o.q[1] - o.qb[1] : o.q[1], r[2]);
        }
#pragma unroll
        for (int v = 0; v < 5; v++) a.rhs[qb + (size_t)v * NP] = r[v];
      }
    };
    for (int i0 = tid; i0 < nodes; i0 += 2 * T) {
      const int i1 = i0 + T;
      const Old o0 = old(i0), o1 = old(i1 < nodes ? i1 : i0);
      update(i0, o0);
      if (i1 < nodes) update(i1, o1);
    }
    if (MODE != 0 && bad && a.status) *a.status = 1;
    if (TABLE) __syncthreads();  // the sums read
  }
}

template <int N, int MODE, int BG>
cudaError_t launch_volume32(const EsdgGrid& g, const EsdgPhys& P, const EsdgLGL& L,
                            const EsdgVolArgs& a, cudaStream_t s) {
  using SH = typename Mix<N, BG>::SH;
  constexpr auto k = k_volume32<N, MODE, BG, false>;
  const GridCap cap = pipe_grid_cap<k>(SH::THREADS, Mix<N, BG>::SMEM);
  if (cap.ctas < 0) return cudaErrorInvalidConfiguration;
  int ntiles, t1, s1;
  pipe_split(g.E, SH::EPB, cap.ctas, cap.sms / a.share, ntiles, t1, s1);
  if (ntiles == 0) return cudaSuccess;
  // one CTA per tile: the hardware hands tiles out as CTAs end, which beats a
  // persistent loop over a fixed share (32^3 N = 4: 0.363 against 0.391 ms)
  return esdg_launch(k, a.after, ntiles, SH::THREADS, Mix<N, BG>::SMEM, s, pipe_member(g, P, a),
                     nullptr, nullptr, nullptr, ntiles, L, a.rkA, a.rkB, esdg_take_phantom(), t1, s1);
}

// batched (TABLE) launches (members with a background at rest); what: 0 launch
// (0 / -1), 1 elements per tile, 2 CTAs per SM
template <int N>
int batch_volume32(int what, const EsdgMember* members, const int2* tiles, const int* ntiles,
                   int grid, const EsdgLGL& L, double A, double B, cudaStream_t s) {
  using SH = typename Mix<N, 1>::SH;
  constexpr auto k = k_volume32<N, 1, 1, true>;
  constexpr size_t SMEM = Mix<N, 1>::SMEM;
  if (what == 1) return SH::EPB;
  if (what == 2) {
    int nb = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, SH::THREADS, SMEM) != cudaSuccess) {
      cudaGetLastError();
      return 1;
    }
    return nb > 0 ? nb : 1;
  }
  static bool configured = false;  // one-time attribute set per instantiation
  if (!configured) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM) != cudaSuccess)
      return -1;
    configured = true;
  }
  EsdgMember none;
  memset(&none, 0, sizeof(none));
  k<<<grid, SH::THREADS, SMEM, s>>>(none, members, tiles, ntiles, 0, L, A, B, 0u, 0, 0);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace esdg_vol
