// volume_fp64.cuh -- the FP64 volume kernel: one CTA per tile of a few elements
// (a batch: persistent CTAs over its work table), pairs in fixed point
// (volume_fx.cuh) or, for elements outside its range, FP64.
//
// A tile's phases use different pipes: the prologue and the epilogue the FP64
// pipe and memory, the pair pass the integer pipes.  The tile is therefore
// small (64 to 224 threads) and several CTAs share an SM, so that one CTA's
// prologue and epilogue run under another's pair pass.
#pragma once
#include "volume_pipe.cuh"

namespace esdg_vol {

// Elements per tile and the CTAs planned per SM (MINB; it sets the register
// budget).  One launch, ms (EPB/MINB): N = 4, 32^3: 3/2 0.951, 2/3 0.972, 4/2 1.004, 2/4
// 1.065, 2/2 1.154, 1/6 1.278; N = 5, 20^3: 2/2 0.455, 1/4 0.482; N = 6, 20^3: 1/2 1.010,
// 2/1 1.189; N = 7, 16^3: 1/2 0.762, 1/3 0.928.  Up to N = 3 more and smaller CTAs are
// faster on large meshes (N = 1, 64^3: 8/7 0.368 against 16/2 0.538; N = 2, 48^3: 2/10
// 0.590 against 7/2 0.685; N = 3, 32^3: 2/6 0.498 against 4/2 0.530) but their fewer
// registers lengthen a tile, which a mesh of one round of tiles waits for (N = 3, 6^3:
// 0.0207 against 0.0162; N = 1, 13^3: 0.0123 against 0.0105; a 4^3 N = 3 step 126 against
// 116 us), so the tiles with registers stay.
template <int N> struct F64Cfg;
template <> struct F64Cfg<1> { static constexpr int EPB = 16, MINB = 2; };
template <> struct F64Cfg<2> { static constexpr int EPB = 7, MINB = 2; };
template <> struct F64Cfg<3> { static constexpr int EPB = 4, MINB = 2; };
template <> struct F64Cfg<4> { static constexpr int EPB = 2, MINB = 3; };
template <> struct F64Cfg<5> { static constexpr int EPB = 2, MINB = 2; };
template <> struct F64Cfg<6> { static constexpr int EPB = 1, MINB = 2; };
template <> struct F64Cfg<7> { static constexpr int EPB = 1, MINB = 2; };

template <int N>
struct F64 {
  using SH = Shape<N, false, 0, F64Cfg<N>::EPB>;
  static constexpr int P = SH::NP * SH::EPB;  // nodes per tile
  static constexpr int NF = SH::NF + 1;
  static constexpr int S0 = 0;                // [el][NF][NP] node fields; sums (1..3) in the Ja slots
  // [el][6][NP] sums 0 and 4; first the copy of q (a bulk-copy target: 16-byte aligned)
  static constexpr int X0 = (NF * P + 1) / 2 * 2;
  static constexpr size_t SMEM = sizeof(double) * (size_t)(X0 + 6 * P + 4);
  static_assert(SH::NF == 18, "FP64 node fields");
};

// ONE: the same kernel with the registers of a whole SM per CTA, for meshes of no more
// tiles than SMs.  At N = 6 and 7 a lone CTA of 168 registers a thread leaves the pipes
// waiting (N = 7, 4^3, one right-hand side, us, ONE against not: FP64 pairs at Mach 1 117
// and 213, fixed point 46 and 62; with two CTAs an SM it is the slower one: 6^3 231 and
// 220, 14^3 817 and 629 in fixed point); below, a tile has the registers it can use.
template <int N>
constexpr bool HAS_ONE = N >= 6;

template <int N, int MODE, bool TABLE, bool ONE>
__global__ void __launch_bounds__(F64<N>::SH::THREADS, ONE ? 1 : F64Cfg<N>::MINB)
    k_volume64(const __grid_constant__ EsdgMember one, const EsdgMember* __restrict__ members,
               const int2* __restrict__ tiles, const int* __restrict__ ntiles_d, int ntiles_1,
               const __grid_constant__ EsdgLGL L, double rkA, double rkB, unsigned phantom, int t1,
               int s1) {
  static_assert(!TABLE || MODE == 1, "the batched kernel applies an RK stage");
  using SH = typename F64<N>::SH;
  constexpr int Nq = SH::Nq, NP = SH::NP, NPEN = SH::NPEN, EPB = SH::EPB, NF = F64<N>::NF;
  constexpr int T = SH::THREADS;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long bar;
  __shared__ esdg_fx::FxElement fxe[EPB];
  // per element: its path; the pencils (three directions, 64
  // bits) whose interface terms leave its range
  __shared__ unsigned gen[EPB], far_lift[EPB][3][2];
  __shared__ bool logs[EPB];  // a node outside the narrow path's range
  double* const sm = reinterpret_cast<double*>(smraw) + F64<N>::S0;
  double* const xs = reinterpret_cast<double*>(smraw) + F64<N>::X0;
  const int tid = threadIdx.x;
  if constexpr (!TABLE) {
    esdg_wait_before();
    if (one.a.early) esdg_start_next();
  }
  const int ntiles = TABLE ? *ntiles_d : ntiles_1;
  if (tid == 0) {
    esdg_mbar_init(&bar, 1);
    esdg_fence_mbar_init();
  }
  __syncthreads();
  unsigned parity = 0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, parity ^= 1u) {
    // the descriptor stays in the constant bank (or global memory: a batch); in
    // shared memory every store there would force its fields to be read again
    const EsdgMember& M = TABLE ? members[tiles[tile].x] : one;
    const EsdgGrid& g = M.g;
    const EsdgPhys& P = M.P;
    const EsdgVolArgs& a = M.a;
    const int4 tr = pipe_tile<TABLE, EPB>(tiles, tile, t1, s1, g.E);
    const int e0 = tr.y, ne = tr.z;
    const double* const vg = reinterpret_cast<const double*>(a.vgeo);
    const int* const nscale = esdg_fx::metric_scales(vg, g.E, NP);
    if (tid == 0) {
      const double* q = a.q_in + (size_t)e0 * 5 * NP;
      pipe_issue(BlockCopy{xs, q, a.q_in + (size_t)g.E * 5 * NP, ne * 5 * NP}, &bar, phantom);
      phantom = 0;
    }
    if (tid < EPB) {
      fxe[tid].mu = 0;
      fxe[tid].mf = 0u;
      gen[tid] = 0u;
      logs[tid] = false;
      for (int w = 0; w < 6; w++) far_lift[tid][w / 2][w % 2] = 0u;
    }
    // the metric limbs and (in the spare field) the geopotential
    for (int idx = tid; idx < ne * NP; idx += T) {
      const int el = idx / NP, n = idx - el * NP;
      double* S = sm + (size_t)el * NF * NP + n;
      const double* gr = vg + (size_t)(e0 + el) * ESDG_NVGEO * NP + n;
#pragma unroll
      for (int k = 0; k < 9; k++) esdg_cp_async(S + (SH::F_NH + k) * NP, gr + k * NP);
      esdg_cp_async(S + 18 * NP, gr + 10 * NP);
    }
    if (tid < ne) esdg_fx::fx_metric(fxe[tid], nscale + 3 * (size_t)(e0 + tid));
    esdg_cp_async_wait_all();  // these, and thread 0's edge elements of q
    const bool ok = tile_wait(&bar, parity, a.timeout);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) atomicExch(a.timeout, 1);
      return;
    }
    // ---- prologue: node fields (FP64) and the elements' largest values ------------
    {
      const double* qr0 = xs + esdg_block_shift(a.q_in + (size_t)e0 * 5 * NP);
      const double gm1 = P.gamma - 1.0;
      for (int idx = tid; idx < ne * NP; idx += T) {
        const int el = idx / NP, n = idx - el * NP;
        double* S = sm + (size_t)el * NF * NP;
        const double* qr = qr0 + (size_t)el * 5 * NP;
        prims64<NP>(qr[n], qr[NP + n], qr[2 * NP + n], qr[3 * NP + n], qr[4 * NP + n],
                    S[18 * NP + n], S[18 * NP], gm1, S, n);
        const int* k = fxe[el].sc.k;
        using esdg_fx::stretched;
        atomicMax(&fxe[el].mu, max(stretched(S[3 * NP + n], k[0]), max(stretched(S[4 * NP + n], k[1]),
                                                                       stretched(S[5 * NP + n], k[2]))));
        atomicMax(&fxe[el].mf, (unsigned)__double2hiint(S[6 * NP + n]) & 0x7fffffffu);
      }
    }
    __syncthreads();  // the copy of q consumed
    // ---- which elements take the fixed-point pairs, and their scales ---------------
    for (int idx = tid; idx < ne * NP; idx += T) {
      const int el = idx / NP, n = idx - el * NP;
      const double* S = sm + (size_t)el * NF * NP;
      const unsigned path = esdg_fx::fx_path(S[n], S[2 * NP + n], S[0], S[2 * NP]);
      if (path != esdg_fx::FX_NARROW) {
        atomicMax(&gen[el], path);
        logs[el] = true;
      }
      if (n == 0) {
        esdg_fx::fx_scales(fxe[el], S[0], S[2 * NP], S[18 * NP], P.gamma - 1.0, P.igm1, L.wm);
        if (!fxe[el].sc.ok) atomicMax(&gen[el], (unsigned)esdg_fx::FX_GENERAL);
        else if (fxe[el].sc.tall()) atomicMax(&gen[el], (unsigned)esdg_fx::FX_TALL);
      }
    }
    __syncthreads();
    for (int idx = tid; idx < ne * NP; idx += T) {
      const int el = idx / NP, n = idx - el * NP;
      double* S = sm + (size_t)el * NF * NP;
      if (gen[el] == esdg_fx::FX_GENERAL)
        prims64_general<NP>(S, n, a.Ja + (size_t)(e0 + el) * 9 * NP, logs[el]);
      else esdg_fx::fx_convert<NP>(S, n, fxe[el], gen[el], 0.5 * P.igm1);
    }
    __syncthreads();

    // ---- pair pass: this thread's pencil --------------------------------------------
    bool far = false;
    const int el = tid / (3 * NPEN);
    if (tid < SH::PENCILS && el < ne) {
      const int rr = tid - el * 3 * NPEN;
      const int d = rr / NPEN;
      const int pen = rr - d * NPEN;
      const int ps = pen % Nq, pt = pen / Nq;
      const int stride = (d == 0) ? 1 : ((d == 1) ? Nq : Nq * Nq);
      const int base = (d == 0) ? Nq * (ps + Nq * pt) : ((d == 1) ? (ps + Nq * Nq * pt) : (ps + Nq * pt));
      double* const S = sm + (size_t)el * NF * NP;
      // this pencil's sums leave through its own Ja slots (momentum) and the
      // spare slots (mass, energy) as the nodes complete
      double* const om = S + (SH::F_NH + 3 * d) * NP + base;
      double* const ox = xs + ((size_t)el * 6 + 2 * d) * NP + base;
      FaceTerms<double> ft = face_fetch<N, double>(g, a, e0 + el, d, ps + Nq * pt);
      if (gen[el] != esdg_fx::FX_GENERAL) {
        using esdg_fx::i64;
        const esdg_fx::FxElement& E2 = fxe[el];
        const int s1 = E2.sc.s1[0];
        i64 acc[Nq][5];
        // energy fluxes relative to the element's geopotential (update restores it)
        ft.m[4] = fma(-E2.phi0, ft.m[0], ft.m[4]);
        ft.p[4] = fma(-E2.phi0, ft.p[0], ft.p[4]);
#pragma unroll
        for (int v = 0; v < 5; v++) {
          const int so = E2.out[v];
          far |= esdg_fx::fx_over(ft.m[v], so, 3) || esdg_fx::fx_over(ft.p[v], so, 3);
#pragma unroll
          for (int i = 0; i < Nq; i++) acc[i][v] = 0;
          acc[0][v] = -esdg_fx::fx_lift(ft.m[v], so, L);
          acc[N][v] = esdg_fx::fx_lift(ft.p[v], so, L);
        }
        if (far) {  // the epilogue adds them in FP64
          atomicOr(&far_lift[el][d][pen >> 5], 1u << (pen & 31));
#pragma unroll
          for (int v = 0; v < 5; v++) acc[0][v] = acc[N][v] = 0;
        }
        const auto load = [&](int i) { return esdg_fx::fx_load<NP>(S, base + i * stride, d); };
        const auto done = [&](int i, const i64* s) {
          auto out = [&](int v) {
            return __longlong_as_double(
                esdg_fx::mul(esdg_fx::limbs4(s[v]), esdg_fx::Fx{L.Wh[i], L.Wl[i]}, L.rnd[0]));
          };
          const int n = i * stride;
          ox[n] = out(0);
          ox[NP + n] = out(4);
          om[n] = out(1);
          om[NP + n] = out(2);
          om[2 * NP + n] = out(3);
        };
        auto pass = [&](auto path) {
          pencil_rolled<N>(acc, load,
                           [&](const esdg_fx::FxNode& A, const esdg_fx::FxNode& B, int i, int l,
                               i64* ai, i64* al) {
                             const int* sp = decltype(path)::value == esdg_fx::FX_TALL ? E2.sc.s1 : &s1;
                             esdg_fx::pair_fx<decltype(path)::value>(
                                 A, B, esdg_fx::Fx{L.Qh[i][l], L.Ql[i][l]}, sp, E2.sc.dp,
                                 esdg_fx::Round{L.rnd[0], L.rnd[1]}, ai, al);
                           }, done);
        };
        using namespace esdg_fx;
        if (gen[el] == FX_NARROW) pass(std::integral_constant<int, FX_NARROW>{});
        else if (gen[el] == FX_WIDE) pass(std::integral_constant<int, FX_WIDE>{});
        else pass(std::integral_constant<int, FX_TALL>{});
      } else {
        double acc[Nq][5];
#pragma unroll
        for (int i = 0; i < Nq; i++)
#pragma unroll
          for (int v = 0; v < 5; v++) acc[i][v] = i == 0 ? -ft.m[v] : (i == N ? ft.p[v] : 0.0);
        const CeSeries cs = ce_series(0.5 * P.igm1);
        // unrolled: independent pairs side by side, as the FP64 pipe's latency needs (rolled,
        // 24^3 N = 4 and 14^3 N = 7 at Mach 1, one right-hand side: 1.720 and 2.113 ms
        // against 1.666 and 1.995)
        pencil_unrolled<N>(
            acc,
            [&](int i) { return load_node<double, true, SH::F_NH, NP, 0>(S, base + i * stride, d); },
            [&](const Node<double>& A, const Node<double>& B, int i, int l, double* ai, double* al) {
              pair64(A, B, L.Dt[i][l], L.Dt[l][i], cs, ai, al);
            },
            [&](int i, const double* s) {
              const int n = i * stride;
              ox[n] = s[0];
              ox[NP + n] = s[4];
              om[n] = s[1];
              om[NP + n] = s[2];
              om[2 * NP + n] = s[3];
            });
      }
    }
    const bool any_far = __syncthreads_or(far);

    // ---- epilogue ------------------------------------------------------------------
    const double dt = a.dt;
    const double* const qin = a.q_in;
    double* const dqp = reinterpret_cast<double*>(a.dq);
    double* const qio = a.q_io;
    double* const rhsp = a.rhs;
    bool bad = false;
    const bool rot = P.f0 != 0.0 || P.beta != 0.0;
    // one thread per node; the loads of two nodes are in flight together
    struct Old {
      double q[5], d[5], iJ, y;
    };
    auto fetch = [&](int idx) {
      const int el2 = idx / NP, n = idx - el2 * NP, e2 = e0 + el2;
      const size_t qv = (size_t)e2 * 5 * NP + n;
      Old o;
      o.iJ = vg[((size_t)e2 * ESDG_NVGEO + 9) * NP + n];
#pragma unroll
      for (int v = 0; v < 5; v++) {
        if (MODE != 0 || (rot && (v == 1 || v == 2))) o.q[v] = qin[qv + v * NP];
        if (MODE != 0 && rkA != 0.0) o.d[v] = dqp[qv + v * NP];
      }
      if (rot) o.y = a.x[((size_t)e2 * 3 + 1) * NP + n];
      return o;
    };
    auto update = [&](int idx, const Old& o) {
      const int el2 = idx / NP, n = idx - el2 * NP, e2 = e0 + el2;
      const size_t qv = (size_t)e2 * 5 * NP + n;
      const bool general = gen[el2] == esdg_fx::FX_GENERAL;
      // -1/J, times dt for a stage update (r then holds dt times the right-hand side)
      const double sJ = MODE != 0 ? -o.iJ * dt : -o.iJ;
      double f = 0.0;
      if (rot) {
        f = P.f0 + P.beta * (o.y - P.y0);
        if (MODE != 0) f *= dt;
      }
      double mass = 0.0;
#pragma unroll
      for (int v = 0; v < 5; v++) {
        const bool mom = v >= 1 && v <= 3;
        const double* Z = mom ? sm + ((size_t)el2 * NF + SH::F_NH + v - 1) * NP + n
                              : xs + ((size_t)el2 * 6 + (v ? 1 : 0)) * NP + n;
        const int zs = mom ? 3 * NP : 2 * NP;
        const double z0 = Z[0], z1 = Z[zs], z2 = Z[2 * zs];
        double r;
        if (!general) {
          r = sJ * esdg_fx::from_fx(__double_as_longlong(z0) + __double_as_longlong(z1) +
                                        __double_as_longlong(z2), fxe[el2].out[v]);
          if (v == 0) mass = r;
          if (v == 4) r = fma(fxe[el2].phi0, mass, r);
          if (any_far) r = fma(sJ, far_terms<N>(g, a, e2, n, v, far_lift[el2]), r);
        } else {
          r = sJ * (z0 + z1 + z2);
        }
        if (rot && v == 1) r = fma(f, o.q[2], r);
        if (rot && v == 2) r = fma(-f, o.q[1], r);
        if constexpr (MODE == 0) {
          rhsp[qv + v * NP] = r;
        } else {
          // first stage (A = 0): the register is not read (see stage32)
          const double dv = rkA == 0.0 ? r : fma(rkA, o.d[v], r);
          dqp[qv + v * NP] = dv;
          const double qn = fma(rkB, dv, o.q[v]);
          qio[qv + v * NP] = qn;
          bad |= esdg_bad_state(qn, v == 0);
        }
      }
    };
    for (int i0 = tid; i0 < ne * NP; i0 += 2 * T) {
      const int i1 = i0 + T;
      const Old o0 = fetch(i0), o1 = fetch(i1 < ne * NP ? i1 : i0);
      update(i0, o0);
      if (i1 < ne * NP) update(i1, o1);
    }
    if (MODE != 0 && bad && a.status) *a.status = 1;
    __syncthreads();  // the sums and the element data read
  }
}

template <int N, int MODE>
cudaError_t launch_volume64(const EsdgGrid& g, const EsdgPhys& P, const EsdgLGL& L,
                            const EsdgVolArgs& a, cudaStream_t s) {
  using SH = typename F64<N>::SH;
  constexpr auto k = k_volume64<N, MODE, false, false>, one = k_volume64<N, MODE, false, HAS_ONE<N>>;
  const GridCap cap = pipe_grid_cap<k>(SH::THREADS, F64<N>::SMEM);
  if (cap.ctas < 0 || pipe_grid_cap<one>(SH::THREADS, F64<N>::SMEM).ctas < 0)
    return cudaErrorInvalidConfiguration;
  int ntiles, t1, s1;
  pipe_split(g.E, SH::EPB, cap.ctas, cap.sms / a.share, ntiles, t1, s1);
  if (ntiles == 0) return cudaSuccess;
  EsdgMember m = pipe_member(g, P, a);
  m.a.early = a.share == 1 && (2 * ntiles <= cap.sms || ntiles >= 4 * cap.ctas);
  // one CTA per tile: the hardware hands tiles out as CTAs end, so tiles of unequal
  // cost (path, clock) leave no SM waiting for the CTA with the costliest share, as a
  // persistent loop over a fixed share did (32^3 N = 4: 1.124 -> 0.976 ms; 16^3 N = 7:
  // 0.790 -> 0.763)
  return esdg_launch(ntiles <= cap.sms / a.share ? one : k, a.after, ntiles, SH::THREADS,
                     F64<N>::SMEM, s, m, nullptr, nullptr, nullptr, ntiles, L, a.rkA, a.rkB,
                     esdg_take_phantom(), t1, s1);
}

// batched (TABLE) launches; what: 0 launch (0 / -1), 1 elements per tile, 2 CTAs per SM
template <int N>
int batch_volume64(int what, const EsdgMember* members, const int2* tiles, const int* ntiles,
                   int grid, const EsdgLGL& L, double A, double B, cudaStream_t s) {
  using SH = typename F64<N>::SH;
  constexpr auto k = k_volume64<N, 1, true, false>;
  if (what == 1) return SH::EPB;
  if (what == 2) {
    int nb = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F64<N>::SMEM) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, SH::THREADS, F64<N>::SMEM) !=
            cudaSuccess) {
      cudaGetLastError();
      return 1;
    }
    return nb > 0 ? nb : 1;
  }
  static bool configured = false;  // one-time attribute set per instantiation
  if (!configured) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F64<N>::SMEM) !=
        cudaSuccess)
      return -1;
    configured = true;
  }
  EsdgMember none;
  memset(&none, 0, sizeof(none));
  k<<<grid, SH::THREADS, F64<N>::SMEM, s>>>(none, members, tiles, ntiles, 0, L, A, B, 0u, 0, 0);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace esdg_vol
