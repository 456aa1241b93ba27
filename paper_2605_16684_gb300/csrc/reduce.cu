// reduce.cu -- global reductions over the state: the CFL time step and the
// conservation/entropy integrals (the monitors of Section 5.2).
//
// Both were bound by the FP64 pipe (64 cycles per warp instruction): divisions,
// square roots and logarithms of CUDA's library cost some 20 to 35 of them
// each.  The CFL bound needs them only near its maximum, so an FP32 pass
// screens the elements and FP64 evaluates the few that can hold it; the
// integrals use short FP64 sequences for the reciprocal and the logarithms.
// 32^3 N = 4, both calls together: 1.77 -> 0.47 ms.
#include "esdg_internal.cuh"

namespace {

constexpr int RT = 256;         // threads of the folding pass
constexpr int SUM_CTAS = 1216;  // CTAs of the integrals (8 per SM)

__device__ __forceinline__ double block_reduce(double v, double* sh) {
  // warp level, then across warps through shared memory
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  if (threadIdx.x == 0) {
    double r = sh[0];
    for (int k = 1; k < nw; k++) r += sh[k];
    sh[0] = r;
  }
  __syncthreads();
  return sh[0];
}

// The largest reference-space signal speed
//   lambda = max_n max_d (|u . Ja^d| + c |Ja^d|) / J;
// the time step is C (xi_1 - xi_0) / lambda (on an affine element this is the
// node-spacing rule C h (xi_1 - xi_0) / (2 (|u_d| + c))).
//
// Screen, one warp per element: lambda in FP32 (the pressure E - rho phi - KE in
// FP64, KE in FP32), off by at most 2e-6 where KE < 8 p; an element with a node
// where it may be off by more (faster, no positive pressure, values out of the
// float range, NaNs) is marked with an infinity.  top is the largest unmarked
// value (positive floats order as integers).
__global__ void __launch_bounds__(256) k_cfl_screen(EsdgGrid g, EsdgPhys P,
                                                    const double* __restrict__ q,
                                                    const double* __restrict__ x,
                                                    const double* __restrict__ J,
                                                    const double* __restrict__ Ja,
                                                    float* __restrict__ lam32, unsigned* top) {
  const int np = g.np, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const double gm1 = P.gamma - 1.0;
  const float gamma = esdg_d2f(P.gamma);
  unsigned best = 0u;
  for (int e = blockIdx.x * nw + (threadIdx.x >> 5); e < g.E; e += gridDim.x * nw) {
    const double* qe = q + (size_t)e * 5 * np;
    const double* ze = x + ((size_t)e * 3 + 2) * np;
    const double* Je = J + (size_t)e * np;
    const double* ja = Ja + (size_t)e * 9 * np;
    float l = 0.0f;
    bool unsure = false;
#pragma unroll 2
    for (int n = lane; n < np; n += 32) {
      double v[5];
      unsigned hi = 0u;
#pragma unroll
      for (int k = 0; k < 5; k++) {
        v[k] = qe[k * np + n];
        hi = max(hi, (unsigned)__double2hiint(v[k]) & 0x7fffffffu);
      }
      const double Jn = Je[n];
      float a[9];
#pragma unroll
      for (int k = 0; k < 9; k++) {
        const double t = ja[k * np + n];
        hi = max(hi, (unsigned)__double2hiint(t) & 0x7fffffffu);
        a[k] = esdg_d2f(t);
      }
      const float rho = esdg_d2f(v[0]), Jf = esdg_d2f(Jn);
      const float ir = esdg_rcpf(rho), iJ = esdg_rcpf(Jf);
      const float m0 = esdg_d2f(v[1]), m1 = esdg_d2f(v[2]), m2 = esdg_d2f(v[3]);
      const float u0 = m0 * ir, u1 = m1 * ir, u2 = m2 * ir;
      const float ke = 0.5f * fmaf(m2, u2, fmaf(m1, u1, m0 * u0));
      const double pd = gm1 * (fma(-v[0], P.g * ze[n], v[4]) - esdg_f2d(ke));
      hi = max(hi, (unsigned)__double2hiint(pd) & 0x7fffffffu);
      hi = max(hi, (unsigned)__double2hiint(Jn));
      const float p = esdg_d2f(pd);
      const float c = sqrtf(gamma * p * ir);
      float ln = 0.0f;
#pragma unroll
      for (int d = 0; d < 3; d++) {
        const float* b = a + 3 * d;
        const float un = fmaf(u2, b[2], fmaf(u1, b[1], u0 * b[0]));
        ln = fmaxf(ln, fmaf(c, sqrtf(fmaf(b[2], b[2], fmaf(b[1], b[1], b[0] * b[0]))), fabsf(un)));
      }
      ln *= iJ;
      // magnitudes below 2^100, density and J above 2^-100
      unsure |= !(hi < 0x46300000u && rho > 1e-30f && Jf > 1e-30f && p > 0.0f && ke < 8.0f * p &&
                  ln > 1e-25f && ln < 1e30f);
      l = fmaxf(l, ln);
    }
    const bool any = __any_sync(0xffffffffu, unsure);
    const unsigned lm = __reduce_max_sync(0xffffffffu, any ? 0u : __float_as_uint(l));
    if (lane == 0) lam32[e] = any ? __int_as_float(0x7f800000) : __uint_as_float(lm);
    best = max(best, lm);
  }
  if (lane == 0 && best) atomicMax(top, best);
}

// lambda in FP64 of the elements that can hold the maximum; out: its bits.  One
// CTA per element (grid-stride), so that many candidates (a layer of a box at rest)
// spread over the GPU.
__global__ void __launch_bounds__(128) k_cfl_exact(EsdgGrid g, EsdgPhys P,
                                                   const double* __restrict__ q,
                                                   const double* __restrict__ x,
                                                   const double* __restrict__ J,
                                                   const double* __restrict__ Ja,
                                                   const float* __restrict__ lam32,
                                                   const unsigned* __restrict__ top,
                                                   unsigned long long* __restrict__ out) {
  const int np = g.np;
  const float least = __uint_as_float(*top) * (1.0f - 1.0f / 16384.0f);
  double lmax = 0.0;
#pragma unroll 4
  for (int ei = blockIdx.x; ei < g.E; ei += gridDim.x) {
    if (!(lam32[ei] >= least)) continue;
    const size_t e = ei;
    for (int n = threadIdx.x; n < np; n += blockDim.x) {
      const double* qe = q + e * 5 * np;
      const double rho = qe[n], ir = 1.0 / rho;
      const double u0 = qe[np + n] * ir, u1 = qe[2 * np + n] * ir, u2 = qe[3 * np + n] * ir;
      const double z = x[(e * 3 + 2) * np + n];
      const double p = (P.gamma - 1.0) *
                       (qe[4 * np + n] - 0.5 * rho * (u0 * u0 + u1 * u1 + u2 * u2) - rho * P.g * z);
      const double cs = sqrt(P.gamma * p * ir);
      const double iJ = 1.0 / J[e * np + n];
      for (int d = 0; d < 3; d++) {
        const double* ja = Ja + (e * 3 + d) * 3 * np + n;
        const double a0 = ja[0], a1 = ja[np], a2 = ja[2 * np];
        const double lam = (fabs(u0 * a0 + u1 * a1 + u2 * a2) + cs * sqrt(a0 * a0 + a1 * a1 + a2 * a2)) * iJ;
        lmax = fmax(lmax, lam);
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
  if ((threadIdx.x & 31) == 0 && lmax > 0.0)
    atomicMax(out, (unsigned long long)__double_as_longlong(lmax));
}

// ln x by a table of reciprocals (P. T. P. Tang, "Table-driven implementation of
// the logarithm function in IEEE floating-point arithmetic", 1990): x = 2^k m with
// m in [1, 2), r_j = 1/(1 + (j + 1/2)/64) for m's top six bits j,
//   ln x = k ln 2 - ln r_j + ln(1 + a),  a = m r_j - 1, |a| < 0.0079,
// the series beyond a^4 in FP32: 9 FP64 instructions.  tab[j] = (r_j, -ln r_j).
__device__ __forceinline__ double log_tab(double x, const double2* tab) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // not positive, subnormal, inf, NaN
  const int k = (hi >> 20) - 1023;
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(x));
  const double2 t = tab[(hi >> 14) & 63];
  const double a = fma(m, t.x, -1.0);
  const float af = esdg_d2f(a);
  const float tail = af * af * fmaf(af, fmaf(af, 1.0f / 7.0f, -1.0f / 6.0f), 0.2f);
  const double c = fma(a, -0.25, 1.0 / 3.0) + esdg_f2d(tail);
  const double l = fma(a * a, fma(a, c, -0.5), a);
  return fma((double)k, 0.693147180559945309417, t.y) + l;
}

// Quadrature of rho, E and eta = -rho s/(gamma-1) over the elements of a CTA
// (grid-stride), one partial triple per CTA; every thread adds its nodes in a
// fixed order.
__global__ void __launch_bounds__(256) k_integrals(EsdgGrid g, EsdgLGL L, EsdgPhys P,
                                                   const double* __restrict__ q,
                                                   const double* __restrict__ J,
                                                   const double* __restrict__ x,
                                                   double* __restrict__ part) {
  __shared__ double sh[32];
  __shared__ double w3[ESDG_MAXNQ * ESDG_MAXNQ * ESDG_MAXNQ];
  __shared__ double2 tab[64];
  const int np = g.np, Nq = g.Nq;
  for (int n = threadIdx.x; n < np; n += blockDim.x)
    w3[n] = L.w[n % Nq] * L.w[(n / Nq) % Nq] * L.w[n / (Nq * Nq)];
  for (int j = threadIdx.x; j < 64; j += blockDim.x) {
    const double r = 1.0 / (1.0 + (j + 0.5) / 64.0);
    tab[j] = make_double2(r, -log(r));
  }
  __syncthreads();
  const double gm1 = P.gamma - 1.0;
  double m = 0.0, en = 0.0, ent = 0.0;
  for (int e = blockIdx.x; e < g.E; e += gridDim.x) {
    const double* qe = q + (size_t)e * 5 * np;
    for (int n = threadIdx.x; n < np; n += blockDim.x) {
      const double rho = qe[n], m0 = qe[np + n], m1 = qe[2 * np + n], m2 = qe[3 * np + n],
                   E = qe[4 * np + n];
      const double wJ = w3[n] * J[(size_t)e * np + n];
      const double z = x[((size_t)e * 3 + 2) * np + n];
      const double ke2 = fma(m2, m2, fma(m1, m1, m0 * m0)) * esdg_rcp(rho);
      const double p = gm1 * fma(-0.5, ke2, fma(-rho, P.g * z, E));
      const double wr = wJ * rho;
      m += wr;
      en = fma(wJ, E, en);
      ent = fma(wr, fma(-P.gamma, log_tab(rho, tab), log_tab(p, tab)), ent);
    }
  }
  m = block_reduce(m, sh);
  en = block_reduce(en, sh);
  ent = block_reduce(-P.igm1 * ent, sh);
  if (threadIdx.x == 0) {
    part[(size_t)blockIdx.x * 3 + 0] = m;
    part[(size_t)blockIdx.x * 3 + 1] = en;
    part[(size_t)blockIdx.x * 3 + 2] = ent;
  }
}

// out[c] = sum of the n partials of component c (c = blockIdx.x)
__global__ void k_fold(const double* __restrict__ part, int n, double* __restrict__ out) {
  __shared__ double sh[32];
  double v = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x; k < n; k += blockDim.x) v += part[(size_t)k * 3 + blockIdx.x];
  v = block_reduce(v, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = v;
}

}  // namespace

size_t esdg_reduce_scratch(const EsdgGrid& g) { return (size_t)g.E * 3; }

cudaError_t esdg_launch_cfl(const EsdgGrid& g, const EsdgPhys& P, const double* q, const double* x,
                            const double* J, const double* Ja, double* scratch, double* out,
                            cudaStream_t s) {
  // scratch: lambda per element in FP32; its largest value behind the result, so that
  // one memset clears both
  float* lam32 = reinterpret_cast<float*>(scratch);
  unsigned* top = reinterpret_cast<unsigned*>(out + 1);
  cudaError_t err = cudaMemsetAsync(out, 0, 2 * sizeof(double), s);
  if (err != cudaSuccess) return err;
  const int warps = 8, most = SUM_CTAS;
  const int screen = (g.E + warps - 1) / warps;
  k_cfl_screen<<<screen < most ? screen : most, 32 * warps, 0, s>>>(g, P, q, x, J, Ja, lam32, top);
  err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  k_cfl_exact<<<g.E < most ? g.E : most, 128, 0, s>>>(
      g, P, q, x, J, Ja, lam32, top, reinterpret_cast<unsigned long long*>(out));
  return cudaGetLastError();
}

cudaError_t esdg_launch_integrals(const EsdgGrid& g, const EsdgLGL& L, const EsdgPhys& P,
                                  const double* q, const double* J, const double* x,
                                  double* scratch, double* out, cudaStream_t s) {
  const int thr = g.np >= 256 ? 256 : ((g.np + 31) / 32) * 32;
  const int ctas = g.E < SUM_CTAS ? g.E : SUM_CTAS;
  k_integrals<<<ctas, thr, 0, s>>>(g, L, P, q, J, x, scratch);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  k_fold<<<3, RT, 0, s>>>(scratch, ctas, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the integrals reduction (es_dg_integrals_noalloc).
//
// Some callers cannot allocate device memory at all: code running under a
// memory pool it does not own, inside a framework that forbids cudaMalloc on
// its hot path, or in a process whose allocator is already exhausted.  For
// them the partial sums (one triple per CTA) live in the file-scope array below
// instead of a handle's scratch buffer.  The array is created with the module on every
// device that loads this library and stays there until the process exits.
// ---------------------------------------------------------------------------
#include <mutex>

#include "../../include/es_dg.h"

namespace {

static __device__ __align__(256) double g_noalloc_partials[3 * SUM_CTAS];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double* g_noalloc_addr[kMaxDevices] = {nullptr};

// Device address of g_noalloc_partials on the current device.  In host code the
// symbol is only a host-side stand-in, so the address must come from
// cudaGetSymbolAddress with that device current.  It is looked up again on
// every call made while the stream is not capturing (a device reset reloads
// the module, possibly at another address); a call made during a capture uses
// the address found by the last call outside one.
int noalloc_scratch(cudaStream_t stream, double** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return ES_DG_ECUDA;
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess) {
    cudaGetLastError();
    return ES_DG_ECUDA;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (cap == cudaStreamCaptureStatusNone || !g_noalloc_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_partials) != cudaSuccess || !p) {
      cudaGetLastError();
      return ES_DG_ECUDA;
    }
    g_noalloc_addr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_addr[dev];
  return ES_DG_OK;
}

}  // namespace

extern "C" int es_dg_integrals_noalloc(const es_dg_mesh* mesh, int N, const es_dg_physics* physics,
                                       const double* q, const double* J, const double* x,
                                       double* out3, void* cuda_stream) {
  if (!mesh || !q || !J || !x || !out3 || N < 1 || N > 7) return ES_DG_EINVAL;
  if (mesh->kx < 1 || mesh->ky < 1 || mesh->kz < 1) return ES_DG_EINVAL;
  const long long E = (long long)mesh->kx * mesh->ky * mesh->kz;
  if (E > ES_DG_NOALLOC_MAX_ELEMS) return ES_DG_EINVAL;  // the documented limit
  EsdgGrid g{};
  g.K[0] = mesh->kx;
  g.K[1] = mesh->ky;
  g.K[2] = mesh->kz;
  g.N = N;
  g.Nq = N + 1;
  g.np = g.Nq * g.Nq * g.Nq;
  g.E = (int)E;
  EsdgLGL L;
  if (esdg_lgl_build(N, &L)) return ES_DG_EINVAL;
  EsdgPhys P{1.4, 9.81, 287.0, 1.0e5, 0.0, 0.0, 0.0, 1, 0.0, 0.0};
  if (physics) {
    P.gamma = physics->gamma;
    P.g = physics->g;
    P.R = physics->R;
    P.p0 = physics->p0;
    P.f0 = physics->f0;
    P.beta = physics->beta;
    P.y0 = physics->y0;
    P.dissipation = physics->dissipation;
  }
  // the checks es_dg_create applies: a bad gas constant would make every
  // integral NaN without any error being reported
  if (!(P.gamma > 1.0) || !(P.R > 0.0) || !(P.p0 > 0.0)) return ES_DG_EINVAL;
  esdg_phys_derive(&P);
  double* scratch = nullptr;
  int st = noalloc_scratch((cudaStream_t)cuda_stream, &scratch);
  if (st) return st;
  // every partial the fold reads (one triple per CTA) is written by this call,
  // so nothing needs clearing between calls
  cudaError_t e = esdg_launch_integrals(g, L, P, q, J, x, scratch, out3, (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? ES_DG_ENOMEM : ES_DG_ECUDA;
  return ES_DG_OK;
}
