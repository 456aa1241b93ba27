// volume_pipe.cuh -- tiles, bulk copies and bounded waits of the volume kernels.
#pragma once
#include "volume_pairs.cuh"

namespace esdg_vol {

// Tiles come from one mesh (SINGLE: one CTA each) or from a device work table of
// (member, first element) entries over member descriptors, which persistent CTAs walk
// (TABLE: the batched server).  A tile's bulk copies complete on an mbarrier.
#define ESDG_WAIT_LIMIT (1u << 18)  // polls; about 1 s on GB300
// Wait for a tile's copies; false when the limit ran out, here or (flag, which the
// caller sets, looked at every 1024 polls) in another CTA: the tiles after a failure do
// not each wait out the limit.
__device__ __forceinline__ bool tile_wait(unsigned long long* bar, unsigned parity, const int* flag) {
  for (unsigned it = 0; it < ESDG_WAIT_LIMIT; it += 1024u) {
    if (esdg_mbar_wait(bar, parity, 1024u)) return true;
    if (*(const volatile int*)flag) break;
  }
  return false;
}

// The tile with index t: (member, first element, elements).  TABLE: from the
// work table (EPB elements, fewer at a member's end).  SINGLE: EPB-element
// tiles up to tile t1, then tiles of s1 elements, so that the last partial
// round is spread over all SMs instead of a few.
template <bool TABLE, int EPB>
__device__ __forceinline__ int4 pipe_tile(const int2* tiles, int t, int t1, int s1, int E) {
  int e0, ne;
  if constexpr (TABLE) {
    const int2 tr = tiles[t];
    return make_int4(tr.x, tr.y, min(EPB, E - tr.y), 0);
  } else {
    if (t < t1) {
      e0 = t * EPB;
      ne = EPB;
    } else {
      e0 = t1 * EPB + (t - t1) * s1;
      ne = s1;
    }
    return make_int4(0, e0, min(ne, E - e0), 0);
  }
}

// One block copy of a tile: n doubles at src, an array that
// ends at lim, into shared memory at dst + sh with sh = (src mod 16)/8.  The
// bulk copy covers the 16-byte-aligned span enclosing the block (it reads up
// to 15 bytes before and after the block, all inside the array: array bases
// are 256-byte aligned allocations or interior pointers of them); only a block
// whose aligned end would pass lim copies its last elements with cp.async.
// dst must be 16-byte aligned with room for n + 4 elements.
struct BlockCopy {
  void* dst;
  const void* src;
  const void* lim;
  int n;
};
struct BlockSpan {
  unsigned long long a, b;  // bulk span [a, b)
  int sh, tail0;            // shift; first element copied with cp.async (n if none)
};
__device__ __forceinline__ BlockSpan bc_span(const BlockCopy& c) {
  constexpr unsigned lg = 3u;  // doubles
  const unsigned long long src = reinterpret_cast<unsigned long long>(c.src);
  const unsigned long long end = src + ((unsigned long long)c.n << lg);
  const unsigned long long lim = reinterpret_cast<unsigned long long>(c.lim);
  BlockSpan s;
  s.a = src & ~15ull;
  s.sh = (int)((unsigned)(src - s.a) >> lg);
  const unsigned long long up = (end + 15ull) & ~15ull;
  s.b = up <= lim ? up : (end & ~15ull);
  if (s.b < s.a) s.b = s.a;
  s.tail0 = s.b >= end ? c.n : (s.b > src ? (int)((s.b - src) >> lg) : 0);
  return s;
}

// Thread 0 copies a tile's block (pipe_issue registers its bytes on the barrier
// before it issues; the last elements with cp.async).  phantom: bytes registered
// but never copied (a test hook that makes the barrier's bounded wait run out; 0
// in normal operation).
__device__ __forceinline__ void pipe_issue(const BlockCopy& c, unsigned long long* bar,
                                           unsigned phantom) {
  const BlockSpan sp = bc_span(c);
  esdg_mbar_arrive_tx(bar, (unsigned)(sp.b - sp.a) + phantom);
  esdg_fence_proxy_async();
  if (sp.b > sp.a)
    esdg_bulk_g2s(c.dst, reinterpret_cast<const void*>(sp.a), (unsigned)(sp.b - sp.a), bar);
  for (int i = sp.tail0; i < c.n; i++)
    esdg_cp_async(static_cast<double*>(c.dst) + sp.sh + i, static_cast<const double*>(c.src) + i);
}

inline EsdgMember pipe_member(const EsdgGrid& g, const EsdgPhys& P, const EsdgVolArgs& a) {
  EsdgMember m;
  memset(&m, 0, sizeof(m));
  m.g = g;
  m.P = P;
  m.a = a;
  m.bg = a.bg;
  return m;
}

}  // namespace esdg_vol
