// cc_tiny.cu - a whole cc_run in one block, for graphs whose parent array fits
// its shared memory and whose edges are too few to fill more than one SM.
//
// Such a run is launches and their gaps: R-MAT scale 12 with 12K edges took 86
// us in eleven kernels and five memsets, although the edges are read in less
// than one. Here one block of 1024 threads counts degrees, picks m, hooks,
// compresses and writes the labels, with the degree counters and then the
// parent array in shared memory, where a search step takes tens of cycles.
// What bounds it: the chains of shared-memory accesses of a thread's edges, one
// after another, and the launch.
#include <cuda_runtime.h>
#include <stdint.h>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {

namespace {

constexpr int kTinyBlock = 1024, kTinyWalk = 16;

// Root name of the vertex named c, with path splitting.
template <class F>
__device__ __forceinline__ uint32_t tiny_root(volatile uint32_t *p, uint32_t c) {
  if (c == 0u) return 0u;  // the permanent root
  uint32_t pc = p[c - F::kOff];
  while (pc != c) {
    if (pc == 0u) return 0u;
    const uint32_t pw = p[pc - F::kOff];
    if (pw != pc) p[c - F::kOff] = pw;
    c = pc;
    pc = pw;
  }
  return c;
}

template <class F>
__device__ __forceinline__ void tiny_unite(uint32_t *p, const F fn, uint32_t a, uint32_t b, uint32_t n, Ctrl *ctrl) {
  if (a >= n || b >= n) {
    set_err(ctrl, kErrRange);
    return;
  }
  uint32_t ca = fn.f(a), cb = fn.f(b);
  while (true) {
    ca = tiny_root<F>(p, ca);
    cb = tiny_root<F>(p, cb);
    if (ca == cb) return;
    const uint32_t hi = max(ca, cb), lo = min(ca, cb);
    const uint32_t old = atomicCAS(p + (hi - F::kOff), hi, lo);
    if (old == hi) return;
    ca = lo;  // that root was hooked meanwhile: continue from its new parent
    cb = old;
  }
}

// Lowers the parent of the vertex of larger name to the smaller one. A link that
// another one overwrites is lost.
template <class F>
__device__ __forceinline__ void tiny_link(uint32_t *p, const F fn, uint32_t a, uint32_t b, uint32_t n) {
  if (a >= n || b >= n) return;  // (reported when the edge is joined)
  const uint32_t ca = fn.f(a), cb = fn.f(b), hi = max(ca, cb), lo = min(ca, cb);
  volatile uint32_t *const slot = p + (hi - F::kOff);
  if (hi != lo && *slot > lo) *slot = lo;
}

// Two edges that follow one another in the list start at close ids.
constexpr uint32_t kTinyClose = 64;
__device__ __forceinline__ bool tiny_close(const uint4 &e) { return max(e.x, e.z) - min(e.x, e.z) <= kTinyClose; }

// Every vertex takes its root; a long chain takes several turns.
template <class F>
__device__ __forceinline__ void tiny_compress(uint32_t *p, const F fn, uint32_t n) {
  bool deep;
  do {
    deep = false;
    for (uint32_t v = threadIdx.x; v < n; v += kTinyBlock) {
      const uint32_t c0 = *(volatile uint32_t *)(p + v);
      uint32_t c = c0;
      int steps = 0;
      for (; c != 0u && steps < kTinyWalk; ++steps) {
        const uint32_t up = *(volatile uint32_t *)(p + (c - F::kOff));
        if (up == c) break;
        c = up;
      }
      if (c != c0) *(volatile uint32_t *)(p + v) = c;
      deep |= steps == kTinyWalk;
    }
  } while (__syncthreads_or(deep));
}

// count_stride: 0 no degree count (f = id, or m given); 1 all edges; k > 1 one
// group of kSampleGroup edges in k.
// (28,672 / 1024, in whole steps of 8 registers: it fits beside the serving executor)
constexpr int kTinyRegs = kBesideExecutorRegs / kTinyBlock / 8 * 8;
static_assert(beside_executor(kTinyBlock, kTinyRegs), "and so do its warps' registers");
static_assert(kTinyVertices * sizeof(uint32_t) + 512 <= kBesideExecutorSmem, "and so do the parents");

template <class F>
__global__ void __maxnreg__(kTinyRegs)
    k_tiny(const uint4 *__restrict__ e4, uint32_t n_quads, const uint2 *head, const uint2 *tail, uint32_t *P,
           uint32_t n, Ctrl *ctrl, uint32_t count_stride, uint32_t m_hint, int min_id, uint32_t *__restrict__ L) {
  extern __shared__ uint32_t p[];  // degrees, then parents
  __shared__ unsigned long long s_key[kTinyBlock / 32];
  __shared__ uint32_t s_gmin, s_roots;
  const uint32_t t = threadIdx.x, h = head ? 1u : 0u;
  uint32_t m = m_hint;
  if (F::kRF && count_stride) {
    for (uint32_t v = t; v < n; v += kTinyBlock) p[v] = 0u;
    __syncthreads();
    auto count = [&](uint32_t i, uint32_t a, uint32_t b) {  // edge i of the list
      if ((i >> kSampleGroupShift) % count_stride) return;
      if (a < n) atomicAdd(p + a, 1u);
      if (b < n) atomicAdd(p + b, 1u);
    };
    if (t == 0 && head) count(0, head->x, head->y);
    if (t == 1 && tail) count(h + 2 * n_quads, tail->x, tail->y);
    for (uint32_t q = t; q < n_quads; q += kTinyBlock) {
      const uint4 e = __ldg(e4 + q);
      count(h + 2 * q, e.x, e.y);
      count(h + 2 * q + 1, e.z, e.w);
    }
    __syncthreads();
    unsigned long long key = 0;  // the largest degree, of those the smallest id
    for (uint32_t v = t; v < n; v += kTinyBlock) {
      const unsigned long long k = ((unsigned long long)p[v] << 32) | (uint32_t)~v;
      key = k > key ? k : key;
    }
    key = warp_max_u64(key);
    if ((t & 31u) == 0u) s_key[t >> 5] = key;
    __syncthreads();
    key = warp_max_u64(s_key[t & 31u]);
    m = ~(uint32_t)key;
  }
  F fn;
  if constexpr (F::kRF) fn.m = m;
  for (uint32_t v = t; v < n; v += kTinyBlock) p[v] = fn.f(v);
  if (t == 0) {
    s_gmin = m;
    s_roots = 0u;
  }
  // Link first, one round, where it saves time. A list in the order of a path or a
  // lattice builds its long chains while every thread walks down them: path of
  // 20000 vertices (f = id) 630 us without and 78 with it, 130 in the general
  // pass; of 4000 103, 27 and 36. With more edges than vertices most of the joining
  // is done at once: R-MAT scale 12, 3 edges a vertex, 33.4 -> 29.3. In other lists
  // the round costs more than it saves: 32,767 uniform edges on 48K vertices 77 and 111.
  const uint32_t first = min(n_quads, (uint32_t)kTinyBlock);
  const int close = __syncthreads_count(t < first && tiny_close(__ldg(e4 + t)));
  if (2u * n_quads > n || (first && 4u * close >= first)) {
    for (uint32_t q = t; q < n_quads; q += kTinyBlock) {
      const uint4 e = __ldg(e4 + q);
      tiny_link(p, fn, e.x, e.y, n);
      tiny_link(p, fn, e.z, e.w, n);
    }
    __syncthreads();
    tiny_compress(p, fn, n);
  }
  if (t == 0 && head) tiny_unite(p, fn, head->x, head->y, n, ctrl);
  if (t == 1 && tail) tiny_unite(p, fn, tail->x, tail->y, n, ctrl);
  for (uint32_t q = t; q < n_quads; q += kTinyBlock) {
    const uint4 e = __ldg(e4 + q);
    tiny_unite(p, fn, e.x, e.y, n, ctrl);
    tiny_unite(p, fn, e.z, e.w, n, ctrl);
  }
  __syncthreads();
  uint32_t roots = 0, least = 0xFFFFFFFFu;
  for (uint32_t v = t; v < n; v += kTinyBlock) {
    const uint32_t c = fn.f(v), r = tiny_root<F>(p, c);
    if (r == c)
      ++roots;
    else
      *(volatile uint32_t *)(p + v) = r;
    if (r == 0u && v < least) least = v;
  }
  roots = __reduce_add_sync(0xFFFFFFFFu, roots);
  least = __reduce_min_sync(0xFFFFFFFFu, least);
  if ((t & 31u) == 0u) {
    atomicAdd(&s_roots, roots);
    atomicMin(&s_gmin, least);
  }
  __syncthreads();
  const uint32_t gmin = s_gmin;
  for (uint32_t v = t; v < n; v += kTinyBlock) {
    // (a split of the loop above may have put back an older ancestor)
    const uint32_t r = tiny_root<F>(p, fn.f(v));
    P[v] = r;
    if (L) L[v] = F::kRF && min_id ? (r == 0u ? gmin : r - 1u) : r;
  }
  if (t == 0) {
    ctrl->m = F::kRF ? m : 0u;
    ctrl->gmin = F::kRF && min_id && L ? gmin : (F::kRF ? m : 0u);
    ctrl->ncomp = s_roots;
    ctrl->cert = 0u;  // no certificate: inserts take the form for any graph
  }
}

}  // namespace

bool tiny_fits(uint64_t n_vertices, uint64_t n_edges) {
  return n_vertices >= 1 && n_vertices <= kTinyVertices && n_edges <= kTinyEdges;
}

cudaError_t launch_tiny(bool rf, const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl, uint32_t count_stride,
                        uint32_t m_hint, int label_space, uint32_t *L, cudaStream_t s) {
  static std::atomic<unsigned long long> set_r{0}, set_i{0};
  const void *k = rf ? (const void *)k_tiny<RootR> : (const void *)k_tiny<RootId>;
  const cudaError_t err = ensure_func_attr(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)(kTinyVertices * sizeof(uint32_t)), rf ? set_r : set_i);
  if (err != cudaSuccess) return err;
  const size_t smem = (size_t)n * sizeof(uint32_t);
  const int min_id = label_space == kLabelMinId;
  if (rf)
    k_tiny<RootR><<<1, kTinyBlock, smem, s>>>(e.quads, (uint32_t)e.n_quads, e.head, e.tail, P, n, ctrl, count_stride,
                                              m_hint, min_id, L);
  else
    k_tiny<RootId><<<1, kTinyBlock, smem, s>>>(e.quads, (uint32_t)e.n_quads, e.head, e.tail, P, n, ctrl, 0u, 0u, min_id,
                                               L);
  note_launch();
  return cudaGetLastError();
}

}  // namespace cc
