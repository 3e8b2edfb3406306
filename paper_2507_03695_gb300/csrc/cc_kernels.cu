// cc_kernels.cu - CUDA kernels of the connected-components hot path for
// sm_103a and their launchers:
//   root selection  degree histogram + argmax (Algorithm 4, max_degree())
//   init            P_v = f(v)                 (Algorithm 3, initialisation)
//   edge pass       one hooking pass           (Algorithm 3, hooking)
//   min-id probe    smallest vertex of m's component (min-id labels under R)
//   flatten         labels + compression       (Algorithm 3, pointer jumping)
//   count, connected, validate                 (queries and insert checks)
#include <cuda_runtime.h>
#include <stdint.h>

#include <array>
#include <atomic>
#include <map>
#include <mutex>
#include <shared_mutex>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {

namespace {

int g_num_sms = 0;

// ------------------------------------------------------------------- init

template <class F>
__global__ void __launch_bounds__(256) k_init(uint32_t *__restrict__ P, uint32_t n, Ctrl *ctrl,
                                              int m_src, uint32_t m_hint, const uint32_t *skip) {
  if (skip && ld_volatile_u32(skip)) return;
  uint32_t m = 0;
  if (F::kRF) {
    if (m_src == kMFromHint)
      m = m_hint;
    else
      m = ~(uint32_t)(*(volatile unsigned long long *)&ctrl->maxkey);
    if (m >= n) m = 0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctrl->m = m;
    ctrl->gmin = m;
    ctrl->ncomp = 0ULL;
  }
  const uint64_t n4 = n / 4u;
  uint4 *P4 = reinterpret_cast<uint4 *>(P);
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n4;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = (uint32_t)(4 * i);
    uint4 r;
    if (F::kRF) {
      r = make_uint4(v + 1u, v + 2u, v + 3u, v + 4u);
      if (m - v < 4u) {
        if (m == v) r.x = 0u;
        if (m == v + 1u) r.y = 0u;
        if (m == v + 2u) r.z = 0u;
        if (m == v + 3u) r.w = 0u;
      }
    } else {
      r = make_uint4(v, v + 1u, v + 2u, v + 3u);
    }
    P4[i] = r;
  }
  if (blockIdx.x == 0 && threadIdx.x < (n & 3u)) {
    const uint32_t v = (uint32_t)(4 * n4) + threadIdx.x;
    P[v] = F::kRF ? (v == m ? 0u : v + 1u) : v;
  }
}

// --------------------------------------------------------------- edge pass

// Direct form: each thread takes Q 128-bit loads (2Q edges) per iteration,
// issues all 4Q parent loads together, then resolves its edges one by one.
template <class F, int Q>
__global__ void __launch_bounds__(512) k_edge_pass_direct(const uint4 *__restrict__ e4,
                                                          uint64_t n_quads, const uint2 *head,
                                                          const uint2 *tail, uint32_t *P,
                                                          uint32_t n, Ctrl *ctrl, const uint32_t *skip) {
  if (skip && ld_volatile_u32(skip)) return;
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  const uint64_t pol = policy_evict_first();
  const uint64_t T = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (t == 0 && head) single_edge(P, fn, head, n, ctrl);
  if (t == 1 % T && tail) single_edge(P, fn, tail, n, ctrl);
  for (uint64_t base = t; base < n_quads; base += T * Q) {
    uint4 e[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      const uint64_t q = base + (uint64_t)j * T;
      e[j] = q < n_quads ? ld_edges(e4 + q, pol) : make_uint4(0u, 0u, 0u, 0u);
    }
    uint32_t p[4 * Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      guard(e[j].x, e[j].y, n, ctrl);
      guard(e[j].z, e[j].w, n, ctrl);
      p[4 * j + 0] = ldP(P + e[j].x);
      p[4 * j + 1] = ldP(P + e[j].y);
      p[4 * j + 2] = ldP(P + e[j].z);
      p[4 * j + 3] = ldP(P + e[j].w);
    }
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      unite(S, fn.f(e[j].x), p[4 * j + 0], fn.f(e[j].y), p[4 * j + 1]);
      unite(S, fn.f(e[j].z), p[4 * j + 2], fn.f(e[j].w), p[4 * j + 3]);
    }
  }
}

// Filtered form: the parent loads of a warp's edges feed the warp ring
// (cc_device.cuh), which drops edges whose endpoints already share a parent
// and resolves the survivors in dense warps.
//
// kZ: the zero-tree bitmap Z (one bit per name, 1/32 of P) stands in front of
// P. An endpoint whose bit is set belongs to the tree of name 0, so its parent
// value is taken as 0 without loading P; an edge with both bits set costs no
// parent load at all. When P is larger than L2 and the giant component hangs
// under name 0 (R with a dominant hub), this turns most random DRAM reads of
// P into L2 hits on Z. Bits are set when a parent value of 0 is read and when
// an edge ends in the tree of name 0.
//
// Instances, chosen at run time by the word *sel (the certificate flag):
//   kZ (with kDirect): the zero-tree form, for a certified hub when Z exists;
//   !kZ, !kDirect: the plain form that always queues, for a certified hub
//     whose P fits L2 (resolving in place cost a few percent there);
//   !kZ, kDirect: the plain form that resolves nearly full warps in place,
//     for graphs without a certified hub; capped at 32 registers, because
//     that search-bound pass gains more from resident warps than it loses
//     to a few spilled registers.
// The register caps (the launch bounds' minimum blocks) were measured.
// The hub-serving instances run only when *sel is nonzero, the other only
// when it is zero; with sel null the launched instance runs.
//
// skip: nothing is done when the word is 1; k + 1: about k of the blocks work, and
// claim (work is then given); 0: all.
// work: the dynamic schedule. Warps claim `grab` steps of 32 * Q consecutive
// quads at a time from *work, so warps whose edges need long searches do not
// set the end of the kernel; null: each warp takes a fixed stride of steps.
// The claim size is chosen by the launcher (grab_for). fixed: they do so only when
// the skip word lets few blocks work.
//
// hot (hub instances only): the hot-vertex table of the root selection
// (CertScratch::hot). Each block copies its vertex ids into shared memory
// after the ring and learns, per entry, whether that vertex is known to be in
// the tree of name 0; an endpoint known so skips its bitmap or parent load.
// The table covers 3-8% of R-MAT endpoint occurrences at 4096 entries
// (measured edge pass, R-MAT 28: 32.50 -> 31.61 ms, R-MAT 24: 1.94 -> 1.79);
// 8192 entries lost occupancy and ran slower.

template <class F, int Q, bool kZ, bool kDirect, bool kL2 = false>
__global__ void __launch_bounds__(512, Q >= 4 ? (kZ ? 1 : 2) : (kZ ? 2 : (kDirect ? 4 : 3)))
    k_edge_pass_filtered(const uint4 *__restrict__ e4, uint64_t n_quads, const uint2 *head, const uint2 *tail,
                         uint32_t *P, uint32_t n, Ctrl *ctrl, const uint32_t *skip, uint32_t *Z,
                         const uint32_t *sel, uint32_t *log, unsigned long long *work, uint32_t grab,
                         const unsigned long long *hot, bool fixed = false) {
  static_assert(kDirect || !kZ, "the zero-tree form resolves in place");
  // kL2 (the queue form on a parent array of at least kL2MinVertices): P is
  // read through L2 only. Its random parent loads almost never hit L1 then,
  // and skipping L1 allocation measured faster (R-MAT scale 24: 2.02 -> 1.94
  // ms); a small P lives in L1 (R-MAT 16's 256 KB: 0.077 ms with L1, 0.13
  // without), and the grid's searches hit L1 (1.27 ms without it, 0.94 with).
  static_assert(!kL2 || (!kZ && !kDirect), "L2-only loads only in the queue form");
  constexpr bool kCG = kL2;
  extern __shared__ uint32_t ring_smem[];
  // (read through L1: every warp of the grid does)
  bool all = true;
  if (skip) {
    const uint32_t w = __ldca(skip), few = w - 1u;
    all = w == 0u || few >= gridDim.x;
    // about that many, spread at uneven distances over the grid, so over the SMs
    // (every eighth block of 512 ran half as fast); block 0 is one of them
    if (!all && __umulhi(blockIdx.x * 2654435769u, gridDim.x) >= few) return;
  }
  if (sel && ((__ldca(sel) != 0u) != (kZ || !kDirect))) return;
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  const uint64_t pol = policy_evict_first();
  WarpRing ring;
  ring.init(ring_smem, kZ ? Z : nullptr, log, kDirect ? kDirectMin : kNeverDirect);
  const uint64_t T = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  // the table: entry v + 1 of a hot vertex v, top bit once v is known to be
  // in the tree of name 0 (0: an empty slot)
  constexpr bool kHub = F::kRF && (kZ || !kDirect);
  uint32_t *const H = ring_smem + (blockDim.x >> 5) * 4 * kRing;
  const bool use_hot = kHub && hot != nullptr;
  if (use_hot) {
    for (uint32_t i = threadIdx.x; i < kHot; i += blockDim.x) H[i] = (uint32_t)hot[i];
    __syncthreads();
  }
  if (t == 0 && head) single_edge(P, fn, head, n, ctrl, log);
  if (t == 1 % T && tail) single_edge(P, fn, tail, n, ctrl, log);
  // One warp step: lane l takes quads base + j * stride (j < Q), base being
  // the warp's first quad plus l; the trip counts stay warp-uniform.
  auto step = [&](uint64_t base, uint64_t stride) {
    uint4 e[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      const uint64_t q = base + (uint64_t)j * stride;
      e[j] = q < n_quads ? ld_edges(e4 + q, pol) : make_uint4(0u, 0u, 0u, 0u);
    }
    uint32_t p[4 * Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      guard(e[j].x, e[j].y, n, ctrl);
      guard(e[j].z, e[j].w, n, ctrl);
    }
    // bit i of hz: endpoint i is known (by the table) to be in the tree of
    // name 0; of hk: endpoint i is its slot's vertex
    uint32_t hz = 0, hk = 0;
    if (use_hot) {
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        const uint32_t xs[4] = {e[j].x, e[j].y, e[j].z, e[j].w};
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
          const uint32_t ent = H[hot_slot(xs[k2])];
          hz |= (uint32_t)(ent == ((xs[k2] + 1u) | 0x80000000u)) << (4 * j + k2);
          hk |= (uint32_t)((ent & 0x7FFFFFFFu) == xs[k2] + 1u) << (4 * j + k2);
        }
      }
    }
    if (kZ) {
      uint32_t z = hz;  // bit i: endpoint i is known to be in the tree of name 0
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        if (!((hz >> (4 * j + 0)) & 1u)) z |= (uint32_t)zbit(Z, fn.f(e[j].x)) << (4 * j + 0);
        if (!((hz >> (4 * j + 1)) & 1u)) z |= (uint32_t)zbit(Z, fn.f(e[j].y)) << (4 * j + 1);
        if (!((hz >> (4 * j + 2)) & 1u)) z |= (uint32_t)zbit(Z, fn.f(e[j].z)) << (4 * j + 2);
        if (!((hz >> (4 * j + 3)) & 1u)) z |= (uint32_t)zbit(Z, fn.f(e[j].w)) << (4 * j + 3);
      }
      if (use_hot) {  // learn: a hot endpoint whose bitmap bit is set
        const uint32_t learn = z & hk & ~hz;
        if (learn) {
#pragma unroll
          for (int j = 0; j < Q; ++j) {
            const uint32_t xs[4] = {e[j].x, e[j].y, e[j].z, e[j].w};
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2)
              if ((learn >> (4 * j + k2)) & 1u) H[hot_slot(xs[k2])] = (xs[k2] + 1u) | 0x80000000u;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        p[4 * j + 0] = (z >> (4 * j + 0)) & 1u ? 0u : ldP(P + e[j].x);
        p[4 * j + 1] = (z >> (4 * j + 1)) & 1u ? 0u : ldP(P + e[j].y);
        p[4 * j + 2] = (z >> (4 * j + 2)) & 1u ? 0u : ldP(P + e[j].z);
        p[4 * j + 3] = (z >> (4 * j + 3)) & 1u ? 0u : ldP(P + e[j].w);
      }
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        if (!((z >> (4 * j + 0)) & 1u) && p[4 * j + 0] == 0u) zset(Z, fn.f(e[j].x));
        if (!((z >> (4 * j + 1)) & 1u) && p[4 * j + 1] == 0u) zset(Z, fn.f(e[j].y));
        if (!((z >> (4 * j + 2)) & 1u) && p[4 * j + 2] == 0u) zset(Z, fn.f(e[j].z));
        if (!((z >> (4 * j + 3)) & 1u) && p[4 * j + 3] == 0u) zset(Z, fn.f(e[j].w));
      }
    } else {
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        p[4 * j + 0] = ((hz >> (4 * j + 0)) & 1u) ? 0u : ldP_t<kCG>(P + e[j].x);
        p[4 * j + 1] = ((hz >> (4 * j + 1)) & 1u) ? 0u : ldP_t<kCG>(P + e[j].y);
        p[4 * j + 2] = ((hz >> (4 * j + 2)) & 1u) ? 0u : ldP_t<kCG>(P + e[j].z);
        p[4 * j + 3] = ((hz >> (4 * j + 3)) & 1u) ? 0u : ldP_t<kCG>(P + e[j].w);
      }
      if (use_hot) {  // learn: a hot endpoint whose parent is name 0
#pragma unroll
        for (int j = 0; j < Q; ++j) {
          const uint32_t xs[4] = {e[j].x, e[j].y, e[j].z, e[j].w};
#pragma unroll
          for (int k2 = 0; k2 < 4; ++k2)
            if (((hk & ~hz) >> (4 * j + k2)) & 1u && p[4 * j + k2] == 0u)
              H[hot_slot(xs[k2])] = (xs[k2] + 1u) | 0x80000000u;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 2 * Q; ++k) {
      const uint32_t a = (k & 1) ? e[k >> 1].z : e[k >> 1].x;
      const uint32_t b = (k & 1) ? e[k >> 1].w : e[k >> 1].y;
      const uint32_t pa = p[2 * k], pb = p[2 * k + 1];
      ring.push<kCG>(S, pa != pb, fn.f(a), pa, fn.f(b), pb);
    }
  };
  if (work && !(fixed && all)) {
    // dynamic: warps claim `grab` steps of 32 * Q consecutive quads at a time,
    // so warps whose edges need longer searches do not set the kernel's end
    const uint64_t steps = (n_quads + 32u * Q - 1) / (32u * Q);
    for (;;) {
      unsigned long long g0 = 0;
      if (ring.lane == 0) g0 = atomicAdd(work, (unsigned long long)grab);
      g0 = __shfl_sync(0xFFFFFFFFu, g0, 0);
      if (g0 >= steps) break;
      const uint64_t g1 = g0 + grab < steps ? g0 + grab : steps;
      for (uint64_t g = g0; g < g1; ++g) step(g * 32u * Q + ring.lane, 32u);
    }
  } else {
    const uint64_t warp_t0 = t - (uint64_t)ring.lane;
    for (uint64_t wbase = warp_t0; wbase < n_quads; wbase += T * Q) step(wbase + ring.lane, T);
  }
  ring.drain<kCG>(S);
}

// The edge pass of a certified hub on a large graph (from 2^22 vertices up,
// default launch shape): as the hub forms above, with the wide hot-vertex
// table (WideHot) in place of the 4096-entry one. Its blocks do not fit beside the
// serving executor's, so without the bitmap it runs only while no server is
// open (ExecutorBlocks) and in no captured run; the bitmap's other form (64 registers a thread, blocks
// of 512) does not fit there either. Smaller blocks lose more than the table
// gives: R-MAT scale 24, whole call, 1830 us with 1024 threads, 2274 with 512 of
// 56 registers, 2395 with 576 of 48, 2500 with 704 of 40, 2176 without the table.
//
// What bounds it: the endpoint lookups, one L2 request each, at most 0.96 per
// SM and clock; random shared-memory loads beside them cost nothing (16 per 8
// lookups left the rate at 0.96). So one block of 1024 threads per SM gives
// 128 KB of its shared memory to the table, which answers 32 warps' lookups
// of the hottest vertices: on R-MAT scale 24 (98K entries) L2 requests fell
// from 489M to 348M. Edge pass before and after: R-MAT scale 28 31.24 -> 27.5
// ms, 26 (edge factor 16) 7.64 -> 6.68, 24 1.70 -> 1.37, 22 with 2^27 edges
// 0.86 -> 0.59.
//
// A bucket is one word of up to four fields; a field holds the identifying
// bits of one vertex and, in its top bit, whether this block knows the vertex
// to be in the tree of name 0. One exact test covers all fields: after the
// exclusive or with the wanted bits and with every top bit set, subtracting
// one from each field clears its top bit exactly where the bits agree.
// Empty fields hold bits of a vertex of the same bucket (or of none below n)
// and no flag, so they cannot answer wrongly.
//
// Flags are learnt in bulk: after its 2nd, 8th, 32nd ... claim a warp looks up
// its share of the table's vertices. A round costs up to 98K lookups a block,
// most of a claim's: R-MAT scale 24 takes 1.42 ms with rounds after the 1st,
// 2nd, 4th, 8th ... claim, 1.37 after the 1st, 4th, 16th ..., 1.35 like this and
// 1.36 after the 4th, 16th, 64th. Learning inside the loop, for
// every lookup that found 0, cost more instructions than the table saved
// requests (1.74 ms on R-MAT scale 24); only the queue form does it, and only
// during its first claim, when the hubs have just joined and their lookups
// would all meet in one L2 sector (rmat 22: 0.49 -> 0.44 ms).
//
// kZ: with the zero-tree bitmap. The loop then only reads bits, Q = 4 quads
// per step, and an edge whose endpoints are not both known goes to the queue as
// two ids; a full queue loads the parents of 32 edges at once (27.5 ms on R-MAT
// scale 28 against 28.4 with predicated parent loads in every step).
// Without Z the parents are the filter, loaded through L2 only, and the next
// step's edges are loaded ahead (1.52 -> 1.47 ms on R-MAT scale 24; with Z
// the registers for it cost more than it gave).
constexpr int kHubBlock = 1024;
constexpr uint32_t kHubClaimQuads = 1024;  // quads a warp claims at a time (512 and 2048 were slower)
constexpr size_t kHubSmem = (size_t)(kHubBlock / 32) * 4 * kRing * sizeof(uint32_t) + kWideBuckets * sizeof(uint32_t);

template <bool kZ>
__global__ void __launch_bounds__(kHubBlock, 1)
    k_edge_pass_hub(const uint4 *__restrict__ e4, uint64_t n_quads, const uint2 *head, const uint2 *tail, uint32_t *P,
                    uint32_t n, Ctrl *ctrl, uint32_t *Z, const uint32_t *sel, unsigned long long *work,
                    const uint32_t *__restrict__ wide, uint32_t s_bits, uint32_t ways) {
  constexpr int Q = kZ ? 4 : 2;
  constexpr bool kAhead = !kZ;
  extern __shared__ uint32_t ring_smem[];
  if (ld_volatile_u32(sel) == 0u) return;
  const RootR fn = RootR::load(ctrl);
  uint32_t *const S = slots<RootR>(P);
  const uint64_t pol = policy_evict_first();
  WideTable table;
  table.load(ring_smem, wide, s_bits, ways);
  WarpRing ring;
  ring.init(ring_smem + kWideBuckets, nullptr, nullptr, kNeverDirect);
  __syncthreads();
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (t == 0 && head) single_edge(P, fn, head, n, ctrl);
  if (t == 1 && tail) single_edge(P, fn, tail, n, ctrl);
  auto load = [&](uint4 (&e)[Q], uint64_t base) {
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      const uint64_t q = base + (uint64_t)j * 32u;
      e[j] = q < n_quads ? ld_edges_now(e4 + q, pol) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  // kZ: joins `count` queued edges (ids; top bit: known to be in the tree of name 0).
  auto resolve = [&](uint32_t count) {
    __syncwarp();
    const uint32_t slot = (ring.head + ring.lane) & (kRing - 1);
    const uint32_t xa = ring.cu[slot], xb = ring.cv[slot];
    __syncwarp();
    if (ring.lane < count) {
      const bool ka = xa >> 31, kb = xb >> 31;
      const uint32_t va = xa & 0x7FFFFFFFu, vb = xb & 0x7FFFFFFFu;
      uint32_t pa = 0u, pb = 0u;
      if (!ka) pa = ldP(P + va);
      if (!kb) pb = ldP(P + vb);
      bool za = !ka && pa == 0u, zb = !kb && pb == 0u;
      if (pa != pb) {
        const UniteResult res = unite(S, fn.f(va), pa, fn.f(vb), pb);
        za |= res.zero && !ka;
        zb |= res.zero && !kb;
      }
      if (za) zset(Z, fn.f(va));
      if (zb) zset(Z, fn.f(vb));
    }
    ring.head += count;
  };
  auto step = [&](uint4 (&e)[Q], bool learning) {
    uint32_t x[4 * Q], p[4 * Q];  // endpoints; bitmap words (kZ) or parent values
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      if (max(max(e[j].x, e[j].y), max(e[j].z, e[j].w)) >= n) {
        guard(e[j].x, e[j].y, n, ctrl);
        guard(e[j].z, e[j].w, n, ctrl);
      }
      x[4 * j + 0] = e[j].x;
      x[4 * j + 1] = e[j].y;
      x[4 * j + 2] = e[j].z;
      x[4 * j + 3] = e[j].w;
    }
#pragma unroll
    for (int i = 0; i < 4 * Q; ++i) {
      const bool known = table.known(x[i]);
      if (kZ) {
        p[i] = 0xFFFFFFFFu;
        if (!known) p[i] = ldP(Z + (fn.f(x[i]) >> 5));
      } else {
        p[i] = 0u;
        if (!known) p[i] = ldP_cg(P + x[i]);
      }
    }
    if (!kZ && learning) {
#pragma unroll
      for (int i = 0; i < 4 * Q; ++i)
        if (p[i] == 0u) table.learn(x[i]);
    }
#pragma unroll
    for (int k = 0; k < 2 * Q; ++k) {
      const uint32_t xa = x[2 * k], xb = x[2 * k + 1];
      if (kZ) {
        const uint32_t ka = (p[2 * k] >> (fn.f(xa) & 31u)) & 1u, kb = (p[2 * k + 1] >> (fn.f(xb) & 31u)) & 1u;
        const bool keep = !(ka & kb) && xa != xb;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
        if (!bal) continue;
        if (keep) {
          const uint32_t slot = (ring.tail + __popc(bal & ring.lt_mask)) & (kRing - 1);
          ring.cu[slot] = xa | (ka << 31);
          ring.cv[slot] = xb | (kb << 31);
        }
        ring.tail += __popc(bal);
        if (ring.tail - ring.head >= 32u) resolve(32u);
      } else {
        ring.push<true>(S, p[2 * k] != p[2 * k + 1], fn.f(xa), p[2 * k], fn.f(xb), p[2 * k + 1]);
      }
    }
  };
  constexpr uint32_t kGrab = kHubClaimQuads / (32u * Q);
  const uint32_t steps = (uint32_t)((n_quads + 32u * Q - 1) / (32u * Q));  // below 2^32 (kHubMaxQuads)
  for (uint32_t claims = 0, learn_at = 2;;) {
    uint32_t g0 = 0;
    if (ring.lane == 0) g0 = (uint32_t)min(atomicAdd(work, (unsigned long long)kGrab), (unsigned long long)steps);
    g0 = __shfl_sync(0xFFFFFFFFu, g0, 0);
    if (g0 >= steps) break;
    const uint32_t g1 = min(g0 + kGrab, steps);
    uint4 e[Q];
    if (kAhead) load(e, (uint64_t)g0 * (32u * Q) + ring.lane);
    for (uint32_t g = g0; g < g1; ++g) {
      uint4 cur[Q];
      if (kAhead) {
#pragma unroll
        for (int j = 0; j < Q; ++j) cur[j] = e[j];
        if (g + 1u < g1) load(e, (uint64_t)(g + 1u) * (32u * Q) + ring.lane);
      } else {
        load(cur, (uint64_t)g * (32u * Q) + ring.lane);
      }
      step(cur, claims == 0u);
    }
    ++claims;
    if (claims == learn_at) {
      learn_at *= 4;
      table.learn_share<kHubBlock / 32>(
          n, [&](uint32_t v) { return kZ ? zbit(Z, fn.f(v)) : ldP_cg(P + v) == 0u; });
    }
  }
  if (kZ) {
    if (ring.tail != ring.head) resolve(ring.tail - ring.head);
  } else {
    ring.drain<true>(S);
  }
}

// kProbe: one more block looks at kProbes pairs of quads spread over the list.
// Where half of them join two vertices that nothing has joined yet, that part of
// the graph still has to grow its trees, and only `few` blocks of the edge pass
// are to work, so that fewer edges meet on the first roots. It clears the edge
// pass's counter too. An id out of range lets no block work.
constexpr uint32_t kProbes = 256;

template <class F, bool kProbe>
__global__ void __launch_bounds__(256) k_validate(const uint4 *__restrict__ e4, uint64_t n_quads,
                                                  const uint2 *head, const uint2 *tail, uint32_t n,
                                                  Ctrl *ctrl, uint32_t *reject, const uint32_t *P, uint32_t few) {
  if (kProbe && blockIdx.x == gridDim.x - 1u) {
    static_assert(kProbes == 256, "one per thread");
    const F fn = F::load(ctrl);
    const uint4 e = __ldg(e4 + n_quads * threadIdx.x / kProbes);
    const bool fresh = e.x < n && e.y < n && ldP_cg(P + e.x) == fn.f(e.x) && ldP_cg(P + e.y) == fn.f(e.y);
    const int grows = __syncthreads_count(fresh);
    if (threadIdx.x == 0) {
      ctrl->work = 0ULL;
      if (2 * grows >= (int)kProbes) atomicCAS(reject, 0u, few + 1u);
    }
    return;
  }
  const uint64_t pol = policy_evict_first();
  const uint64_t T = (uint64_t)(gridDim.x - (kProbe ? 1u : 0u)) * blockDim.x;
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  bool bad = false;
  if (t == 0 && head) {
    uint2 e = ld_edge(head);
    bad |= e.x >= n || e.y >= n;
  }
  if (t == 1 % T && tail) {
    uint2 e = ld_edge(tail);
    bad |= e.x >= n || e.y >= n;
  }
  for (uint64_t q = t; q < n_quads; q += T) {
    const uint4 e = ld_edges(e4 + q, pol);
    bad |= (e.x >= n) | (e.y >= n) | (e.z >= n) | (e.w >= n);
  }
  if (__any_sync(0xFFFFFFFFu, bad) && (threadIdx.x & 31) == 0) {
    atomicExch(reject, 1u);
    set_err(ctrl, kErrRange);
  }
}

// A short insert in one block, which validates all pairs, loads all parents, then
// hooks the pairs. Four launches and two memsets otherwise took longer than the
// work. The parents are those from before any hook: loaded later, the pairs of a
// path in order walk down the chain that the others have built (4096 of them: 568
// us instead of 14). They are kept in shared memory: the registers that are left
// beside the serving executor do not hold them. 1024 threads fit beside three of
// its blocks per SM, 512 beside four.
template <int kInsertBlock>
constexpr int kInsertRegs = kInsertBlock == 1024 ? kBesideExecutorRegs / 1024 / 8 * 8 : kSmallBlockRegs;

template <class F, int kInsertBlock>
__global__ void __maxnreg__(kInsertRegs<kInsertBlock>) k_insert_small(const uint2 *__restrict__ e, uint32_t n_edges, uint32_t *P,
                                                        uint32_t n, Ctrl *ctrl) {
  extern __shared__ uint4 pairs[];  // the ids, then the parents
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  bool bad = false;
#pragma unroll 2
  for (uint32_t i = threadIdx.x; i < n_edges; i += kInsertBlock) {
    const uint2 x = ld_edge(e + i);
    const bool ok = x.x < n && x.y < n;
    bad |= !ok;
    pairs[i] = make_uint4(x.x, x.y, ok ? ldP_cg(P + x.x) : 0u, ok ? ldP_cg(P + x.y) : 0u);
  }
  if (__syncthreads_or(bad)) {  // nothing is applied
    if (threadIdx.x == 0) set_err(ctrl, kErrRange);
    return;
  }
  for (uint32_t i = threadIdx.x; i < n_edges; i += kInsertBlock) {
    const uint4 x = pairs[i];
    unite<true>(S, fn.f(x.x), x.z, fn.f(x.y), x.w);
  }
}

// ------------------------------------------------------------------ flatten

// Smallest vertex whose root value is 0 under R. Its answer is at most m, so
// only [0, m) is scanned, in chunks of increasing id; a block stops as soon as
// its next chunk starts above the best candidate found so far.
__global__ void __launch_bounds__(256) k_gmin_probe(uint32_t *P, uint32_t n, Ctrl *ctrl) {
  const RootR fn = RootR::load(ctrl);
  const uint32_t m = fn.m;
  __shared__ uint32_t s_stop, s_best;
  const uint64_t chunk = 4ull * blockDim.x;
  for (uint64_t c = blockIdx.x;; c += gridDim.x) {
    const uint64_t start = c * chunk;
    if (threadIdx.x == 0) {
      s_stop = (start >= m) || (start > ld_volatile_u32(&ctrl->gmin));
      s_best = 0xFFFFFFFFu;
    }
    __syncthreads();
    const bool stop = s_stop;
    __syncthreads();
    if (stop) return;
    uint32_t best = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint64_t v = start + (uint64_t)k * blockDim.x + threadIdx.x;
      if (v < m && v < best) {
        const uint32_t pv = ldP(P + v);
        if (root_name(slots<RootR>(P), fn.f((uint32_t)v), pv) == 0u) best = (uint32_t)v;
      }
    }
    // one global atomic per block and chunk at most: the first chunks nearly
    // always hold the answer, and an atomic per warp of the whole grid on the
    // one word took longer than the scan (R-MAT scale 20: 9.9 us, 24: 14.3)
    best = __reduce_min_sync(0xFFFFFFFFu, best);
    if ((threadIdx.x & 31) == 0 && best != 0xFFFFFFFFu) atomicMin(&s_best, best);
    __syncthreads();
    if (threadIdx.x == 0 && s_best < ld_volatile_u32(&ctrl->gmin)) atomicMin(&ctrl->gmin, s_best);
  }
}

// Adds the block's roots to ctrl->ncomp, one global atomic per block: one per
// warp met on the one word for longer than a small flatten takes (R-MAT scale
// 20, flatten: 16.3 us). Every thread of the block calls it.
__device__ __forceinline__ void add_roots(unsigned long long roots, Ctrl *ctrl) {
  __shared__ unsigned long long s_roots;
  if (threadIdx.x == 0) s_roots = 0ULL;
  __syncthreads();
  roots = warp_sum_u64(roots);
  if ((threadIdx.x & 31) == 0 && roots) atomicAdd(&s_roots, roots);
  __syncthreads();
  if (threadIdx.x == 0 && s_roots) atomicAdd(&ctrl->ncomp, s_roots);
}

// Pointer jumping (Algorithm 3): every vertex finds its root name c with
// path splitting, stores c into P (compression; roots are never written) and,
// when L is given, writes its label: the root's name (root-value labels, and
// min-id labels under f = id), or under f = R the root's id c - 1 for c != 0
// and the smallest vertex of m's component for c == 0. Roots are counted.
template <class F, int LABEL>
__device__ __forceinline__ uint32_t label_of(uint32_t c, uint32_t gmin) {
  if (LABEL == kLabelRootValue || !F::kRF) return c;
  return c == 0u ? gmin : c - 1u;
}

template <class F>
__device__ __forceinline__ uint32_t flatten_one(uint32_t *S, const F fn, uint32_t v, uint32_t pv,
                                                unsigned long long &roots) {
  const uint32_t cv = fn.f(v);
  if (pv == cv) {
    ++roots;
    return pv;
  }
  return root_name(S, cv, pv);
}

// 16-byte load of four consecutive parent values.
__device__ __forceinline__ uint4 ldP4(const uint32_t *p) {
  uint4 r;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p) : "memory");
  return r;
}

// Root names of W vertices (names c, parent values pc), walked in lock step:
// each round issues the next parent load of every walk still running, so the
// dependent chains overlap instead of following one another. Path splitting
// as in root_name(); r receives the root names.
template <int W>
__device__ __forceinline__ void root_names_lockstep(uint32_t *S, uint32_t (&c)[W], uint32_t (&pc)[W],
                                                    uint32_t (&r)[W], unsigned long long &roots) {
  unsigned running = 0;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    if (pc[k] == c[k]) {
      ++roots;
      r[k] = pc[k];
    } else if (pc[k] == 0u) {
      r[k] = 0u;
    } else {
      running |= 1u << k;
    }
  }
  while (running) {
    uint32_t pw[W];
#pragma unroll
    for (int k = 0; k < W; ++k)
      if (running & (1u << k)) pw[k] = ldP(S + pc[k]);
#pragma unroll
    for (int k = 0; k < W; ++k) {
      if (!(running & (1u << k))) continue;
      if (pw[k] == pc[k]) {  // pc[k] is a root
        r[k] = pc[k];
        running &= ~(1u << k);
        continue;
      }
      stP(S + c[k], pw[k]);  // the parent is not a root: split past it
      c[k] = pc[k];
      pc[k] = pw[k];
      if (pc[k] == 0u) {  // the permanent root
        r[k] = 0u;
        running &= ~(1u << k);
      }
    }
  }
}

// Four consecutive vertices per thread: 16-byte loads of P, 16-byte stores of
// the compressed names (only when one changed; every name written is a valid
// ancestor, and roots are never changed) and of the labels.
template <class F, int LABEL>
__global__ void __launch_bounds__(256) k_flatten4(uint32_t *P, uint32_t n, uint32_t *__restrict__ L,
                                                  Ctrl *ctrl) {
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  uint32_t gmin = 0;
  if (F::kRF && LABEL == kLabelMinId) gmin = ld_volatile_u32(&ctrl->gmin);
  unsigned long long roots = 0;
  const uint64_t n4 = n / 4u;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n4;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = (uint32_t)(4 * i);
    const uint4 p = ldP4(P + v);
    uint32_t c[4] = {fn.f(v), fn.f(v + 1u), fn.f(v + 2u), fn.f(v + 3u)};
    uint32_t pc[4] = {p.x, p.y, p.z, p.w};
    uint32_t r[4];
    root_names_lockstep<4>(S, c, pc, r, roots);
    const uint4 cq = make_uint4(r[0], r[1], r[2], r[3]);
    if (cq.x != p.x || cq.y != p.y || cq.z != p.z || cq.w != p.w)
      asm volatile("st.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(P + v), "r"(cq.x), "r"(cq.y), "r"(cq.z),
                   "r"(cq.w)
                   : "memory");
    if (L)
      __stcs(reinterpret_cast<uint4 *>(L + v),
             make_uint4(label_of<F, LABEL>(cq.x, gmin), label_of<F, LABEL>(cq.y, gmin),
                        label_of<F, LABEL>(cq.z, gmin), label_of<F, LABEL>(cq.w, gmin)));
  }
  // the last n % 4 vertices
  if (blockIdx.x == 0 && threadIdx.x < (n & 3u)) {
    const uint32_t v = (uint32_t)(4 * n4) + threadIdx.x;
    const uint32_t pv = ldP(P + v);
    const uint32_t c = flatten_one(S, fn, v, pv, roots);
    if (c != pv) stP(P + v, c);
    if (L) L[v] = label_of<F, LABEL>(c, gmin);
  }
  add_roots(roots, ctrl);
}

// One vertex per thread, for label buffers that are not 16-byte aligned.
template <class F, int LABEL>
__global__ void __launch_bounds__(256) k_flatten(uint32_t *P, uint32_t n, uint32_t *__restrict__ L,
                                                 Ctrl *ctrl) {
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  uint32_t gmin = 0;
  if (F::kRF && LABEL == kLabelMinId) gmin = ld_volatile_u32(&ctrl->gmin);
  unsigned long long roots = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = (uint32_t)i;
    const uint32_t pv = ldP(P + v);
    const uint32_t c = flatten_one(S, fn, v, pv, roots);
    if (c != pv) stP(P + v, c);
    if (L) __stcs(L + v, label_of<F, LABEL>(c, gmin));
  }
  add_roots(roots, ctrl);
}

template <class F>
__global__ void __launch_bounds__(256) k_count_roots(const uint32_t *__restrict__ P, uint32_t n,
                                                     Ctrl *ctrl) {
  const F fn = F::load(ctrl);
  unsigned long long roots = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    roots += (P[i] == fn.f((uint32_t)i));
  add_roots(roots, ctrl);
}

template <class F>
__global__ void __launch_bounds__(256) k_connected(uint32_t *P, uint32_t n,
                                                   const uint2 *__restrict__ pairs, uint64_t n_pairs,
                                                   uint8_t *__restrict__ out, Ctrl *ctrl) {
  const F fn = F::load(ctrl);
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n_pairs;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint2 q = ld_edge(pairs + i);
    uint8_t r = 0;
    if (q.x >= n || q.y >= n) {
      set_err(ctrl, kErrRange);
    } else {
      const uint32_t cu = root_name(slots<F>(P), fn.f(q.x), ldP(P + q.x));
      const uint32_t cv = root_name(slots<F>(P), fn.f(q.y), ldP(P + q.y));
      r = cu == cv;
    }
    out[i] = r;
  }
}

// The forest as edges (the pairs (v, P_v) that each machine sends to the
// Reducer, Section III): a non-root v (P[v] != f(v)) gives (v, f^-1(P[v])),
// the vertex its parent name names. Each thread takes 4 consecutive vertices
// (one 16-byte load); a warp scan and a block prefix place the block's pairs
// behind one atomic per block and round (one per warp serialised on the one
// counter: 5.7 ms for 2^28 vertices).
template <class F>
__global__ void __launch_bounds__(256) k_forest_pairs(const uint32_t *__restrict__ P, uint32_t n, uint2 *out,
                                                      uint64_t cap, Ctrl *ctrl) {
  __shared__ unsigned int s_cnt[8];
  __shared__ unsigned long long s_base[8];
  const F fn = F::load(ctrl);
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, n_w = blockDim.x >> 5;
  const uint64_t per_block = 4ull * blockDim.x;
  for (uint64_t b0 = (uint64_t)blockIdx.x * per_block; b0 < n; b0 += (uint64_t)gridDim.x * per_block) {
    const uint64_t v0 = b0 + 4ull * threadIdx.x;  // block-uniform trip count
    uint32_t pv[4] = {0u, 0u, 0u, 0u};
    if (v0 + 3 < n) {
      const uint4 q = *reinterpret_cast<const uint4 *>(P + v0);  // P is 256-byte aligned
      pv[0] = q.x;
      pv[1] = q.y;
      pv[2] = q.z;
      pv[3] = q.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (v0 + j < n) pv[j] = P[v0 + j];
    }
    uint32_t mine = 0, k = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool nr = v0 + j < n && pv[j] != fn.f((uint32_t)(v0 + j));
      mine |= (uint32_t)nr << j;
      k += nr ? 1u : 0u;
    }
    uint32_t incl = k;  // inclusive warp scan of the pair counts
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_cnt[wid] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long tot = 0;
      for (uint32_t w = 0; w < n_w; ++w) {
        s_base[w] = tot;
        tot += s_cnt[w];
      }
      const unsigned long long g = tot ? atomicAdd(&ctrl->pairs, tot) : 0ULL;
      for (uint32_t w = 0; w < n_w; ++w) s_base[w] += g;
    }
    __syncthreads();
    uint64_t slot = s_base[wid] + (incl - k);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if ((mine >> j) & 1u) {
        if (slot < cap) out[slot] = make_uint2((uint32_t)(v0 + j), fn.finv(pv[j]));
        ++slot;
      }
    }
    __syncthreads();  // s_cnt and s_base are reused next round
  }
}

}  // namespace

// ======================================================================= host

namespace {
std::atomic<unsigned long long> g_launches{0};
}

void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
unsigned long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

namespace {
struct Servers {
  std::shared_mutex mu;
  std::map<int, std::array<uint32_t, 9>> open;  // per device, servers by executor blocks per SM
  uint32_t most(int device) const {
    uint32_t n = 0;
    const auto it = open.find(device);
    if (it != open.end())
      for (uint32_t k = 1; k < it->second.size(); ++k)
        if (it->second[k]) n = k;
    return n;
  }
};
Servers &servers() {
  static Servers *s = new Servers();  // outlives every server
  return *s;
}
}  // namespace

ExecutorBlocks::ExecutorBlocks(int device) {
  servers().mu.lock_shared();
  n_ = servers().most(device);
}
ExecutorBlocks::~ExecutorBlocks() { servers().mu.unlock_shared(); }

uint32_t executor_announce(int device, uint32_t blocks_per_sm) {
  Servers &s = servers();
  std::lock_guard<std::shared_mutex> lk(s.mu);
  const uint32_t before = s.most(device);
  s.open[device][blocks_per_sm < 8 ? blocks_per_sm : 8]++;
  return before;
}
void executor_withdraw(int device, uint32_t blocks_per_sm) {
  Servers &s = servers();
  std::lock_guard<std::shared_mutex> lk(s.mu);
  s.open[device][blocks_per_sm < 8 ? blocks_per_sm : 8]--;
}

uint64_t persistent_cap(const void *kernel, int block, size_t smem) {
  struct Key {
    const void *k;
    int block, dev;
    size_t smem;
    bool operator<(const Key &o) const {
      if (k != o.k) return k < o.k;
      if (block != o.block) return block < o.block;
      if (dev != o.dev) return dev < o.dev;
      return smem < o.smem;
    }
  };
  static std::mutex mu;
  static std::map<Key, int> cache;
  int dev = 0;
  cudaGetDevice(&dev);
  const Key key{kernel, block, dev, smem};
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return (uint64_t)num_sms() * (uint64_t)it->second;
  }
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, block, smem) != cudaSuccess || occ < 1) occ = 1;
  {
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = occ;
  }
  return (uint64_t)num_sms() * (uint64_t)occ;
}

int num_sms() {
  if (g_num_sms == 0) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) v = 1;
    g_num_sms = v;
  }
  return g_num_sms;
}

EdgeSpan split_edges(const uint32_t *edges, uint64_t n_edges) {
  EdgeSpan s;
  if (n_edges == 0) return s;
  const uint2 *e2 = reinterpret_cast<const uint2 *>(edges);
  uint64_t h = ((uintptr_t)edges & 15u) ? 1u : 0u;
  if (h) s.head = e2;
  const uint64_t body = n_edges - h;
  s.n_quads = body / 2u;
  s.quads = reinterpret_cast<const uint4 *>(e2 + h);
  if (body & 1u) s.tail = e2 + h + 2u * s.n_quads;
  return s;
}

cudaError_t launch_init(bool rf, uint32_t *P, uint32_t n, Ctrl *ctrl, int m_src, uint32_t m_hint,
                        cudaStream_t s, const uint32_t *skip) {
  const uint64_t work = n / 4u + 1u;
  if (rf) {
    const unsigned g = clamp_grid((work + 255) / 256, persistent_cap((const void *)k_init<RootR>, 256, 0));
    k_init<RootR><<<g, 256, 0, s>>>(P, n, ctrl, m_src, m_hint, skip); note_launch();
  } else {
    const unsigned g = clamp_grid((work + 255) / 256, persistent_cap((const void *)k_init<RootId>, 256, 0));
    k_init<RootId><<<g, 256, 0, s>>>(P, n, ctrl, m_src, m_hint, skip); note_launch();
  }
  return cudaGetLastError();
}

namespace {
constexpr uint64_t kMinWaves = 8;
// The queue form reads P through L2 only from this many vertices up (16 MB).
constexpr uint32_t kL2MinVertices = 1u << 22;

constexpr uint64_t kHubMaxQuads = 1ULL << 37;

// Claim size of the dynamic schedule, in warp steps. From 2^20 edges up,
// 16 steps at a time (measured best there: fewer warps start on the hub's
// trees at once, so fewer CAS collide). Below that, a smaller graph would
// leave most warps of the grid idle, so the claim shrinks to about half the
// steps per warp (at least one).
uint32_t grab_for(uint64_t n_quads, int Q, unsigned grid, int block) {
  constexpr uint32_t kGrabMax = 16;
  if (n_quads >= (1ULL << 19)) return kGrabMax;
  const uint64_t steps = (n_quads + 32u * Q - 1) / (32u * Q);
  const uint64_t warps = (uint64_t)grid * (uint64_t)(block / 32);
  const uint64_t g = steps / (2 * (warps ? warps : 1));
  return g < 1 ? 1u : (g > kGrabMax ? kGrabMax : (uint32_t)g);
}

template <class F, int Q>
cudaError_t edge_pass_q(int filter, int block, const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl,
                        const uint32_t *skip, uint32_t *Z, const uint32_t *zsel, bool one_shot, uint32_t *log,
                        const uint32_t *hub, bool dyn, cudaStream_t s, const unsigned long long *hot,
                        const WideHot *wide_hot, bool settled) {
  const uint64_t per_block = (uint64_t)block * Q;
  // At least kMinWaves grid iterations per thread: when a whole graph fits
  // one wave, every edge reads P before any hooking and duplicate hub edges
  // then CAS the same roots at once (R-MAT scale 16: 97% of the CAS failed);
  // later waves find most edges already joined. one_shot: no cap at the
  // resident blocks, so blocks retire after their kMinWaves iterations and
  // kernels of other streams get SMs while this one runs.
  // Into settled trees one iteration per thread does: ten inserts of 10^3 to
  // 10^6 pairs into R-MAT scale 20 took 51 us each on 1 to 62 blocks.
  const uint64_t per = per_block * (settled ? 1 : kMinWaves);
  const uint64_t want = (e.n_quads + per - 1) / per;
  const uint64_t cap_big = 0x7FFFFFFFull;
  if (filter) {
    unsigned long long *work = nullptr;
    if (dyn) {  // one counter serves both instances: only one of them runs
      cudaError_t err = cudaMemsetAsync(&ctrl->work, 0, sizeof(unsigned long long), s);
      if (err != cudaSuccess) return err;
      work = &ctrl->work;
    }
    const size_t smem = (size_t)(block / 32) * 4 * kRing * sizeof(uint32_t);
    static_assert((512 / 32) * 4 * kRing * sizeof(uint32_t) + kHot * sizeof(uint32_t) <= 48 * 1024,
                  "the ring of a 512-thread block and the hot table fit the default dynamic shared memory limit");
    // the hub instances also hold the hot-vertex table
    const size_t smem_hub = smem + (F::kRF && hot ? kHot * sizeof(uint32_t) : 0);
    // the certificate word chooses among the launched instances (see
    // k_edge_pass_filtered); zsel: with Z, hub: without it
    const uint32_t *wsel = Z ? zsel : hub;
    if (F::kRF && wide_hot && wsel && work && !log && !skip && !one_shot && e.n_quads < kHubMaxQuads) {
      const uint32_t sb = id_bits(n);
      const void *k = Z ? (const void *)k_edge_pass_hub<true> : (const void *)k_edge_pass_hub<false>;
      static std::atomic<unsigned long long> set_z{0}, set_p{0};
      const cudaError_t err =
          ensure_func_attr(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHubSmem, Z ? set_z : set_p);
      if (err != cudaSuccess) return err;
      const unsigned g = (unsigned)persistent_cap(k, kHubBlock, kHubSmem);
      if (Z)
        k_edge_pass_hub<true><<<g, kHubBlock, kHubSmem, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n, ctrl, Z, wsel,
                                                             work, wide_hot->word, sb, wide_ways(sb));
      else
        k_edge_pass_hub<false><<<g, kHubBlock, kHubSmem, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n, ctrl, nullptr,
                                                              wsel, work, wide_hot->word, sb, wide_ways(sb));
      note_launch();
    } else if (Z) {
      const void *k = (const void *)k_edge_pass_filtered<F, Q, true, true>;
      const unsigned g = clamp_grid(want, one_shot ? cap_big : persistent_cap(k, block, smem_hub));
      const uint32_t grab = grab_for(e.n_quads, Q, g, block);
      k_edge_pass_filtered<F, Q, true, true><<<g, block, smem_hub, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n,
                                                                        ctrl, skip, Z, zsel, log, work, grab, hot);
      note_launch();
    } else if (hub) {
      const bool l2 = n >= kL2MinVertices;
      const void *k = l2 ? (const void *)k_edge_pass_filtered<F, Q, false, false, true>
                         : (const void *)k_edge_pass_filtered<F, Q, false, false, false>;
      const unsigned g = clamp_grid(want, one_shot ? cap_big : persistent_cap(k, block, smem_hub));
      const uint32_t grab = grab_for(e.n_quads, Q, g, block);
      if (l2)
        k_edge_pass_filtered<F, Q, false, false, true><<<g, block, smem_hub, s>>>(
            e.quads, e.n_quads, e.head, e.tail, P, n, ctrl, skip, nullptr, hub, log, work, grab, hot);
      else
        k_edge_pass_filtered<F, Q, false, false, false><<<g, block, smem_hub, s>>>(
            e.quads, e.n_quads, e.head, e.tail, P, n, ctrl, skip, nullptr, hub, log, work, grab, hot);
      note_launch();
    }
    if (!Z || zsel) {
      const void *k = (const void *)k_edge_pass_filtered<F, Q, false, true>;
      const unsigned g = clamp_grid(want, one_shot ? cap_big : persistent_cap(k, block, smem));
      const uint32_t grab = grab_for(e.n_quads, Q, g, block);
      k_edge_pass_filtered<F, Q, false, true><<<g, block, smem, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n,
                                                                     ctrl, skip, nullptr, Z ? zsel : hub, log,
                                                                     work, grab, nullptr);
      note_launch();
    }
  } else {
    const void *k = (const void *)k_edge_pass_direct<F, Q>;
    const unsigned g = clamp_grid(want, one_shot ? cap_big : persistent_cap(k, block, 0));
    k_edge_pass_direct<F, Q><<<g, block, 0, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n, ctrl,
                                                 skip); note_launch();
  }
  return cudaGetLastError();
}

template <class F>
cudaError_t edge_pass_f(int filter, int ept, int block, const EdgeSpan &e, uint32_t *P, uint32_t n,
                        Ctrl *ctrl, const uint32_t *skip, uint32_t *Z, const uint32_t *zsel, bool one_shot,
                        uint32_t *log, const uint32_t *hub, bool dyn, cudaStream_t s, const unsigned long long *hot,
                        const WideHot *wide_hot, bool settled) {
  switch (ept) {
    case 2: return edge_pass_q<F, 1>(filter, block, e, P, n, ctrl, skip, Z, zsel, one_shot, log, hub, dyn, s, hot, nullptr, settled);
    case 8: return edge_pass_q<F, 4>(filter, block, e, P, n, ctrl, skip, Z, zsel, one_shot, log, hub, dyn, s, hot, nullptr, settled);
    default: return edge_pass_q<F, 2>(filter, block, e, P, n, ctrl, skip, Z, zsel, one_shot, log, hub, dyn, s, hot, wide_hot, settled);
  }
}
}  // namespace

cudaError_t launch_edge_pass(bool rf, int filter, int ept, int block, const EdgeSpan &e, uint32_t *P,
                             uint32_t n, Ctrl *ctrl, const uint32_t *skip, cudaStream_t s, uint32_t *Z,
                             const uint32_t *zsel, bool one_shot, uint32_t *log, const uint32_t *hub, bool dyn,
                             const unsigned long long *hot, const WideHot *wide_hot, bool settled) {
  if (block != 128 && block != 256 && block != 512) block = 256;
  if (e.n_quads == 0 && !e.head && !e.tail) return cudaSuccess;
  if (log) filter = 1;  // the log is kept by the filtered form
  return rf ? edge_pass_f<RootR>(filter, ept, block, e, P, n, ctrl, skip, Z, zsel, one_shot, log, hub, dyn, s, hot,
                                   wide_hot, settled)
            : edge_pass_f<RootId>(filter, ept, block, e, P, n, ctrl, skip, Z, zsel, one_shot, log, hub, dyn, s,
                                  nullptr, nullptr, settled);
}

template <class F>
cudaError_t edge_pass_general(const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl, const uint32_t *skip,
                              cudaStream_t s, bool settled) {
  constexpr int block = 512, Q = 2;
  const size_t smem = (size_t)(block / 32) * 4 * kRing * sizeof(uint32_t);
  const void *k = (const void *)k_edge_pass_filtered<F, Q, false, true>;
  const uint64_t per = (uint64_t)block * Q;
  const uint64_t cap = persistent_cap(k, block, smem);
  const unsigned few = clamp_grid((e.n_quads + per * kMinWaves - 1) / (per * kMinWaves), cap);
  const unsigned g = settled ? clamp_grid((e.n_quads + per - 1) / per, cap) : few;
  k_edge_pass_filtered<F, Q, false, true><<<g, block, smem, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n, ctrl, skip,
                                                                 nullptr, nullptr, nullptr, &ctrl->work,
                                                                 grab_for(e.n_quads, Q, few, block), nullptr, settled);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_edge_pass_general(bool rf, const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl,
                                     const uint32_t *skip, cudaStream_t s, bool settled) {
  return rf ? edge_pass_general<RootR>(e, P, n, ctrl, skip, s, settled)
            : edge_pass_general<RootId>(e, P, n, ctrl, skip, s, settled);
}

cudaError_t launch_validate(const EdgeSpan &e, uint32_t n, Ctrl *ctrl, cudaStream_t s, uint32_t *reject) {
  if (e.n_quads == 0 && !e.head && !e.tail) return cudaSuccess;
  const unsigned g = clamp_grid((e.n_quads + 255) / 256, persistent_cap((const void *)k_validate<RootId, false>, 256, 0));
  k_validate<RootId, false><<<g, 256, 0, s>>>(e.quads, e.n_quads, e.head, e.tail, n, ctrl,
                                              reject ? reject : &ctrl->reject, nullptr, 0u);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_validate_probe(bool rf, const EdgeSpan &e, const uint32_t *P, uint32_t n, Ctrl *ctrl, cudaStream_t s) {
  const uint64_t per = 512ull * 2 * kMinWaves;  // as edge_pass_q's, for its default shape
  const uint32_t few = clamp_grid((e.n_quads + per - 1) / per, 1u << 20);
  const unsigned g = 1u + clamp_grid((e.n_quads + 255) / 256, persistent_cap((const void *)k_validate<RootR, true>, 256, 0));
  if (rf)
    k_validate<RootR, true><<<g, 256, 0, s>>>(e.quads, e.n_quads, e.head, e.tail, n, ctrl, &ctrl->reject, P, few);
  else
    k_validate<RootId, true><<<g, 256, 0, s>>>(e.quads, e.n_quads, e.head, e.tail, n, ctrl, &ctrl->reject, P, few);
  note_launch();
  return cudaGetLastError();
}

namespace {
template <class F, int kBlock>
cudaError_t insert_small(const uint2 *first, uint32_t count, uint32_t *P, uint32_t n, Ctrl *ctrl, cudaStream_t s) {
  static_assert(beside_executor(kBlock, kInsertRegs<kBlock>), "inserts run beside a busy server");
  static std::atomic<unsigned long long> smem_set{0};
  const cudaError_t err =
      ensure_func_attr((const void *)k_insert_small<F, kBlock>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(kInsertOneBlock * sizeof(uint4)), smem_set);
  if (err != cudaSuccess) return err;
  k_insert_small<F, kBlock><<<1, kBlock, count * sizeof(uint4), s>>>(first, count, P, n, ctrl);
  note_launch();
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_insert_small(bool rf, const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl, cudaStream_t s,
                                bool large_block) {
  const uint2 *first = e.head ? e.head : (e.n_quads ? reinterpret_cast<const uint2 *>(e.quads) : e.tail);
  const uint32_t count = (uint32_t)(2 * e.n_quads + (e.head ? 1 : 0) + (e.tail ? 1 : 0));
  if (large_block)
    return rf ? insert_small<RootR, 1024>(first, count, P, n, ctrl, s) : insert_small<RootId, 1024>(first, count, P, n, ctrl, s);
  return rf ? insert_small<RootR, 512>(first, count, P, n, ctrl, s) : insert_small<RootId, 512>(first, count, P, n, ctrl, s);
}

// The kernels that single-graph calls take only while a server is open. With lazy
// module loading a first launch may wait for the device to be idle, which beside an
// executor it is not; asking for the attributes loads them.
cudaError_t load_kernels_beside_executor() {
  const void *const kernels[] = {
      (const void *)k_edge_pass_filtered<RootR, 2, false, false, false>,
      (const void *)k_edge_pass_filtered<RootR, 2, false, false, true>,
      (const void *)k_edge_pass_filtered<RootR, 2, false, true>,
      (const void *)k_edge_pass_filtered<RootId, 2, false, true>,
      (const void *)k_insert_small<RootR, 512>,
      (const void *)k_insert_small<RootId, 512>,
  };
  for (const void *k : kernels) {
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, k);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_gmin_probe(uint32_t *P, uint32_t n, Ctrl *ctrl, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t want = ((uint64_t)n + 255) / 256;
  const unsigned gp = clamp_grid(want / 4 + 1, persistent_cap((const void *)k_gmin_probe, 256, 0));
  k_gmin_probe<<<gp, 256, 0, s>>>(P, n, ctrl);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_flatten(bool rf, int label_space, uint32_t *P, uint32_t n, uint32_t *L, Ctrl *ctrl,
                           cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t want = ((uint64_t)n + 255) / 256;
  if (rf && label_space == kLabelMinId && L) {
    const unsigned gp = clamp_grid(want / 4 + 1, persistent_cap((const void *)k_gmin_probe, 256, 0));
    k_gmin_probe<<<gp, 256, 0, s>>>(P, n, ctrl); note_launch();
  }
#define CC_FLAT(F_, LAB_)                                                                         \
  do {                                                                                            \
    if (vec) {                                                                                    \
      const unsigned g = clamp_grid(want / 4 + 1, persistent_cap((const void *)k_flatten4<F_, LAB_>, 256, 0)); \
      k_flatten4<F_, LAB_><<<g, 256, 0, s>>>(P, n, L, ctrl);                                      \
    } else {                                                                                      \
      const unsigned g = clamp_grid(want, persistent_cap((const void *)k_flatten<F_, LAB_>, 256, 0)); \
      k_flatten<F_, LAB_><<<g, 256, 0, s>>>(P, n, L, ctrl);                                       \
    }                                                                                             \
    note_launch();                                                                                \
  } while (0)
  const bool vec = ((uintptr_t)L & 15u) == 0;  // P itself is 256-byte aligned
  if (rf) {
    if (label_space == kLabelRootValue) CC_FLAT(RootR, kLabelRootValue);
    else CC_FLAT(RootR, kLabelMinId);
  } else {
    if (label_space == kLabelRootValue) CC_FLAT(RootId, kLabelRootValue);
    else CC_FLAT(RootId, kLabelMinId);
  }
#undef CC_FLAT
  return cudaGetLastError();
}

cudaError_t launch_count_roots(bool rf, const uint32_t *P, uint32_t n, Ctrl *ctrl, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t want = ((uint64_t)n + 255) / 256;
  if (rf) {
    const unsigned g = clamp_grid(want, persistent_cap((const void *)k_count_roots<RootR>, 256, 0));
    k_count_roots<RootR><<<g, 256, 0, s>>>(P, n, ctrl); note_launch();
  } else {
    const unsigned g = clamp_grid(want, persistent_cap((const void *)k_count_roots<RootId>, 256, 0));
    k_count_roots<RootId><<<g, 256, 0, s>>>(P, n, ctrl); note_launch();
  }
  return cudaGetLastError();
}

cudaError_t launch_forest_pairs(bool rf, const uint32_t *P, uint32_t n, uint32_t *out, uint64_t cap, Ctrl *ctrl,
                                cudaStream_t s) {
  cudaError_t err = cudaMemsetAsync(&ctrl->pairs, 0, sizeof(unsigned long long), s);
  if (err != cudaSuccess || n == 0) return err;
  const uint64_t want = ((uint64_t)n + 1023) / 1024;  // 4 vertices per thread
  uint2 *o = reinterpret_cast<uint2 *>(out);
  if (rf) {
    const unsigned g = clamp_grid(want, persistent_cap((const void *)k_forest_pairs<RootR>, 256, 0));
    k_forest_pairs<RootR><<<g, 256, 0, s>>>(P, n, o, cap, ctrl);
  } else {
    const unsigned g = clamp_grid(want, persistent_cap((const void *)k_forest_pairs<RootId>, 256, 0));
    k_forest_pairs<RootId><<<g, 256, 0, s>>>(P, n, o, cap, ctrl);
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_connected(bool rf, uint32_t *P, uint32_t n, const uint2 *pairs, uint64_t n_pairs,
                             uint8_t *out, Ctrl *ctrl, cudaStream_t s) {
  if (n_pairs == 0) return cudaSuccess;
  const uint64_t want = (n_pairs + 255) / 256;
  if (rf) {
    const unsigned g = clamp_grid(want, persistent_cap((const void *)k_connected<RootR>, 256, 0));
    k_connected<RootR><<<g, 256, 0, s>>>(P, n, pairs, n_pairs, out, ctrl); note_launch();
  } else {
    const unsigned g = clamp_grid(want, persistent_cap((const void *)k_connected<RootId>, 256, 0));
    k_connected<RootId><<<g, 256, 0, s>>>(P, n, pairs, n_pairs, out, ctrl); note_launch();
  }
  return cudaGetLastError();
}

}  // namespace cc

#ifdef CC_STATS
// Diagnostics builds only: read and clear the search counters.
extern "C" __attribute__((visibility("default"))) int cc_stats_read(unsigned long long out[4]) {
  cudaError_t e = cudaMemcpyFromSymbol(out, cc::g_cc_stats, 4 * sizeof(unsigned long long));
  unsigned long long z[4] = {0, 0, 0, 0};
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(cc::g_cc_stats, z, sizeof(z));
  return (int)e;
}
#endif
