// cc_batched.cu - connected components of many independent graphs in one
// call (include/cc_batch.h).
//
// All graphs share one name space: vertex i of graph g is named
// vtx_off[g] + i and f is the identity (Algorithm 1), so each graph's forest
// lives in its own range and the root of a component is its smallest global
// name; minus vtx_off[g] that is the graph-local min-id label. The label array
// is the parent array during the run. Phases, each a launch of its own so that
// each has the registers and shared memory it needs (as one kernel the hooking
// ran at half its occupancy):
//   0. one block checks the offsets and turns them into tile offsets; after a
//      grid barrier every vertex gets P[x] = x (k_batch_begin, cooperative);
//   1. hooking: edge tiles (each inside one graph) through the warp ring or
//      per lane; of a graph with many edges per vertex only one chunk in
//      sample_stride, which is enough to form its giant component;
//   2. compression: every vertex stores its root's name, and each sampled
//      graph gets a reference, the root that most of its edges' endpoints have;
//   3. the chunks left over, against one bit per vertex in shared memory: an
//      edge inside the reference's tree costs two shared-memory loads (where that
//      tree is small, the edges are hooked as in phase 1);
//   4. compression;
//   5. labels: vertex tiles turn root names into graph-local ids in place.
// Measured in ms, before (every edge hooked, one cooperative kernel) and now:
// 4096 mixed graphs (1.18G edges) 12.2 -> 8.2, 400 graphs 2.0 -> 1.26, 40
// graphs 0.89 -> 0.46, one graph of 38K edges 0.39 -> 0.08; lattices of 200 x 200
// 0.62 either way. Phase 1 waits for the dependent loads and compare-and-swaps of
// the searches, phase 3 issues 3.3 instructions per clock.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <new>

#include "cc_batch.h"
#include "cc_chunks.h"
#include "cc_chunks.h"
#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {

struct alignas(128) BatchCtrl {
  unsigned int bar_count;    // cumulative arrivals at grid barriers   } reset
  unsigned int bar_gen;      // barriers completed                     } before
  unsigned int abort;        // nonzero: every block leaves at the next barrier } each run
  unsigned int err;          // kErr* bits (sticky until cc_batch_sync)
  unsigned int bad_offsets;  // malformed offsets (sticky until cc_batch_sync)
  unsigned int tile_chunks;  // chunks per hooking tile of this run
  unsigned long long segs;   // segments of the filtered phase claimed so far (reset before each run)
};

struct BatchArgs {
  uint32_t n_graphs;
  const uint64_t *vtx_off;
  const uint64_t *edge_off;
  const uint2 *edges;
  uint32_t *P;  // the label array
  uint64_t *etile_off;  // n_graphs + 1
  uint64_t *vtile_off;  // n_graphs + 1
  uint64_t *chunk_off;  // n_graphs + 1: chunks of the graphs that the filtered phase takes
  uint32_t *ref;        // n_graphs: the root of each such graph's reference tree, and kScattered
  uint32_t tile_edges, tile_vertices;
  uint32_t hook_warps;  // warps of the hooking launch
  unsigned long long barrier_ns;  // bounded wait of every grid barrier
  BatchCtrl *ctrl;
};

namespace {

constexpr unsigned long long kBarrierTimeoutNs = 4000000000ULL;  // 4 s: default barrier wait

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int *p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier for a cooperative launch (all blocks co-resident). Arrivals
// are counted cumulatively, so barrier k completes when the count reaches
// k * gridDim.x. Every wait gives up after limit_ns, flags kErrTimeout and
// aborts the run (every block then leaves at its next barrier). Returns false
// when the run must stop.
__device__ bool grid_barrier(BatchCtrl *c, unsigned int &gen, unsigned long long limit_ns) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int target = gen + 1u;
    int ok = 1;
    __threadfence();
    const unsigned int arrived = atomicAdd(&c->bar_count, 1u) + 1u;
    if (arrived == gridDim.x * target) {
      __threadfence();
      atomicExch(&c->bar_gen, target);
    } else {
      const unsigned long long t0 = globaltimer();
      while (ld_acquire_u32(&c->bar_gen) < target) {
        if (globaltimer() - t0 > limit_ns) {
          atomicOr(&c->err, kErrTimeout);
          atomicExch(&c->abort, 1u);
          ok = 0;
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
    if (*(volatile unsigned int *)&c->abort) ok = 0;
    s_ok = ok;
  }
  __syncthreads();
  ++gen;
  return s_ok != 0;
}

// Edges are taken in chunks of kChunkEdges, four per lane of a warp.
constexpr uint32_t kChunkEdges = 128;
// The filtered phase keeps a bit per vertex of one graph in shared memory: 32
// KB per block leave room for 48 warps per SM.
constexpr uint32_t kBitsMax = 1u << 18;
// Graphs with fewer edges, or fewer than three per vertex, are hooked whole:
// the sample that forms their giant component would be most of them.
constexpr uint64_t kFilterMinEdges = 1u << 15;
constexpr uint64_t kFilterMinDegree = 3;
constexpr uint64_t kStrideMax = 64;

// One chunk in sample_stride is hooked first; 1: all of them. The sample
// holds 1.5 edges per vertex: with one per vertex the giant component of a
// uniform graph is still missing a fifth of the vertices and the filter lets
// too many edges through (2000 mixed graphs: 4.05 ms with one, 3.91 with 1.5,
// 4.14 with two).
__device__ __forceinline__ uint32_t sample_stride(uint64_t n_edges, uint64_t nv) {
  if (nv == 0 || nv > kBitsMax || n_edges < kFilterMinEdges || n_edges < kFilterMinDegree * nv) return 1u;
  const uint64_t s = 2 * n_edges / (3 * nv);
  return (uint32_t)(s < kStrideMax ? s : kStrideMax);
}

// Largest g in [0, n) with off[g] <= t (off nondecreasing, off[0] == 0), by a
// whole warp: every lane calls it, 32 candidates per round.
__device__ __forceinline__ uint32_t owner_warp(const uint64_t *off, uint32_t n, uint64_t t) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t lo = 0, hi = n;  // answer in [lo, hi)
  while (hi - lo > 1u) {
    const uint32_t step = (hi - lo + 31u) / 32u;
    const uint64_t i = lo + (uint64_t)lane * step;
    const uint32_t at_most = __ballot_sync(0xFFFFFFFFu, i < hi && off[i] <= t);  // lane 0 always
    lo += (31u - (uint32_t)__clz((int)at_most)) * step;
    hi = hi - lo > step ? lo + step : hi;
  }
  return lo;
}

// Chunks that a hooking tile holds: 3/8 of the configured tile's (the default
// 8192 edges: 24 chunks), or fewer where that would leave warps without a tile.
// Between 15 and 30 chunks 4096 graphs take 8.4 to 8.6 ms, with 61 10.2 (the last
// tiles leave most warps idle). Smaller tiles, four per warp, spread each graph
// over more SMs, whose warps then meet on its roots: 100 R-MAT graphs of 2^18 edges
// 924 us, 444 like this; 200 uniform ones of 65,536 vertices with 2.5 edges each
// 1365 and 936. One graph of 38K edges took 0.39 ms in five tiles of 8192 edges
// and takes 0.08.
constexpr uint64_t kTilesPerWarp = 1;
constexpr uint32_t kTileMinChunks = 2;

// Chunks of graph g that phase 1 hooks (0 when its offsets decrease).
__device__ __forceinline__ uint64_t hooked_chunks(const BatchArgs &a, uint32_t g) {
  const uint64_t v0 = a.vtx_off[g], v1 = a.vtx_off[g + 1], e0 = a.edge_off[g], e1 = a.edge_off[g + 1];
  if (v1 < v0 || e1 < e0) return 0;
  const uint32_t stride = sample_stride(e1 - e0, v1 - v0);
  return ((e1 - e0 + kChunkEdges - 1) / kChunkEdges + stride - 1) / stride;
}

// Phase 0 (one block): validate the offsets and write exclusive prefix sums
// of the per-graph tile counts.
__device__ void scan_tiles(const BatchArgs &a) {
  constexpr int K = 3;  // hooking tiles, vertex tiles, chunks of the filtered phase
  __shared__ unsigned long long s_carry[K], s_w[K][32];
  __shared__ int s_bad;
  uint64_t *const out[K] = {a.etile_off, a.vtile_off, a.chunk_off};
  if (threadIdx.x < K) s_carry[threadIdx.x] = 0ULL;
  if (threadIdx.x == 0) s_bad = (a.vtx_off[0] != 0ULL || a.edge_off[0] != 0ULL);
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // the chunks to hook, all graphs together, and from them a tile's size
  __shared__ unsigned long long s_hooked;
  if (threadIdx.x == 0) s_hooked = 0ULL;
  __syncthreads();
  unsigned long long hooked = 0;
  for (uint32_t g = threadIdx.x; g < a.n_graphs; g += blockDim.x) hooked += hooked_chunks(a, g);
  hooked = warp_sum_u64(hooked);
  if (lane == 0) atomicAdd(&s_hooked, hooked);
  __syncthreads();
  const uint64_t even = s_hooked / (kTilesPerWarp * a.hook_warps);
  const uint32_t share = a.tile_edges / kChunkEdges * 3u / 8u, most = share > kTileMinChunks ? share : kTileMinChunks;
  const uint32_t per_tile = even >= most ? most : (even < kTileMinChunks ? kTileMinChunks : (uint32_t)even);
  if (threadIdx.x == 0) a.ctrl->tile_chunks = per_tile;
  for (uint32_t base = 0; base < a.n_graphs; base += blockDim.x) {
    const uint32_t g = base + threadIdx.x;
    unsigned long long own[K] = {0, 0, 0}, incl[K];
    if (g < a.n_graphs) {
      const uint64_t v0 = a.vtx_off[g], v1 = a.vtx_off[g + 1];
      const uint64_t e0 = a.edge_off[g], e1 = a.edge_off[g + 1];
      if (v1 < v0 || e1 < e0) {
        s_bad = 1;
      } else {
        const uint64_t chunks = (e1 - e0 + kChunkEdges - 1) / kChunkEdges;
        const uint32_t stride = sample_stride(e1 - e0, v1 - v0);
        own[0] = ((chunks + stride - 1) / stride + per_tile - 1) / per_tile;
        own[1] = (v1 - v0 + a.tile_vertices - 1) / a.tile_vertices;
        own[2] = stride > 1u ? chunks : 0u;
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {  // inclusive warp scans
      incl[k] = own[k];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl[k], o);
        if (lane >= (uint32_t)o) incl[k] += y;
      }
      if (lane == 31) s_w[k][wid] = incl[k];
    }
    __syncthreads();
    if (wid < K) {  // warp k scans the warp totals of quantity k
      unsigned long long x = lane < nw ? s_w[wid][lane] : 0ULL;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      __syncwarp();
      if (lane < nw) s_w[wid][lane] = x;  // inclusive prefix over warps
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (g < a.n_graphs) out[k][g] = s_carry[k] + (wid ? s_w[k][wid - 1] : 0ULL) + incl[k] - own[k];
    __syncthreads();
    if (threadIdx.x < K) s_carry[threadIdx.x] += s_w[threadIdx.x][nw - 1];
    __syncthreads();
  }
  if (threadIdx.x < K) out[threadIdx.x][a.n_graphs] = s_carry[threadIdx.x];
  if (threadIdx.x == 0) {
    if (a.vtx_off[a.n_graphs] > 0x7FFFFFFFULL) s_bad = 1;
    if (s_bad) {
      a.ctrl->bad_offsets = 1u;
      atomicExch(&a.ctrl->abort, 1u);
    }
  }
}

// Root of vertex x by a read-only walk through L2.
__device__ __forceinline__ uint32_t walk_root(const uint32_t *P, uint32_t x) {
  uint32_t r = x, pr = ldP_cg(P + r);
  while (pr != r) {
    r = pr;
    pr = ldP_cg(P + r);
  }
  return r;
}

// Every vertex stores its root's name: read-only walks, four per thread in
// lock step, so that their dependent loads overlap; each entry is written
// only by its owner.
__device__ void compress(uint32_t *P, uint64_t V, uint64_t tid, uint64_t T) {
  const uint64_t head = ((16u - ((uintptr_t)P & 15u)) & 15u) / 4u;  // entries before the first 16-byte boundary
  const uint64_t h = head < V ? head : V, n4 = (V - h) / 4u;
  for (uint64_t i = tid; i < n4; i += T) {
    const uint64_t x0 = h + 4u * i;
    uint32_t r[4], p[4];
    asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "l"(P + x0)
                 : "memory");
    uint32_t run = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      p[k] = r[k];
      run |= (uint32_t)(r[k] != (uint32_t)(x0 + k)) << k;
    }
    while (run) {
      uint32_t q[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if ((run >> k) & 1u) q[k] = ldP_cg(P + r[k]);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if ((run >> k) & 1u) {
          if (q[k] == r[k]) run &= ~(1u << k);
          r[k] = q[k];
        }
    }
    if (r[0] != p[0] || r[1] != p[1] || r[2] != p[2] || r[3] != p[3])
      *reinterpret_cast<uint4 *>(P + x0) = make_uint4(r[0], r[1], r[2], r[3]);
  }
  const uint64_t rest = V - 4u * n4;  // the entries before and after the aligned body
  if (tid < rest) {
    const uint64_t x = tid < h ? tid : tid + 4u * n4;
    const uint32_t px = ldP_cg(P + x), r = walk_root(P, px);
    if (r != px) stP(P + x, r);
  }
}

// Segments of consecutive chunks per block, claimed from a counter: more
// segments balance better, but each starts by building its graph's bits (2000
// mixed graphs, this phase: 1.24, 1.27 and 1.68 ms with 4, 8 and 16).
constexpr uint32_t kSegs = 4;

// The filtered phase: the chunks of each graph that the hooking phase left,
// against one bit per vertex in shared memory, set for the members of the
// graph's reference tree. Where that holds less than half of the graph's sampled
// edges (kScattered in ref), the bits would let nearly every edge through, and
// the edges are hooked as they come.
constexpr uint32_t kMinVotes = 16;             // of 32
constexpr uint32_t kScattered = 0x80000000u;  // names stay below 2^31

__device__ void filtered_phase(const BatchArgs &a, uint32_t *bits, uint32_t *ring_words) {
  __shared__ unsigned long long s_claim;
  __shared__ uint32_t s_graph;
  BatchCtrl *const c = a.ctrl;
  uint32_t *const P = a.P;
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  // a queue of ids per warp: a's id in the first half, b's in the second
  uint32_t *const qa = ring_words + wid * 2 * kRing, *const qb = qa + kRing;
  const uint64_t total = a.chunk_off[a.n_graphs];
  if (total == 0) return;
  uint64_t seg = (total + (uint64_t)gridDim.x * kSegs - 1) / ((uint64_t)gridDim.x * kSegs);
  if (seg < 64) seg = 64;
  uint32_t built = 0xFFFFFFFFu;  // the graph whose bits are in shared memory
  for (;;) {
    if (threadIdx.x == 0) s_claim = atomicAdd(&c->segs, 1ULL);
    __syncthreads();
    uint64_t t = s_claim * seg;
    const uint64_t t1 = t + seg < total ? t + seg : total;
    if (t >= total) return;
    while (t < t1) {
      if (wid == 0) {
        const uint32_t found = owner_warp(a.chunk_off, a.n_graphs, t);
        if (lane == 0) s_graph = found;
      }
      __syncthreads();
      const uint32_t g = s_graph;
      const uint64_t base64 = a.vtx_off[g];
      const uint32_t base = (uint32_t)base64, nv = (uint32_t)(a.vtx_off[g + 1] - base64);
      const uint64_t e0 = a.edge_off[g], n_e = a.edge_off[g + 1] - e0;
      const uint32_t c0 = (uint32_t)(t - a.chunk_off[g]);
      const uint64_t t_end = a.chunk_off[g + 1] < t1 ? a.chunk_off[g + 1] : t1;
      const uint32_t c1 = (uint32_t)(t_end - a.chunk_off[g]);
      t = t_end;
      const uint32_t stride = sample_stride(n_e, nv);
      const uint32_t ref = a.ref[g];
      const bool scattered = (ref & kScattered) != 0u;
      if (built != g && !scattered) {
        const uint32_t words = (nv + 31u) / 32u;
        for (uint32_t w0 = wid * 4u; w0 < words; w0 += nw * 4u) {
          uint32_t p[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t v = (w0 + k) * 32u + lane;
            p[k] = v < nv ? ldP_cg(P + base + v) : ~ref;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, p[k] == ref);
            if (lane == 0 && w0 + k < words) bits[w0 + k] = word;
          }
        }
        built = g;
        __syncthreads();
      }
      uint32_t head = 0, tail = 0;
      auto resolve = [&](uint32_t count) {
        __syncwarp();
        const uint32_t slot = (head + lane) & (kRing - 1);
        const uint32_t xa = qa[slot], xb = qb[slot];
        __syncwarp();
        if (lane < count) {
          const uint32_t va = xa & 0x7FFFFFFFu, vb = xb & 0x7FFFFFFFu;
          uint32_t pa = ref, pb = ref;  // a marked endpoint's parent was ref once
          if (!(xa >> 31)) pa = ldP_cg(P + base + va);
          if (!(xb >> 31)) pb = ldP_cg(P + base + vb);
          if (!(xa >> 31) && pa == ref) atomicOr(bits + (va >> 5), 1u << (va & 31u));
          if (!(xb >> 31) && pb == ref) atomicOr(bits + (vb >> 5), 1u << (vb & 31u));
          if (pa != pb) unite<true>(P, base + va, pa, base + vb, pb);
        }
        head += count;
      };
      // this warp's chunks that were not sampled, the next one loaded ahead
      const uint32_t full = (uint32_t)(n_e / kChunkEdges);  // chunks before a ragged last one
      const uint2 *const e_lane = a.edges + e0 + lane;
      UnsampledChunks mine(c0, stride, wid, nw);
      uint32_t ch = mine.chunk();
      uint2 e[4];
      auto load = [&]() {
        const uint2 *const p = e_lane + (uint64_t)ch * kChunkEdges;
        if (ch < full) {
#pragma unroll
          for (int j = 0; j < 4; ++j) e[j] = ld_edge_now(p + 32 * j);
        } else {
          const uint32_t left = (uint32_t)(n_e - (uint64_t)ch * kChunkEdges);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            e[j] = make_uint2(0u, 0u);
            if (lane + 32u * j < left) e[j] = ld_edge_now(p + 32 * j);
          }
        }
      };
      if (ch < c1) load();
      while (ch < c1) {
        uint2 cur[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) cur[j] = e[j];
        mine.next();
        ch = mine.chunk();
        if (ch < c1) load();
        const uint32_t top = max(max(max(cur[0].x, cur[0].y), max(cur[1].x, cur[1].y)),
                                 max(max(cur[2].x, cur[2].y), max(cur[3].x, cur[3].y)));
        if (top >= nv) {
          atomicOr(&c->err, kErrRange);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (max(cur[j].x, cur[j].y) >= nv) cur[j] = make_uint2(0u, 0u);
        }
        if (scattered) {
          uint32_t pa[4], pb[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            pa[j] = ldP(P + base + cur[j].x);
            pb[j] = ldP(P + base + cur[j].y);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) unite(P, base + cur[j].x, pa[j], base + cur[j].y, pb[j]);
          continue;
        }
        uint32_t wa[4], wb[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          wa[j] = bits[cur[j].x >> 5];
          wb[j] = bits[cur[j].y >> 5];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // the vertex's bit comes to the bottom (the rotation takes the count modulo 32)
          const uint32_t ka = __funnelshift_r(wa[j], wa[j], cur[j].x), kb = __funnelshift_r(wb[j], wb[j], cur[j].y);
          const bool keep = !(ka & kb & 1u);
          const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
          if (!bal) continue;
          if (keep) {
            const uint32_t slot = (tail + __popc(bal & lt_mask)) & (kRing - 1);
            qa[slot] = cur[j].x | (ka << 31);
            qb[slot] = cur[j].y | (kb << 31);
          }
          tail += __popc(bal);
          if (tail - head >= 32u) resolve(32u);
        }
      }
      if (tail != head) resolve(tail - head);
      __syncthreads();  // the bits and s_graph are rewritten next
    }
  }
}

// Phases 0 and 1, one cooperative launch: the offsets, then P[x] = x.
__global__ void __launch_bounds__(512) k_batch_begin(BatchArgs a) {
  unsigned int gen = 0;
  if (blockIdx.x == 0) scan_tiles(a);
  if (!grid_barrier(a.ctrl, gen, a.barrier_ns)) return;
  const uint64_t V = a.vtx_off[a.n_graphs];
  const uint64_t T = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < V; x += T) a.P[x] = (uint32_t)x;
}

__device__ __forceinline__ bool aborted(const BatchArgs &a) { return *(volatile unsigned int *)&a.ctrl->abort != 0u; }

// Phase 1. Bound by latency (52 of 64 cycles between a warp's instructions wait
// for a load or a compare-and-swap), so 64 warps per SM at 32 registers: 2.03
// ms on 2000 mixed graphs against 2.45 with 48 warps and 2.87 with 32. Several
// edges per lane in lock step measured slower (2.3 to 2.5 ms), and so did
// hooking every vertex under its smallest sampled neighbour first.
template <int EPT, bool FILTER>
__global__ void __launch_bounds__(512, 4) k_batch_hook(BatchArgs a) {
  extern __shared__ uint32_t ring_smem[];
  if (aborted(a)) return;
  BatchCtrl *const c = a.ctrl;
  // One warp per tile, so no block barrier is taken per tile (a block would
  // wait for its slowest warp's searches). Tile t goes to warp t % warps of
  // block t / warps % gridDim.x: consecutive tiles, often of one graph, stay
  // on one SM and share its L1.
  uint32_t *const P = a.P;  // names are global ids: the slot of name x is P[x]
  WarpRing ring;
  if (FILTER) ring.init(ring_smem);
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t wpb = blockDim.x >> 5;
  const uint64_t wid = (uint64_t)blockIdx.x * wpb + (threadIdx.x >> 5);  // block-major
  const uint64_t n_warps = wpb * gridDim.x;
  const uint64_t n_etiles = a.etile_off[a.n_graphs];
  const uint32_t per_tile = c->tile_chunks;
  for (uint64_t t = wid; t < n_etiles; t += n_warps) {
    const uint32_t g = owner_warp(a.etile_off, a.n_graphs, t);
    const uint64_t e0 = a.edge_off[g], n_e = a.edge_off[g + 1] - e0;
    const uint64_t base64 = a.vtx_off[g], nv = a.vtx_off[g + 1] - base64;
    const uint32_t base = (uint32_t)base64, stride = sample_stride(n_e, nv);
    const uint64_t step = (uint64_t)stride * kChunkEdges;
    uint64_t first = (t - a.etile_off[g]) * per_tile * step;
    for (uint32_t k = 0; k < per_tile && first < n_e; ++k, first += step) {
      const uint64_t last = first + kChunkEdges < n_e ? first + kChunkEdges : n_e;
      for (uint64_t r0 = first; r0 < last; r0 += 32u * EPT) {
        uint32_t u[EPT], v[EPT], pu[EPT], pv[EPT];
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
          const uint64_t i = r0 + (uint64_t)j * 32u + lane;
          uint2 ed = make_uint2(0u, 0u);
          bool ok = false;
          if (i < last) {
            ed = ld_edge(a.edges + e0 + i);
            ok = ed.x < nv && ed.y < nv;
            if (!ok) atomicOr(&c->err, kErrRange);
          }
          // an empty or invalid slot touches no memory: equal parents drop it
          u[j] = ok ? base + ed.x : 0u;
          v[j] = ok ? base + ed.y : 0u;
          pu[j] = ok ? 1u : 0u;
          pv[j] = pu[j];
        }
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
          if (pu[j]) {
            pu[j] = ldP(P + u[j]);
            pv[j] = ldP(P + v[j]);
          }
        }
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
          if (FILTER)
            ring.push(P, pu[j] != pv[j], u[j], pu[j], v[j], pv[j]);
          else
            unite(P, u[j], pu[j], v[j], pv[j]);
        }
      }
    }
  }
  if (FILTER) ring.drain(P);
}

// Compression; kRefs: also each graph's reference, and nothing when no graph has a filtered phase.
template <bool kRefs>
__global__ void __launch_bounds__(256) k_batch_compress(BatchArgs a) {
  if (aborted(a)) return;
  uint32_t *const P = a.P;
  const uint64_t T = (uint64_t)gridDim.x * blockDim.x, tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (kRefs) {
    if (a.chunk_off[a.n_graphs] == 0) return;
    const uint32_t lane = threadIdx.x & 31u;
    for (uint64_t g = tid / 32u; g < a.n_graphs; g += T / 32u) {
      const uint64_t v0 = a.vtx_off[g], nv = a.vtx_off[g + 1] - v0;
      if (sample_stride(a.edge_off[g + 1] - a.edge_off[g], nv) == 1u) continue;
      const uint64_t e0 = a.edge_off[g];
      uint32_t x = a.edges[e0 + (a.edge_off[g + 1] - e0) * lane / 32u].x;  // (of edges: many vertices may have none)
      if (x >= nv) x = 0u;
      const uint32_t r = walk_root(P, (uint32_t)v0 + x);
      const uint32_t votes = (uint32_t)__popc(__match_any_sync(0xFFFFFFFFu, r));
      const uint32_t best = __reduce_max_sync(0xFFFFFFFFu, votes * 32u + lane);
      const uint32_t ref = __shfl_sync(0xFFFFFFFFu, r, (int)(best & 31u));
      if (lane == 0) a.ref[g] = ref | (best / 32u < kMinVotes ? kScattered : 0u);
    }
  }
  compress(P, a.vtx_off[a.n_graphs], tid, T);
}

__global__ void __launch_bounds__(512, 3) k_batch_filtered(BatchArgs a) {
  extern __shared__ uint32_t ring_smem[];  // the bits, then the queues
  if (aborted(a)) return;
  filtered_phase(a, ring_smem, ring_smem + kBitsMax / 32u);
}

// Graph-local labels, in place.
__global__ void __launch_bounds__(512) k_batch_labels(BatchArgs a) {
  __shared__ uint64_t s_tile[4];
  if (aborted(a)) return;
  uint32_t *const P = a.P;
  const uint64_t n_vtiles = a.vtile_off[a.n_graphs];
  for (uint64_t t = blockIdx.x; t < n_vtiles; t += gridDim.x) {
    if (threadIdx.x < 32) {
      const uint32_t g = owner_warp(a.vtile_off, a.n_graphs, t);
      const uint64_t x0 = a.vtx_off[g] + (t - a.vtile_off[g]) * a.tile_vertices;
      const uint64_t x1 = a.vtx_off[g + 1];
      s_tile[1] = x0;
      s_tile[2] = x0 + a.tile_vertices < x1 ? x0 + a.tile_vertices : x1;
      s_tile[3] = a.vtx_off[g];
    }
    __syncthreads();
    const uint64_t x0 = s_tile[1], x1 = s_tile[2];
    const uint32_t base = (uint32_t)s_tile[3];
    __syncthreads();
    for (uint64_t x = x0 + threadIdx.x; x < x1; x += blockDim.x) P[x] = ldP_strong(P + x) - base;
  }
}

}  // namespace
}  // namespace cc

using cc::BatchArgs;
using cc::BatchCtrl;

struct cc_batch {
  int device = 0;
  uint32_t max_graphs = 0;
  cc_batch_config cfg{};
  BatchCtrl *ctrl = nullptr;
  BatchCtrl *host_ctrl = nullptr;
  uint64_t *tile_off = nullptr;  // 3 * (max_graphs + 1), then max_graphs references (uint32)
  cudaStream_t last = nullptr;
  // the last cc_batch_tune: every candidate with its best time
  cc_batch_config tuned[64];
  float tuned_ms[64];
  uint32_t n_tuned = 0;
};

namespace {

bool cfg_valid(const cc_batch_config &c) {
  if (c.block_size != 256 && c.block_size != 512) return false;
  if (c.edges_per_thread != 1 && c.edges_per_thread != 2 && c.edges_per_thread != 4) return false;
  if (c.filter != 0 && c.filter != 1) return false;
  if (c.tile_edges < 256 || c.tile_edges % 256 || c.tile_vertices < 256) return false;
  if (c.barrier_wait_us > 60u * 1000u * 1000u) return false;
  for (int r : c.reserved)
    if (r) return false;
  return true;
}

// The configuration (4096 mixed graphs: 8.2 ms) that is
// used until cc_batch_tune or cc_batch_set_config chooses another.
cc_batch_config default_cfg() {
  cc_batch_config c{};
  c.block_size = 512;
  c.edges_per_thread = 1;
  c.filter = 1;
  c.tile_edges = 8192;
  c.tile_vertices = 4096;
  return c;
}

template <int EPT, bool FILTER>
cudaError_t launch_hook(const cc_batch_config &cfg, const BatchArgs &a, cudaStream_t s) {
  const size_t smem = FILTER ? (size_t)(cfg.block_size / 32) * 4 * cc::kRing * sizeof(uint32_t) : 0;
  const unsigned grid = (unsigned)cc::persistent_cap((const void *)cc::k_batch_hook<EPT, FILTER>, cfg.block_size, smem);
  cc::k_batch_hook<EPT, FILTER><<<grid, cfg.block_size, smem, s>>>(a);
  cc::note_launch();
  return cudaGetLastError();
}

cudaError_t launch_batched(const cc_batch_config &cfg, BatchArgs &a, cudaStream_t s) {
  cudaError_t e;
  {
    const void *k = (const void *)cc::k_batch_begin;
    const unsigned grid = (unsigned)cc::persistent_cap(k, 512, 0);
    void *args[] = {&a};
    if ((e = cudaLaunchCooperativeKernel(k, dim3(grid), dim3(512), args, 0, s)) != cudaSuccess) return e;
    cc::note_launch();
  }
  const unsigned gc = (unsigned)cc::persistent_cap((const void *)cc::k_batch_compress<true>, 256, 0);
  switch (cfg.edges_per_thread * 2 + cfg.filter) {
    case 2: e = launch_hook<1, false>(cfg, a, s); break;
    case 3: e = launch_hook<1, true>(cfg, a, s); break;
    case 4: e = launch_hook<2, false>(cfg, a, s); break;
    case 5: e = launch_hook<2, true>(cfg, a, s); break;
    case 8: e = launch_hook<4, false>(cfg, a, s); break;
    default: e = launch_hook<4, true>(cfg, a, s); break;
  }
  if (e != cudaSuccess) return e;
  cc::k_batch_compress<true><<<gc, 256, 0, s>>>(a);
  cc::note_launch();
  const size_t smem = cc::kBitsMax / 8 + (size_t)(512 / 32) * 2 * cc::kRing * sizeof(uint32_t);
  static std::atomic<unsigned long long> smem_set{0};
  const void *kf = (const void *)cc::k_batch_filtered;
  if ((e = cc::ensure_func_attr(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem, smem_set)) != cudaSuccess) return e;
  cc::k_batch_filtered<<<(unsigned)cc::persistent_cap(kf, 512, smem), 512, smem, s>>>(a);
  cc::note_launch();
  cc::k_batch_compress<false><<<gc, 256, 0, s>>>(a);
  cc::note_launch();
  const unsigned gl = (unsigned)cc::persistent_cap((const void *)cc::k_batch_labels, 512, 0);
  cc::k_batch_labels<<<gl, 512, 0, s>>>(a);
  cc::note_launch();
  return cudaGetLastError();
}

cc_status from_cuda(cudaError_t e) {
  if (e == cudaSuccess) return CC_OK;
  if (e == cudaErrorMemoryAllocation) return CC_ERR_OOM;
  return CC_ERR_CUDA;
}

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int d) {
    int cur = -1;
    if (cudaGetDevice(&cur) == cudaSuccess && cur != d) {
      prev = cur;
      cudaSetDevice(d);
    }
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

cc_status enqueue(cc_batch *b, const cc_batch_config &cfg, uint32_t n_graphs, const uint64_t *vtx_off,
                  const uint64_t *edge_off, const uint32_t *edges, uint32_t *L, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(b->ctrl, 0, 3 * sizeof(unsigned int), s);  // barrier state and abort
  if (e == cudaSuccess) e = cudaMemsetAsync(&b->ctrl->segs, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return from_cuda(e);
  BatchArgs a;
  a.n_graphs = n_graphs;
  a.vtx_off = vtx_off;
  a.edge_off = edge_off;
  a.edges = reinterpret_cast<const uint2 *>(edges);
  a.P = L;
  a.etile_off = b->tile_off;
  a.vtile_off = a.etile_off + (b->max_graphs + 1);
  a.chunk_off = a.vtile_off + (b->max_graphs + 1);
  a.ref = reinterpret_cast<uint32_t *>(a.chunk_off + (b->max_graphs + 1));
  a.tile_edges = cfg.tile_edges;
  a.tile_vertices = cfg.tile_vertices;
  a.hook_warps = (uint32_t)(cc::num_sms() * 64);
  a.barrier_ns = cfg.barrier_wait_us ? (unsigned long long)cfg.barrier_wait_us * 1000ULL : cc::kBarrierTimeoutNs;
  a.ctrl = b->ctrl;
  return from_cuda(launch_batched(cfg, a, s));
}

cc_status check_args(cc_batch *b, uint32_t n_graphs, const uint64_t *vtx_off, const uint64_t *edge_off,
                     const uint32_t *edges, uint32_t *L) {
  if (!b) return CC_ERR_INVALID_ARGUMENT;
  if (n_graphs > b->max_graphs) return CC_ERR_TOO_LARGE;
  if (n_graphs == 0) return CC_OK;
  if (!vtx_off || !edge_off || !L || ((uintptr_t)vtx_off & 7u) || ((uintptr_t)edge_off & 7u) ||
      ((uintptr_t)L & 3u) || (edges && ((uintptr_t)edges & 7u)))
    return CC_ERR_INVALID_ARGUMENT;
  return CC_OK;
}

}  // namespace

extern "C" {

cc_status cc_batch_create(uint32_t max_graphs, cc_batch **out) {
  if (!out) return CC_ERR_INVALID_ARGUMENT;
  *out = nullptr;
  if (max_graphs == 0 || max_graphs > (1u << 28)) return CC_ERR_INVALID_ARGUMENT;
  cc_batch *b = new (std::nothrow) cc_batch();
  if (!b) return CC_ERR_OOM;
  b->max_graphs = max_graphs;
  b->cfg = default_cfg();
  cudaError_t e = cudaGetDevice(&b->device);
  if (e == cudaSuccess) e = cudaMalloc((void **)&b->ctrl, sizeof(BatchCtrl));
  if (e == cudaSuccess) e = cudaMallocHost((void **)&b->host_ctrl, sizeof(BatchCtrl));
  if (e == cudaSuccess) e = cudaMalloc((void **)&b->tile_off, 3 * ((size_t)max_graphs + 1) * sizeof(uint64_t) + (size_t)max_graphs * sizeof(uint32_t));
  if (e == cudaSuccess) e = cudaMemset(b->ctrl, 0, sizeof(BatchCtrl));
  if (e != cudaSuccess) {
    cc_batch_destroy(b);
    return from_cuda(e);
  }
  *out = b;
  return CC_OK;
}

void cc_batch_destroy(cc_batch *b) {
  if (!b) return;
  DeviceGuard dg(b->device);
  cudaDeviceSynchronize();
  if (b->ctrl) cudaFree(b->ctrl);
  if (b->host_ctrl) cudaFreeHost(b->host_ctrl);
  if (b->tile_off) cudaFree(b->tile_off);
  delete b;
}

cc_status cc_run_batched(cc_batch *b, uint32_t n_graphs, const uint64_t *vtx_off_dev,
                         const uint64_t *edge_off_dev, const uint32_t *edges_dev, uint32_t *L_out_dev,
                         cc_stream_t stream) {
  cc_status st = check_args(b, n_graphs, vtx_off_dev, edge_off_dev, edges_dev, L_out_dev);
  if (st != CC_OK || n_graphs == 0) return st;
  DeviceGuard dg(b->device);
  b->last = (cudaStream_t)stream;
  return enqueue(b, b->cfg, n_graphs, vtx_off_dev, edge_off_dev, edges_dev, L_out_dev, b->last);
}

cc_status cc_batch_tune_results(const cc_batch *b, cc_batch_config *cfgs, float *ms, uint32_t cap,
                                uint32_t *count) {
  if (!b || !count || (cap && (!cfgs || !ms))) return CC_ERR_INVALID_ARGUMENT;
  const uint32_t k = b->n_tuned < cap ? b->n_tuned : cap;
  for (uint32_t i = 0; i < k; ++i) {
    cfgs[i] = b->tuned[i];
    ms[i] = b->tuned_ms[i];
  }
  *count = b->n_tuned;
  return CC_OK;
}

cc_status cc_batch_set_config(cc_batch *b, const cc_batch_config *cfg) {
  if (!b || !cfg || !cfg_valid(*cfg)) return CC_ERR_INVALID_ARGUMENT;
  b->cfg = *cfg;
  return CC_OK;
}

cc_status cc_batch_get_config(const cc_batch *b, cc_batch_config *cfg) {
  if (!b || !cfg) return CC_ERR_INVALID_ARGUMENT;
  *cfg = b->cfg;
  return CC_OK;
}

cc_status cc_batch_sync(cc_batch *b) {
  if (!b) return CC_ERR_INVALID_ARGUMENT;
  DeviceGuard dg(b->device);
  cudaStream_t s = b->last;
  cudaError_t e = cudaMemcpyAsync(b->host_ctrl, b->ctrl, sizeof(BatchCtrl), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return from_cuda(e);
  const BatchCtrl h = *b->host_ctrl;
  if (h.err || h.abort || h.bad_offsets) {
    e = cudaMemsetAsync(b->ctrl, 0, sizeof(BatchCtrl), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
  }
  if (h.bad_offsets) return CC_ERR_INVALID_ARGUMENT;
  if (h.err & cc::kErrTimeout) return CC_ERR_TIMEOUT;
  if (h.err & cc::kErrRange) return CC_ERR_OUT_OF_RANGE;
  return CC_OK;
}

cc_status cc_batch_tune(cc_batch *b, uint32_t n_graphs, const uint64_t *vtx_off_dev,
                        const uint64_t *edge_off_dev, const uint32_t *edges_dev, uint32_t *L_out_dev,
                        cc_stream_t stream, cc_batch_config *best, float *best_ms) {
  cc_status st = check_args(b, n_graphs, vtx_off_dev, edge_off_dev, edges_dev, L_out_dev);
  if (st != CC_OK) return st;
  if (n_graphs == 0) return CC_ERR_INVALID_ARGUMENT;
  DeviceGuard dg(b->device);
  cudaStream_t s = (cudaStream_t)stream;
  b->last = s;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return CC_ERR_CUDA;
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return CC_ERR_CUDA;
  }
  const int blocks[] = {256, 512};
  const int epts[] = {1, 2, 4};
  const int filters[] = {1, 0};
  const uint32_t tiles[] = {4096, 8192, 16384, 65536};  // edges per warp tile
  cc_batch_config top = b->cfg;
  float top_ms = 1e30f;
  b->n_tuned = 0;
  for (int blk : blocks)
    for (int ept : epts)
      for (int flt : filters)
        for (uint32_t te : tiles) {
          cc_batch_config c = default_cfg();
          c.barrier_wait_us = b->cfg.barrier_wait_us;
          c.block_size = blk;
          c.edges_per_thread = ept;
          c.filter = flt;
          c.tile_edges = te;
          float ms_min = 1e30f;
          for (int rep = 0; rep < 3 && st == CC_OK; ++rep) {
            cudaEventRecord(e0, s);
            st = enqueue(b, c, n_graphs, vtx_off_dev, edge_off_dev, edges_dev, L_out_dev, s);
            cudaEventRecord(e1, s);
            if (st != CC_OK) break;
            if (cudaEventSynchronize(e1) != cudaSuccess) {
              st = CC_ERR_CUDA;
              break;
            }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0 && ms < ms_min) ms_min = ms;  // the first run warms up
          }
          if (st != CC_OK) break;
          if (b->n_tuned < 64) {
            b->tuned[b->n_tuned] = c;
            b->tuned_ms[b->n_tuned++] = ms_min;
          }
          if (ms_min < top_ms) {
            top_ms = ms_min;
            top = c;
          }
        }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != CC_OK) return st;
  st = cc_batch_sync(b);
  if (st != CC_OK) return st;
  b->cfg = top;
  if (best) *best = top;
  if (best_ms) *best_ms = top_ms;
  return CC_OK;
}

}  // extern "C"
