// cc_bits.cu - the edge pass on graphs whose vertices fit, a bit each, in one
// block's shared memory (at most kBitsVertices) and that have at least
// kBitsMinDegree edges per vertex.
//
// The general pass is slow there for two reasons. It looks up both endpoints
// of every edge in L2, although after a small part of the edges nearly all of
// them lie inside the giant component. And that small part takes most of the
// time: all searches meet on the few roots of the growing trees, and loads and
// compare-and-swaps of one L2 sector are served one after another (R-MAT
// scale 16 under f = id: 1.0M of its 1.05M edges in flight at once take 0.55
// ms, and the general pass throttles itself to 512 warps to reach 0.09). So:
//   1. linking rounds. Each takes a sample of the edges and lowers the parent
//      of the larger of the two endpoints' roots to the smaller one, by a
//      reduction that nothing waits for; the lanes of a warp that lower one
//      root do it once. A link that another one overwrites is lost, which is
//      harmless: step 3 goes through every edge. After each round all vertices
//      are compressed to their roots. The samples shrink fourfold per round
//      while the trees grow more than that, so a root gets enough edges to be
//      linked and too few to queue up behind. Where a round has left deep trees
//      (rows of a lattice, paths), the next rounds only go on compressing, with
//      longer walks, until they are flat: compressing chains of thousands of
//      links in one go took longer than the whole general pass.
//   2. the last compression also writes one bit per vertex: whether it is in
//      the reference tree, the one that most of 32 sampled endpoints are in.
//   3. every block copies the bits into its shared memory and streams the
//      edges: one whose endpoints are both marked is inside the reference tree
//      for good, and costs two shared-memory loads. The others are queued and
//      joined exactly as in the general pass.
//   4. where the reference tree holds less than half of the sampled endpoints
//      (many components of one size, meshes that the rounds joined in part), the
//      filter would queue nearly every edge: the general pass takes its place.
//      The choice is made on the device.
// Whole calls under f = id, us, general pass and this one: R-MAT scale 16 88 -> 74,
// 18 178 -> 92, 20 with 2^26 edges 1200 -> 308; uniform, 1.5M vertices with three
// edges each 350 -> 158; lattice of 1000 x 1000 with eight neighbours 198 -> 100, of
// 100^3 with 26 182 -> 200; star whose centre has the largest id 370 -> 198; cliques
// of ten 196 -> 222. What bounds it: at scale 16 the launches (eleven of 2 to 4 us,
// the first sample's and step 3's loads aside), at scale 20 step 3 (a tenth of the
// edges still leads to a search).
#include <cuda_runtime.h>
#include <stdint.h>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {

namespace {

constexpr uint32_t kChunkQuads = 64;  // 128 edges, four per lane of a warp
constexpr int kFilterBlock = 640, kFilterRegs = 40;
static_assert(beside_executor(kFilterBlock, kFilterRegs), "the filter runs beside a busy server");
constexpr int kLinkBlock = 256;
constexpr size_t filter_queue_bytes(int block) { return (size_t)(block / 32) * 2 * kRing * sizeof(uint32_t); }
static_assert(kBitsVertices / 8 + filter_queue_bytes(kFilterBlock) <= kBesideExecutorSmem, "the bits and the queues fit beside the executor");
// Two blocks on an SM where their bits fit, then of 512 threads: R-MAT scale 18 (f =
// id) 119 us with two of 640, 111 with these.
constexpr int kFilterPairBlock = 512;
constexpr size_t kFilterPairBytes = kSmemPerSM / 2 - kSmemPerBlock;

// Linking rounds and their samples: two edges per vertex in the first round, a
// quarter of that in each of the next. Edge pass in microseconds on uniform
// graphs of 2^20 vertices with 3 / 10 edges per vertex and R-MAT scales 16 and
// 18 under f = id: 117 / 135 / 66 / 75. With one edge per vertex 380 / 956 /
// 70 / 99 and with three rounds 302 / 662 / 57 / 64, because step 3 then meets
// many trees; with three edges per vertex 118 / 135 / 65 / 104.
constexpr uint32_t kRounds = 4;
static_assert(kRounds == sizeof(Ctrl::deep) / sizeof(uint32_t), "a word per round");
constexpr uint64_t kFirstSample = 2, kShrink = 4;
constexpr uint64_t kMinSampleChunks = 32;

// Samples of the linking rounds: one chunk in chunk_stride[k] for the k-th round
// that links.
struct Rounds {
  uint32_t chunk_stride[kRounds];
};

// Linking round r over the chunks k * stride + r % stride, unless round r - 1 left
// deep trees. kFirst: P holds every vertex's own name, so the endpoints need no
// parent loads. The lanes of a warp that lower one root do it once; in the first
// round, where nearly all targets are distinct and finding equal ones takes longer
// than the atomics (uniform graph of 1.5M vertices: 28 -> 75 us), only those whose
// target is often met by the block's first edges: 2^21 edges of a star whose
// centre has the largest id took 2548 us with an atomic each.
__device__ __forceinline__ uint4 ld_quad_now(const uint4 *a) {  // kept where it stands in the program
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(a));
  return v;
}

constexpr uint32_t kCentreBits = 8, kCentreCount = kLinkBlock / 32;
__device__ __forceinline__ uint32_t centre_slot(uint32_t x) { return (x * 2654435761u) >> (32u - kCentreBits); }

template <class F, bool kFirst>
__global__ void __launch_bounds__(kLinkBlock) k_bits_link(const uint4 *__restrict__ e4, uint64_t n_quads, Rounds rounds,
                                                          uint32_t r, uint32_t *P, uint32_t n, Ctrl *ctrl) {
  __shared__ uint32_t centre[1u << kCentreBits];
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  const uint32_t lane = threadIdx.x & 31u;
  uint64_t step, q0;
  uint4 e[2];
  auto start = [&](uint32_t stride) {  // other edges than the round before
    step = (uint64_t)stride * kChunkQuads;
    q0 = ((uint64_t)blockIdx.x * (kLinkBlock / 32) + (threadIdx.x >> 5)) * step + r % stride * kChunkQuads;
  };
  auto load = [&]() {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint64_t q = q0 + 32u * j + lane;
      e[j] = q < n_quads ? ld_quad_now(e4 + q) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  start(rounds.chunk_stride[r]);
  load();  // while it is found whether the rounds before have all linked
  if (!kFirst) {
    uint32_t linked = 0;  // rounds that have linked
    bool flat = true;
    uint32_t deep[kRounds];  // through L1: every warp reads them
#pragma unroll
    for (uint32_t j = 0; j < kRounds; ++j) deep[j] = ldP(&ctrl->deep[j]);
#pragma unroll
    for (uint32_t j = 0; j + 1u < kRounds; ++j) {
      if (j >= r) break;
      linked += flat ? 1u : 0u;
      flat = deep[j] == 0u;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->deep[r] = 0u;
    if (!flat) return;
    if (linked != r) {
      start(rounds.chunk_stride[linked]);
      load();
    }
  } else {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->deep[r] = 0u;
    for (uint32_t i = threadIdx.x; i < 1u << kCentreBits; i += kLinkBlock) centre[i] = 0u;
    __syncthreads();
  }
  const uint64_t hop = (uint64_t)gridDim.x * (kLinkBlock / 32) * step;
  bool counted = !kFirst;
  while (q0 < n_quads || !counted) {
    uint32_t x[8], p[8];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (max(max(e[j].x, e[j].y), max(e[j].z, e[j].w)) >= n) e[j] = make_uint4(0u, 0u, 0u, 0u);  // reported by the filter
      x[4 * j] = e[j].x;
      x[4 * j + 1] = e[j].y;
      x[4 * j + 2] = e[j].z;
      x[4 * j + 3] = e[j].w;
    }
    q0 += hop;
    load();
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = kFirst ? fn.f(x[i]) : ldP(P + x[i]);
    if (!counted) {  // once per block, by every thread
      if (p[0] != p[1]) atomicAdd(centre + centre_slot(max(p[0], p[1])), 1u);
      __syncthreads();
      counted = true;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t a = p[2 * k], b = p[2 * k + 1], hi = max(a, b), lo = min(a, b);
      const bool share = hi != lo && (!kFirst || centre[centre_slot(hi)] >= kCentreCount);
      const uint32_t act = __ballot_sync(0xFFFFFFFFu, share);
      if (share) {
        const uint32_t peers = __match_any_sync(act, hi);
        const uint32_t least = __reduce_min_sync(peers, lo);
        if ((peers & ((1u << lane) - 1u)) == 0u) atomicMin(S + hi, least);
      } else if (kFirst && hi != lo) {
        atomicMin(S + hi, lo);
      }
    }
  }
}

// Compression, four vertices per thread: every vertex walks up to its root and
// stores it, or after kShortWalk steps (kLongWalk where the round before left
// deep trees) the ancestor that it has come to. The walks only read, so that
// only its owner writes a vertex (a split stored late would put an older ancestor
// back, and a vertex that does not name its root spoils the next round: uniform
// graphs then reached step 3 in many trees, 415 us instead of 117), and read
// through L1, which answers the many loads of one root. A round that leaves a
// quarter of some 128 vertices on their way has left deep trees. A lattice of 1000
// x 1000 with eight neighbours makes chains of 1000 links: walks that split their
// path past 16 steps met in L2 for 410 us there, and this takes four short rounds.
// kBits: also the reference and the bits (32 per word, the words of a warp step's
// 128 vertices together; bits from n on are 0).
constexpr int kShortWalk = 16, kLongWalk = 64;
constexpr uint32_t kMinVotes = 16;  // of 32

template <class F, bool kBits>
__global__ void __launch_bounds__(256) k_bits_build(const uint4 *__restrict__ e4, uint64_t n_quads, uint32_t r,
                                                    uint32_t *P, uint32_t n, Ctrl *ctrl, uint32_t *bits) {
  __shared__ uint32_t s_ref, s_deep;
  const int longest = r && ldP(&ctrl->deep[r - 1u]) ? kLongWalk : kShortWalk;
  if (threadIdx.x == 0) s_deep = 0u;
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  const uint32_t lane = threadIdx.x & 31u;
  if (kBits && threadIdx.x < 32) {
    // compression moves no vertex to another root, so every block finds the
    // same reference whatever the others have done already
    uint32_t x = __ldg(e4 + n_quads * lane / 32u).x;
    if (x >= n) x = 0u;
    const uint32_t root = root_name(S, fn.f(x), ldP(P + x));
    const uint32_t votes = (uint32_t)__popc(__match_any_sync(0xFFFFFFFFu, root));
    const uint32_t best = __reduce_max_sync(0xFFFFFFFFu, votes * 32u + lane), best_votes = best / 32u;
    const uint32_t ref = __shfl_sync(0xFFFFFFFFu, root, (int)(best & 31u));
    if (lane == 0) {
      s_ref = ref;
      if (blockIdx.x == 0) {
        ctrl->ref = ref;
        ctrl->marked = best_votes >= kMinVotes ? 1u : 0u;
        ctrl->work = 0ULL;  // step 3's claims
      }
    }
  }
  __syncthreads();
  const uint32_t ref = kBits ? s_ref : 0u;
  const uint32_t groups = (n + 127u) / 128u;  // of 128 vertices, one per warp step
  for (uint32_t g = blockIdx.x * 8u + (threadIdx.x >> 5); g < groups; g += gridDim.x * 8u) {
    const uint32_t v = g * 128u + 4u * lane;
    uint32_t nib = 0, run = 0;
    if (v < n) {  // P is padded to a multiple of four entries
      uint32_t p0[4], up[4];
      asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(p0[0]), "=r"(p0[1]), "=r"(p0[2]), "=r"(p0[3])
                   : "l"(P + v)
                   : "memory");
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        up[k] = p0[k];
        run |= (uint32_t)(v + k < n && up[k] != fn.f(v + k) && up[k] != 0u) << k;
      }
      for (int steps = 0; run && steps < longest; ++steps) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((run >> k) & 1u) w[k] = ldP(S + up[k]);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((run >> k) & 1u) {
            if (w[k] == up[k] || w[k] == 0u) run &= ~(1u << k);
            up[k] = w[k];
          }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (v + k >= n) continue;
        if (up[k] != p0[k]) stP(P + v + k, up[k]);
        nib |= (uint32_t)(up[k] == ref) << k;
      }
    }
    if (__reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(run)) >= 32u) s_deep = 1u;
    if (kBits) {
      const uint32_t word = __reduce_or_sync(0xFFu << (lane & 24u), nib << (4u * (lane & 7u)));
      if ((lane & 7u) == 0u) bits[g * 4u + (lane >> 3)] = word;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_deep) ctrl->deep[r] = 1u;
}

// Step 3. One block of 20 warps on an SM, or two of 16, because one of 32 would not
// fit beside the serving executor's; a warp's next chunk is loaded while it works on
// one. Long lists are claimed kGrab chunks at a time: with a fixed split into one
// block per SM the pass took either 235 or 550 us on R-MAT scale 20 with 2^26 edges,
// from run to run. Whole calls with one block of 32 warps and a fixed split, and like
// this, us: R-MAT scale 18 (f = id) 111 and 106, 19 206 and 192, 20 with 2^26 edges 538
// and 480, 1,000,003 vertices with 16M edges 270 and 260; with one block of 28 warps of
// 32 registers, which spill, 116 / 197 / 466 / 270.
template <class F>
__global__ void __maxnreg__(kFilterRegs)
    k_bits_filter(const uint4 *__restrict__ e4, uint64_t n_quads, const uint2 *head, const uint2 *tail, uint32_t *P,
                  uint32_t n, Ctrl *ctrl, const uint32_t *__restrict__ all_bits, uint32_t grab) {
  extern __shared__ uint32_t smem[];
  if (ldP(&ctrl->marked) == 0u) return;  // (through L1: every warp reads it)
  const F fn = F::load(ctrl);
  uint32_t *const S = slots<F>(P);
  const uint32_t ref = ldP(&ctrl->ref);
  const uint32_t groups = (n + 127u) / 128u;
  uint32_t *const bits = smem;
  for (uint32_t i = threadIdx.x; i < groups; i += blockDim.x)
    reinterpret_cast<uint4 *>(bits)[i] = __ldg(reinterpret_cast<const uint4 *>(all_bits) + i);
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, lt_mask = (1u << lane) - 1u;
  // a queue of ids per warp (top bit: marked), as deep as the warp ring's
  uint32_t *const qa = smem + 4u * groups + wid * 2 * kRing, *const qb = qa + kRing;
  uint32_t q_head = 0, q_tail = 0;
  __syncthreads();
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (t == 0 && head) single_edge<F, true>(P, fn, head, n, ctrl);
  if (t == 1 && tail) single_edge<F, true>(P, fn, tail, n, ctrl);
  auto resolve = [&](uint32_t count) {
    __syncwarp();
    const uint32_t slot = (q_head + lane) & (kRing - 1);
    const uint32_t xa = qa[slot], xb = qb[slot];
    __syncwarp();
    if (lane < count) {
      const bool ka = xa >> 31, kb = xb >> 31;
      const uint32_t va = xa & 0x7FFFFFFFu, vb = xb & 0x7FFFFFFFu;
      uint32_t pa = ref, pb = ref;  // a marked vertex's parent was the reference
      if (!ka) pa = ldP_cg(P + va);
      if (!kb) pb = ldP_cg(P + vb);
      if (!ka && pa == ref) atomicOr(bits + (va >> 5), 1u << (va & 31u));
      if (!kb && pb == ref) atomicOr(bits + (vb >> 5), 1u << (vb & 31u));
      if (pa != pb) unite<true>(S, fn.f(va), pa, fn.f(vb), pb);
    }
    q_head += count;
  };
  const uint64_t pol = policy_evict_first();
  const uint32_t chunks = (uint32_t)((n_quads + kChunkQuads - 1) / kChunkQuads);  // (at most 2^29)
  // grab > 1: chunks [ch, end) are claimed from a counter, and the claim after
  // them is asked for when they begin; else a fixed stride of chunks
  uint32_t ch = wid * gridDim.x + blockIdx.x, end = ch + 1u, next = 0;
  auto claim = [&]() {
    ch = __shfl_sync(0xFFFFFFFFu, next, 0);
    end = ch + grab;
    if (lane == 0) next = (uint32_t)atomicAdd(&ctrl->work, (unsigned long long)grab);
  };
  if (grab > 1u) {
    if (lane == 0) next = (uint32_t)atomicAdd(&ctrl->work, (unsigned long long)grab);
    claim();
  }
  uint4 e[2];
  auto load = [&]() {
    const uint4 *const p = e4 + (uint64_t)ch * kChunkQuads + lane;
    if (ch + 1u < chunks) {
      e[0] = ld_edges_now(p, pol);
      e[1] = ld_edges_now(p + 32, pol);
    } else {
      const uint32_t left = (uint32_t)(n_quads - (uint64_t)ch * kChunkQuads);
      e[0] = lane < left ? ld_edges_now(p, pol) : make_uint4(0u, 0u, 0u, 0u);
      e[1] = lane + 32u < left ? ld_edges_now(p + 32, pol) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  if (ch < chunks) load();
  while (ch < chunks) {
    uint32_t x[8] = {e[0].x, e[0].y, e[0].z, e[0].w, e[1].x, e[1].y, e[1].z, e[1].w};
    if (++ch == end) {
      if (grab > 1u) {
        claim();
      } else {
        ch += gridDim.x * (blockDim.x / 32u) - 1u;
        end = ch + 1u;
      }
    }
    if (ch < chunks) load();
    const uint32_t top = max(max(max(x[0], x[1]), max(x[2], x[3])), max(max(x[4], x[5]), max(x[6], x[7])));
    if (top >= n) {
#pragma unroll
      for (int k = 0; k < 4; ++k) guard(x[2 * k], x[2 * k + 1], n, ctrl);
    }
#pragma unroll
    for (int h = 0; h < 8; h += 4) {  // two edges at a time: all four took the registers of more warps
      uint32_t w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = bits[x[h + i] >> 5];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t xa = x[h + 2 * k], xb = x[h + 2 * k + 1];
        // the vertex's bit comes to the bottom (the rotation takes the count modulo 32)
        const uint32_t ka = __funnelshift_r(w[2 * k], w[2 * k], xa), kb = __funnelshift_r(w[2 * k + 1], w[2 * k + 1], xb);
        const bool keep = !(ka & kb & 1u);
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
        if (!bal) continue;
        if (keep) {
          const uint32_t slot = (q_tail + __popc(bal & lt_mask)) & (kRing - 1);
          qa[slot] = xa | (ka << 31);
          qb[slot] = xb | (kb << 31);
        }
        q_tail += __popc(bal);
        if (q_tail - q_head >= 32u) resolve(32u);
      }
    }
  }
  if (q_tail != q_head) resolve(q_tail - q_head);
}

constexpr uint32_t kGrab = 8;

template <class F>
cudaError_t bits_pass(const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl, uint32_t *bits, cudaStream_t s) {
  const uint64_t chunks = (e.n_quads + kChunkQuads - 1) / kChunkQuads;
  const unsigned gb = clamp_grid(((uint64_t)n + 1023) / 1024, persistent_cap((const void *)k_bits_build<F, true>, 256, 0));
  uint64_t sample = kFirstSample * n / (2 * kChunkQuads) + 1;  // in chunks
  Rounds rounds;
  uint64_t taken[kRounds];  // chunks
  for (uint32_t j = 0; j < kRounds; ++j, sample = sample / kShrink > kMinSampleChunks ? sample / kShrink : kMinSampleChunks) {
    rounds.chunk_stride[j] = (uint32_t)(chunks > sample ? chunks / sample : 1);
    taken[j] = (chunks + rounds.chunk_stride[j] - 1) / rounds.chunk_stride[j];
  }
  for (uint32_t r = 0; r < kRounds; ++r) {
    const void *k = r ? (const void *)k_bits_link<F, false> : (const void *)k_bits_link<F, true>;
    const unsigned gl = clamp_grid((taken[r] + kLinkBlock / 32 - 1) / (kLinkBlock / 32), persistent_cap(k, kLinkBlock, 0));
    if (r == 0)
      k_bits_link<F, true><<<gl, kLinkBlock, 0, s>>>(e.quads, e.n_quads, rounds, r, P, n, ctrl);
    else
      k_bits_link<F, false><<<gl, kLinkBlock, 0, s>>>(e.quads, e.n_quads, rounds, r, P, n, ctrl);
    note_launch();
    if (r + 1 < kRounds)
      k_bits_build<F, false><<<gb, 256, 0, s>>>(e.quads, e.n_quads, r, P, n, ctrl, nullptr);
    else
      k_bits_build<F, true><<<gb, 256, 0, s>>>(e.quads, e.n_quads, r, P, n, ctrl, bits);
    note_launch();
  }
  const void *k = (const void *)k_bits_filter<F>;
  static std::atomic<unsigned long long> smem_set{0};
  const cudaError_t err = ensure_func_attr(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)(kBitsVertices / 8 + filter_queue_bytes(kFilterBlock)), smem_set);
  if (err != cudaSuccess) return err;
  const bool pair = bits_bytes(n) + filter_queue_bytes(kFilterPairBlock) <= kFilterPairBytes;
  const unsigned block = pair ? kFilterPairBlock : kFilterBlock, warps = block / 32;
  const size_t smem = bits_bytes(n) + filter_queue_bytes(block);
  const unsigned gf = clamp_grid((chunks + warps - 1) / warps, (uint64_t)num_sms() * (pair ? 2u : 1u));
  const uint32_t grab = chunks >= (uint64_t)gf * warps * 4u * kGrab ? kGrab : 1u;
  k_bits_filter<F><<<gf, block, smem, s>>>(e.quads, e.n_quads, e.head, e.tail, P, n, ctrl, bits, grab);
  note_launch();
  // step 4, or nothing (the counter was reset with step 3's)
  return launch_edge_pass_general(F::kRF, e, P, n, ctrl, &ctrl->marked, s);
}

}  // namespace

bool bits_pass_fits(uint64_t n_vertices, uint64_t n_edges) {
  return n_vertices >= 1 && n_vertices <= kBitsVertices && n_edges >= kBitsMinEdges && n_edges < kBitsMaxEdges &&
         n_edges >= kBitsMinDegree * n_vertices;
}

cudaError_t launch_edge_pass_bits(bool rf, const EdgeSpan &e, uint32_t *P, uint32_t n, Ctrl *ctrl, uint32_t *bits,
                                  cudaStream_t s) {
  return rf ? bits_pass<RootR>(e, P, n, ctrl, bits, s) : bits_pass<RootId>(e, P, n, ctrl, bits, s);
}

}  // namespace cc
