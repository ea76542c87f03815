// Dimension 0 (Section 4, "Persistence pairs": the paper uses Kruskal's
// algorithm with union-find).  The persistence pairs of dimension 0 are the
// edges of the minimum spanning forest of the threshold graph under the refined
// filtration order, each paired with the vertex whose component dies (elder
// rule: of the two merging components, the one whose oldest vertex -- the
// largest index, Section 2 -- is younger dies).
//
// GB300 design: after the edge sort each cloud's edges are contiguous and in
// filtration order, so an edge's position is a unique weight realising the total
// order.  A cloud of up to H0_BLOCK_MAX_N vertices runs in one block (all clouds
// of a batch in one launch), which takes its edges from the front of the list,
// a batch at a time, and finds forest and elder rule together by contraction
// (h0_block_kernel); it stops reading when one component is left.  A larger
// cloud uses grid-wide Boruvka rounds and then the elder rule over the forest.
#include <atomic>

#include "rips_internal.cuh"

namespace rips {

namespace {

constexpr int H0_BLOCK_MAX_N = 12800;  // 12 bytes of shared memory per vertex, beside the edge list

__device__ __forceinline__ void edge_vertices_u32(uint64_t idx, uint32_t* a, uint32_t* b) {
  uint32_t x = (uint32_t)((1.0f + sqrtf(1.0f + 8.0f * (float)idx)) * 0.5f);
  while ((uint64_t)x * (x - 1) / 2 > idx) --x;
  while ((uint64_t)(x + 1) * x / 2 <= idx) ++x;
  *a = x;
  *b = (uint32_t)(idx - (uint64_t)x * (x - 1) / 2);
}

__device__ __forceinline__ uint64_t key_edge_index(uint64_t key, int eb) {
  const uint64_t emask = (1ull << eb) - 1;
  return emask - (key & emask);
}
__device__ __forceinline__ float key_length(uint64_t key, int eb) {
  return __uint_as_float((uint32_t)(key >> eb));
}

__device__ void emit_bar(rips_bar_t* bars, uint32_t* nbars, uint32_t cap, int cloud, float death, uint64_t birth_v,
                         uint64_t death_s) {
  const uint32_t pos = atomicAdd(nbars, 1u);
  if (pos < cap) {
    rips_bar_t b;
    b.dim = 0;
    b.birth = 0.0f;
    b.death = death;
    b.cloud = cloud;
    b.birth_simplex = birth_v;
    b.death_simplex = death_s;
    bars[pos] = b;
  }
}

// Elder rule over the forest edges fpos[0..nf) (increasing positions) of one
// cloud, by the calling thread, with parent/top already initialised.
__device__ void elder_rule(const uint64_t* __restrict__ keys, int eb, const uint32_t* __restrict__ eu,
                           const uint32_t* __restrict__ ev, const uint32_t* __restrict__ fpos, uint32_t nf, int n,
                           uint32_t* parent, uint32_t* top, int cloud, rips_bar_t* bars, uint32_t* nbars,
                           uint32_t cap, unsigned long long* st) {
  unsigned long long zero = 0;
  for (uint32_t q = 0; q < nf; ++q) {
    const uint32_t e = fpos[q];
    uint32_t ru = eu[e], rv = ev[e];
    while (parent[ru] != ru) {
      parent[ru] = parent[parent[ru]];
      ru = parent[ru];
    }
    while (parent[rv] != rv) {
      parent[rv] = parent[parent[rv]];
      rv = parent[rv];
    }
    if (ru == rv) continue;  // cannot happen on a forest edge
    const uint32_t die = min(top[ru], top[rv]);
    const uint32_t live = max(top[ru], top[rv]);
    parent[ru] = rv;
    top[rv] = live;
    const float death = key_length(keys[e], eb);
    if (death == 0.0f) {
      ++zero;
      continue;
    }
    emit_bar(bars, nbars, cap, cloud, death, die, key_edge_index(keys[e], eb));
  }
  unsigned long long ess = 0;
  for (int v = 0; v < n; ++v)
    if (parent[v] == (uint32_t)v) {
      emit_bar(bars, nbars, cap, cloud, __int_as_float(0x7f800000), top[v], ~0ull);
      ++ess;
    }
  st[0] = nf;
  st[1] = zero;
  st[2] = ess;
}

// local endpoints of every sorted edge
__global__ void edge_endpoints_kernel(const uint64_t* __restrict__ keys, uint32_t m, int eb, uint32_t* __restrict__ eu,
                                      uint32_t* __restrict__ ev) {
  uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m) return;
  uint32_t a, b;
  edge_vertices_u32(key_edge_index(keys[e], eb), &a, &b);
  eu[e] = a;
  ev[e] = b;
}

// local endpoints (a > b) of an edge of a cloud of at most H0_BLOCK_MAX_N
// vertices: an FP32 square root is within one of a there (indices below 2^27)
__device__ __forceinline__ uint32_t edge_vertices_u16(uint32_t idx) {
  uint32_t x = (uint32_t)((1.0f + sqrtf(1.0f + 8.0f * (float)idx)) * 0.5f);
  while (x * (x - 1) / 2 > idx) --x;
  while ((x + 1) * x / 2 <= idx) ++x;
  return (x << 16) | (idx - x * (x - 1) / 2);
}

// One cloud per block.  A component is named by its oldest (largest) vertex.
// Contraction: let e be the first edge, in filtration order, that leaves
// component C, and D the component across it.  If D's name is larger, C's name
// dies at e: every part of C that the edges before e join to C's end of e has
// C's name in it (a part of C was attached by its own first edge, which comes
// before any other edge that leaves it, e included), nothing outside C is joined
// to it before e, and likewise D's end is joined to D's name; so at e the
// component of C's name meets an older one, which is the elder rule.  C may then
// be merged into D, since its other edges come after e.  All components do this
// at once, round after round; the first edge left is always some component's, so
// a round merges at least one, and on unordered points half of them.  Edges are
// taken in batches of the shortest that still join two components; when a batch
// goes on for more than H0_ROUNDS rounds (an ordered chain of growing gaps merges
// one component a round), one thread finishes it in filtration order.
//
// The block before this one read all the edges about log2(n) times and then let
// one thread apply the elder rule from global memory: 34.5 ms for 4,096 points
// (8.4 M edges), 1.8 ms for 1,000.  Bound now by the latency of the shared-memory
// rounds.
constexpr int H0_ROUNDS = 40;
constexpr int H0_STEP = 4;  // edges a thread looks at in one step

__global__ void __launch_bounds__(1024) h0_block_kernel(const CloudInfo* __restrict__ clouds,
                                                        const uint64_t* __restrict__ keys, int eb,
                                                        uint8_t* __restrict__ in_forest_all,
                                                        rips_bar_t* __restrict__ bars, uint32_t* __restrict__ nbars,
                                                        uint32_t bar_cap, unsigned long long* __restrict__ stats,
                                                        int stats_stride, uint32_t list_cap) {
  extern __shared__ uint32_t sm[];
  const int cloud = blockIdx.x;
  const CloudInfo ci = clouds[cloud];
  const int n = ci.n;
  const uint32_t m = ci.m;
  const uint64_t* ek = keys + ci.eoff;
  uint8_t* in_forest = in_forest_all + ci.eoff;
  uint32_t* comp = sm;            // component of a vertex
  uint32_t* best = sm + n;        // a component's first edge; of one that is gone, the edge it died at
  uint32_t* parent = sm + 2 * n;  // itself, or the component it was merged into
  uint32_t* le = sm + 3 * n;      // the batch: edges
  uint32_t* lv = le + list_cap;   // and their endpoints, 16 bits each
  __shared__ uint32_t cnt, any, roots, tally[3];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const uint64_t emask = (1ull << eb) - 1;
  for (int v = tid; v < n; v += nt) {
    comp[v] = parent[v] = v;
    best[v] = 0xFFFFFFFFu;
  }
  if (tid == 0) {
    roots = n;
    tally[0] = tally[1] = tally[2] = 0;
  }
  __syncthreads();
  const uint32_t step = H0_STEP * nt;
  uint32_t pos = 0;
  while (pos < m && roots > 1) {  // block-uniform: both change between barriers only
    if (tid == 0) cnt = 0;
    __syncthreads();
    while (pos < m && cnt + step <= list_cap) {
      uint64_t key[H0_STEP];
#pragma unroll
      for (int u = 0; u < H0_STEP; ++u) {
        const uint32_t e = pos + u * nt + tid;
        key[u] = e < m ? ek[e] : 0;
      }
      __syncthreads();  // every thread has read cnt
#pragma unroll
      for (int u = 0; u < H0_STEP; ++u) {
        const uint32_t e = pos + u * nt + tid;
        const uint32_t uv = e < m ? edge_vertices_u16((uint32_t)(emask - (key[u] & emask))) : 0u;
        const bool keep = e < m && comp[uv >> 16] != comp[uv & 0xFFFFu];
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        uint32_t base = 0;
        if (lane == 0 && bal) base = atomicAdd(&cnt, (uint32_t)__popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(bal & ((1u << lane) - 1u));
        if (keep) {
          le[base] = e;
          lv[base] = uv;
        }
      }
      pos += step;
      __syncthreads();
    }
    const uint32_t L = cnt;
    for (int round = 0;; ++round) {
      if (tid == 0) any = 0;
      __syncthreads();
      bool mine = false;
      for (uint32_t i = tid; i < L; i += nt) {
        const uint32_t cu = comp[lv[i] >> 16], cv = comp[lv[i] & 0xFFFFu];
        if (cu != cv) {
          atomicMin(&best[cu], le[i]);
          atomicMin(&best[cv], le[i]);
          mine = true;
        }
      }
      if (mine) any = 1;
      __syncthreads();
      if (!any) break;
      if (round == H0_ROUNDS) {  // the rest of the batch in order: sort it, then one thread
        uint32_t n2 = 2;
        while (n2 < L) n2 <<= 1;  // at most list_cap, a power of two
        for (uint32_t i = L + tid; i < n2; i += nt) le[i] = 0xFFFFFFFFu;
        __syncthreads();
        for (uint32_t size = 2; size <= n2; size <<= 1)
          for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
            for (uint32_t i = tid; i < n2 / 2; i += nt) {
              const uint32_t x = 2 * i - (i & (stride - 1)), y = x + stride;
              const uint32_t ex = le[x], ey = le[y];
              if ((ex > ey) == ((x & size) == 0)) {
                const uint32_t t = lv[x];
                le[x] = ey;
                le[y] = ex;
                lv[x] = lv[y];
                lv[y] = t;
              }
            }
            __syncthreads();
          }
        if (tid == 0)
          for (uint32_t i = 0; i < L; ++i) {
            uint32_t cu = comp[lv[i] >> 16], cv = comp[lv[i] & 0xFFFFu];
            while (parent[cu] != cu) cu = parent[cu] = parent[parent[cu]];
            while (parent[cv] != cv) cv = parent[cv] = parent[parent[cv]];
            if (cu == cv) continue;
            const uint32_t die = min(cu, cv);
            parent[die] = max(cu, cv);
            best[die] = le[i];
            --roots;
          }
      } else {
        uint32_t hooked = 0;
        for (uint32_t i = tid; i < L; i += nt) {
          const uint32_t cu = comp[lv[i] >> 16], cv = comp[lv[i] & 0xFFFFu], die = min(cu, cv);
          if (cu != cv && best[die] == le[i]) {
            parent[die] = max(cu, cv);
            ++hooked;
          }
        }
        hooked = __reduce_add_sync(0xffffffffu, hooked);
        if (lane == 0 && hooked) atomicSub(&roots, hooked);
      }
      __syncthreads();
      for (int v = tid; v < n; v += nt) {
        uint32_t x = comp[v];
        while (parent[x] != x) x = parent[x];
        comp[v] = x;
        if (parent[v] == (uint32_t)v) best[v] = 0xFFFFFFFFu;
      }
      __syncthreads();
    }
    __syncthreads();  // cnt is reset
  }
  // bars: a vertex whose component is gone died at its edge (zero-length ones are counted only)
  for (int v0 = tid - lane; v0 < n; v0 += nt) {
    const int v = v0 + lane;
    const bool dead = v < n && parent[v] != (uint32_t)v, ess = v < n && !dead;
    const uint64_t key = dead ? ek[best[v]] : 0;
    const float death = dead ? key_length(key, eb) : __int_as_float(0x7f800000);
    if (dead) in_forest[best[v]] = 1;
    const bool zero = dead && death == 0.0f, put = (dead && !zero) || ess;
    const unsigned md = __ballot_sync(0xffffffffu, dead), mz = __ballot_sync(0xffffffffu, zero),
                   me = __ballot_sync(0xffffffffu, ess), mp = __ballot_sync(0xffffffffu, put);
    uint32_t base = 0;
    if (lane == 0) {
      if (md) atomicAdd(&tally[0], (uint32_t)__popc(md));
      if (mz) atomicAdd(&tally[1], (uint32_t)__popc(mz));
      if (me) atomicAdd(&tally[2], (uint32_t)__popc(me));
      if (mp) base = atomicAdd(nbars, (uint32_t)__popc(mp));
    }
    base = __shfl_sync(0xffffffffu, base, 0) + __popc(mp & ((1u << lane) - 1u));
    if (put && base < bar_cap) {
      rips_bar_t b;
      b.dim = 0;
      b.birth = 0.0f;
      b.death = death;
      b.cloud = cloud;
      b.birth_simplex = (uint64_t)v;
      b.death_simplex = dead ? key_edge_index(key, eb) : ~0ull;
      bars[base] = b;
    }
  }
  __syncthreads();
  if (tid < 3) stats[(size_t)cloud * stats_stride + tid] = tally[tid];
}

// ---------------------------------------------------------------- one large cloud

__global__ void init_components_kernel(int n, uint32_t* __restrict__ comp, uint32_t* __restrict__ best) {
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  comp[v] = v;
  best[v] = 0xFFFFFFFFu;
}

__global__ void boruvka_min_edge_kernel(const uint32_t* __restrict__ eu, const uint32_t* __restrict__ ev,
                                        uint32_t m, const uint32_t* __restrict__ comp, uint32_t* __restrict__ best) {
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < m; e += gridDim.x * blockDim.x) {
    uint32_t cu = comp[eu[e]], cv = comp[ev[e]];
    if (cu != cv) {
      atomicMin(&best[cu], e);
      atomicMin(&best[cv], e);
    }
  }
}

// every root hooks onto the component across its cheapest edge; of two
// components that chose the same edge, the larger label hooks
__global__ void boruvka_hook_kernel(int n, const uint32_t* __restrict__ eu, const uint32_t* __restrict__ ev,
                                    const uint32_t* __restrict__ comp, const uint32_t* __restrict__ best,
                                    uint32_t* __restrict__ parent, uint8_t* __restrict__ in_forest) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n || comp[c] != (uint32_t)c) return;
  uint32_t e = best[c];
  if (e == 0xFFFFFFFFu) {
    parent[c] = c;
    return;
  }
  uint32_t a = comp[eu[e]], b = comp[ev[e]];
  uint32_t other = (a == (uint32_t)c) ? b : a;
  if (best[other] == e && (uint32_t)c < other) {
    parent[c] = c;
  } else {
    parent[c] = other;
    in_forest[e] = 1;
  }
}

__global__ void boruvka_jump_kernel(int n, uint32_t* __restrict__ comp, const uint32_t* __restrict__ parent,
                                    uint32_t* __restrict__ best, uint32_t* __restrict__ err) {
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  uint32_t x = comp[v];
  int guard = 0;
  while (parent[x] != x) {
    x = parent[x];
    if (++guard > n) {
      set_error(err, ERRF_TIMEOUT);
      break;
    }
  }
  comp[v] = x;
  best[v] = 0xFFFFFFFFu;
}

__global__ void elder_rule_kernel(int n, const uint32_t* __restrict__ fpos, const uint32_t* __restrict__ nf,
                                  const uint32_t* __restrict__ eu, const uint32_t* __restrict__ ev,
                                  const uint64_t* __restrict__ keys, int eb, uint32_t* __restrict__ parent,
                                  uint32_t* __restrict__ top, rips_bar_t* __restrict__ bars,
                                  uint32_t* __restrict__ nbars, uint32_t bar_cap, unsigned long long* __restrict__ st) {
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    parent[v] = v;
    top[v] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) elder_rule(keys, eb, eu, ev, fpos, *nf, n, parent, top, 0, bars, nbars, bar_cap, st);
}

__global__ void flags_from_bytes_kernel(const uint8_t* __restrict__ b, uint32_t m, uint32_t* __restrict__ f) {
  uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < m) f[e] = b[e];
}

__global__ void compact_positions_kernel(const uint8_t* __restrict__ in_forest, const uint32_t* __restrict__ excl,
                                         uint32_t m, uint32_t* __restrict__ out) {
  uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < m && in_forest[e]) out[excl[e]] = e;
}

}  // namespace

bool h0_blocks_fit(int n_max) { return n_max <= H0_BLOCK_MAX_N; }

cudaError_t launch_h0_blocks(const CloudInfo* clouds, int nclouds, int n_max, const uint64_t* sorted_keys,
                             int edge_bits, uint32_t m_total, uint8_t* in_forest, rips_bar_t* bars, uint32_t* nbars,
                             uint32_t bar_cap, unsigned long long* stats, int stats_stride, cudaStream_t s) {
  cudaError_t e;
  if (m_total && (e = cudaMemsetAsync(in_forest, 0, m_total, s)) != cudaSuccess) return e;
  // Threads and list for the cloud size: a batch of 8,192 edges (two steps of 1,024 threads) costs 64 KB beside the
  // 12 bytes a vertex; small clouds, many to a launch, take 256 threads and 2,048 edges, so that several blocks share
  // an SM.
  const int threads = n_max <= 256 ? 256 : 1024;
  const uint32_t list_cap = 2u * H0_STEP * (uint32_t)threads;
  const size_t smem = (size_t)12 * (n_max > 0 ? n_max : 1) + (size_t)8 * list_cap;
  if (smem > 48 * 1024) {
    // once per device and to the largest size any call needs: calls of other threads are between setting and launching
    static std::atomic<bool> opted[64];
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !opted[dev].load(std::memory_order_acquire)) {
      constexpr int most = 12 * H0_BLOCK_MAX_N + 8 * 2 * H0_STEP * 1024;
      if ((e = cudaFuncSetAttribute(h0_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess)
        return e;
      if (dev >= 0 && dev < 64) opted[dev].store(true, std::memory_order_release);
    }
  }
  h0_block_kernel<<<nclouds, threads, smem, s>>>(clouds, sorted_keys, edge_bits, in_forest, bars, nbars, bar_cap, stats,
                                                 stats_stride, list_cap);
  note_launch();
  return cudaGetLastError();
}

cudaError_t run_h0_large(int n, const uint64_t* sorted_keys, uint32_t m, int edge_bits, uint32_t* eu, uint32_t* ev,
                         uint32_t* comp, uint32_t* best, uint32_t* parent, uint8_t* in_forest, uint32_t* flags,
                         uint32_t* fpos, void* scan_tmp, uint32_t* d_nf, uint32_t* gtop, rips_bar_t* bars,
                         uint32_t* nbars, uint32_t bar_cap, unsigned long long* stats, uint32_t* err, cudaStream_t s) {
  cudaError_t e;
  if ((e = cudaMemsetAsync(in_forest, 0, m ? m : 1, s)) != cudaSuccess) return e;
  if (m) {
    edge_endpoints_kernel<<<(m + 255) / 256, 256, 0, s>>>(sorted_keys, m, edge_bits, eu, ev);
    note_launch();
  }
  init_components_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, comp, best);
  note_launch();
  int rounds = 1;
  while ((1 << (rounds - 1)) < n) ++rounds;
  int eblocks = (int)((m + 255) / 256);
  if (eblocks > 152 * 8) eblocks = 152 * 8;
  if (eblocks < 1) eblocks = 1;
  for (int r = 0; m && r < rounds; ++r) {
    boruvka_min_edge_kernel<<<eblocks, 256, 0, s>>>(eu, ev, m, comp, best);
    note_launch();
    boruvka_hook_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, eu, ev, comp, best, parent, in_forest);
    note_launch();
    boruvka_jump_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, comp, parent, best, err);
    note_launch();
  }
  if (m) {
    flags_from_bytes_kernel<<<(m + 255) / 256, 256, 0, s>>>(in_forest, m, flags);
    note_launch();
    if ((e = launch_exclusive_scan(flags, flags, m, scan_tmp, d_nf, s)) != cudaSuccess) return e;
    compact_positions_kernel<<<(m + 255) / 256, 256, 0, s>>>(in_forest, flags, m, fpos);
    note_launch();
  } else {
    if ((e = cudaMemsetAsync(d_nf, 0, sizeof(uint32_t), s)) != cudaSuccess) return e;
  }
  // the forest has at most n - 1 edges; the elder rule reads the count on the device
  elder_rule_kernel<<<1, 256, 0, s>>>(n, fpos, d_nf, eu, ev, sorted_keys, edge_bits, parent, gtop, bars, nbars, bar_cap,
                                      stats);
  note_launch();
  return cudaGetLastError();
}

}  // namespace rips
