// One dimension d >= 1 of the cohomology computation (Section 3.3) for every
// cloud of a batch at once: columns are the d-simplices, rows the
// (d+1)-simplices, columns are processed youngest first (diameter down, then
// index up, Section 3.5 "Shortcuts" and Section 4 "Pivot extraction"), and a
// column's pivot is its OLDEST nonzero row (smallest diameter, then largest
// index).  Every work item carries its cloud in the top bits of its key.
//
// Kernels (warp-cooperative; lanes take consecutive entries of a vertex's
// neighbour list, so every cofacet tile is 32 candidates wide):
//
//  enumerate_kernel   all d-simplices <= t, each made once as (j, rho) with
//                     j above the top vertex of a (d-1)-simplex rho (Section 4,
//                     "Assembling column indices").
//  test_kernel        drops a d-simplex if it is cleared (a pivot of the
//                     (d-1)-reduction: Section 3.2 / Algorithm 2), if it has a
//                     zero-persistence apparent cofacet, or a zero-persistence
//                     apparent facet (Proposition in Section 3.5 and the
//                     procedure in its "Shortcuts" paragraph); survivors are
//                     compacted with their processing-order key.
//  reduce_persistent_kernel  one cooperative launch per dimension:
//     first pivots    the cofacets are scanned in decreasing index order and
//                     the first one with the column's own diameter is the pivot
//                     (the emergent-pair shortcut, Section 3.5); only when there
//                     is none is the whole coboundary scanned for its minimum;
//     claim           columns claim their pivot in an open-addressing table by
//                     atomicCAS on the key and atomicMin on the column ordinal:
//                     the earliest column in processing order owns a pivot;
//     reduce          every column whose pivot is owned by an earlier column
//                     adds that column (R_j -= lambda R_k, Algorithm 1) and keeps
//                     going while the new pivot is owned by an earlier column; a
//                     pivot with a zero apparent facet is owned by that facet's
//                     column (Section 4, "Persistence pairs": apparent pairs are
//                     not in the table).  A warp makes short chains, one
//                     addition after the other, at most DimArgs::chain_limit a
//                     round; the columns it gives up, and all of them once there
//                     are few, are reduced by blocks or teams of blocks that add
//                     many columns at a time (rips_wide.cuh).
//
// The coboundary stays implicit (Section 3.4) for every column that is never
// added to -- apparent, emergent and unreduced owners: their coboundary is
// generated from the combinatorial number system when it is needed.  A column
// that is reduced keeps its working column R_j materialised (sorted row keys,
// nonzero coefficients), so later additions of it cost a merge instead of a
// regeneration; V is not stored since only pairs are reported.
//
// Parallel reduction and correctness.  Claims and reductions alternate in
// rounds separated by grid barriers.  A column only ever adds a column that
// precedes it in processing order (or an apparent facet's column, which
// precedes every column with that pivot), so R = D V with V upper
// unitriangular; pivots only move to younger rows, so the rounds end; at the
// end every nonzero column owns its pivot alone, i.e. R is reduced, and by the
// pivot proposition of Section 3.1 the pairs are exactly those of the
// sequential algorithm (the pairing of a reduced matrix is unique).
#include <mutex>
#include <vector>

#include "rips_internal.cuh"

namespace rips {

namespace {

constexpr int WARPS_PER_BLOCK = 8;
constexpr uint32_t MAX_PIVOT_PASSES = 1u << 30;  // additions in one chain before giving up
constexpr uint32_t FIRST_CHAIN = 8;               // additions a warp makes on a column with its first pivot
constexpr uint8_t HEAVY = 2;                      // flag in RedState::reduced: reduced by blocks
constexpr uint8_t UNSORTED = 4;                   // flag: its stored run is not in key order (and it is heavy)

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct Binom {
  const uint64_t* t;
  int s;
  __device__ __forceinline__ uint64_t operator()(int i, int k) const { return t[(size_t)k * s + i]; }
};

__device__ __forceinline__ Binom stage_binom(const DimArgs& a, uint64_t* smem) {
  Binom b{a.binom, a.bn + 1};
  if (a.smem_binom) {
    const int total = (a.kmax + 1) * (a.bn + 1);
    for (int i = threadIdx.x; i < total; i += blockDim.x) smem[i] = a.binom[i];
    __syncthreads();
    b.t = smem;
  }
  return b;
}

// ---------------------------------------------------------------- clouds
// A cloud's view: its size, rank matrix and neighbour-list offsets (indexed by
// local vertex) into the shared list array.
// R is null for a sparse input: the rank of an edge then comes from the
// neighbour lists (nrank[q] = rank of the edge to nbr[q]).
struct CV {
  int n;
  const uint32_t* R;
  const uint32_t* off;
  const uint32_t* nbr;
  const uint32_t* nrank;
};

__device__ __forceinline__ CV cloud_view(const DimArgs& a, uint32_t c) {
  const CloudInfo ci = a.clouds[c];
  return CV{ci.n, a.R ? a.R + ci.roff : nullptr, a.nbr_off + ci.voff, a.nbr, a.nrank};
}

// Rank of the edge (x, y), RANK_INF when it is above the threshold or x == y:
// one read of the rank matrix, or with a sparse input a binary search for y in
// x's neighbour list (vertices in decreasing order).
__device__ __forceinline__ uint32_t rank_of(const CV& cv, int x, int y) {
  if (cv.R) return cv.R[(size_t)x * cv.n + y];
  const uint32_t end = cv.off[x + 1];
  uint32_t lo = cv.off[x], hi = end;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (cv.nbr[mid] > (uint32_t)y) lo = mid + 1;
    else hi = mid;
  }
  return lo < end && cv.nbr[lo] == (uint32_t)y ? cv.nrank[lo] : RANK_INF;
}

__device__ __forceinline__ uint64_t low_mask(int bits) { return bits >= 64 ? ~0ull : ((1ull << bits) - 1); }
__device__ __forceinline__ uint32_t high_part(uint64_t x, int bits) { return bits >= 64 ? 0u : (uint32_t)(x >> bits); }

// ---------------------------------------------------------------- simplex helpers

struct Simplex {
  int v[MAX_DIM + 2];  // vertices, decreasing
  uint64_t idx;
  uint32_t rank;
};

// largest v in [lo, hi] with C(v, k) <= N, by bisection
__device__ __forceinline__ int max_vertex_bisect(const Binom& B, int k, int lo, int hi, uint64_t N) {
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B(mid, k) <= N) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Largest v in [k-1, hi] with C(v, k) <= N (k >= 2), i.e. the top vertex of the
// k-subset with index N (Section 4, "combinatorial number system").  Since
// C(v, k) is about (v - (k-1)/2)^k / k!, a float root of k! N gives v to within
// one or two; four neighbouring table entries (one or two cache lines) settle
// it, and bisection takes over if the estimate was further off.
__device__ __forceinline__ int max_vertex(const Binom& B, int k, int hi, uint64_t N) {
  float kf = 1.0f;
  for (int i = 2; i <= k; ++i) kf *= (float)i;
  const float est = exp2f(log2f(__ull2float_rn(N) * kf) / (float)k) + 0.5f * (float)(k - 1);
  int v = est >= (float)hi ? hi : (int)est;
  if (v < k - 1) v = k - 1;
  const uint64_t b0 = B(v, k);
  const uint64_t bm = B(v > 0 ? v - 1 : 0, k);
  const uint64_t b1 = B(v + 1 <= hi ? v + 1 : hi, k);
  const uint64_t b2 = B(v + 2 <= hi ? v + 2 : hi, k);
  if (b0 <= N) {
    if (v == hi || b1 > N) return v;
    if (v + 1 == hi || b2 > N) return v + 1;
    return max_vertex_bisect(B, k, v + 2, hi, N);
  }
  // b0 > N implies v >= k, so v - 1 >= k - 1
  if (bm <= N) return v - 1;
  return max_vertex_bisect(B, k, k - 1, v - 2, N);
}

__device__ __forceinline__ void decode(const Binom& B, int n, uint64_t N, int d, int* v) {
  int hi = n - 1;
  for (int k = d + 1; k >= 1; --k) {
    const int x = k == 1 ? (int)N : max_vertex(B, k, hi, N);
    v[d + 1 - k] = x;
    N -= k == 1 ? N : B(x, k);
    hi = x - 1;
  }
}

// Vertices of a d-simplex given by a reference: its index, or (packed) its
// vertices packed vbits apiece as the pair map stores them.
__device__ __forceinline__ void simplex_vertices(const Binom& B, int n, uint64_t ref, bool packed, int vbits, int d,
                                                 int* v) {
  if (!packed) {
    decode(B, n, ref, d, v);
    return;
  }
  const uint64_t m = (1ull << vbits) - 1;
  for (int l = 0; l <= d; ++l) v[l] = (int)((ref >> (l * vbits)) & m);
}

// rank of sigma with vertex v[l] removed, for every l (d >= 1)
__device__ __forceinline__ void ranks_minus_one(const CV& cv, const int* v, int d, uint32_t* out) {
  for (int l = 0; l <= d; ++l) out[l] = 0;
  for (int a = 0; a <= d; ++a)
    for (int b = a + 1; b <= d; ++b) {
      uint32_t r = rank_of(cv, v[a], v[b]);
      for (int l = 0; l <= d; ++l)
        if (l != a && l != b) out[l] = max(out[l], r);
    }
}

// vertex of sigma (index into v) with the shortest neighbour list
__device__ __forceinline__ int min_degree_vertex(const CV& cv, const int* v, int cnt) {
  int best = 0;
  uint32_t bd = cv.off[v[0] + 1] - cv.off[v[0]];
  for (int l = 1; l < cnt; ++l) {
    uint32_t dg = cv.off[v[l] + 1] - cv.off[v[l]];
    if (dg < bd) {
      bd = dg;
      best = l;
    }
  }
  return best;
}

// Cofacet tau = sigma + j of a d-simplex with vertices v (decreasing).  c = number
// of vertices above j.  idx(tau) = above[c] + C(j, d+2-c) + below[c], where
// above[c] = sum_{l<c} C(v[l], d+2-l), below[c] = sum_{l>=c} C(v[l], d+1-l)
// (Section 4, "Enumerating cofacets": the two running partial sums).
struct CofacetSums {
  uint64_t above[MAX_DIM + 2];
  uint64_t below[MAX_DIM + 2];
};

__device__ __forceinline__ void cofacet_sums(const Binom& B, const int* v, int d, CofacetSums& cs) {
  uint64_t acc = 0;
  for (int c = 0; c <= d + 1; ++c) {
    cs.above[c] = acc;
    if (c <= d) acc += B(v[c], d + 2 - c);
  }
  acc = 0;
  for (int c = d + 1; c >= 0; --c) {
    cs.below[c] = acc;
    if (c >= 1) acc += B(v[c - 1], d + 2 - c);
  }
}

// Evaluate candidate j for the cofacets of sigma: returns false if sigma + j is not
// a simplex <= t (including j in sigma).  On success gives rank, index and the
// number c of vertices of sigma above j.
__device__ __forceinline__ bool cofacet_of(const CV& cv, const Binom& B, const int* v, int d, uint32_t srank,
                                           const CofacetSums& cs, int j, uint32_t* rank, uint64_t* idx, int* cpos) {
  uint32_t r = srank;
  int c = 0;
  bool ok = true;
  for (int l = 0; l <= d; ++l) {  // no early exit: the loads are independent
    const uint32_t x = rank_of(cv, v[l], j);
    ok &= x != RANK_INF;
    r = max(r, x);
    c += v[l] > j;
  }
  const uint64_t bj = B(j, d + 2 - c);  // loaded beside the rank lookups, not after them
  if (!ok) return false;
  *rank = r;
  *cpos = c;
  *idx = cs.above[c] + bj + cs.below[c];
  return true;
}

__device__ __forceinline__ uint64_t row_key(const DimArgs& a, uint32_t rank, uint64_t idx) {
  const uint64_t mask = (a.row_bits >= 64) ? ~0ull : ((1ull << a.row_bits) - 1);
  return ((uint64_t)rank << a.row_bits) | (mask - idx);
}
__device__ __forceinline__ uint64_t row_key_idx(const DimArgs& a, uint64_t key) {
  const uint64_t mask = (a.row_bits >= 64) ? ~0ull : ((1ull << a.row_bits) - 1);
  return mask - (key & mask);
}
__device__ __forceinline__ uint32_t row_key_rank(const DimArgs& a, uint64_t key) {
  return (uint32_t)(key >> a.row_bits);
}

// Largest-index cofacet of sigma with the same diameter rank (the candidate tau of
// the Proposition on zero apparent pairs), found by scanning cofacets in
// decreasing index order.  Warp-cooperative; every lane gets the result.
// Returns the vertex j (or -1) and, on the owning lane, fills the ranks of j to
// the vertices of sigma.
__device__ int first_equal_cofacet(const CV& cv, const int* v, int d, uint32_t srank, int lane,
                                   uint32_t* rj /* d+1, valid on the returned lane */, int* hit_lane) {
  int av = v[min_degree_vertex(cv, v, d + 1)];
  const uint32_t beg = cv.off[av], end = cv.off[av + 1];
  for (uint32_t q0 = beg; q0 < end; q0 += 32) {
    const uint32_t q = q0 + lane;
    bool hit = false;
    int j = -1;
    if (q < end) {
      j = (int)cv.nbr[q];
      hit = true;
      for (int l = 0; l <= d; ++l) {
        uint32_t x = rank_of(cv, v[l], j);
        rj[l] = x;
        if (x > srank) hit = false;  // also rejects RANK_INF and j in sigma
      }
    }
    unsigned m = __ballot_sync(0xffffffffu, hit);
    if (m) {
      int src = __ffs(m) - 1;
      *hit_lane = src;
      return __shfl_sync(0xffffffffu, j, src);
    }
  }
  *hit_lane = -1;
  return -1;
}

// Zero apparent facet of a k-simplex tau with vertices w (decreasing) and rank r
// (Section 3.5): rho = the smallest-index facet with the same rank (facets in
// increasing index order drop the largest vertices first); apparent iff tau is
// the largest-index cofacet of rho with that rank, i.e. no vertex u > w[l]
// outside tau gives rank(rho + u) <= r.  Warp-cooperative.  Returns l (the
// dropped vertex position) or -1.
__device__ int zero_apparent_facet(const CV& cv, const int* w, int k, uint32_t r, const uint32_t* minus,
                                   int lane) {
  int l = -1;
  for (int x = 0; x <= k; ++x)
    if (minus[x] == r) {
      l = x;
      break;
    }
  if (l < 0) return -1;
  const int drop = w[l];
  // vertices of rho
  int rv[MAX_DIM + 2];
  int m = 0;
  for (int x = 0; x <= k; ++x)
    if (x != l) rv[m++] = w[x];
  int av = rv[min_degree_vertex(cv, rv, k)];
  const uint32_t beg = cv.off[av], end = cv.off[av + 1];
  for (uint32_t q0 = beg; q0 < end; q0 += 32) {
    const uint32_t q = q0 + lane;
    bool above = false, hit = false;
    if (q < end) {
      int u = (int)cv.nbr[q];
      above = u > drop;
      if (above) {
        hit = true;
        for (int x = 0; x < k; ++x) hit &= rank_of(cv, rv[x], u) <= r;
        // u is not a vertex of tau: the dropped vertex is excluded by u > drop, the
        // others by R = RANK_INF on the diagonal
      }
    }
    if (__any_sync(0xffffffffu, hit)) return -1;
    if (!__all_sync(0xffffffffu, above || q >= end)) break;  // the list went below drop
  }
  return l;
}

// ---------------------------------------------------------------- hash table
__device__ __forceinline__ uint64_t mix(uint64_t x) {
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  x *= 0xc4ceb9fe1a85ec53ull;
  x ^= x >> 33;
  return x;
}

// slot of key, inserting it if absent; -1 when the probe limit is hit
__device__ __forceinline__ int64_t table_insert(uint64_t* keys, uint64_t cap_mask, uint64_t key) {
  uint64_t h = mix(key) & cap_mask;
  for (uint64_t probe = 0; probe <= cap_mask; ++probe) {
    uint64_t cur = keys[h];
    if (cur == key) return (int64_t)h;
    if (cur == IDX_NONE) {
      uint64_t old = atomicCAS((unsigned long long*)&keys[h], (unsigned long long)IDX_NONE, (unsigned long long)key);
      if (old == IDX_NONE || old == key) return (int64_t)h;
    }
    h = (h + 1) & cap_mask;
  }
  return -1;
}

// (key, value) pair tables: slot h is kv[2h] (key, IDX_NONE when empty) and
// kv[2h + 1] (value), so a probe reads both in one 16-byte load
__device__ __forceinline__ int64_t pair_insert(uint64_t* kv, uint64_t cap_mask, uint64_t key) {
  uint64_t h = mix(key) & cap_mask;
  for (uint64_t probe = 0; probe <= cap_mask; ++probe) {
    const uint64_t cur = kv[2 * h];
    if (cur == key) return (int64_t)h;
    if (cur == IDX_NONE) {
      const uint64_t old =
          atomicCAS((unsigned long long*)&kv[2 * h], (unsigned long long)IDX_NONE, (unsigned long long)key);
      if (old == IDX_NONE || old == key) return (int64_t)h;
    }
    h = (h + 1) & cap_mask;
  }
  return -1;
}

__device__ __forceinline__ bool pair_find(const uint64_t* kv, uint64_t cap_mask, uint64_t key, uint64_t* val) {
  uint64_t h = mix(key) & cap_mask;
  for (uint64_t probe = 0; probe <= cap_mask; ++probe) {
    const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(kv + 2 * h);
    if (e.x == key) {
      *val = e.y;
      return true;
    }
    if (e.x == IDX_NONE) return false;
    h = (h + 1) & cap_mask;
  }
  return false;
}

__device__ __forceinline__ int64_t table_find(const uint64_t* keys, uint64_t cap_mask, uint64_t key) {
  if (cap_mask == 0 && keys == nullptr) return -1;
  uint64_t h = mix(key) & cap_mask;
  for (uint64_t probe = 0; probe <= cap_mask; ++probe) {
    uint64_t cur = keys[h];
    if (cur == key) return (int64_t)h;
    if (cur == IDX_NONE) return -1;
    h = (h + 1) & cap_mask;
  }
  return -1;
}

}  // namespace

// ====================================================================== enumeration

__global__ void __launch_bounds__(256) enumerate_kernel(DimArgs a, const uint64_t* __restrict__ pidx,
                                                        const uint32_t* __restrict__ prank, uint32_t np, int pbits,
                                                        uint64_t* __restrict__ out_idx, uint32_t* __restrict__ out_rank,
                                                        unsigned long long* __restrict__ count,
                                                        unsigned long long cap) {
  extern __shared__ uint64_t smem[];
  Binom B = stage_binom(a, smem);
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int d = a.d;  // new simplices are d-simplices, made from (d-1)-simplices
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < np; s += warps) {
    const uint64_t g = pidx[s];
    const uint32_t cl = high_part(g, pbits);
    const uint64_t local = g & low_mask(pbits);
    const CV cv = cloud_view(a, cl);
    const uint64_t chi = a.col_bits >= 64 ? 0ull : ((uint64_t)cl << a.col_bits);
    int v[MAX_DIM + 2];
    decode(B, cv.n, local, d - 1, v);
    const uint32_t r0 = prank[s];
    const int top = v[0];
    const int av = v[min_degree_vertex(cv, v, d)];
    const uint32_t beg = cv.off[av], end = cv.off[av + 1];
    for (uint32_t q0 = beg; q0 < end; q0 += 32) {
      const uint32_t q = q0 + lane;
      int j = q < end ? (int)cv.nbr[q] : -1;
      bool ok = j > top;
      uint32_t r = r0;
      if (ok)
        for (int l = 0; l < d; ++l) {
          uint32_t x = rank_of(cv, v[l], j);
          if (x == RANK_INF) {
            ok = false;
            break;
          }
          r = max(r, x);
        }
      unsigned m = __ballot_sync(0xffffffffu, ok);
      if (m) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(count, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (ok) {
          unsigned long long pos = base + __popc(m & lt);
          if (pos < cap) {
            out_idx[pos] = chi | (local + B(j, d + 1));
            out_rank[pos] = r;
          }
        }
      }
      if (!__all_sync(0xffffffffu, j > top)) break;  // the list went below the top vertex
    }
  }
}

// edges (sorted) -> simplex list of dimension 1
__global__ void edges_to_simplices_kernel(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ erank,
                                          uint32_t m, int eb, int col_bits, uint64_t* __restrict__ sidx,
                                          uint32_t* __restrict__ srank) {
  uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m) return;
  const uint64_t key = keys[e];
  if (key == ~0ull) {  // padding past the edge count (batch plans): skipped by the test
    sidx[e] = ~0ull;
    srank[e] = 0;
    return;
  }
  const uint64_t emask = (1ull << eb) - 1;
  const uint64_t c = key >> (32 + eb);
  sidx[e] = (col_bits >= 64 ? 0ull : (c << col_bits)) | (emask - (key & emask));
  srank[e] = erank[e];
}

// ====================================================================== apparent + clearing test

// pivot-table key of a row: (cloud << row_bits) | local row index
__device__ __forceinline__ uint64_t table_key(const DimArgs& a, uint32_t cloud, uint64_t row_idx) {
  return (a.row_bits >= 64 ? 0ull : ((uint64_t)cloud << a.row_bits)) | row_idx;
}

// A lane takes a simplex.  Most simplices are settled by one or two hash probes
// or by the first few candidates of their neighbour list (a cofacet of their own
// diameter), so 32 of them side by side need a fraction of the instructions of a
// warp on each; a lane that finds none among FIRST_CANDIDATES leaves the rest of
// its list to the whole warp, 32 candidates at a time.  Bound by the L1 on dense
// inputs that fit it and by the gathers through the rank matrix on others
// (scattered 32-byte sectors).  D = d keeps a simplex's vertices in registers;
// 0: any d.
constexpr uint32_t FIRST_CANDIDATES = 32;

template <int D>
__global__ void __launch_bounds__(256) test_kernel(DimArgs a, const uint64_t* __restrict__ sidx,
                                                   const uint32_t* __restrict__ srank, uint32_t ns,
                                                   const uint8_t* __restrict__ cleared_flag /* d == 1 */,
                                                   const uint64_t* __restrict__ prev_keys, uint64_t prev_mask,
                                                   uint64_t* __restrict__ col_keys, uint32_t* __restrict__ ncols,
                                                   uint32_t col_cap, unsigned long long* __restrict__ st,
                                                   int st_stride) {
  const Binom B{a.binom, a.bn + 1};
  const int lane = threadIdx.x & 31;
  const int d = D ? D : a.d;
  constexpr int NV = D ? D + 1 : MAX_DIM + 2;
  // cofacet side: (sigma, tau) zero apparent pair?  (not with the apparent-pair
  // shortcut switched off: every simplex that is not cleared is then a column)
  const bool apparent = !(a.opts & RIPS_OPT_NO_APPARENT);
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  // counters are flushed to the cloud's statistics whenever the warp moves to another cloud
  unsigned n_cof = 0, n_fac = 0, n_clr = 0;
  uint32_t cur_cloud = 0xFFFFFFFFu;
  auto flush = [&](uint32_t next) {
    if (lane == 0 && cur_cloud != 0xFFFFFFFFu) {
      unsigned long long* q = st + (size_t)cur_cloud * st_stride;
      if (n_cof) atomicAdd(&q[4], (unsigned long long)n_cof);
      if (n_fac) atomicAdd(&q[5], (unsigned long long)n_fac);
      if (n_clr) atomicAdd(&q[6], (unsigned long long)n_clr);
    }
    n_cof = n_fac = n_clr = 0;
    cur_cloud = next;
  };
  for (uint64_t s0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; s0 < ns; s0 += warps * 32) {
    const uint64_t s = s0 + lane;
    const uint64_t g = s < ns ? sidx[s] : ~0ull;
    const bool act = g != ~0ull;  // else past the end, or padding (batch plans)
    const unsigned am = __ballot_sync(0xffffffffu, act);
    if (!am) continue;
    const uint32_t cl = act ? high_part(g, a.col_bits) : 0u;
    const uint64_t idx = g & low_mask(a.col_bits);
    // clearing: pivots of the previous dimension
    bool clr = false, fac = false;
    if (act) {
      if (d == 1) clr = cleared_flag[s] != 0;
      else clr = prev_keys != nullptr && table_find(prev_keys, prev_mask, g) >= 0;
      // facet side (d >= 2; in dimension 1 such edges are spanning-forest edges): the previous dimension's test
      // recorded every zero apparent pair.  A simplex is in one pair at most, so this side may go first.
      if (!clr && apparent && d >= 2 && a.pmap) {
        uint64_t unused;
        fac = pair_find(a.pmap, a.pmap_mask, g, &unused);
      }
    }
    const bool rem = act && !clr && !fac;
    const CV cv = cloud_view(a, cl);
    int v[NV];
    uint32_t rj[NV];
    uint32_t r = 0, q = 0, end = 0;
    int j = -1;
    if (rem) {
      r = srank[s];
      int hi = cv.n - 1;
      uint64_t N = idx;
#pragma unroll
      for (int l = 0; l < NV; ++l)
        if (l <= d) {
          const int k = d + 1 - l;
          v[l] = k == 1 ? (int)N : max_vertex(B, k, hi, N);
          N -= k == 1 ? N : B(v[l], k);
          hi = v[l] - 1;
        }
      if (apparent) {
        q = cv.off[v[0]];
        end = cv.off[v[0] + 1];
#pragma unroll
        for (int l = 1; l < NV; ++l)
          if (l <= d) {
            const uint32_t o0 = cv.off[v[l]], o1 = cv.off[v[l] + 1];
            if (o1 - o0 < end - q) {
              q = o0;
              end = o1;
            }
          }
        const uint32_t lim = min(end, q + FIRST_CANDIDATES);
        for (; q < lim; ++q) {
          const int c = (int)cv.nbr[q];
          bool ok = true;
#pragma unroll
          for (int l = 0; l < NV; ++l)
            if (l <= d) {
              rj[l] = rank_of(cv, v[l], c);
              ok &= rj[l] <= r;  // also rejects RANK_INF and vertices of sigma
            }
          if (ok) {
            j = c;
            break;
          }
        }
      }
    }
    unsigned m = __ballot_sync(0xffffffffu, rem && apparent && j < 0 && q < end);
    while (m) {  // the rest of a lane's list, by the whole warp
      const int L = __ffs(m) - 1;
      m &= m - 1;
      const CV cb = cloud_view(a, __shfl_sync(0xffffffffu, cl, L));
      const uint32_t rb = __shfl_sync(0xffffffffu, r, L), eb = __shfl_sync(0xffffffffu, end, L);
      int vb[NV];
#pragma unroll
      for (int l = 0; l < NV; ++l) vb[l] = l <= d ? __shfl_sync(0xffffffffu, v[l], L) : 0;
      for (uint32_t q0 = __shfl_sync(0xffffffffu, q, L); q0 < eb; q0 += 32) {
        const int c = q0 + lane < eb ? (int)cb.nbr[q0 + lane] : vb[0];  // a vertex of sigma is no candidate
        bool ok = true;
        uint32_t rc[NV];
#pragma unroll
        for (int l = 0; l < NV; ++l)
          if (l <= d) {
            rc[l] = rank_of(cb, vb[l], c);
            ok &= rc[l] <= rb;
          }
        const unsigned hit = __ballot_sync(0xffffffffu, ok);
        if (hit) {
          const int src = __ffs(hit) - 1;
          const int jc = __shfl_sync(0xffffffffu, c, src);
          if (lane == L) j = jc;
#pragma unroll
          for (int l = 0; l < NV; ++l)
            if (l <= d) {
              const uint32_t x = __shfl_sync(0xffffffffu, rc[l], src);
              if (lane == L) rj[l] = x;
            }
          break;
        }
      }
    }
    bool app = false;
    if (j >= 0) {
      app = true;
      // facets of tau dropping a vertex above j come before sigma in index order: none may have its diameter
      int c = 0;
#pragma unroll
      for (int l = 0; l < NV; ++l)
        if (l <= d && v[l] > j) {
          ++c;
          uint32_t fr = 0;
#pragma unroll
          for (int x = 0; x < NV; ++x)
            if (x <= d && x != l) {
              fr = max(fr, rj[x]);
#pragma unroll
              for (int y = x + 1; y < NV; ++y)
                if (y <= d && y != l) fr = max(fr, rank_of(cv, v[x], v[y]));
            }
          if (fr == r) app = false;
        }
      if (app && a.amap) {  // tau -> sigma, for the reduction and the next dimension
        uint64_t tidx = B(j, d + 2 - c);
#pragma unroll
        for (int l = 0; l < NV; ++l)
          if (l <= d) tidx += B(v[l], l < c ? d + 2 - l : d + 1 - l);
        const int64_t slot = pair_insert(a.amap, a.amap_mask, table_key(a, cl, tidx));
        if (slot < 0) {
          set_error(a.err, ERRF_TABLE_FULL);
        } else {
          uint64_t ref = idx;
          if (a.vbits) {
            ref = 0;
#pragma unroll
            for (int l = 0; l < NV; ++l)
              if (l <= d) ref |= (uint64_t)v[l] << (l * a.vbits);
          }
          a.amap[2 * slot + 1] = (ref << 4) | (uint64_t)c;
        }
      }
    }
    if (apparent && d >= 2 && !a.pmap) {  // no recorded pairs: a warp looks for each remaining simplex's facet
      m = __ballot_sync(0xffffffffu, rem && !app);
      while (m) {
        const int L = __ffs(m) - 1;
        m &= m - 1;
        const CV cb = cloud_view(a, __shfl_sync(0xffffffffu, cl, L));
        int w[MAX_DIM + 2];
#pragma unroll
        for (int l = 0; l < NV; ++l) w[l] = l <= d ? __shfl_sync(0xffffffffu, v[l], L) : 0;
        uint32_t minus[MAX_DIM + 2];
        ranks_minus_one(cb, w, d, minus);
        const bool f = zero_apparent_facet(cb, w, d, __shfl_sync(0xffffffffu, r, L), minus, lane) >= 0;
        if (lane == L) fac = f;
      }
    }
    const bool col = rem && !app && !fac;
    const unsigned mc = __ballot_sync(0xffffffffu, app), mf = __ballot_sync(0xffffffffu, fac && !app),
                   ml = __ballot_sync(0xffffffffu, clr), mk = __ballot_sync(0xffffffffu, col);
    const uint32_t c0 = __shfl_sync(0xffffffffu, cl, __ffs(am) - 1);
    if (__all_sync(0xffffffffu, !act || cl == c0)) {
      if (c0 != cur_cloud) flush(c0);
      n_cof += __popc(mc);
      n_fac += __popc(mf);
      n_clr += __popc(ml);
    } else if (app || fac || clr) {  // clouds meet within the warp's simplices
      atomicAdd(st + (size_t)cl * st_stride + (app ? 4 : clr ? 6 : 5), 1ull);
    }
    if (mk) {
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(ncols, (uint32_t)__popc(mk));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (col) {
        const uint32_t pos = base + __popc(mk & ((1u << lane) - 1u));
        if (pos < col_cap) {
          const int hb = a.rank_bits + a.col_bits;
          col_keys[pos] = (hb >= 64 ? 0ull : ((uint64_t)cl << hb)) | ((uint64_t)(a.rank_max - r) << a.col_bits) | idx;
        } else {
          set_error(a.err, ERRF_OUT_OVERFLOW);
        }
      }
    }
  }
  flush(0xFFFFFFFFu);
}

// ====================================================================== reduction

namespace {

__device__ __forceinline__ void column_simplex(const DimArgs& a, const RedState& s, uint32_t j, uint64_t* idx,
                                               uint32_t* rank, uint32_t* cloud) {
  const uint64_t key = s.col_keys[j];
  *idx = key & low_mask(a.col_bits);
  *rank = a.rank_max - (uint32_t)((key >> a.col_bits) & low_mask(a.rank_bits));
  *cloud = high_part(key, a.rank_bits + a.col_bits);
}


// Minimum over the cofacet entries of sum_{(s,c) in V} c * delta(s) restricted to
// row keys > after: returns the key (IDX_NONE if none) and the summed
// coefficient at that key (mod p).  Warp-cooperative.
__device__ void min_entry(const DimArgs& a, const CV& cv, const Binom& B, int lane, const uint64_t* vidx,
                          const uint32_t* vrank,
                          const uint32_t* vcoef, uint32_t vlen, uint64_t self_idx, uint32_t self_rank,
                          uint64_t after, bool has_after, uint64_t* out_key, uint32_t* out_coef) {
  const int d = a.d;
  uint64_t best = IDX_NONE;
  uint32_t sum = 0;
  const uint32_t cnt = vlen ? vlen : 1;
  for (uint32_t e = 0; e < cnt; ++e) {
    const uint64_t sidx = vlen ? vidx[e] : self_idx;
    const uint32_t sr = vlen ? vrank[e] : self_rank;
    const uint32_t sc = vlen ? vcoef[e] : 1u;
    int v[MAX_DIM + 2];
    decode(B, cv.n, sidx, d, v);
    CofacetSums cs;
    cofacet_sums(B, v, d, cs);
    const int av = v[min_degree_vertex(cv, v, d + 1)];
    const uint32_t beg = cv.off[av], end = cv.off[av + 1];
    for (uint32_t q = beg + lane; q < end; q += 32) {
      const int j = (int)cv.nbr[q];
      uint32_t r;
      uint64_t tidx;
      int c;
      if (!cofacet_of(cv, B, v, d, sr, cs, j, &r, &tidx, &c)) continue;
      const uint64_t key = row_key(a, r, tidx);
      if (has_after && key <= after) continue;
      // paper's orientation: (-1)^k with k = #vertices below j minus one = d - c
      const uint32_t sgn = ((d - c) & 1) ? a.p - 1 : 1u;
      const uint32_t cf = (uint32_t)(((uint64_t)sgn * sc) % a.p);
      if (key < best) {
        best = key;
        sum = cf;
      } else if (key == best) {
        sum = (sum + cf) % a.p;
      }
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    uint64_t ob = __shfl_xor_sync(0xffffffffu, best, o);
    uint32_t os = __shfl_xor_sync(0xffffffffu, sum, o);
    if (ob < best) {
      best = ob;
      sum = os;
    } else if (ob == best) {
      sum = (sum + os) % a.p;
    }
  }
  *out_key = best;
  *out_coef = best == IDX_NONE ? 0 : sum;
}

// Apparent facet of the pivot row tau (a (d+1)-simplex): returns the facet's
// reference (IDX_NONE if none; packed vertices when the pair map holds them,
// see DimArgs::vbits, else its index), its rank and the coefficient of tau in
// its coboundary.
__device__ uint64_t pivot_apparent_facet(const DimArgs& a, const CV& cv, const Binom& B, int lane, uint32_t cl,
                                         uint64_t key, uint32_t* frank, uint32_t* tcoef) {
  const int k = a.d + 1;
  if (a.amap) {  // recorded by this dimension's test kernel
    uint64_t v;
    if (!pair_find(a.amap, a.amap_mask, table_key(a, cl, row_key_idx(a, key)), &v)) return IDX_NONE;
    *frank = row_key_rank(a, key);
    *tcoef = ((a.d - (int)(v & 15)) & 1) ? a.p - 1 : 1u;
    return v >> 4;
  }
  const uint64_t tidx = row_key_idx(a, key);
  const uint32_t tr = row_key_rank(a, key);
  int w[MAX_DIM + 2];
  decode(B, cv.n, tidx, k, w);
  uint32_t minus[MAX_DIM + 2];
  ranks_minus_one(cv, w, k, minus);
  int l = zero_apparent_facet(cv, w, k, tr, minus, lane);
  if (l < 0) return IDX_NONE;
  // facet index: drop w[l]; vertices above it keep C(w, k+1-pos) -> C(w, k-pos)
  uint64_t fidx = 0;
  int pos = 0;
  for (int x = 0; x <= k; ++x) {
    if (x == l) continue;
    fidx += B(w[x], k - pos);
    ++pos;
  }
  *frank = tr;
  // in the coboundary of the facet, tau = facet + w[l] with c = l vertices above
  const int c = l;
  *tcoef = ((a.d - c) & 1) ? a.p - 1 : 1u;
  return fidx;
}

// Owner of the pivot row `key` of a column of cloud cl: the zero apparent facet
// of the row (Section 4, "Persistence pairs": apparent pairs are not in the
// table; its reference as pivot_apparent_facet gives it), else the table's
// owner (0xFFFFFFFF: none).  With the recorded pair
// map the two lookups run at once on lanes 0 and 1.  Warp-cooperative; every
// lane gets the results.
__device__ __forceinline__ uint64_t pivot_owner(const DimArgs& a, const RedState& s, const CV& cv, const Binom& B,
                                                int lane, uint32_t cl, uint64_t key, uint32_t* frank, uint32_t* tcoef,
                                                uint32_t* owner) {
  const uint64_t tkey = table_key(a, cl, row_key_idx(a, key));
  if (a.opts & RIPS_OPT_NO_APPARENT) {  // apparent pairs are ordinary columns: the table owns every pivot
    const int64_t slot = table_find(s.t_keys, s.t_mask, tkey);
    *owner = slot >= 0 ? s.t_vals[slot] : 0xFFFFFFFFu;
    return IDX_NONE;
  }
  if (a.amap) {
    // lane 0 probes the pair map, lane 1 the pivot table, with the same load
    // instructions, so the two lookups take the time of one
    // (each probe loads the slot's value with its key)
    uint64_t val = 0;
    int found = 0;
    if (lane < 2) {
      const uint64_t mask = lane == 0 ? a.amap_mask : s.t_mask;
      uint64_t h = mix(tkey) & mask;
      for (uint64_t probe = 0; probe <= mask; ++probe) {
        uint64_t cur, cv2;
        if (lane == 0) {
          const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(a.amap + 2 * h);
          cur = e.x;
          cv2 = e.y;
        } else {
          cur = s.t_keys[h];
          cv2 = s.t_vals[h];
        }
        if (cur == tkey) {
          found = 1;
          val = cv2;
          break;
        }
        if (cur == IDX_NONE) break;
        h = (h + 1) & mask;
      }
    }
    const int ffound = __shfl_sync(0xffffffffu, found, 0);
    const uint64_t v = __shfl_sync(0xffffffffu, val, 0);
    const int tfound = __shfl_sync(0xffffffffu, found, 1);
    const uint64_t tv = __shfl_sync(0xffffffffu, val, 1);
    *owner = tfound ? (uint32_t)tv : 0xFFFFFFFFu;
    if (!ffound) return IDX_NONE;
    *frank = row_key_rank(a, key);
    *tcoef = ((a.d - (int)(v & 15)) & 1) ? a.p - 1 : 1u;
    return v >> 4;
  }
  const uint64_t fidx = pivot_apparent_facet(a, cv, B, lane, cl, key, frank, tcoef);
  *owner = 0xFFFFFFFFu;
  if (fidx == IDX_NONE) {
    const int64_t slot = table_find(s.t_keys, s.t_mask, tkey);
    *owner = slot >= 0 ? s.t_vals[slot] : 0xFFFFFFFFu;
  }
  return fidx;
}

// ---------------------------------------------------------------- working columns
// A column that has to be reduced keeps R_j = D V_j materialised in the R arena,
// sorted by row key (oldest row first) with nonzero coefficients: the GPU form of
// the paper's working coboundary (Section 4, "Pivot extraction").  Columns that
// never get reduced (apparent, emergent) never build theirs; the coboundary of an
// unreduced owner or of an apparent facet is generated on the fly into a per-warp
// scratch slice and sorted there.

// all cofacets of the d-simplex (idx, rank) with their paper-orientation signs,
// unsorted, into buf; returns the count (warp-uniform).  idx is a reference as
// simplex_vertices takes it.
__device__ uint32_t gen_coboundary(const DimArgs& a, const CV& cv, const Binom& B, int lane, uint64_t idx,
                                   bool packed, uint32_t rank, uint32_t scale, uint64_t* bkey, uint32_t* bcoef,
                                   uint32_t cap) {
  const int d = a.d;
  const unsigned lt = (1u << lane) - 1u;
  int v[MAX_DIM + 2];
  simplex_vertices(B, cv.n, idx, packed, a.vbits, d, v);
  CofacetSums cs;
  cofacet_sums(B, v, d, cs);
  const int av = v[min_degree_vertex(cv, v, d + 1)];
  const uint32_t beg = cv.off[av], end = cv.off[av + 1];
  uint32_t cnt = 0;
  for (uint32_t q0 = beg; q0 < end; q0 += 32) {
    const uint32_t q = q0 + lane;
    uint32_t r = 0;
    uint64_t tidx = 0;
    int c = 0;
    const bool ok = q < end && cofacet_of(cv, B, v, d, rank, cs, (int)cv.nbr[q], &r, &tidx, &c);
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    if (ok) {
      const uint32_t pos = cnt + __popc(m & lt);
      if (pos < cap) {
        const uint32_t sgn = ((d - c) & 1) ? a.p - 1 : 1u;
        bkey[pos] = row_key(a, r, tidx);
        bcoef[pos] = (uint32_t)(((uint64_t)sgn * scale) % a.p);
      }
    }
    cnt += __popc(m);
  }
  if (cnt > cap) set_error(a.err, ERRF_INTERNAL);
  return cnt < cap ? cnt : cap;
}

// ascending bitonic sort of (key, coef) pairs in a buffer of at least
// next_pow2(n) entries; the padding takes key ~0 (never a row key)
__device__ void warp_sort_pairs(uint64_t* key, uint32_t* coef, uint32_t n, int lane) {
  uint32_t p2 = 1;
  while (p2 < n) p2 <<= 1;
  for (uint32_t i = n + lane; i < p2; i += 32) {
    key[i] = ~0ull;
    coef[i] = 0;
  }
  __syncwarp();
  for (uint32_t k = 2; k <= p2; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t i = lane; i < p2; i += 32) {
        const uint32_t l = i ^ j;
        if (l > i) {
          const uint64_t ki = key[i], kl = key[l];
          const bool up = (i & k) == 0;
          if ((ki > kl) == up) {
            key[i] = kl;
            key[l] = ki;
            const uint32_t t = coef[i];
            coef[i] = coef[l];
            coef[l] = t;
          }
        }
      }
      __syncwarp();
    }
  }
}

// ---------------------------------------------------------------- lazy working column
// During a chain of additions the working column is a sum of sorted runs, one
// per lane (at most 32), each with its own Z/p scale: R_j's own entries and the
// columns added to it.  Adding a column appends a run (no copy of R_j); the
// pivot is the smallest head key whose combined coefficient is nonzero, found by
// warp reductions, and the heads at a key whose coefficients cancel move on:
// the paper's lazily evaluated working coboundary (Section 4, "Pivot
// extraction"), with sorted runs in place of its heap.  Runs are merged size-
// tiered: when four runs (eight short ones) fall in the same size class
// (sizes within a factor of four), they become one, so an entry is merged a
// logarithmic number of times however long the chain; at the end of a chain
// the column is merged into one run, which later columns add.
//
// Each run keeps the RUN_AHEAD entries after its head (key and stored
// coefficient) in registers, loaded that many steps before they are needed.
constexpr int RUN_AHEAD = 1;

struct Run {
  const uint64_t* key;
  const uint32_t* coef;
  uint32_t len, cur, scale;
  uint64_t hk;             // head key, ~0 once the run is used up
  uint32_t hc;             // head coefficient times scale, mod p (1 over Z/2)
  uint64_t nk[RUN_AHEAD];  // the keys after the head (~0 past the end)
  uint32_t nc[RUN_AHEAD];  // and their stored coefficients (not loaded over Z/2)
};

// c * scale mod p; both below p < 2^16, so the product fits in 32 bits
__device__ __forceinline__ uint32_t scaled(uint32_t c, uint32_t scale, uint32_t p) {
  return p == 2 ? 1u : (c * scale) % p;
}

// head and look-ahead from the cursor on
__device__ __forceinline__ void run_head(Run& r, uint32_t p) {
  r.hk = r.cur < r.len ? r.key[r.cur] : ~0ull;
  r.hc = r.cur < r.len ? scaled(p == 2 ? 1u : r.coef[r.cur], r.scale, p) : 0u;
#pragma unroll
  for (int i = 0; i < RUN_AHEAD; ++i) {
    const bool in = r.cur + 1 + i < r.len;
    r.nk[i] = in ? r.key[r.cur + 1 + i] : ~0ull;
    r.nc[i] = in && p != 2 ? r.coef[r.cur + 1 + i] : 1u;
  }
}

// move to the next entry, loaded ahead; the entry RUN_AHEAD past it is requested now
__device__ __forceinline__ void run_next(Run& r, uint32_t p) {
  ++r.cur;
  r.hk = r.nk[0];
  r.hc = r.cur < r.len ? scaled(r.nc[0], r.scale, p) : 0u;
#pragma unroll
  for (int i = 0; i + 1 < RUN_AHEAD; ++i) {
    r.nk[i] = r.nk[i + 1];
    r.nc[i] = r.nc[i + 1];
  }
  const bool in = r.cur + RUN_AHEAD < r.len;
  r.nk[RUN_AHEAD - 1] = in ? r.key[r.cur + RUN_AHEAD] : ~0ull;
  r.nc[RUN_AHEAD - 1] = in && p != 2 ? r.coef[r.cur + RUN_AHEAD] : 1u;
}

__device__ __forceinline__ Run empty_run() {
  Run r;
  r.key = nullptr;
  r.coef = nullptr;
  r.len = r.cur = 0;
  r.scale = 1;
  r.hk = ~0ull;
  r.hc = 0;
#pragma unroll
  for (int i = 0; i < RUN_AHEAD; ++i) {
    r.nk[i] = ~0ull;
    r.nc[i] = 1u;
  }
  return r;
}

// A run over n arena entries.  When the block has the first entries in shared
// memory (sk, sc: the same keys and coefficients), the head and look-ahead are
// taken from there instead of waiting for the arena.
__device__ __forceinline__ Run make_run(const uint64_t* k, const uint32_t* c, uint32_t n, uint32_t scale,
                                        uint32_t p, const uint64_t* sk = nullptr, const uint32_t* sc = nullptr) {
  Run r = empty_run();
  r.key = k;
  r.coef = c;
  r.len = n;
  r.scale = scale;
  if (sk) {
    r.hk = n ? sk[0] : ~0ull;
    r.hc = n ? scaled(sc[0], scale, p) : 0u;
#pragma unroll
    for (int i = 0; i < RUN_AHEAD; ++i) {
      const bool in = 1u + i < n;
      r.nk[i] = in ? sk[1 + i] : ~0ull;
      r.nc[i] = in ? sc[1 + i] : 1u;
    }
  } else {
    run_head(r, p);
  }
  return r;
}

// run_next on the lanes where `at` holds, without a divergent branch: every
// lane computes its next state (its loads stay inside its run) and keeps it or not
__device__ __forceinline__ void advance_if(Run& r, bool at, uint32_t p) {
  Run t = r;
  run_next(t, p);
  if (at) r = t;
}

// combined coefficient of the lanes at the current minimum (`at`)
__device__ __forceinline__ uint32_t warp_coef_sum(bool at, uint32_t hc, uint32_t p) {
  if (p == 2) return __popc(__ballot_sync(0xffffffffu, at)) & 1u;
  return __reduce_add_sync(0xffffffffu, at ? hc : 0u) % p;
}

// size class of the run's remaining entries (-1 when used up)
__device__ __forceinline__ int run_tier(const Run& r) {
  const uint32_t n = r.len - r.cur;
  return n ? (31 - __clz(n)) >> 1 : -1;
}

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t x) {
  const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32));
  const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32) == hi ? (uint32_t)x : 0xffffffffu);
  return ((uint64_t)hi << 32) | lo;
}

// arena allocation by lane 0, broadcast; false when the arena is full
__device__ __forceinline__ bool arena_alloc(const RedState& s, int lane, unsigned long long count,
                                            unsigned long long* off) {
  unsigned long long o = 0;
  if (lane == 0) o = atomicAdd(s.r_top, count);
  o = __shfl_sync(0xffffffffu, o, 0);
  *off = o;
  return o + count <= s.r_cap;
}

// per-warp shared-memory tile for sorting generated coboundaries
constexpr uint32_t SORT_TILE = 256;
struct SortTile {
  uint64_t* key;
  uint32_t* coef;
};

// coboundary of the d-simplex (idx, rank), generated, sorted (in the warp's
// shared-memory tile when it fits) and stored in the arena
__device__ bool gen_sorted(const DimArgs& a, const RedState& s, const CV& cv, const Binom& B, int lane,
                           const SortTile& tile, uint64_t idx, bool packed, uint32_t rank, const uint64_t** k,
                           const uint32_t** c, uint32_t* n) {
  unsigned long long off;
  if (s.scr_slice <= SORT_TILE) {
    const uint32_t cnt = gen_coboundary(a, cv, B, lane, idx, packed, rank, 1u, tile.key, tile.coef, SORT_TILE);
    __syncwarp();
    warp_sort_pairs(tile.key, tile.coef, cnt, lane);
    if (!arena_alloc(s, lane, cnt ? cnt : 1, &off)) return false;
    for (uint32_t i = lane; i < cnt; i += 32) {
      s.r_key[off + i] = tile.key[i];
      s.r_coef[off + i] = tile.coef[i];
    }
    __syncwarp();
    *k = s.r_key + off;
    *c = s.r_coef + off;
    *n = cnt;
    return true;
  }
  if (!arena_alloc(s, lane, s.scr_slice, &off)) return false;
  uint64_t* kk = s.r_key + off;
  uint32_t* cc = s.r_coef + off;
  const uint32_t cnt = gen_coboundary(a, cv, B, lane, idx, packed, rank, 1u, kk, cc, s.scr_slice);
  __syncwarp();
  warp_sort_pairs(kk, cc, cnt, lane);
  *k = kk;
  *c = cc;
  *n = cnt;
  return true;
}

// Pivot of the run set: the smallest head key with a nonzero combined
// coefficient.  Heads at a key whose coefficients cancel are advanced.
template <bool Z2>
__device__ __forceinline__ uint64_t runs_pivot(Run& rs, uint32_t p, uint32_t* coef_out) {
  Run r = rs;  // the search works on registers; the chain's copy may live in local memory
  for (;;) {
    const uint64_t m = warp_min_u64(r.hk);
    if (m == ~0ull) {
      rs = r;
      *coef_out = 0;
      return IDX_NONE;
    }
    const bool at = r.hk == m;
    const uint32_t c = warp_coef_sum(at, r.hc, Z2 ? 2u : p);
    if (c) {
      rs = r;
      *coef_out = c;
      return m;
    }
    advance_if(r, at, Z2 ? 2u : p);
  }
}

// move the runs that are not used up to lanes 0 .. nr-1
__device__ void runs_pack(Run& r, int lane, int* nr) {
  const unsigned live = __ballot_sync(0xffffffffu, r.hk != ~0ull);
  const int cnt = __popc(live);
  const int src = lane < cnt ? (int)__fns(live, 0, lane + 1) : lane;
  Run t;
  t.key = (const uint64_t*)__shfl_sync(0xffffffffu, (unsigned long long)r.key, src);
  t.coef = (const uint32_t*)__shfl_sync(0xffffffffu, (unsigned long long)r.coef, src);
  t.len = __shfl_sync(0xffffffffu, r.len, src);
  t.cur = __shfl_sync(0xffffffffu, r.cur, src);
  t.scale = __shfl_sync(0xffffffffu, r.scale, src);
  t.hk = __shfl_sync(0xffffffffu, r.hk, src);
  t.hc = __shfl_sync(0xffffffffu, r.hc, src);
#pragma unroll
  for (int i = 0; i < RUN_AHEAD; ++i) {
    t.nk[i] = __shfl_sync(0xffffffffu, r.nk[i], src);
    t.nc[i] = __shfl_sync(0xffffffffu, r.nc[i], src);
  }
  r = lane < cnt ? t : empty_run();
  *nr = cnt;
}

// Runs to merge now: a size class holding MERGE_GROUP runs (MERGE_GROUP_SHORT
// for the classes of runs shorter than 4^(SHORT_TIERS), where a merge costs
// more than the entries it saves), or, when all 32 lanes are taken, the size
// class holding the most runs (the shortest of those); 0 when none.
constexpr int MERGE_GROUP = 4;
constexpr int MERGE_GROUP_SHORT = 8;
constexpr int SHORT_TIERS = 4;  // runs of fewer than 256 entries

__device__ unsigned runs_merge_mask(const Run& r, int lane, int nr) {
  const int t = lane < nr ? run_tier(r) : -1;
  const unsigned grp = __match_any_sync(0xffffffffu, t >= 0 ? t : -2 - lane);
  const unsigned elig =
      __ballot_sync(0xffffffffu, t >= 0 && __popc(grp) >= (t < SHORT_TIERS ? MERGE_GROUP_SHORT : MERGE_GROUP));
  if (elig) return __shfl_sync(0xffffffffu, grp, __ffs(elig) - 1);
  if (nr == 32) {
    const unsigned score = t >= 0 ? ((unsigned)__popc(grp) << 8) | (255u - (unsigned)t) : 0u;
    const unsigned best = __reduce_max_sync(0xffffffffu, score);
    return __shfl_sync(0xffffffffu, grp, __ffs(__ballot_sync(0xffffffffu, score == best)) - 1);
  }
  return 0;
}

// Merges the runs of the lanes in `mask` (from their cursors) into one run in
// the arena, scale 1, held by the lowest of those lanes; the others are used
// up.  One merged entry per step of the warp.  False when the arena is full.
__device__ bool runs_merge_warp(const RedState& s, Run& r, int lane, uint32_t p, unsigned mask) {
  const bool in = (mask >> lane) & 1u;
  const uint32_t rest = __reduce_add_sync(0xffffffffu, in ? r.len - r.cur : 0u);
  unsigned long long off;
  if (!arena_alloc(s, lane, rest ? rest : 1, &off)) return false;
  uint64_t* ok = s.r_key + off;
  uint32_t* oc = s.r_coef + off;
  uint32_t out = 0;
  for (;;) {
    const uint64_t h = in ? r.hk : ~0ull;
    const uint64_t m = warp_min_u64(h);
    if (m == ~0ull) break;
    const bool at = h == m;
    const uint32_t c = warp_coef_sum(at, r.hc, p);
    advance_if(r, at, p);
    if (c) {
      if (lane == 0) {
        ok[out] = m;
        oc[out] = c;
      }
      ++out;
    }
  }
  __syncwarp();
  if (lane == 0) atomicAdd(s.compacted, (unsigned long long)rest);
  if (lane == __ffs(mask) - 1) r = make_run(ok, oc, out, 1, p);
  else if (in) r = empty_run();
  return true;
}

// State of column j's chain of additions, held by the warp that runs it.
struct Chain {
  Run r;          // this lane's run
  int nr;         // lanes in use
  uint32_t step;  // additions so far
  uint64_t key;   // current pivot, IDX_NONE once the column is zero
  uint32_t coef;
  int64_t owner;  // table owner of the pivot, or -1 to look it up
  bool started;   // R_j's own run is in place
  unsigned long long t0;  // globaltimer when the chain passed 255 additions
};

enum : int { CH_DONE = 0, CH_MERGE = 1, CH_ARENA = 2, CH_LONG = 3, CH_INTERNAL = 4, CH_GEN = 5, CH_GEN_SELF = 6,
             CH_HEAVY = 7 };

// work handed from warp 0 to its block: runs to merge, or a coboundary to generate
struct ChainReq {
  unsigned mask;  // CH_MERGE: lanes of the runs
  uint64_t gidx;  // CH_GEN, CH_GEN_SELF: the simplex (a reference as simplex_vertices takes it)
  uint32_t grank;
  bool gpacked;
};

// R_j <- R_j - lambda C, lambda = pivot coefficient ratio (Algorithm 1): the run
// of C joins the set, then the new pivot is found
__device__ __forceinline__ void chain_add(const DimArgs& a, const RedState& s, Chain& ch, int lane,
                                          const uint64_t* wk, const uint32_t* wc, uint32_t wn, uint32_t wcoef,
                                          const uint64_t* sk = nullptr, const uint32_t* sc = nullptr) {
  const uint32_t lam = (uint32_t)(((uint64_t)ch.coef * mod_inv(wcoef, a.p)) % a.p);
  if (lane == ch.nr) ch.r = make_run(wk, wc, wn, (a.p - lam) % a.p, a.p, sk, sc);
  ++ch.nr;
  ++ch.step;
  if (lane == 0) {
    atomicAdd(s.added, (unsigned long long)wn);
    if ((ch.step & 15) == 0) atomicAdd(s.heartbeat, 1u);  // progress, for the grid barrier
  }
  ch.key = a.p == 2 ? runs_pivot<true>(ch.r, a.p, &ch.coef) : runs_pivot<false>(ch.r, a.p, &ch.coef);
  ch.owner = -1;
}

// Column j adds the columns owning its pivot until the pivot is free, owned by
// a later column, or the column is zero (Algorithm 1's inner loop with R = D V,
// Sections 3.1 and 3.4).  Owners found in the table are stable while the
// reduce phase runs (an owner is never on the reduce list), so the chain may
// take several steps in one round.  A pivot with a zero apparent facet is owned
// by that facet's column (Section 4, "Persistence pairs").  In warp mode a
// chain longer than `limit` additions, or one needing a merge of more than
// DimArgs::merge_max entries, stops with CH_HEAVY before anything is written back:
// a block then reduces the column from its last stored state (rips_wide.cuh).
__device__ int chain_advance(const DimArgs& a, const RedState& s, const CV& cv, const Binom& B, int lane,
                             const SortTile& tile, uint32_t j, uint64_t jidx, uint32_t jrank, uint32_t cl,
                             uint32_t limit, Chain& ch) {
  for (;;) {
    if (ch.nr == 32) runs_pack(ch.r, lane, &ch.nr);  // every lane taken: drop the used-up runs
    const unsigned mm = runs_merge_mask(ch.r, lane, ch.nr);
    if (mm) {
      if (__reduce_add_sync(0xffffffffu, (mm >> lane) & 1u ? ch.r.len - ch.r.cur : 0u) > a.merge_max)
        return CH_HEAVY;
      if (!runs_merge_warp(s, ch.r, lane, a.p, mm)) return CH_ARENA;
      runs_pack(ch.r, lane, &ch.nr);
      continue;
    }
    if (ch.key == IDX_NONE) return CH_DONE;
    if (ch.step > MAX_PIVOT_PASSES) return CH_LONG;
    if ((ch.step & 255) == 255) {  // the chain's wall-clock bound
      const unsigned long long now = __shfl_sync(0xffffffffu, global_ns(), 0);
      if (ch.t0 == 0) ch.t0 = now;
      else if (now - ch.t0 > s.chain_ns) return CH_LONG;
    }
    // the column owning the current pivot: an apparent facet, or the table's owner
    const uint64_t* wk;
    const uint32_t* wc;
    uint32_t wn, wcoef;
    if (ch.owner < 0) {
      uint32_t frank, tcoef, k;
      const uint64_t fidx = pivot_owner(a, s, cv, B, lane, cl, ch.key, &frank, &tcoef, &k);
      if (fidx == IDX_NONE) {
        if (k >= j) return CH_DONE;             // free, or owned by a later column: claim it next round
        if (ch.step >= limit) return CH_HEAVY;  // long chain: a block takes the column over
        ch.owner = k;
        continue;
      }
      if (ch.step >= limit) return CH_HEAVY;
      if (!gen_sorted(a, s, cv, B, lane, tile, fidx, a.vbits != 0, frank, &wk, &wc, &wn)) return CH_ARENA;
      wcoef = tcoef;
    } else {
      const uint32_t k = (uint32_t)ch.owner;
      // the owner's coefficient, stored run and simplex, read at once
      wcoef = s.piv_coef[k];
      const uint32_t kn = s.r_len[k];
      const unsigned long long ko = s.r_off[k];
      const uint64_t kkey = s.col_keys[k];
      if (kn) {
        if (s.reduced[k] & UNSORTED) return CH_HEAVY;  // a long run, not in key order
        wk = s.r_key + ko;
        wc = s.r_coef + ko;
        wn = kn;
      } else {
        const uint64_t kidx = kkey & low_mask(a.col_bits);
        const uint32_t kr = a.rank_max - (uint32_t)((kkey >> a.col_bits) & low_mask(a.rank_bits));
        if (!gen_sorted(a, s, cv, B, lane, tile, kidx, false, kr, &wk, &wc, &wn)) return CH_ARENA;
      }
    }
    // the working column's own entries, on first use
    if (!ch.started) {
      const uint64_t* jk = nullptr;
      const uint32_t* jc = nullptr;
      uint32_t jn = s.r_len[j];
      if (jn) {
        jk = s.r_key + s.r_off[j];
        jc = s.r_coef + s.r_off[j];
      } else if (!gen_sorted(a, s, cv, B, lane, tile, jidx, false, jrank, &jk, &jc, &jn)) {
        return CH_ARENA;
      }
      if (lane == 0) ch.r = make_run(jk, jc, jn, 1, a.p);
      ch.nr = 1;
      ch.started = true;
    }
    chain_add(a, s, ch, lane, wk, wc, wn, wcoef);
  }
}

// Lanes whose runs must be merged before the column is stored as one run (0:
// it already is one run of scale 1).
__device__ __forceinline__ unsigned chain_store_mask(const Chain& ch, int lane) {
  const unsigned live = __ballot_sync(0xffffffffu, lane < ch.nr && ch.r.hk != ~0ull);
  const unsigned scaled = __ballot_sync(0xffffffffu, lane < ch.nr && ch.r.hk != ~0ull && ch.r.scale != 1);
  return (__popc(live) > 1 || scaled) ? live : 0u;
}

// Results of a finished chain: statistics, R_j (lane 0's run after
// chain_store_mask came back 0) when the column changed and is not zero, the
// pivot, and the claim list.
__device__ void chain_finish(const RedState& s, const Chain& ch, int lane, uint32_t j, uint32_t* claim_count) {
  Run r = ch.r;
  const uint32_t src = __ffs(__ballot_sync(0xffffffffu, lane < ch.nr && r.hk != ~0ull)) - 1;
  const unsigned long long off = __shfl_sync(0xffffffffu, (unsigned long long)(r.key + r.cur), src & 31);
  const uint32_t len = __shfl_sync(0xffffffffu, r.len - r.cur, src & 31);
  if (lane != 0) return;
  if (ch.step) {
    s.reduced[j] |= 1;
    atomicAdd(s.steps, (unsigned long long)ch.step);
    atomicMax(s.max_chain, ch.step);
    if (ch.key != IDX_NONE) {
      s.r_off[j] = (unsigned long long)((const uint64_t*)off - s.r_key);
      s.r_len[j] = len;
    }
  }
  s.piv_key[j] = ch.key;
  s.piv_coef[j] = ch.coef;
  if (ch.key != IDX_NONE) s.claim_list[atomicAdd(claim_count, 1u)] = j;
}

// warp mode: run the chain to its end and store the column
__device__ int chain_warp(const DimArgs& a, const RedState& s, const CV& cv, const Binom& B, int lane,
                          const SortTile& tile, uint32_t j, uint64_t jidx, uint32_t jrank, uint32_t cl, uint32_t limit,
                          Chain& ch) {
  int st = chain_advance(a, s, cv, B, lane, tile, j, jidx, jrank, cl, limit, ch);
  if (st != CH_DONE) return st;
  if (ch.step && ch.key != IDX_NONE) {
    const unsigned m = chain_store_mask(ch, lane);
    if (m) {
      if (__reduce_add_sync(0xffffffffu, (m >> lane) & 1u ? ch.r.len - ch.r.cur : 0u) > a.merge_max)
        return CH_HEAVY;
      if (!runs_merge_warp(s, ch.r, lane, a.p, m)) return CH_ARENA;
      runs_pack(ch.r, lane, &ch.nr);
    }
  }
  return CH_DONE;
}

// A warp gives a heavy column up before changing any of its state: the column
// is flagged and queued for a block in the next round.
__device__ __forceinline__ void chain_give_up(const RedState& s, int lane, uint32_t j, uint32_t* heavy_count,
                                              uint32_t* heavy_list) {
  if (lane == 0) {
    s.reduced[j] |= HEAVY;
    heavy_list[atomicAdd(heavy_count, 1u)] = j;
  }
}

__device__ __forceinline__ void chain_error(const DimArgs& a, int st) {
  set_error(a.err, st == CH_ARENA ? ERRF_ARENA : st == CH_LONG ? ERRF_TIMEOUT : ERRF_INTERNAL);
}

// First pivot of column j: the cofacets are scanned in decreasing index order and
// the first with the column's own diameter is the pivot (emergent shortcut,
// Section 3.5); only when there is none is the whole coboundary scanned for its
// oldest entry.  A pivot with a zero apparent facet is eliminated at once.  A
// column with a pivot is appended to the claim list.
__device__ void init_column(const DimArgs& a, const RedState& s, const Binom& B, int lane, const SortTile& tile,
                            uint32_t j, uint32_t limit, uint32_t* claim_count, uint32_t* heavy_count,
                            uint32_t* heavy_list) {
  const int d = a.d;
  uint64_t idx;
  uint32_t r, cl;
  column_simplex(a, s, j, &idx, &r, &cl);
  const CV cv = cloud_view(a, cl);
  int v[MAX_DIM + 2];
  decode(B, cv.n, idx, d, v);
  uint32_t rj[MAX_DIM + 2];
  int hl;
  // the first cofacet with the column's own diameter is its pivot; with the
  // emergent shortcut switched off the whole coboundary is scanned instead
  const int jv = (a.opts & RIPS_OPT_NO_EMERGENT) ? -1 : first_equal_cofacet(cv, v, d, r, lane, rj, &hl);
  uint64_t key;
  uint32_t coef;
  if (jv >= 0) {
    CofacetSums cs;
    cofacet_sums(B, v, d, cs);
    int c = 0;
    for (int l = 0; l <= d; ++l) c += v[l] > jv;
    const uint64_t tidx = cs.above[c] + B(jv, d + 2 - c) + cs.below[c];
    key = row_key(a, r, tidx);
    coef = ((d - c) & 1) ? a.p - 1 : 1u;
  } else {
    min_entry(a, cv, B, lane, nullptr, nullptr, nullptr, 0, idx, r, 0, false, &key, &coef);
  }
  if (lane == 0) {
    s.r_len[j] = 0;
    s.reduced[j] = 0;
  }
  __syncwarp();
  // during the first phase the table is empty: only apparent facets can own a pivot
  Chain ch{empty_run(), 0, 0, key, coef, -1, false, 0};
  const int st = chain_warp(a, s, cv, B, lane, tile, j, idx, r, cl, limit, ch);
  if (st == CH_HEAVY) {  // the block will start over from the first pivot
    if (lane == 0) {
      s.piv_key[j] = key;
      s.piv_coef[j] = coef;
    }
    chain_give_up(s, lane, j, heavy_count, heavy_list);
    return;
  }
  if (st != CH_DONE) {
    chain_error(a, st);  // an arena overflow restarts this dimension with a larger arena
    return;
  }
  chain_finish(s, ch, lane, j, claim_count);
}

// Column j claims its pivot: the smallest ordinal owns it; the loser (j, or the
// displaced former owner) goes to the reduce list.
__device__ __forceinline__ void to_reduce(const RedState& s, uint32_t j, uint32_t* reduce_count, uint32_t* heavy_count,
                                          uint32_t* heavy_list) {
  if (s.reduced[j] & HEAVY) heavy_list[atomicAdd(heavy_count, 1u)] = j;
  else s.reduce_list[atomicAdd(reduce_count, 1u)] = j;
}

__device__ void claim_one(const DimArgs& a, const RedState& s, uint32_t j, uint32_t* reduce_count,
                          uint32_t* heavy_count, uint32_t* heavy_list) {
  const uint64_t key = s.piv_key[j];
  const uint32_t cl = high_part(s.col_keys[j], a.rank_bits + a.col_bits);
  const int64_t slot = table_insert(s.t_keys, s.t_mask, table_key(a, cl, row_key_idx(a, key)));
  if (slot < 0) {
    set_error(a.err, ERRF_TABLE_FULL);
    return;
  }
  const uint32_t old = atomicMin(&s.t_vals[slot], j);
  if (old < j) to_reduce(s, j, reduce_count, heavy_count, heavy_list);
  else if (old != 0xFFFFFFFFu && old != j) to_reduce(s, old, reduce_count, heavy_count, heavy_list);
}

// owner of column j's current pivot in the table, which must precede j
__device__ __forceinline__ int64_t reduce_owner(const DimArgs& a, const RedState& s, uint32_t j, uint32_t cl,
                                                uint64_t key) {
  const int64_t slot = table_find(s.t_keys, s.t_mask, table_key(a, cl, row_key_idx(a, key)));
  const uint32_t k = slot >= 0 ? s.t_vals[slot] : 0xFFFFFFFFu;
  return k < j ? (int64_t)k : -1;
}

// Column j (its pivot owned by an earlier column) reduces as far as it can in
// this round, one warp, at most DimArgs::chain_limit additions, and goes back to
// the claim list unless it became zero.
__device__ void reduce_one(const DimArgs& a, const RedState& s, const Binom& B, int lane, const SortTile& tile,
                           uint32_t j, uint32_t* claim_count, uint32_t* heavy_count, uint32_t* heavy_list) {
  uint64_t jidx;
  uint32_t jr, cl;
  column_simplex(a, s, j, &jidx, &jr, &cl);
  const CV cv = cloud_view(a, cl);
  Chain ch{empty_run(), 0, 0, s.piv_key[j], s.piv_coef[j], -1, false, 0};
  ch.owner = reduce_owner(a, s, j, cl, ch.key);
  if (ch.owner < 0) {
    set_error(a.err, ERRF_INTERNAL);
    return;
  }
  const int st = chain_warp(a, s, cv, B, lane, tile, j, jidx, jr, cl, a.chain_limit, ch);
  if (st == CH_HEAVY) {
    chain_give_up(s, lane, j, heavy_count, heavy_list);
    return;
  }
  if (st != CH_DONE) {
    chain_error(a, st);
    return;
  }
  chain_finish(s, ch, lane, j, claim_count);
}

// ---------------------------------------------------------------- blocks and teams
constexpr size_t RED_SMEM_BYTES = (size_t)WARPS_PER_BLOCK * SORT_TILE * 12;  // the warps' sort tiles

// ascending bitonic sort of n2 (a power of two) (key, coef) pairs by the whole block
__device__ void block_bitonic(uint64_t* key, uint32_t* coef, uint32_t n2) {
  for (uint32_t k = 2; k <= n2; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t i = threadIdx.x; i < n2; i += blockDim.x) {
        const uint32_t l = i ^ j;
        if (l > i) {
          const uint64_t ki = key[i], kl = key[l];
          if ((ki > kl) == ((i & k) == 0)) {
            key[i] = kl;
            key[l] = ki;
            const uint32_t t = coef[i];
            coef[i] = coef[l];
            coef[l] = t;
          }
        }
      }
      __syncthreads();
    }
  }
}

}  // namespace

#include "rips_wide.cuh"

namespace {

static_assert(SORT_RUN * 12 <= RED_SMEM_BYTES && WIDE_SAMPLES * 8 <= RED_SMEM_BYTES, "sorts of wide mode fit the tiles");

// Grid-wide barrier for a cooperative launch (all blocks co-resident).  The
// wait is bounded: when limit_ns pass with no block making progress
// (the heartbeat counter, bumped by long chains of additions, stands still) the
// block records ERRF_TIMEOUT and returns false, and the caller leaves the
// kernel.
__device__ bool grid_barrier(unsigned* count, unsigned* gen, const RedState& s, uint32_t* err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    const unsigned g = *(volatile unsigned*)gen;
    __threadfence();
    if (atomicAdd(count, 1u) == gridDim.x - 1) {
      atomicExch(count, 0u);
      __threadfence();
      atomicAdd(gen, 1u);
    } else {
      unsigned long long t0 = global_ns();
      unsigned hb = *(volatile const unsigned*)s.heartbeat;
      while (*(volatile unsigned*)gen == g) {
        __nanosleep(32);
        const unsigned long long now = global_ns();
        if (now - t0 > s.barrier_ns) {
          const unsigned h = *(volatile const unsigned*)s.heartbeat;
          if (h == hb) {
            set_error(err, ERRF_TIMEOUT);
            ok = 0;
            break;
          }
          hb = h;  // another block is still working
          t0 = now;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace

// The whole reduction of one dimension in one cooperative launch: the first
// pivots of all columns, then claim / reduce rounds separated by grid
// barriers, until no column is left to claim or reduce.  The losers of a
// round's claims are reduced in its reduce phase: heavy columns (flagged when a
// warp gave them up) one block each, the others one warp each, both handed out
// by atomic counters; when there are no more columns than blocks, every column
// gets a block, and when there are no more than a quarter as many and one is
// large, a team of blocks.  Once three blocks of four have nothing left to do, the columns
// still running are suspended and each goes on with a team of as many blocks as
// the grid has for it, in as many steps as it takes (wide_advance).  Work-list
// counters are double buffered by round parity (ctl[0..1] claim, ctl[2..3]
// reduce, ctl[16..17] heavy); ctl[4..5] are the barrier's counter and
// generation, ctl[6] receives the number of rounds, ctl[12] is the progress
// heartbeat, ctl[18..19] the light and heavy work cursors; ctl[20..22] count
// the suspended columns (listed from ctl[64] on) and ctl[24..26] the teams done.
__global__ void __launch_bounds__(256, 2) reduce_persistent_kernel(DimArgs a, RedState s, unsigned* ctl) {
  extern __shared__ uint64_t smem[];
  Binom B = stage_binom(a, smem);
  const int lane = threadIdx.x & 31;
  const uint32_t warp_id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t threads = gridDim.x * blockDim.x;
  __shared__ __align__(16) unsigned char red_smem[RED_SMEM_BYTES];
  __shared__ WideState ws, wt;  // this block's own column; the column of its team
  __shared__ WideShared wsh;
  __shared__ uint32_t take;
  uint64_t* const sm = (uint64_t*)red_smem;
  if (threadIdx.x == 0) {  // visible to the block after the first grid barrier
    ws = WideState{};
    for (int q = 0; q < 3; ++q) wide_clear(&wsh.c[q]);
  }
  const uint32_t w = threadIdx.x >> 5;
  const SortTile tile{(uint64_t*)red_smem + w * SORT_TILE,
                      (uint32_t*)(red_smem + (size_t)WARPS_PER_BLOCK * SORT_TILE * 8) + w * SORT_TILE};
  unsigned* claim_cnt = ctl;
  unsigned* red_cnt = ctl + 2;
  unsigned* bar_count = ctl + 4;
  unsigned* bar_gen = ctl + 5;
  unsigned* heavy_cnt = ctl + 16;
  unsigned* light_next = ctl + 18;
  unsigned* heavy_next = ctl + 19;
  unsigned* susp_cnt = ctl + 20;
  unsigned* team_done = ctl + 24;
  unsigned* susp_list = ctl + 64;
  uint32_t* heavy[2] = {s.heavy_list, s.heavy_list + (size_t)s.ncols + 1};
  const uint32_t ncols = s.ncols_dev ? *s.ncols_dev : s.ncols;

  // additions a warp makes on a column in this phase: none when there is a block for every column
  const uint32_t first_limit = ncols <= gridDim.x ? 0u : min(a.chain_limit, FIRST_CHAIN);
  for (uint32_t j = warp_id; j < ncols; j += warps)
    init_column(a, s, B, lane, tile, j, first_limit, &claim_cnt[0], &heavy_cnt[0], heavy[0]);
  if (!grid_barrier(bar_count, bar_gen, s, a.err)) return;
  uint32_t r = 0, it = 0;
  for (;; ++r) {
    const int src = r & 1, dst = src ^ 1;
    const uint32_t nclaim = *(volatile unsigned*)&claim_cnt[src];
    const uint32_t nqueued = *(volatile unsigned*)&heavy_cnt[src];
    // the error word changes under other blocks: thread 0 reads it for the
    // whole block, so its threads leave the loop together
    __shared__ uint32_t errs_seen;
    if (threadIdx.x == 0) errs_seen = *(volatile uint32_t*)a.err;
    __syncthreads();
    const uint32_t errs = errs_seen;
    if ((nclaim == 0 && nqueued == 0) || (errs & (ERRF_ARENA | ERRF_TIMEOUT | ERRF_INTERNAL | ERRF_TABLE_FULL)))
      break;
    for (uint32_t t = tid; t < nclaim; t += threads)
      claim_one(a, s, s.claim_list[t], &red_cnt[src], &heavy_cnt[src], heavy[src]);
    if (tid == 0) {  // the next round's heavy list and this round's cursors start empty
      heavy_cnt[dst] = 0;
      *light_next = 0;
      *heavy_next = 0;
    }
    if (!grid_barrier(bar_count, bar_gen, s, a.err)) return;
    if (tid == 0) {
      claim_cnt[src] = 0;
      red_cnt[dst] = 0;
    }
    const uint32_t nred = *(volatile unsigned*)&red_cnt[src];
    const uint32_t nheavy = *(volatile unsigned*)&heavy_cnt[src];
    const bool few = nred + nheavy <= gridDim.x;  // one block per column
    const uint32_t nwide = few ? nred + nheavy : nheavy;
    const uint32_t nlight = few ? 0u : nred;
    // no more than one column for four blocks, and one of them stored with so many rows that it takes a block long to
    // enter them: a team each from the start
    bool direct = nlight == 0 && 4 * nwide <= gridDim.x;
    if (direct) {
      const uint32_t j = threadIdx.x < nheavy ? heavy[src][threadIdx.x]
                         : threadIdx.x < nwide ? s.reduce_list[threadIdx.x - nheavy] : 0u;
      direct = __syncthreads_or(threadIdx.x < nwide && s.r_len[j] > TEAM_MIN_ROWS);
    }
    if (direct && blockIdx.x < nwide && threadIdx.x == 0) {
      WideCtx* c = s.wide + blockIdx.x;
      const int ph = ws.ph;
      c->st = ws;  // with this block's buffers, if it has any
      c->st.j = blockIdx.x < nheavy ? heavy[src][blockIdx.x] : s.reduce_list[blockIdx.x - nheavy];
      c->st.tmask = 0;  // not begun
      for (int q = 0; q < 3; ++q) wide_clear(&c->sh.c[q]);
      c->sh.bar_count = c->sh.bar_gen = 0;
      susp_list[(it % 3) * gridDim.x + atomicAdd(&susp_cnt[it % 3], 1u)] = blockIdx.x;
      ws = WideState{};
      ws.ph = ph;
    }
    // Columns by blocks (queue), then light ones by warps, then what is suspended by teams.  A heavy column given up by
    // a warp may come with a pivot nobody owns yet; it then ends at once and claims it.
    for (bool queue = !direct;;) {
      if (queue) {
        if (threadIdx.x == 0) take = atomicAdd(heavy_next, 1u);
        __syncthreads();
      }
      const uint32_t qt = queue ? take : ~0u;
      __syncthreads();
      if (qt >= nwide && (queue || direct)) {  // the queue is empty (or was never used)
        queue = direct = false;
        for (;;) {  // a warp each
          uint32_t t = 0;
          if (lane == 0) t = nlight ? atomicAdd(light_next, 1u) : 0u;
          t = __shfl_sync(0xffffffffu, t, 0);
          if (t >= nlight) break;
          reduce_one(a, s, B, lane, tile, s.reduce_list[t], &claim_cnt[dst], &heavy_cnt[dst], heavy[dst]);
        }
        if (!grid_barrier(bar_count, bar_gen, s, a.err)) return;
      }
      uint32_t j = 0, nteam = 0;
      WideCtx* c = s.wide + blockIdx.x;
      WideState& w = queue ? ws : wt;
      Team team{1, 0, &wsh};
      GiveWay gw{heavy_next, light_next, bar_count, nwide, nlight, 3 * gridDim.x, TEAM_MIN_STEPS};
      if (queue) {
        j = qt < nheavy ? heavy[src][qt] : s.reduce_list[qt - nheavy];
        if (threadIdx.x == 0) ws.tmask = 0;  // not begun
      } else {
        nteam = *(volatile unsigned*)&susp_cnt[it % 3];
        if (nteam == 0) break;
        if (tid == 0) {  // read last before the previous barrier, used next after the coming one
          susp_cnt[(it + 2) % 3] = 0;
          team_done[(it + 2) % 3] = 0;
        }
        const uint32_t size = gridDim.x / nteam, q = blockIdx.x / size;
        team.size = 0;  // none for this block
        if (q < nteam) {
          c = s.wide + *(volatile unsigned*)&susp_list[(it % 3) * gridDim.x + q];
          if (threadIdx.x == 0) wt = c->st;
          team = Team{(int)size, (int)(blockIdx.x - q * size), &c->sh};
        }
        const volatile unsigned* done = team_done + it % 3;
        gw = GiveWay{done, done, done, nteam > 1 ? 0u : ~0u, 0u, 3 * nteam, 0u};
      }
      __syncthreads();
      if (team.size) {
        if (!queue) j = wt.j;
        uint64_t jidx, piv;
        uint32_t jr, cl, coef;
        column_simplex(a, s, j, &jidx, &jr, &cl);
        const CV cv = cloud_view(a, cl);
        int st = CH_DONE;
        if (w.tmask == 0) st = wide_begin(a, s, team, w, cv, B, j, cl, jidx, jr);
        if (st == CH_DONE) st = wide_advance(a, s, team, w, cv, B, sm, &piv, &coef, gw);
        if (st == CH_DONE) st = wide_finish(a, s, team, w, sm, piv, coef, !few, &claim_cnt[dst]);
        if (threadIdx.x == 0 && team.rank == 0) {
          if (st == CH_HEAVY) {
            c->st = w;
            const uint32_t to = queue ? it % 3 : (it + 1) % 3;
            susp_list[to * gridDim.x + atomicAdd(&susp_cnt[to], 1u)] = (unsigned)(c - s.wide);
            if (queue) {
              for (int q = 0; q < 3; ++q) wide_clear(&c->sh.c[q]);
              c->sh.bar_count = c->sh.bar_gen = 0;
              const int ph = ws.ph;  // its buffers went with the column
              ws = WideState{};
              ws.ph = ph;
            }
          } else {
            if (!queue) atomicAdd(&team_done[it % 3], 1u);
            if (st != CH_DONE) {
              chain_error(a, st);
            } else if (!queue && ws.tab[0].cap + ws.tab[1].cap == 0) {  // the buffers serve this block's next column
              const int ph = ws.ph;
              ws = wt;
              ws.ph = ph;
            }
          }
        }
        __syncthreads();
      }
      if (!queue) {
        if (!grid_barrier(bar_count, bar_gen, s, a.err)) return;
        ++it;
      }
    }
  }
  if (tid == 0) ctl[6] = r;
}

// bars of this dimension and the statistics
__global__ void readout_kernel(DimArgs a, RedState s, const float* __restrict__ rank_value,
                               rips_bar_t* __restrict__ bars, uint32_t* __restrict__ nbars, uint32_t bar_cap,
                               unsigned long long* __restrict__ stats, int st_stride) {
  const uint32_t ncols = s.ncols_dev ? *s.ncols_dev : s.ncols;
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < ncols; j += gridDim.x * blockDim.x) {
    uint64_t idx;
    uint32_t r, cl;
    column_simplex(a, s, j, &idx, &r, &cl);
    // per-cloud counters: [0] pairs, [1] zero pairs, [2] essential, [3] emergent
    unsigned long long* st = stats + (size_t)cl * st_stride;
    const uint64_t key = s.piv_key[j];
    rips_bar_t b;
    b.dim = a.d;
    b.cloud = (int32_t)cl;
    b.birth = rank_value[r];
    b.birth_simplex = idx;
    if (s.reduced[j] == 0 && key != IDX_NONE) atomicAdd(&st[3], 1ull);
    if (key == IDX_NONE) {
      atomicAdd(&st[2], 1ull);
      b.death = __int_as_float(0x7f800000);
      b.death_simplex = ~0ull;
    } else {
      atomicAdd(&st[0], 1ull);
      const uint32_t tr = row_key_rank(a, key);
      if (tr == r) {
        atomicAdd(&st[1], 1ull);
        continue;
      }
      if (tr > a.rank_max) {  // not a row of this filtration: a broken reduction, not a bar
        set_error(a.err, ERRF_INTERNAL);
        continue;
      }
      b.death = rank_value[tr];
      b.death_simplex = row_key_idx(a, key);
    }
    uint32_t pos = atomicAdd(nbars, 1u);
    if (pos < bar_cap) bars[pos] = b;
  }
}

// ---------------------------------------------------------------- host launchers

static int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess || sms < 1)
      sms = 152;
  }
  return sms;
}

// one warp per item, at most per_sm blocks on every SM (the rest loop)
static int grid_for_warps(uint64_t items, int per_sm) {
  uint64_t blocks = (items + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK;
  const uint64_t cap = (uint64_t)sm_count() * (uint64_t)(per_sm > 0 ? per_sm : 16);
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

static size_t binom_smem(const DimArgs& a) {
  return a.smem_binom ? (size_t)(a.kmax + 1) * (a.bn + 1) * sizeof(uint64_t) : 0;
}

// Opt in to more than 48 KB of shared memory when the kernel's static plus
// dynamic shared memory needs it.  The attributes are queried and set once per
// kernel, device and size, so launches that are being captured into a CUDA
// graph make no such calls.
struct PreparedKernel {
  const void* fn;
  int device;
  size_t smem;
};
static std::mutex g_prep_mu;
static std::vector<PreparedKernel> g_prepared;

template <typename K>
static cudaError_t prepare(K kernel, size_t smem) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> g(g_prep_mu);
  for (const PreparedKernel& pk : g_prepared)
    if (pk.fn == (const void*)kernel && pk.device == dev && pk.smem >= smem) return cudaSuccess;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  if (smem + fa.sharedSizeBytes > 48 * 1024)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) g_prepared.push_back(PreparedKernel{(const void*)kernel, dev, smem});
  return e;
}

cudaError_t launch_enumerate(const DimArgs& a, const uint64_t* pidx, const uint32_t* prank, uint32_t np,
                             int prev_col_bits, uint64_t* out_idx, uint32_t* out_rank, unsigned long long* count,
                             unsigned long long cap, cudaStream_t st) {
  if (np == 0) return cudaSuccess;
  size_t sm = binom_smem(a);
  cudaError_t e = prepare(enumerate_kernel, sm);
  if (e != cudaSuccess) return e;
  enumerate_kernel<<<grid_for_warps(np, a.scan_blocks_per_sm), 256, sm, st>>>(a, pidx, prank, np, prev_col_bits, out_idx, out_rank, count,
                                                        cap);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_edges_to_simplices(const uint64_t* keys, const uint32_t* erank, uint32_t m, int edge_bits,
                                      int col_bits, uint64_t* sidx, uint32_t* srank, cudaStream_t st) {
  if (m == 0) return cudaSuccess;
  edges_to_simplices_kernel<<<(m + 255) / 256, 256, 0, st>>>(keys, erank, m, edge_bits, col_bits, sidx, srank);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_test(const DimArgs& a, const uint64_t* sidx, const uint32_t* srank, uint32_t ns,
                        const uint8_t* cleared_flag, const uint64_t* prev_keys, uint64_t prev_mask,
                        uint64_t* col_keys, uint32_t* ncols, uint32_t col_cap, unsigned long long* stats,
                        int stats_stride, cudaStream_t st) {
  if (ns == 0) return cudaSuccess;
  const int grid = grid_for_warps((ns + 31) / 32, a.scan_blocks_per_sm);
#define TEST(D) \
  test_kernel<D><<<grid, 256, 0, st>>>(a, sidx, srank, ns, cleared_flag, prev_keys, prev_mask, col_keys, ncols, col_cap, \
                                       stats, stats_stride)
  switch (a.d) {
    case 1: TEST(1); break;
    case 2: TEST(2); break;
    case 3: TEST(3); break;
    default: TEST(0);
  }
#undef TEST
  note_launch();
  return cudaGetLastError();
}

size_t wide_ctx_bytes(int blocks) { return (size_t)blocks * sizeof(WideCtx); }

int reduction_blocks(const DimArgs& a, uint32_t ncols) {
  const size_t sm = binom_smem(a);
  if (prepare(reduce_persistent_kernel, sm) != cudaSuccess) return -1;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, reduce_persistent_kernel, 256, sm) != cudaSuccess)
    return -1;
  if (per_sm < 1) return -1;
  // as many blocks as fit, up to one per column: a block takes a column at a time
  uint64_t want = ncols;
  if (a.reduce_blocks_per_sm > 0 && a.reduce_blocks_per_sm < per_sm) per_sm = a.reduce_blocks_per_sm;
  uint64_t maxb = (uint64_t)sms * per_sm;
  if (maxb > (uint64_t)WIDE_MAX_BLOCKS) maxb = WIDE_MAX_BLOCKS;
  int blocks = (int)(want < maxb ? want : maxb);
  return blocks < 1 ? 1 : blocks;
}

cudaError_t launch_reduction(const DimArgs& a, const RedState& s, int blocks, unsigned* ctl, cudaStream_t st) {
  if (s.ncols == 0) return cudaSuccess;
  if (blocks < 1) return cudaErrorInvalidValue;
  const size_t sm = binom_smem(a);
  cudaError_t e = prepare(reduce_persistent_kernel, sm);
  if (e != cudaSuccess) return e;
  DimArgs aa = a;
  RedState ss = s;
  void* args[] = {&aa, &ss, &ctl};
  e = cudaLaunchCooperativeKernel((const void*)reduce_persistent_kernel, dim3(blocks), dim3(256), args, sm, st);
  note_launch();
  return e;
}

cudaError_t launch_readout(const DimArgs& a, const RedState& s, const float* rank_value, rips_bar_t* bars,
                           uint32_t* nbars, uint32_t bar_cap, unsigned long long* stats, int stats_stride,
                           cudaStream_t st) {
  if (s.ncols == 0) return cudaSuccess;
  int blocks = (int)((s.ncols + 255) / 256);
  if (blocks > 152 * 8) blocks = 152 * 8;
  readout_kernel<<<blocks, 256, 0, st>>>(a, s, rank_value, bars, nbars, bar_cap, stats, stats_stride);
  note_launch();
  return cudaGetLastError();
}

}  // namespace rips
