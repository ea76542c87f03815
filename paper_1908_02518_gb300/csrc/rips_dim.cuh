// Device helpers of one dimension's kernels (rips_dim.cu, rips_reduce.cuh): cloud
// views, simplex indices and vertices, row keys, hash tables.
#pragma once
#include "rips_internal.cuh"

namespace rips {

namespace {

constexpr int WARPS_PER_BLOCK = 8;
constexpr uint32_t MAX_PIVOT_PASSES = 1u << 30;  // additions in one chain before giving up
constexpr uint32_t FIRST_CHAIN = 6;               // additions a warp makes on a column with its first pivot
// Columns a block for which blocks take all columns of a round: a block reduces a short chain in 50 to 100 us, a warp
// needs 30 us an addition (2,048 rotations, 305 columns on 304 blocks: 1.4 ms by warps)
constexpr uint32_t BLOCK_COLUMNS = 4;
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

// pivot-table key of a row: (cloud << row_bits) | local row index
__device__ __forceinline__ uint64_t table_key(const DimArgs& a, uint32_t cloud, uint64_t row_idx) {
  return (a.row_bits >= 64 ? 0ull : ((uint64_t)cloud << a.row_bits)) | row_idx;
}

__device__ __forceinline__ void column_simplex(const DimArgs& a, const RedState& s, uint32_t j, uint64_t* idx,
                                               uint32_t* rank, uint32_t* cloud) {
  const uint64_t key = s.col_keys[j];
  *idx = key & low_mask(a.col_bits);
  *rank = a.rank_max - (uint32_t)((key >> a.col_bits) & low_mask(a.rank_bits));
  *cloud = high_part(key, a.rank_bits + a.col_bits);
}


}  // namespace

}  // namespace rips
