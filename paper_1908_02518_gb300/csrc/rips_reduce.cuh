// The reduction of one dimension (see rips_dim.cu for the whole): one cooperative
// kernel, compiled for each D (columns are D-simplices; 0: any d) in a file of its
// own, rips_reduce_d*.cu.  D fixes the lengths of the loops over a simplex's
// vertices, which then live in registers.
#pragma once
#include "rips_dim.cuh"
#include "rips_wide_types.cuh"

namespace rips {

namespace {

// The coboundary of a d-simplex, walked by a warp along the neighbour list of the
// vertex with the fewest: lanes take U candidates each at a time, whose loads are
// under way together, so a coboundary is a few dependent memory round trips.

template <int D>
struct Coboundary {
  static constexpr int NV = D ? D + 1 : MAX_DIM + 2;
  static constexpr int U = D ? 4 : 1;
  int x[NV];             // vertices, decreasing
  uint64_t sum[NV + 1];  // [c]: of the cofacet's index, all but the new vertex's binomial, with c vertices above it
  int best;
  uint32_t beg, end;

  // ref: the simplex's index, or its packed vertices
  __device__ __forceinline__ void set(const DimArgs& a, const CV& cv, const Binom& B, uint64_t ref, bool packed) {
    const int d = D ? D : a.d;
    if (packed) {
      const uint64_t m = (1ull << a.vbits) - 1;
#pragma unroll
      for (int l = 0; l < NV; ++l)
        if (l <= d) x[l] = (int)((ref >> (l * a.vbits)) & m);
    } else {
      int hi = cv.n - 1;
      uint64_t N = ref;
#pragma unroll
      for (int l = 0; l < NV; ++l)
        if (l <= d) {
          const int k = d + 1 - l;
          x[l] = k == 1 ? (int)N : max_vertex(B, k, hi, N);
          N -= k == 1 ? N : B(x[l], k);
          hi = x[l] - 1;
        }
    }
    uint64_t acc = 0;
#pragma unroll
    for (int l = NV - 1; l >= 0; --l)
      if (l <= d) acc += B(x[l], d + 1 - l);
    sum[0] = acc;
#pragma unroll
    for (int l = 0; l < NV; ++l)
      if (l <= d) sum[l + 1] = sum[l] - B(x[l], d + 1 - l) + B(x[l], d + 2 - l);
    best = 0;
    beg = cv.off[x[0]];
    end = cv.off[x[0] + 1];
#pragma unroll
    for (int l = 1; l < NV; ++l)
      if (l <= d) {
        const uint32_t o0 = cv.off[x[l]], o1 = cv.off[x[l] + 1];
        if (o1 - o0 < end - beg) {
          best = l;
          beg = o0;
          end = o1;
        }
      }
  }

  // the lane's candidates from q0 on: whether each is a cofacet, its row key and the number of vertices above it
  __device__ __forceinline__ void eval(const DimArgs& a, const CV& cv, const Binom& B, uint32_t rank, uint32_t q0,
                                       int lane, bool (&ok)[U], uint64_t (&key)[U], int (&c)[U]) const {
    const int d = D ? D : a.d;
    int j[U];
    uint32_t r[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t q = q0 + u * 32 + lane;
      ok[u] = q < end;
      j[u] = ok[u] ? (int)cv.nbr[q] : x[0];  // a vertex of the simplex is no candidate
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      r[u] = rank;
      c[u] = 0;
#pragma unroll
      for (int l = 0; l < NV; ++l)
        if (l <= d) {
          const uint32_t q = q0 + u * 32 + lane;
          const uint32_t y = cv.nrank && l == best && q < end ? cv.nrank[q] : rank_of(cv, x[l], j[u]);
          ok[u] &= y != RANK_INF;
          r[u] = max(r[u], y);
          c[u] += x[l] > j[u];
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      uint64_t si = sum[0];
#pragma unroll
      for (int l = 1; l <= NV; ++l)
        if (l <= d + 1) si = c[u] == l ? sum[l] : si;
      key[u] = row_key(a, r[u], si + B(j[u], d + 2 - c[u]));
    }
  }
};

// Apparent facet of the pivot row tau (a (d+1)-simplex), for want of a pair map:
// returns the facet's index (IDX_NONE if none), its rank and the coefficient of
// tau in its coboundary.
__device__ uint64_t pivot_apparent_facet(const DimArgs& a, const CV& cv, const Binom& B, int lane, uint64_t key,
                                         uint32_t* frank, uint32_t* tcoef) {
  const int k = a.d + 1;
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
// table; its packed vertices when the pair map holds them, see DimArgs::vbits,
// else its index), else the table's owner (0xFFFFFFFF: none).  With the recorded
// pair map the two lookups run at once on lanes 0 and 1.  Warp-cooperative; every
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
  const uint64_t fidx = pivot_apparent_facet(a, cv, B, lane, key, frank, tcoef);
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
// unsorted, into buf; returns the count (warp-uniform).  idx: as Coboundary::set takes it.
template <int D>
__device__ uint32_t gen_coboundary(const DimArgs& a, const CV& cv, const Binom& B, int lane, uint64_t idx,
                                     bool packed, uint32_t rank, uint64_t* bkey, uint32_t* bcoef, uint32_t cap) {
  const int d = D ? D : a.d;
  const unsigned lt = (1u << lane) - 1u;
  Coboundary<D> cob;
  cob.set(a, cv, B, idx, packed);
  uint32_t cnt = 0;
  for (uint32_t q0 = cob.beg; q0 < cob.end; q0 += 32 * Coboundary<D>::U) {
    bool ok[Coboundary<D>::U];
    uint64_t key[Coboundary<D>::U];
    int c[Coboundary<D>::U];
    cob.eval(a, cv, B, rank, q0, lane, ok, key, c);
#pragma unroll
    for (int u = 0; u < Coboundary<D>::U; ++u) {
      const unsigned m = __ballot_sync(0xffffffffu, ok[u]);
      const uint32_t pos = cnt + __popc(m & lt);
      if (ok[u] && pos < cap) {
        bkey[pos] = key[u];
        bcoef[pos] = ((d - c[u]) & 1) ? a.p - 1 : 1u;
      }
      cnt += __popc(m);
    }
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

// a run over n arena entries
__device__ __forceinline__ Run make_run(const uint64_t* k, const uint32_t* c, uint32_t n, uint32_t scale,
                                        uint32_t p) {
  Run r = empty_run();
  r.key = k;
  r.coef = c;
  r.len = n;
  r.scale = scale;
  run_head(r, p);
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
template <int D>
__device__ bool gen_sorted(const DimArgs& a, const RedState& s, const CV& cv, const Binom& B, int lane,
                           const SortTile& tile, uint64_t idx, bool packed, uint32_t rank, const uint64_t** k,
                           const uint32_t** c, uint32_t* n) {
  unsigned long long off;
  if (s.scr_slice <= SORT_TILE) {
    const uint32_t cnt = gen_coboundary<D>(a, cv, B, lane, idx, packed, rank, tile.key, tile.coef, SORT_TILE);
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
  const uint32_t cnt = gen_coboundary<D>(a, cv, B, lane, idx, packed, rank, kk, cc, s.scr_slice);
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

// how a chain or one of its sections ends; CH_EMPTY: no rows left to look at
enum : int { CH_DONE = 0, CH_EMPTY, CH_ARENA, CH_LONG, CH_HEAVY };

// R_j <- R_j - lambda C, lambda = pivot coefficient ratio (Algorithm 1): the run
// of C joins the set, then the new pivot is found
__device__ __forceinline__ void chain_add(const DimArgs& a, const RedState& s, Chain& ch, int lane,
                                          const uint64_t* wk, const uint32_t* wc, uint32_t wn, uint32_t wcoef) {
  const uint32_t lam = (uint32_t)(((uint64_t)ch.coef * mod_inv(wcoef, a.p)) % a.p);
  if (lane == ch.nr) ch.r = make_run(wk, wc, wn, (a.p - lam) % a.p, a.p);
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
template <int D>
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
      if (!gen_sorted<D>(a, s, cv, B, lane, tile, fidx, a.vbits != 0, frank, &wk, &wc, &wn)) return CH_ARENA;
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
        if (!gen_sorted<D>(a, s, cv, B, lane, tile, kidx, false, kr, &wk, &wc, &wn)) return CH_ARENA;
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
      } else if (!gen_sorted<D>(a, s, cv, B, lane, tile, jidx, false, jrank, &jk, &jc, &jn)) {
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
template <int D>
__device__ int chain_warp(const DimArgs& a, const RedState& s, const CV& cv, const Binom& B, int lane,
                          const SortTile& tile, uint32_t j, uint64_t jidx, uint32_t jrank, uint32_t cl, uint32_t limit,
                          Chain& ch) {
  int st = chain_advance<D>(a, s, cv, B, lane, tile, j, jidx, jrank, cl, limit, ch);
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

// The columns that blocks reduce in a round, and whether one of that round (heavy
// or not) is stored with so many rows that it takes a block long to enter them.
// Said while columns are listed: a block that looked the rows up in the reduce
// phase would race with blocks that store reduced columns.
constexpr uint32_t TEAM_MIN_ROWS = 1024;  // stored rows from which a column starts with a team
struct HeavyList {
  uint32_t *count, *list;
  unsigned* large;
  __device__ __forceinline__ void put(const RedState& s, uint32_t j) const {
    list[atomicAdd(count, 1u)] = j;
    note(s, j);
  }
  __device__ __forceinline__ void note(const RedState& s, uint32_t j) const {
    if (s.r_len[j] > TEAM_MIN_ROWS) *(volatile unsigned*)large = 1u;
  }
};

// A warp gives a heavy column up before changing any of its state: the column
// is flagged and queued for a block in the next round.
__device__ __forceinline__ void chain_give_up(const RedState& s, int lane, uint32_t j, const HeavyList& heavy) {
  if (lane == 0) {
    s.reduced[j] |= HEAVY;
    heavy.put(s, j);
  }
}

__device__ __forceinline__ void chain_error(const DimArgs& a, int st) {
  set_error(a.err, st == CH_ARENA ? ERRF_ARENA : st == CH_LONG ? ERRF_TIMEOUT : ERRF_INTERNAL);
}

// Oldest cofacet of the d-simplex (idx, rank): its row key (IDX_NONE: there is
// none) and coefficient.  The candidates come in decreasing index order, so once
// a tile holds one of the simplex's own diameter, the tile's minimum is the
// oldest (the emergent shortcut, Section 3.5).  Warp-wide.
template <int D>
__device__ uint64_t first_pivot(const DimArgs& a, const CV& cv, const Binom& B, int lane, uint64_t idx, uint32_t rank,
                                uint32_t* coef) {
  const int d = D ? D : a.d;
  const bool emergent = !(a.opts & RIPS_OPT_NO_EMERGENT);
  Coboundary<D> cob;
  cob.set(a, cv, B, idx, false);
  uint64_t best = IDX_NONE;
  int bc = 0;
  for (uint32_t q0 = cob.beg; q0 < cob.end; q0 += 32 * Coboundary<D>::U) {
    bool ok[Coboundary<D>::U];
    uint64_t key[Coboundary<D>::U];
    int c[Coboundary<D>::U];
    cob.eval(a, cv, B, rank, q0, lane, ok, key, c);
#pragma unroll
    for (int u = 0; u < Coboundary<D>::U; ++u)
      if (ok[u] && key[u] < best) {
        best = key[u];
        bc = c[u];
      }
    if (emergent && __any_sync(0xffffffffu, best != IDX_NONE && row_key_rank(a, best) == rank)) break;
  }
  const uint64_t m = warp_min_u64(best);
  bc = __shfl_sync(0xffffffffu, bc, __ffs(__ballot_sync(0xffffffffu, best == m)) - 1);
  *coef = m == IDX_NONE ? 0u : ((d - bc) & 1) ? a.p - 1 : 1u;
  return m;
}

// First pivot of column j; one with a zero apparent facet is eliminated at once,
// by at most `limit` additions of this warp.  A column with a pivot is appended
// to the claim list.
template <int D>
__device__ void init_column(const DimArgs& a, const RedState& s, const Binom& B, int lane, const SortTile& tile,
                            uint32_t j, uint32_t limit, uint32_t* claim_count, const HeavyList& heavy) {
  uint64_t idx;
  uint32_t r, cl, coef;
  column_simplex(a, s, j, &idx, &r, &cl);
  const CV cv = cloud_view(a, cl);
  const uint64_t key = first_pivot<D>(a, cv, B, lane, idx, r, &coef);
  if (lane == 0) {
    s.r_len[j] = 0;
    s.reduced[j] = 0;
  }
  __syncwarp();
  // during the first phase the table is empty: only apparent facets can own a pivot
  Chain ch{empty_run(), 0, 0, key, coef, -1, false, 0};
  const int st = chain_warp<D>(a, s, cv, B, lane, tile, j, idx, r, cl, limit, ch);
  if (st == CH_HEAVY) {  // the block will start over from the first pivot
    if (lane == 0) {
      s.piv_key[j] = key;
      s.piv_coef[j] = coef;
    }
    chain_give_up(s, lane, j, heavy);
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
__device__ __forceinline__ void to_reduce(const RedState& s, uint32_t j, uint32_t* reduce_count,
                                          const HeavyList& heavy) {
  if (s.reduced[j] & HEAVY) {
    heavy.put(s, j);
  } else {
    s.reduce_list[atomicAdd(reduce_count, 1u)] = j;
    heavy.note(s, j);
  }
}

__device__ void claim_one(const DimArgs& a, const RedState& s, uint32_t j, uint32_t* reduce_count,
                          const HeavyList& heavy) {
  const uint64_t key = s.piv_key[j];
  const uint32_t cl = high_part(s.col_keys[j], a.rank_bits + a.col_bits);
  const int64_t slot = table_insert(s.t_keys, s.t_mask, table_key(a, cl, row_key_idx(a, key)));
  if (slot < 0) {
    set_error(a.err, ERRF_TABLE_FULL);
    return;
  }
  const uint32_t old = atomicMin(&s.t_vals[slot], j);
  if (old < j) to_reduce(s, j, reduce_count, heavy);
  else if (old != 0xFFFFFFFFu && old != j) to_reduce(s, old, reduce_count, heavy);
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
template <int D>
__device__ void reduce_one(const DimArgs& a, const RedState& s, const Binom& B, int lane, const SortTile& tile,
                           uint32_t j, uint32_t* claim_count, const HeavyList& heavy) {
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
  const int st = chain_warp<D>(a, s, cv, B, lane, tile, j, jidx, jr, cl, a.chain_limit, ch);
  if (st == CH_HEAVY) {
    chain_give_up(s, lane, j, heavy);
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

// Entry of the list of suspended columns: the context, and whether the column has
// made TEAM_LARGE_STEPS additions.
constexpr unsigned SUSP_LARGE = 0x80000000u;

// The whole reduction of one dimension in one cooperative launch: the first
// pivots of all columns, then claim / reduce rounds separated by grid
// barriers, until no column is left to claim or reduce.  The losers of a
// round's claims are reduced in its reduce phase: heavy columns (flagged when a
// warp gave them up) one block each, the others one warp each, both handed out
// by atomic counters; when there are no more columns than blocks, every column
// gets a block, and when there are no more than half as many and one is large, a
// team of blocks.  Once half of the blocks have nothing left to do, the columns
// still running are suspended and each goes on with a team of as many blocks as
// the grid has for it, in as many steps as it takes (wide_advance).  Work-list
// counters are double buffered by round parity (ctl[0..1] claim, ctl[2..3]
// reduce, ctl[16..17] heavy); ctl[4..5] are the barrier's counter and
// generation, ctl[6] receives the number of rounds, ctl[12] is the progress
// heartbeat, ctl[18..19] the light and heavy work cursors; ctl[20..22] count
// the suspended columns (listed from ctl[64] on) and ctl[24..26] the teams done;
// ctl[28..29] tell, by round parity, of columns stored with many rows (HeavyList).
template <int D>
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
  __shared__ bool lent;  // ws went into this block's context with a column, and is there again after the round
  uint64_t* const sm = (uint64_t*)red_smem;
  if (threadIdx.x == 0) {  // visible to the block after the first grid barrier
    ws = WideState{};
    lent = false;
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
  unsigned* large = ctl + 28;
  unsigned* susp_list = ctl + 64;
  uint32_t* heavy[2] = {s.heavy_list, s.heavy_list + (size_t)s.ncols + 1};
  const auto heavies = [&](int q) { return HeavyList{heavy_cnt + q, heavy[q], large + q}; };
  const uint32_t ncols = s.ncols_dev ? *s.ncols_dev : s.ncols;

  // Additions a warp makes on a column in this phase: a few while its coboundaries fit the warp's tile, else none
  // (sorting them in the arena takes a warp longer than a block needs for the column).
  const bool tiles = s.scr_slice <= SORT_TILE;
  const uint32_t first_limit = tiles ? min(a.chain_limit, FIRST_CHAIN) : 0u;
  for (uint32_t j = warp_id; j < ncols; j += warps)
    init_column<D>(a, s, B, lane, tile, j, first_limit, &claim_cnt[0], heavies(0));
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
    // (a full table is only found by claims, which other blocks may be at: seen after them)
    if ((nclaim == 0 && nqueued == 0) || (errs & (ERRF_ARENA | ERRF_TIMEOUT | ERRF_INTERNAL))) break;
    for (uint32_t t = tid; t < nclaim; t += threads)
      claim_one(a, s, s.claim_list[t], &red_cnt[src], heavies(src));
    if (tid == 0) {  // the next round's heavy list and this round's cursors start empty
      heavy_cnt[dst] = 0;
      large[dst] = 0;
      *light_next = 0;
      *heavy_next = 0;
    }
    if (!grid_barrier(bar_count, bar_gen, s, a.err)) return;
    if (*(volatile uint32_t*)a.err & ERRF_TABLE_FULL) break;
    if (tid == 0) {
      claim_cnt[src] = 0;
      red_cnt[dst] = 0;
    }
    const uint32_t nred = *(volatile unsigned*)&red_cnt[src];
    const uint32_t nheavy = *(volatile unsigned*)&heavy_cnt[src];
    const bool few = !tiles || nred + nheavy <= BLOCK_COLUMNS * gridDim.x;  // blocks take all columns, a few each
    const uint32_t nwide = few ? nred + nheavy : nheavy;
    const uint32_t nlight = few ? 0u : nred;
    if (lent) {  // the buffers of the column that this block gave to a team, with what it added
      const int ph = ws.ph;
      __syncthreads();
      wide_load(&ws, &s.wide[blockIdx.x].st);
      __syncthreads();
      if (threadIdx.x == 0) {
        ws.ph = ph;
        lent = false;
      }
    }
    // no more than one column for two blocks, and one of them stored with so many rows that it takes a block long to
    // enter them: a team each from the start
    bool direct = nlight == 0 && 2 * nwide <= gridDim.x && *(volatile unsigned*)&large[src];
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
      lent = true;
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
          reduce_one<D>(a, s, B, lane, tile, s.reduce_list[t], &claim_cnt[dst], heavies(dst));
        }
        if (!grid_barrier(bar_count, bar_gen, s, a.err)) return;
      }
      uint32_t j = 0, nteam = 0;
      WideCtx* c = s.wide + blockIdx.x;
      WideState& w = queue ? ws : wt;
      Team team{1, 0, &wsh};
      GiveWay gw{heavy_next, light_next, bar_count, nwide, nlight, gridDim.x, TEAM_MIN_STEPS};
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
        // one team left: a grid-wide barrier pays from rounds of thousands of rows on
        uint32_t size = gridDim.x / nteam;
        // (from the list, which stays as it is in this phase: the team's leader writes the column's state)
        const bool small = nteam == 1 && size > TEAM_SMALL &&
                           !(*(volatile unsigned*)&susp_list[(it % 3) * gridDim.x] & SUSP_LARGE);
        if (small) size = TEAM_SMALL;
        const uint32_t q = blockIdx.x / size;
        team.size = 0;  // none for this block
        if (q < nteam) {
          c = s.wide + (*(volatile unsigned*)&susp_list[(it % 3) * gridDim.x + q] & ~SUSP_LARGE);
          wide_load(&wt, &c->st);
          team = Team{(int)size, (int)(blockIdx.x - q * size), &c->sh};
        }
        const volatile unsigned* done = team_done + it % 3;
        gw = small ? GiveWay{done, done, done, 0u, 0u, 0u, TEAM_LARGE_STEPS}
                   : GiveWay{done, done, done, nteam > 1 ? 0u : ~0u, 0u, nteam, 0u};
      }
      __syncthreads();
      if (team.size) {
        if (!queue) j = wt.j;
        uint64_t jidx, piv;
        uint32_t jr, cl, coef;
        column_simplex(a, s, j, &jidx, &jr, &cl);
        const CV cv = cloud_view(a, cl);
        int st = CH_DONE;
        if (w.tmask == 0) st = wide_begin<D>(a, s, team, w, cv, B, j, cl, jidx, jr);
        if (st == CH_DONE) st = wide_advance<D>(a, s, team, w, cv, B, sm, &piv, &coef, gw);
        if (st == CH_DONE) st = wide_finish(a, s, team, w, sm, piv, coef, !few, &claim_cnt[dst]);
        if (threadIdx.x == 0 && team.rank == 0) {
          if (st == CH_HEAVY) {
            c->st = w;
            const uint32_t to = queue ? it % 3 : (it + 1) % 3;
            susp_list[to * gridDim.x + atomicAdd(&susp_cnt[to], 1u)] =
                (unsigned)(c - s.wide) | (w.step >= TEAM_LARGE_STEPS ? SUSP_LARGE : 0u);
            if (queue) {
              for (int q = 0; q < 3; ++q) wide_clear(&c->sh.c[q]);
              c->sh.bar_count = c->sh.bar_gen = 0;
              const int ph = ws.ph;
              ws = WideState{};
              ws.ph = ph;
              lent = true;
            }
          } else {
            if (!queue) atomicAdd(&team_done[it % 3], 1u);
            if (st != CH_DONE) chain_error(a, st);
            else if (!queue) c->st = w;  // the buffers go back to the block that began the column
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

}  // namespace rips
