// Wide elimination: the reduction of one column by a team of blocks, many
// additions at a time.  Included by rips_reduce.cuh only.
//
// Algorithm 1 adds one column per pivot, and a column's next owner depends on
// its new pivot, so a chain of additions is sequential and costs a round of
// memory latencies per addition.  But an entry of the working column that has
// an owner (a zero apparent facet, Section 4 "Persistence pairs", or an earlier
// column of the pivot table) can be eliminated before it becomes the pivot:
// adding its owner changes that entry and younger rows only, and the owner
// precedes the column, so R = D V with V unitriangular stays true.  Entries
// older than an eliminated one are never touched.  The pivot is then the
// oldest live entry once that one has no owner, whatever was eliminated beyond
// it, and the pairing of a reduced matrix is unique (Section 3.1): the pairs
// are those of the one-at-a-time order.
//
// The working column is a hash table (row key -> coefficient sum) in the arena;
// an addition is a set of atomic adds in any order.  Rows are visited in
// windows of the filtration order:
//   front  a list of the rows up to `bound`, as table slots with their owner kept
//          beside them,
//   mid    an unordered list of the rows from there up to `mbound`, as keys;
// the rows beyond are in the table only.  A round extends the front from the mid
// list, up to a key sampled so that about K rows join it, looks its rows over,
// writes the live owned ones into a work list, and then adds their owners, one
// warp a row.  The mid list is refilled by a scan of the table.  K grows with the
// additions made so far, so a chain of A additions takes on the order of log2(A)
// rounds and the additions wasted on rows past its pivot are a share of A: a
// third of them and at least 8 for a block, since other columns wait for it; for
// a team as many as made, between 32 and 512, and half as many beyond, since half
// of the chip waits for a team and a round costs it a barrier over blocks more.
// That holds while rows stay eliminated; K is therefore also bound by the rows
// that rounds settle (WIDE_AHEAD).  A window whose rows multiply is cut back to K.
// (K counts rows that have an
// owner: the window is extended by the share of such rows the last time.)  Rows
// behind the window are settled; a table that fills up is rebuilt from its live
// rows.
//
// What bounds it: memory latency.  A section is a handful of dependent round
// trips (a row's slot, value and owner: 5 to 7 us; a coboundary's neighbours,
// ranks and table slots: 5 to 15 us at up to a few rows a warp) and a barrier
// (0.5 us in a block, 4 to 8 us over the grid), whatever the number of rows, so
// the gain is in rows per section.  Reduction before (one addition at a time, 10
// to 25 us each) and after, GB300: 2,048 rotations, chains of 16,240 and 15,062
// additions, 319 -> 15 ms; 4,096 rotations, 580,824 and 78,690 additions, 7,328 ->
// 76 ms; torus of 1,000 points, 730 additions, 11.6 -> 2.2 ms (4 % of the cycles
// issue, warps wait at barriers).
//
// A team is one block (counters in shared memory) or several (counters in the
// column's context in global memory); all its threads run the same code on
// replicated state, separated by team barriers.  A column that outlives the
// others is suspended between two rounds and resumed by a larger team.

namespace {

constexpr uint32_t SORT_RUN = 1024;  // stored runs up to this length are sorted (and usable by a warp)

// owner code of a front row: the pair map's value (low four bits: 0..8), or
constexpr uint64_t OWN_TABLE = 13, OWN_NONE = 14, OWN_UNKNOWN = 15;  // OWN_TABLE | (ordinal << 4)

constexpr uint32_t WIDE_K0 = 8;         // rows of the first window
// Rows of a team's window: as many as additions made, between these, and half as many beyond.  Measured against a third
// of them, at least 8, for teams too: torus of 1,000 points to H2 3.58 -> 2.82 ms, 1,500 points of a Clifford torus
// 4.76 -> 3.77, edge list of 4,999 points 13.8 -> 11.7, 2,048 rotations 18.1 -> 16.1, 24-cloud plan 3.22 -> 2.88,
// 32 clouds 24.9 -> 24.0.  Windows this wide in single blocks cost more than they save while blocks are short (32
// clouds 24.9 -> 25.3 to 28.6, 100 points 0.75 -> 0.80 to 0.85), all additions past 512 too (3-sphere of 144 points
// over Z/3 15.7 -> 16.6).
constexpr uint32_t WIDE_TEAM_K0 = 32, WIDE_TEAM_K1 = 512;
// And at most WIDE_AHEAD times the rows that a round has settled of late (rows older than every live one), or as many
// as bring this many entries a block, whose additions a round's latency hides.  On lengths without geometry rows come
// back as often as they are eliminated and a round settles about one, however wide the window: without this bound it
// grows all the same.  Random lengths, 200 points 220 -> 105 ms (1.37 million additions -> 88,000), 300 points of 40
// bits by Hamming distance 82 -> 38, integers up to 9 on 1,000 points 240 to 390 -> 58; with geometry 0.5 % slower.
// 1,024 for teams: 89 and 31 ms, but 4,999 points of a Clifford torus 6 % slower; 16,384: 134 and 58.
constexpr float WIDE_AHEAD = 4.0f;
constexpr float WIDE_FREE = 1024.0f, WIDE_TEAM_FREE = 4096.0f;
constexpr uint32_t WIDE_SAMPLES = 128;   // keys sampled to place a bound, one a thread
constexpr uint32_t TEAM_MIN_STEPS = 32;  // additions a block makes before it gives its column to a team
constexpr uint32_t TEAM_SMALL = 64;         // blocks of a lone team up to
constexpr uint32_t TEAM_LARGE_STEPS = 4096;  // additions
constexpr uint32_t WIDE_LONGS = 256;     // stored runs added by the whole team in one section

struct Team {
  int size, rank;
  WideShared* g;
};

__device__ __forceinline__ void wide_clear(WideCount* c) {
  c->add[0] = c->add[1] = c->fresh = c->todo = 0;
  c->count = c->nlong = c->stop = c->settled = c->ents = 0;
  c->un = c->ow = ~0ull;
  c->longsum = c->longroom = c->tmp = 0;
}

// a column's state from its context into shared memory, a word a thread
__device__ __forceinline__ void wide_load(WideState* to, const WideState* from) {
  static_assert(sizeof(WideState) % 4 == 0, "words");
  for (uint32_t i = threadIdx.x; i < sizeof(WideState) / 4; i += blockDim.x)
    ((unsigned*)to)[i] = ((const unsigned*)from)[i];
}

// Barrier of the team's blocks; bounded like the grid barrier.
__device__ bool team_sync(const Team& t, const RedState& s) {
  if (t.size == 1) {
    __syncthreads();
    return true;
  }
  __shared__ int tok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned* gen = &t.g->bar_gen;
    const unsigned g0 = *gen;
    __threadfence();
    if (atomicAdd(&t.g->bar_count, 1u) == (unsigned)t.size - 1u) {
      atomicExch(&t.g->bar_count, 0u);
      __threadfence();
      atomicAdd(&t.g->bar_gen, 1u);
    } else {
      unsigned long long t0 = global_ns();
      unsigned hb = *(volatile const unsigned*)s.heartbeat;
      for (unsigned it = 1; *gen == g0; ++it) {
        if (it & 63u) continue;
        const unsigned long long now = global_ns();
        if (now - t0 <= s.barrier_ns) continue;
        const unsigned h = *(volatile const unsigned*)s.heartbeat;
        if (h == hb) {
          set_error(s.err, ERRF_TIMEOUT);
          ok = 0;
          break;
        }
        hb = h;
        t0 = now;
      }
    }
    __threadfence();
    tok = ok;
  }
  __syncthreads();
  return tok != 0;
}

// End of a section: barrier, the section's counts into w.d, list lengths moved on.
__device__ bool wide_sync(const Team& t, const RedState& s, WideState& w) {
  const bool ok = team_sync(t, s);
  if (threadIdx.x < 32) {
    // one lane a word, so that a count in global memory costs one round trip
    static_assert(sizeof(WideCount) % 4 == 0 && sizeof(WideCount) <= 128, "one word a lane");
    volatile unsigned* c = (volatile unsigned*)&t.g->c[w.ph];
    if (threadIdx.x < sizeof(WideCount) / 4) ((unsigned*)&w.d)[threadIdx.x] = c[threadIdx.x];
    __syncwarp();
    if (threadIdx.x == 0) {
      w.n[0] += w.d.add[0];
      w.n[1] += w.d.add[1];
      w.used += w.d.fresh;
      if (t.rank == 0) wide_clear(&t.g->c[(w.ph + 2) % 3]);
      w.ph = (w.ph + 1) % 3;
    }
  }
  __syncthreads();
  return ok;
}

// count arena entries for the team, from a multiple of four on (16-byte loads of
// keys and coefficients): CH_DONE, CH_ARENA when the arena is full, CH_LONG when the
// wait for the team ran out (so for all that allocates below)
__device__ int wide_alloc(const Team& t, const RedState& s, WideState& w, unsigned long long count, WideList* out) {
  if (threadIdx.x == 0 && t.rank == 0) {
    const unsigned long long o = (atomicAdd(s.r_top, count + 3) + 3) & ~3ull;
    *(volatile unsigned long long*)&t.g->c[w.ph].tmp = o + count <= s.r_cap ? o : ~0ull;
  }
  if (!wide_sync(t, s, w)) return CH_LONG;
  if (w.d.tmp == ~0ull) return CH_ARENA;
  *out = WideList{w.d.tmp, count};
  return CH_DONE;
}

// `slot` (a buffer of w that holds nothing) becomes one of at least `need` entries:
// the smallest of the spare ones that will do, or `count` new entries, and the old
// one is kept as a spare.
__device__ int wide_grow(const Team& t, const RedState& s, WideState& w, WideList& slot, unsigned long long need,
                         unsigned long long count) {
  int best = -1, least = 0;
  for (int q = 0; q < WIDE_SPARES; ++q) {
    const unsigned long long cap = w.spare[q].cap;
    if (cap >= need && (best < 0 || cap < w.spare[best].cap)) best = q;
    if (cap < w.spare[least].cap) least = q;
  }
  WideList nl = best >= 0 ? w.spare[best] : WideList{0, 0};
  if (best < 0) {
    if (const int e = wide_alloc(t, s, w, count, &nl)) return e;
    if (slot.cap > w.spare[least].cap) best = least;  // the smallest one is given up
  }
  __syncthreads();  // every thread has read the spares
  if (threadIdx.x == 0) {
    if (best >= 0) w.spare[best] = slot;
    slot = nl;
  }
  __syncthreads();
  return CH_DONE;
}

// ---------------------------------------------------------------- lists and table

// Appends U rows a lane (l: the row's list; L_FAR or -1: none): a key, or for
// the front list its table slot and owner code.  Whole warps call it; a list's
// places are taken with one atomic.
template <int U>
__device__ __forceinline__ void wide_append(const RedState& s, WideCount* c, const WideState& w, int lane,
                                            const int (&l)[U], const uint64_t (&kv)[U], const uint32_t (&slot)[U]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    unsigned m[U];
    unsigned total = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      m[u] = __ballot_sync(0xffffffffu, l[u] == q);
      total += __popc(m[u]);
    }
    if (!total) continue;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&c->add[q], total);
    unsigned long long pos = w.list[q][w.cur[q]].off + w.n[q] + __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (l[u] == q) {
        const unsigned long long at = pos + __popc(m[u] & ((1u << lane) - 1u));
        s.r_key[at] = kv[u];
        if (q == L_FRONT) s.r_coef[at] = slot[u];
      }
      pos += __popc(m[u]);
    }
  }
}

// Slots of U keys a lane (where ok) known to be in the table.
template <int U>
__device__ __forceinline__ void wide_find(const RedState& s, unsigned long long toff, uint64_t mask,
                                          const bool (&ok)[U], const uint64_t (&key)[U], uint64_t (&h)[U]) {
  uint64_t got[U];
  bool open[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    h[u] = mix(key[u]) & mask;
    open[u] = ok[u];
  }
  for (uint64_t probe = 0;; ++probe) {
    bool again = false;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (open[u]) got[u] = __ldcg(s.r_key + toff + h[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (open[u]) {
        open[u] = got[u] != key[u];
        if (open[u]) {
          h[u] = (h[u] + 1) & mask;
          again = true;
        }
      }
    if (!again) return;
    if (probe > mask) {
      set_error(s.err, ERRF_INTERNAL);
      return;
    }
  }
}

__device__ __forceinline__ uint64_t wide_find(const RedState& s, unsigned long long toff, uint64_t mask, uint64_t key) {
  const bool ok[1] = {true};
  const uint64_t k[1] = {key};
  uint64_t h[1];
  wide_find(s, toff, mask, ok, k, h);
  return h[0];
}

// Slots of U keys a lane (where ok), entered if absent (fresh); the caller has
// made room.  A probe of every key is under way at a time.
template <int U>
__device__ __forceinline__ void wide_enter(const RedState& s, unsigned long long toff, uint64_t mask,
                                           const bool (&ok)[U], const uint64_t (&key)[U], uint64_t (&h)[U],
                                           bool (&fresh)[U]) {
  unsigned long long* tk = (unsigned long long*)s.r_key + toff;
  uint64_t old[U];
  bool open[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    h[u] = mix(key[u]) & mask;
    open[u] = ok[u];
    fresh[u] = false;
  }
  for (uint64_t probe = 0;; ++probe) {
    bool again = false;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (open[u]) old[u] = atomicCAS(tk + h[u], IDX_NONE, (unsigned long long)key[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (open[u]) {
        fresh[u] = old[u] == IDX_NONE;
        open[u] = !fresh[u] && old[u] != key[u];
        if (open[u]) {
          h[u] = (h[u] + 1) & mask;
          again = true;
        }
      }
    if (!again) break;
    if (probe > mask) {
      set_error(s.err, ERRF_INTERNAL);
      break;
    }
  }
}

__device__ __forceinline__ uint32_t wide_value(const RedState& s, unsigned long long toff, uint64_t slot, uint32_t p) {
  const uint32_t v = __ldcg(s.r_coef + toff + slot);
  return p == 2 ? v & 1u : v % p;
}

// The table and bounds, copied to registers for a section.
struct WideView {
  unsigned long long toff;
  uint64_t mask, bound, mbound;
  WideCount* c;
};

__device__ __forceinline__ WideView wide_view(const Team& t, const WideState& w) {
  return WideView{w.tab[w.tcur].off, w.tmask, w.bound, w.mbound, &t.g->c[w.ph]};
}

// Adds c (mod p) to row `key` of the working column, U rows a lane (where ok);
// a row seen for the first time joins the list of its key.  Returns how many of
// the lane's rows are new.  Sums of coefficients below p < 2^16 stay below 2^32:
// the add that passes 2^31 takes a multiple of p off again, and no more adds of one
// row are under way at a time than there are warps in the team (an added column
// has a row once, is added by one warp, and the warp waits for its adds): 2,432 of
// less than 2^16 each on 304 blocks.
template <int U>
__device__ __forceinline__ unsigned wide_insert(const RedState& s, const WideState& w, const WideView& v, int lane,
                                                uint32_t p, const bool (&ok)[U], const uint64_t (&key)[U],
                                                const uint32_t (&c)[U]) {
  uint64_t h[U];
  bool fresh[U];
  wide_enter(s, v.toff, v.mask, ok, key, h, fresh);
  uint32_t* tv = s.r_coef + v.toff;
  int l[U];
  uint64_t kv[U];
  uint32_t slot[U];
  unsigned cnt = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (ok[u]) {
      if (p == 2) {
        atomicXor(tv + h[u], 1u);
      } else {
        const uint32_t old = atomicAdd(tv + h[u], c[u]);
        if (old < 0x80000000u && old + c[u] >= 0x80000000u) atomicSub(tv + h[u], (0x80000000u / p) * p);
      }
    }
    l[u] = !fresh[u] ? -1 : key[u] <= v.bound ? L_FRONT : key[u] <= v.mbound ? L_MID : L_FAR;
    kv[u] = l[u] == L_FRONT ? OWN_UNKNOWN : key[u];
    slot[u] = (uint32_t)h[u];
    cnt += fresh[u];
  }
  wide_append(s, v.c, w, lane, l, kv, slot);
  return cnt;
}

// the list's other buffer holds at least `cap` entries
__device__ int wide_alt(const Team& t, const RedState& s, WideState& w, int l, unsigned long long cap) {
  WideList& alt = w.list[l][w.cur[l] ^ 1];
  return alt.cap >= cap ? CH_DONE : wide_grow(t, s, w, alt, cap, cap + cap / 2 + 64);
}

// room for `room` more rows in list l
__device__ int wide_room(const Team& t, const RedState& s, WideState& w, int l, unsigned long long room) {
  const uint32_t n = w.n[l];
  const WideList old = w.list[l][w.cur[l]];
  if (n + room <= old.cap) return CH_DONE;
  if (const int e = wide_alt(t, s, w, l, n + room)) return e;
  const WideList to = w.list[l][w.cur[l] ^ 1];
  if (n) {
    const uint32_t step = (uint32_t)t.size * blockDim.x;
    for (uint32_t i = (uint32_t)t.rank * blockDim.x + threadIdx.x; i < n; i += step) {
      s.r_key[to.off + i] = __ldcg(s.r_key + old.off + i);
      if (l == L_FRONT) s.r_coef[to.off + i] = __ldcg(s.r_coef + old.off + i);
    }
    if (!wide_sync(t, s, w)) return CH_LONG;
  } else {
    __syncthreads();  // every thread has read cur
  }
  if (threadIdx.x == 0) w.cur[l] ^= 1;
  __syncthreads();
  return CH_DONE;
}

// an empty table of `cap` (a power of two >= 1024) slots in the other table buffer
__device__ int wide_table(const Team& t, const RedState& s, WideState& w, unsigned long long cap) {
  if (w.tab[w.tcur ^ 1].cap < cap)
    if (const int e = wide_grow(t, s, w, w.tab[w.tcur ^ 1], cap, cap)) return e;
  const unsigned long long off = w.tab[w.tcur ^ 1].off;
  const unsigned long long step = (unsigned long long)t.size * blockDim.x;
  ulonglong2* tk = (ulonglong2*)(s.r_key + off);
  uint4* tv = (uint4*)(s.r_coef + off);
  const unsigned long long first = (unsigned long long)t.rank * blockDim.x + threadIdx.x;
  for (unsigned long long i = first; i < cap / 2; i += step) tk[i] = make_ulonglong2(IDX_NONE, IDX_NONE);
  for (unsigned long long i = first; i < cap / 4; i += step) tv[i] = make_uint4(0, 0, 0, 0);
  return wide_sync(t, s, w) ? CH_DONE : CH_LONG;
}

__device__ __forceinline__ unsigned long long wide_pow2(unsigned long long x) {
  unsigned long long c = 1024;
  while (c < x) c <<= 1;
  return c;
}

// Calls f(keys, value words) for the table's slots, eight a lane and whole warps
// together.
template <class F>
__device__ __forceinline__ void wide_scan(const Team& t, const RedState& s, unsigned long long off,
                                          unsigned long long cap, F f) {
  const unsigned long long step = (unsigned long long)t.size * blockDim.x * 8;
  const ulonglong2* tk = (const ulonglong2*)(s.r_key + off);
  const uint4* tv = (const uint4*)(s.r_coef + off);
  const uint32_t lane = threadIdx.x & 31;
  const unsigned long long w0 = ((unsigned long long)t.rank * blockDim.x + threadIdx.x - lane) * 8;
  for (unsigned long long b = w0; b < cap; b += step) {  // cap is a multiple of 256, a warp's share of a step
    uint64_t key[8];
    uint32_t val[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const unsigned long long at = b + q * 128 + lane * 4;
      const ulonglong2 k0 = __ldcg(tk + at / 2), k1 = __ldcg(tk + at / 2 + 1);
      const uint4 v = __ldcg(tv + at / 4);
      key[4 * q] = k0.x;
      key[4 * q + 1] = k0.y;
      key[4 * q + 2] = k1.x;
      key[4 * q + 3] = k1.y;
      val[4 * q] = v.x;
      val[4 * q + 1] = v.y;
      val[4 * q + 2] = v.z;
      val[4 * q + 3] = v.w;
    }
    f(key, val);
  }
}

__device__ __forceinline__ bool wide_live(uint32_t v, uint32_t p) { return p == 2 ? (v & 1u) != 0 : v % p != 0; }

// Room for `room` more rows: in both lists, and in the table at half load.  A
// table too full is rebuilt from the rows of the front and the live rows beyond
// it (the mid list drops its dead rows with the table), at a size for as many of
// them as a sample of its slots shows, and again if there are more.
__device__ int wide_ensure(const Team& t, const RedState& s, WideState& w, uint32_t p, unsigned long long room) {
  const int lane = threadIdx.x & 31;
  for (int l = 0; l < 2; ++l)
    if (const int e = wide_room(t, s, w, l, room)) return e;
  // (the second time unless a quarter of that is left free, or the next section would be back here)
  bool rebuilt = false;
  while (2 * (w.used + room) > (rebuilt ? (w.tmask + 1) / 4 * 3 : w.tmask + 1)) {
    unsigned long long need = 4 * (w.used + room);
    if (!rebuilt) {  // live rows among WIDE_SAMPLES slots (every block takes the same ones)
      bool live = false;
      if (threadIdx.x < WIDE_SAMPLES) {
        const unsigned long long at = w.tab[w.tcur].off + threadIdx.x * ((w.tmask + 1) / WIDE_SAMPLES);
        const uint64_t key = __ldcg(s.r_key + at);
        live = key != IDX_NONE && key > w.bound && wide_live(__ldcg(s.r_coef + at), p);
      }
      const unsigned long long seen = (unsigned)__syncthreads_count(live) + 4;
      const unsigned long long kept = min((unsigned long long)w.used, seen * ((w.tmask + 1) / WIDE_SAMPLES) + w.n[L_FRONT]);
      need = max(w.used + room, 3 * (kept + room));  // never less than what could be kept
    }
    const unsigned long long cap = wide_pow2(need);
    if (cap > (1ull << 32)) return CH_ARENA;
    if (const int e = wide_table(t, s, w, cap)) return e;
    if (const int e = wide_alt(t, s, w, L_MID, w.n[L_MID] + room)) return e;
    const unsigned long long from = w.tab[w.tcur].off, to = w.tab[w.tcur ^ 1].off;
    const uint64_t fmask = w.tmask, tmask = cap - 1, bound = w.bound;
    const unsigned long long foff = w.list[L_FRONT][w.cur[L_FRONT]].off, moff = w.list[L_MID][w.cur[L_MID]].off;
    const uint32_t nf = w.n[L_FRONT], nm = w.n[L_MID];
    const uint64_t was = w.used;
    __syncthreads();
    if (threadIdx.x == 0) {
      w.cur[L_MID] ^= 1;
      w.n[L_MID] = 0;
      w.tcur ^= 1;
      w.tmask = tmask;
      w.used = nf;
    }
    __syncthreads();
    WideCount* c = &t.g->c[w.ph];
    const uint32_t step = (uint32_t)t.size * blockDim.x, first = (uint32_t)t.rank * blockDim.x + threadIdx.x;
    for (uint32_t i = first; i < nf; i += step) {
      const uint32_t o = __ldcg(s.r_coef + foff + i);
      const bool ok[1] = {true};
      const uint64_t key[1] = {__ldcg(s.r_key + from + o)};
      uint64_t h[1];
      bool fresh[1];
      wide_enter(s, to, tmask, ok, key, h, fresh);
      s.r_coef[to + h[0]] = __ldcg(s.r_coef + from + o);
      s.r_coef[foff + i] = (uint32_t)h[0];
    }
    for (uint32_t i0 = first - lane; i0 < nm; i0 += step) {  // whole warps go round together
      const uint32_t i = i0 + lane;
      int l[1] = {-1};
      uint64_t key[1] = {0};
      const uint32_t none[1] = {0};
      if (i < nm) {
        key[0] = __ldcg(s.r_key + moff + i);
        if (wide_value(s, from, wide_find(s, from, fmask, key[0]), p)) l[0] = L_MID;
      }
      wide_append(s, c, w, lane, l, key, none);
    }
    unsigned kept = 0;
    wide_scan(t, s, from, fmask + 1, [&](const uint64_t (&key)[8], const uint32_t (&val)[8]) {
      bool ok[8], fresh[8];
      uint64_t h[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        ok[u] = key[u] != IDX_NONE && key[u] > bound && wide_live(val[u], p);
        kept += ok[u];
      }
      wide_enter(s, to, tmask, ok, key, h, fresh);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (ok[u]) s.r_coef[to + h[u]] = p == 2 ? 1u : val[u] % p;
    });
    kept = __reduce_add_sync(0xffffffffu, kept);
    if (lane == 0 && kept) atomicAdd(&c->fresh, kept);
    if (threadIdx.x == 0 && t.rank == 0) atomicAdd(s.compacted, (unsigned long long)was);
    if (!wide_sync(t, s, w)) return CH_LONG;
    rebuilt = true;
  }
  return CH_DONE;
}

// ---------------------------------------------------------------- windows

// The q-th smallest (from 0) of the keys the block's first WIDE_SAMPLES threads
// hold: each counts the keys before its own (broadcast reads of shared memory, no
// sort).
__device__ uint64_t wide_select(uint64_t key, uint32_t q, uint64_t* sm) {
  __syncthreads();
  if (threadIdx.x < WIDE_SAMPLES) sm[threadIdx.x] = key;
  __syncthreads();
  if (threadIdx.x < WIDE_SAMPLES) {
    uint32_t before = 0, same = 0;
    const ulonglong2* s2 = (const ulonglong2*)sm;
#pragma unroll 8
    for (uint32_t i = 0; i < WIDE_SAMPLES / 2; ++i) {
      const ulonglong2 x = s2[i];
      before += (x.x < key) + (x.y < key);
      same += (x.x == key) + (x.y == key);
    }
    if (before <= q && q < before + same) sm[WIDE_SAMPLES] = key;  // equal keys write the same
  }
  __syncthreads();
  return sm[WIDE_SAMPLES];
}

// place q of a quantile k / n among S samples
__device__ __forceinline__ uint32_t wide_quantile(unsigned long long k, unsigned long long n, uint32_t S) {
  return (uint32_t)min((float)k * (float)S / (float)n, (float)(S - 1));
}

// A bound with about k rows of list l up to it, from evenly spaced samples (every
// block takes the same ones).  Of the front list only live rows with an owner
// count.
__device__ uint64_t wide_sample(const RedState& s, const WideState& w, uint32_t p, int l, unsigned long long k,
                                uint64_t* sm) {
  const uint32_t n = w.n[l];
  const uint32_t S = min(n, WIDE_SAMPLES);
  const unsigned long long off = w.list[l][w.cur[l]].off, toff = w.tab[w.tcur].off;
  uint64_t key = ~0ull;
  if (threadIdx.x < S) {
    const unsigned long long at =
        off + (n < WIDE_SAMPLES ? threadIdx.x : (uint32_t)(((uint64_t)threadIdx.x * n) / WIDE_SAMPLES));
    if (l == L_FRONT) {
      const uint32_t slot = __ldcg(s.r_coef + at);
      if (wide_value(s, toff, slot, p) && __ldcg(s.r_key + at) != OWN_NONE) key = __ldcg(s.r_key + toff + slot);
    } else {
      key = __ldcg(s.r_key + at);
    }
  }
  return wide_select(key, wide_quantile(k, n, S), sm);
}

// A bound with about k live rows of the table between `after` and it, from
// samples of its slots (hash order, so evenly spaced ones are as good as random):
// ~0 when no more than that seem to be left.
__device__ uint64_t wide_sample_table(const RedState& s, const WideState& w, uint32_t p, uint64_t after,
                                      unsigned long long k, uint64_t* sm) {
  const unsigned long long cap = w.tmask + 1;  // at least 1024
  uint64_t key = ~0ull;
  if (threadIdx.x < WIDE_SAMPLES) {
    const unsigned long long at = w.tab[w.tcur].off + threadIdx.x * (cap / WIDE_SAMPLES);
    key = __ldcg(s.r_key + at);
    if (key == IDX_NONE || key <= after || !wide_live(__ldcg(s.r_coef + at), p)) key = ~0ull;
  }
  return k >= cap ? ~0ull : wide_select(key, wide_quantile(k, cap, WIDE_SAMPLES), sm);
}

// Splits list l at key b: rows up to b go to list lo, which is l itself (its rows
// move to its other buffer), the others to list hi (L_FAR: none).  Rows older
// than `settled` are dropped.
__device__ int wide_split(const Team& t, const RedState& s, WideState& w, int l, uint64_t b, int lo, int hi,
                          uint64_t settled = 0) {
  const int lane = threadIdx.x & 31;
  const uint32_t n = w.n[l];
  if (const int e = wide_alt(t, s, w, l, n)) return e;
  for (int q = 0; q < 2; ++q)
    if (q != l && (q == lo || q == hi))
      if (const int e = wide_room(t, s, w, q, n)) return e;
  const unsigned long long off = w.list[l][w.cur[l]].off;
  __syncthreads();
  if (threadIdx.x == 0) {
    w.cur[l] ^= 1;
    w.n[l] = 0;
  }
  __syncthreads();
  const WideView v = wide_view(t, w);
  const uint32_t step = (uint32_t)t.size * blockDim.x * 4;
  // a warp takes 128 rows at a time, four a lane, whose loads are under way together
  for (uint32_t i0 = ((uint32_t)t.rank * blockDim.x + threadIdx.x - lane) * 4; i0 < n; i0 += step) {
    uint64_t key[4], code[4];
    uint32_t slot[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t i = i0 + u * 32 + lane;
      key[u] = code[u] = 0;
      slot[u] = 0;
      if (i < n) {
        key[u] = __ldcg(s.r_key + off + i);
        if (l == L_FRONT) slot[u] = __ldcg(s.r_coef + off + i);
      }
    }
    if (l == L_FRONT) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        code[u] = key[u];
        if (i0 + u * 32 + lane < n) key[u] = __ldcg(s.r_key + v.toff + slot[u]);
      }
    }
    int to[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      to[u] = -1;
      if (i0 + u * 32 + lane < n && key[u] >= settled) to[u] = key[u] <= b ? lo : hi;
      if (to[u] == L_FRONT) key[u] = code[u];
    }
    wide_append(s, v.c, w, lane, to, key, slot);
  }
  return wide_sync(t, s, w) ? CH_DONE : CH_LONG;
}

// Rows in the mid list for the next part of the window, about k of them: the list
// is refilled from the table with 8 k when it is empty, and cut down to them when
// it has outgrown 24 k.  CH_EMPTY when nothing lies beyond the front.
__device__ int wide_refill(const Team& t, const RedState& s, WideState& w, uint32_t p, unsigned long long k,
                           uint64_t* sm) {
  const int lane = threadIdx.x & 31;
  while (w.n[L_MID] == 0) {
    const uint64_t after = w.mbound;
    if (after == ~0ull) return CH_EMPTY;
    const uint64_t b = wide_sample_table(s, w, p, after, 8 * k, sm);
    if (const int e = wide_room(t, s, w, L_MID, w.used)) return e;
    __syncthreads();
    if (threadIdx.x == 0) w.mbound = b;
    __syncthreads();
    WideCount* c = &t.g->c[w.ph];
    wide_scan(t, s, w.tab[w.tcur].off, w.tmask + 1, [&](const uint64_t (&key)[8], const uint32_t (&val)[8]) {
      int l[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) l[u] = key[u] != IDX_NONE && key[u] > after && key[u] <= b ? L_MID : -1;
      wide_append(s, c, w, lane, l, key, val);
    });
    if (!wide_sync(t, s, w)) return CH_LONG;
  }
  if (w.n[L_MID] > 24 * k) {
    const uint64_t b = wide_sample(s, w, p, L_MID, 8 * k, sm);
    __syncthreads();
    if (threadIdx.x == 0) w.mbound = b;
    __syncthreads();
    return wide_split(t, s, w, L_MID, b, L_MID, L_FAR);
  }
  return CH_DONE;
}

// ---------------------------------------------------------------- additions

// The coboundary of a d-simplex (reference, rank) times f, added to the working
// column by one warp.
template <int D>
__device__ uint32_t wide_gen(const DimArgs& a, const RedState& s, const WideState& w, const WideView& v, const CV& cv,
                             const Binom& B, int lane, uint64_t ref, bool packed, uint32_t rank, uint32_t f,
                             unsigned& fresh) {
  const int d = D ? D : a.d;
  Coboundary<D> cob;
  cob.set(a, cv, B, ref, packed);
  uint32_t cnt = 0;
  for (uint32_t q0 = cob.beg; q0 < cob.end; q0 += 32 * Coboundary<D>::U) {
    bool ok[Coboundary<D>::U];
    uint64_t key[Coboundary<D>::U];
    int c[Coboundary<D>::U];
    uint32_t f4[Coboundary<D>::U];
    cob.eval(a, cv, B, rank, q0, lane, ok, key, c);
#pragma unroll
    for (int u = 0; u < Coboundary<D>::U; ++u) {
      f4[u] = a.p == 2 ? 1u : (((d - c[u]) & 1) ? a.p - f : f);
      cnt += __popc(__ballot_sync(0xffffffffu, ok[u]));
    }
    fresh += wide_insert(s, w, v, lane, a.p, ok, key, f4);
  }
  return cnt;
}

// a stored run times f, added by the `warps` warps of which this is the i-th
__device__ void wide_run(const RedState& s, const WideState& w, const WideView& v, int lane, uint32_t p,
                         unsigned long long off, uint32_t len, uint32_t f, uint32_t i, uint32_t warps,
                         unsigned& fresh) {
  constexpr int U = 4;
  for (uint32_t e0 = i * 32 * U; e0 < len; e0 += warps * 32 * U) {
    bool ok[U];
    uint64_t key[U];
    uint32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t e = e0 + u * 32 + lane;
      ok[u] = e < len;
      key[u] = ok[u] ? s.r_key[off + e] : 0;
      c[u] = ok[u] && p != 2 ? (s.r_coef[off + e] * f) % p : 1u;
    }
    fresh += wide_insert(s, w, v, lane, p, ok, key, c);
  }
}

// Owner code of a live row, looked up by one lane: the pair map and the pivot
// table are probed with their first loads issued together.
__device__ __forceinline__ uint64_t wide_owner(const DimArgs& a, const RedState& s, uint32_t cl, uint32_t j,
                                               uint64_t key) {
  const uint64_t tkey = table_key(a, cl, row_key_idx(a, key));
  const uint64_t hash = mix(tkey);
  uint64_t h = hash & s.t_mask;
  uint64_t tk = s.t_keys[h];
  uint32_t tv = s.t_vals[h];
  if (a.amap) {
    uint64_t val;
    if (pair_find(a.amap, a.amap_mask, tkey, &val)) return val;
  }
  for (uint64_t probe = 0; probe <= s.t_mask; ++probe) {
    if (tk == tkey) return tv < j ? ((uint64_t)tv << 4) | OWN_TABLE : OWN_NONE;
    if (tk == IDX_NONE) break;
    h = (h + 1) & s.t_mask;
    tk = s.t_keys[h];
    tv = s.t_vals[h];
  }
  return OWN_NONE;
}

// two neighbouring counts with one atomic
__device__ __forceinline__ void wide_count2(unsigned* first, unsigned a, unsigned b) {
  if (a | b) atomicAdd((unsigned long long*)first, a | ((unsigned long long)b << 32));
}

// new rows of a warp's lanes and the entries it added, counted once a section
__device__ __forceinline__ void wide_count_fresh(WideCount* c, int lane, unsigned fresh, unsigned ents = 0) {
  fresh = __reduce_add_sync(0xffffffffu, fresh);
  if (lane == 0) wide_count2(&c->fresh, fresh, ents);
}

// kinds of work records (two arena entries: key words ref, kind << 32 | length,
// coefficient words factor, rank)
enum { REC_PACKED = 0, REC_INDEX = 1, REC_RUN = 2 };

// what a warp has seen in a section
struct WideSeen {
  uint64_t un, ow;  // oldest live rows without and with an owner
  unsigned own;     // live rows with one
};

// A row a lane (val: its coefficient, 0 for none): looks its owner up unless
// `code` has it, and writes a work record for a live row that has one (long
// stored runs go on their own list).  Warp-wide; returns the owner code to keep.
__device__ __forceinline__ uint64_t wide_look(const DimArgs& a, const RedState& s, const WideState& w, const WideView& v, const CV& cv,
                              const Binom& B, int lane, uint32_t val, uint64_t key, uint64_t code, WideSeen& seen) {
  const uint32_t p = a.p;
  const bool live = val != 0;
  const bool scan = !a.amap && !(a.opts & RIPS_OPT_NO_APPARENT);  // apparent facets are found by scanning
  uint64_t ref = 0;
  uint32_t f = 0, rlen = 0, pc = 1, kind = REC_INDEX;  // pc: the row's coefficient in its owner's column
  uint32_t rank = live ? row_key_rank(a, key) : 0u;
  bool facet = false;  // found by scanning, not kept
  if (live && code == OWN_UNKNOWN && !scan) code = wide_owner(a, s, w.cl, w.j, key);
  if (scan) {
    unsigned m = __ballot_sync(0xffffffffu, live && code == OWN_UNKNOWN);
    while (m) {
      const int L = __ffs(m) - 1;
      m &= m - 1;
      uint32_t fr, tc;
      const uint64_t fi = pivot_apparent_facet(a, cv, B, lane, __shfl_sync(0xffffffffu, key, L), &fr, &tc);
      if (lane == L) {
        if (fi == IDX_NONE) {
          code = wide_owner(a, s, w.cl, w.j, key);
        } else {
          facet = true;
          ref = fi;
          pc = tc;
        }
      }
    }
  }
  const uint32_t ck = (uint32_t)(code & 15);
  const bool own = live && ck != OWN_NONE;
  bool put = own, lng = false;
  if (own) {
    if (facet) {
    } else if (ck == OWN_TABLE) {
      const uint32_t k = (uint32_t)(code >> 4);
      pc = s.piv_coef[k];
      rlen = s.r_len[k];
      const unsigned long long ro = s.r_off[k];
      const uint64_t kk = s.col_keys[k];
      if (rlen) {
        kind = REC_RUN;
        ref = ro;
        lng = rlen > s.scr_slice;
      } else {
        ref = kk & low_mask(a.col_bits);
        rank = a.rank_max - (uint32_t)((kk >> a.col_bits) & low_mask(a.rank_bits));
      }
    } else {
      ref = code >> 4;
      kind = a.vbits ? REC_PACKED : REC_INDEX;
      pc = ((a.d - (int)ck) & 1) ? p - 1 : 1u;
    }
    f = p == 2 ? 1u : (p - (val * (pc == 1 || pc == p - 1 ? pc : mod_inv(pc, p))) % p) % p;
    seen.ow = min(seen.ow, key);
    ++seen.own;
  } else if (live) {
    seen.un = min(seen.un, key);
  }
  if (lng) {  // added by the whole team, as far as there is room for it this round
    put = false;
    const unsigned long long limit = max(4096ull, (unsigned long long)w.used);
    const unsigned long long o = atomicAdd(&v.c->longsum, (unsigned long long)rlen);
    if (o == 0 || o + rlen <= limit) {
      const unsigned q = atomicAdd(&v.c->nlong, 1u);
      if (q < WIDE_LONGS) {
        s.r_key[w.lng.off + q] = (code >> 4) | ((uint64_t)f << 32);
        atomicAdd(&v.c->longroom, (unsigned long long)rlen);
      }
    }
  }
  const unsigned pm = __ballot_sync(0xffffffffu, put);
  if (pm) {
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&v.c->todo, (unsigned)__popc(pm));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (put) {
      const unsigned long long q = w.todo.off + 2ull * (base + __popc(pm & ((1u << lane) - 1u)));
      s.r_key[q] = ref;
      s.r_coef[q] = f;
      s.r_key[q + 1] = ((uint64_t)kind << 32) | rlen;
      s.r_coef[q + 1] = rank;
    }
  }
  return code;
}

template <typename T>
__device__ __forceinline__ T wide_pick(const T (&x)[4], int u) {
  return u == 0 ? x[0] : u == 1 ? x[1] : u == 2 ? x[2] : x[3];
}

// First section of a round: looks over the front's n rows and over the nm mid
// rows from moff on, of which those up to the bound (set already) join the front
// and the others go to the mid list's other buffer.  A warp takes a tile of 128
// rows of one list at a time, four a lane, whose loads are under way together.
__device__ __forceinline__ void wide_check(const DimArgs& a, const RedState& s, const Team& t, const WideState& w,
                                           const CV& cv, const Binom& B, unsigned long long moff, uint32_t nm) {
  const int lane = threadIdx.x & 31;
  const WideView v = wide_view(t, w);
  const unsigned long long foff = w.list[L_FRONT][w.cur[L_FRONT]].off;
  const uint32_t n = w.n[L_FRONT];
  const uint32_t p = a.p;
  WideSeen seen{~0ull, ~0ull, 0};
  const uint64_t lo = w.lo, hi = w.hi;
  unsigned settled = 0;
  const uint32_t ft = (n + 127) / 128, tiles = ft + (nm + 127) / 128;
  const uint32_t tw = (uint32_t)t.rank + (threadIdx.x >> 5) * (uint32_t)t.size, TW = (uint32_t)t.size * WARPS_PER_BLOCK;
  unsigned joined = 0;
  for (uint32_t tile = tw; tile < tiles; tile += TW) {
    const bool front = tile < ft;
    const uint32_t i0 = (front ? tile : tile - ft) * 128 + lane, end = front ? n : nm;
    uint64_t key[4], code[4];
    uint32_t slot[4], val[4];
    bool near[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t i = i0 + u * 32;
      const bool in = i < end;
      slot[u] = front && in ? __ldcg(s.r_coef + foff + i) : 0u;
      key[u] = in ? __ldcg(s.r_key + (front ? foff : moff) + i) : ~0ull;
      near[u] = in && (front || key[u] <= v.bound);
    }
    if (front) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        code[u] = key[u];
        key[u] = near[u] ? __ldcg(s.r_key + v.toff + slot[u]) : ~0ull;
        settled += key[u] >= lo && key[u] < hi && (code[u] & 15) < OWN_NONE;
      }
    } else {
      uint64_t h[4];
      wide_find(s, v.toff, v.mask, near, key, h);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        code[u] = OWN_UNKNOWN;
        slot[u] = (uint32_t)h[u];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) val[u] = near[u] ? wide_value(s, v.toff, slot[u], p) : 0u;
    const unsigned before = seen.own;
#pragma unroll 1
    for (int u = 0; u < 4; ++u) {
      const uint32_t x = wide_pick(val, u);
      if (!__ballot_sync(0xffffffffu, x != 0)) continue;
      const uint64_t c = wide_look(a, s, w, v, cv, B, lane, x, wide_pick(key, u), wide_pick(code, u), seen);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q == u && x) {
          if (front && c != code[q]) s.r_key[foff + i0 + q * 32] = c;
          code[q] = c;
        }
    }
    if (!front) {
      joined += seen.own - before;
      int to[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        to[u] = i0 + u * 32 >= end ? -1 : near[u] ? L_FRONT : L_MID;
        if (near[u]) key[u] = code[u];
      }
      wide_append(s, v.c, w, lane, to, key, slot);
    }
  }
  const uint64_t un = warp_min_u64(seen.un), ow = warp_min_u64(seen.ow);
  joined = __reduce_add_sync(0xffffffffu, joined);
  settled = __reduce_add_sync(0xffffffffu, settled);
  if (lane == 0) {
    wide_count2(&v.c->count, joined, settled);
    if (ow != ~0ull) atomicMin(&v.c->ow, (unsigned long long)ow);
    if (un != ~0ull) atomicMin(&v.c->un, (unsigned long long)un);
  }
}

// Second section: work records [p0, p1), a warp each.
template <int D>
__device__ void wide_process(const DimArgs& a, const RedState& s, const Team& t, const WideState& w, const CV& cv,
                             const Binom& B, uint32_t p0, uint32_t p1) {
  const int lane = threadIdx.x & 31;
  const uint32_t tw = (uint32_t)t.rank + (threadIdx.x >> 5) * (uint32_t)t.size, TW = (uint32_t)t.size * WARPS_PER_BLOCK;
  const WideView v = wide_view(t, w);
  unsigned long long ents = 0;
  unsigned fresh = 0;
  for (uint32_t i = p0 + tw; i < p1; i += TW) {
    const unsigned long long q = w.todo.off + 2ull * i;
    const uint64_t ref = __ldcg(s.r_key + q), kl = __ldcg(s.r_key + q + 1);
    const uint32_t f = __ldcg(s.r_coef + q), rank = __ldcg(s.r_coef + q + 1), len = (uint32_t)kl;
    const int kind = (int)(kl >> 32);
    if (kind == REC_RUN) {
      wide_run(s, w, v, lane, a.p, ref, len, f, 0, 1, fresh);
      ents += len;
    } else {
      ents += wide_gen<D>(a, s, w, v, cv, B, lane, ref, kind == REC_PACKED, rank, f, fresh);
    }
  }
  wide_count_fresh(v.c, lane, fresh, (unsigned)ents);
  if (lane == 0 && ents) atomicAdd(s.added, ents);
}

// the section's long runs, every one spread over all the team's warps
__device__ void wide_longs(const RedState& s, const Team& t, const WideState& w, uint32_t p, uint32_t count) {
  const int lane = threadIdx.x & 31;
  const uint32_t tw = (uint32_t)t.rank * WARPS_PER_BLOCK + (threadIdx.x >> 5), TW = (uint32_t)t.size * WARPS_PER_BLOCK;
  const WideView v = wide_view(t, w);
  unsigned fresh = 0;
  for (uint32_t i0 = 0; i0 < count; i0 += 32) {
    uint64_t e = 0;
    uint32_t len = 0;
    unsigned long long off = 0;
    if (i0 + lane < count) {
      e = __ldcg(s.r_key + w.lng.off + i0 + lane);
      len = s.r_len[(uint32_t)e];
      off = s.r_off[(uint32_t)e];
    }
    for (uint32_t i = 0; i < 32 && i0 + i < count; ++i)  // each run starts at another warp
      wide_run(s, w, v, lane, p, __shfl_sync(0xffffffffu, off, i), __shfl_sync(0xffffffffu, len, i),
               (uint32_t)(__shfl_sync(0xffffffffu, e, i) >> 32), (tw + (i0 + i) * 37u) % TW, TW, fresh);
  }
  wide_count_fresh(v.c, lane, fresh);
}

// ---------------------------------------------------------------- a column

// Column j's own entries into an empty working column.
template <int D>
__device__ __forceinline__ int wide_begin(const DimArgs& a, const RedState& s, const Team& t, WideState& w, const CV& cv,
                          const Binom& B, uint32_t j, uint32_t cl, uint64_t jidx, uint32_t jrank) {
  const int lane = threadIdx.x & 31;
  const uint32_t jn = s.r_len[j];
  __syncthreads();
  if (threadIdx.x == 0) {
    w.j = j;
    w.cl = cl;
    w.step = 0;
    w.pace = w.each = 0.0f;
    w.lo = w.hi = 0;
    w.dil = 1;
    w.n[0] = w.n[1] = 0;
    w.tmask = 0;
    w.used = 0;
    w.bound = 0;
    w.mbound = ~0ull;
    w.t0 = global_ns();
  }
  __syncthreads();
  const unsigned long long own = jn ? jn : s.scr_slice;
  if (w.lng.cap == 0) {  // a first column: its buffers in one piece
    const unsigned long long cap0 = wide_pow2(2 * (own + (unsigned long long)WIDE_K0 * s.scr_slice)), row = cap0 / 2;
    WideList nl;
    if (const int e = wide_alloc(t, s, w, cap0 + 4 * row + 4 * WIDE_LONGS, &nl)) return e;
    if (threadIdx.x == 0) {
      unsigned long long o = nl.off;
      w.tab[w.tcur ^ 1] = WideList{o, cap0};
      o += cap0;
      for (int l = 0; l < 2; ++l)
        for (int q = 0; q < 2; ++q, o += row) w.list[l][q] = WideList{o, row};
      w.lng = WideList{o, WIDE_LONGS};
      w.todo = WideList{o + WIDE_LONGS, 3 * WIDE_LONGS};
    }
    __syncthreads();
  }
  const unsigned long long cap = wide_pow2(2 * (own + (unsigned long long)WIDE_K0 * s.scr_slice));
  if (cap > (1ull << 32)) return CH_ARENA;
  if (const int e = wide_table(t, s, w, cap)) return e;
  __syncthreads();
  if (threadIdx.x == 0) {
    w.tcur ^= 1;
    w.tmask = cap - 1;
  }
  __syncthreads();
  const int e = wide_ensure(t, s, w, a.p, own);
  if (e != CH_DONE) return e;
  const WideView v = wide_view(t, w);
  const uint32_t tw = (uint32_t)t.rank * WARPS_PER_BLOCK + (threadIdx.x >> 5);
  unsigned fresh = 0;
  if (jn) wide_run(s, w, v, lane, a.p, s.r_off[j], jn, 1, tw, (uint32_t)t.size * WARPS_PER_BLOCK, fresh);
  else if (tw == 0) wide_gen<D>(a, s, w, v, cv, B, lane, jidx, false, jrank, 1, fresh);
  wide_count_fresh(v.c, lane, fresh);
  return wide_sync(t, s, w) ? CH_DONE : CH_LONG;
}

// When a column gives way to a larger team (asked by its leader between rounds):
// a block once it has made TEAM_MIN_STEPS additions, all columns and light ones
// are handed out and half of the blocks wait; a team once half of the teams are
// done.
struct GiveWay {
  const volatile unsigned *a, *b, *c;
  unsigned na, nb, nc, steps;
  __device__ __forceinline__ bool operator()(uint32_t step) const {
    return step >= steps && *a >= na && *b >= nb && 2 * *c >= nc;
  }
};

// Eliminates until the pivot is free, owned by a later column, or the column is
// zero: CH_DONE with the pivot (IDX_NONE: zero) and its coefficient.  CH_HEAVY:
// suspended between two rounds, to be resumed by a larger team.
template <int D>
__device__ __forceinline__ int wide_advance(const DimArgs& a, const RedState& s, const Team& t, WideState& w, const CV& cv,
                                            const Binom& B, uint64_t* sm, uint64_t* piv, uint32_t* coef,
                                            const GiveWay& give_way) {
  const uint32_t p = a.p;
  const uint32_t kmax = 2u * (uint32_t)t.size * WARPS_PER_BLOCK;  // more than this and a round's time is its additions'
  const unsigned long long rows = 1024ull * t.size * WARPS_PER_BLOCK;  // most rows a window is extended by
  const int sbits = 31 - __clz(s.scr_slice);                           // scr_slice is a power of two
  float again = 0.0f;       // share of a round's rows that come back live in the next one
  uint32_t last = 0;        // rows added last round
  float share = 1.0f;       // of k, to extend the window by
  const float free = t.size > 1 ? WIDE_TEAM_FREE * (float)t.size : WIDE_FREE;
  const bool paced = a.amap || (a.opts & RIPS_OPT_NO_APPARENT);  // owners are kept, so that settled rows can be counted
  for (;;) {
    const uint32_t goal = t.size > 1 ? max(w.step / 2, min(max(w.step, WIDE_TEAM_K0), WIDE_TEAM_K1))
                                     : max(w.step / 3, WIDE_K0);
    // rows with an owner wanted in the window
    const float ahead = fmaxf(WIDE_AHEAD * w.pace, free / fmaxf(w.each, 1.0f));
    const uint32_t k = min(min(goal, kmax), paced ? max((uint32_t)ahead, 2u) : ~0u);
    const uint32_t crowd = max(2 * k, min(64u, 8 * k));  // and more than these are too many
    const unsigned long long want = max(1ull, min((unsigned long long)((float)k * share) * w.dil, rows));
    bool extend = false;
    uint64_t b = w.bound;
    if (share > 0.0f || w.n[L_FRONT] == 0) {
      const int e = wide_refill(t, s, w, p, want, sm);
      if (e == CH_DONE) {
        extend = true;
        b = w.n[L_MID] <= 2 * want ? w.mbound : wide_sample(s, w, p, L_MID, want, sm);
      } else if (e != CH_EMPTY) {
        return e;
      } else if (w.n[L_FRONT] == 0) {
        *piv = IDX_NONE;
        *coef = 0;
        return CH_DONE;
      }
    }
    const uint32_t nm = extend ? w.n[L_MID] : 0u;
    if (extend) {
      if (const int e = wide_alt(t, s, w, L_MID, nm)) return e;
      if (const int e = wide_room(t, s, w, L_FRONT, nm)) return e;
    }
    if (w.todo.cap < 2ull * (w.n[L_FRONT] + nm)) {
      const unsigned long long rows = w.n[L_FRONT] + nm;
      if (const int e = wide_grow(t, s, w, w.todo, 2 * rows, 3 * rows + 64)) return e;
    }
    const unsigned long long moff = w.list[L_MID][w.cur[L_MID]].off;
    __syncthreads();
    if (threadIdx.x == 0) {
      if (extend) {
        w.cur[L_MID] ^= 1;
        w.n[L_MID] = 0;
        w.bound = b;
      }
      if (t.rank == 0) {
        unsigned st = 0;
        if (global_ns() - w.t0 > s.chain_ns) st = 1;  // the chain's wall-clock bound
        else if (give_way(w.step)) st = 2;
        if (st) *(volatile unsigned*)&t.g->c[w.ph].stop = st;
        atomicAdd(s.heartbeat, 1u);  // progress, for the barriers
      }
    }
    __syncthreads();
    wide_check(a, s, t, w, cv, B, moff, nm);
    if (!wide_sync(t, s, w)) return CH_LONG;
    const uint32_t todo = w.d.todo, nl = min(w.d.nlong, WIDE_LONGS), joined = w.d.add[L_FRONT], owned = w.d.count;
    const unsigned stop = w.d.stop;
    const uint64_t un = w.d.un, ow = w.d.ow;
    const unsigned long long lr = w.d.longroom;
    if (un < ow) {  // the oldest live row has no owner: it is the pivot
      const unsigned long long toff = w.tab[w.tcur].off;
      *piv = un;
      *coef = wide_value(s, toff, wide_find(s, toff, w.tmask, un), p);
      return CH_DONE;
    }
    if ((stop & 1u) || w.step > MAX_PIVOT_PASSES) return CH_LONG;
    __syncthreads();
    if (threadIdx.x == 0) {
      if (w.hi > w.lo) w.pace = 0.5f * (w.pace + (float)w.d.settled);
      w.lo = w.hi;
      w.hi = ow == ~0ull ? w.bound : ow;
      if (joined) w.dil = max(1u, joined / max(owned, 1u));
      if (ow == ~0ull) w.n[L_FRONT] = 0;  // no live row: all of them are settled
    }
    __syncthreads();
    if (last) again = 0.5f * again + 0.5f * min(4.0f, (float)(todo + nl - owned) / (float)last);
    last = 0;
    if (ow == ~0ull) {
      share = 1.0f;
      if (stop & 2u) return CH_HEAVY;
      continue;
    }
    if (todo > crowd) {  // the window's rows have multiplied: keep about the k oldest
      const uint64_t b2 = min(wide_sample(s, w, p, L_FRONT, k, sm), w.bound);
      if (b2 < w.bound) {
        __syncthreads();
        if (threadIdx.x == 0) w.bound = b2;
        __syncthreads();
        const int e = wide_split(t, s, w, L_FRONT, b2, L_FRONT, L_MID, w.lo);
        if (e != CH_DONE) return e;
        if (stop & 2u) return CH_HEAVY;
        share = 0.0f;
        continue;
      }
      // the bound stays: no block adds to the rows before all have sampled them, or it would find another bound
      if (t.size > 1 && !wide_sync(t, s, w)) return CH_LONG;
    } else if (w.n[L_FRONT] > 4 * min((unsigned long long)k * w.dil, rows) + 1024) {  // mostly settled rows: drop them
      const int e = wide_split(t, s, w, L_FRONT, w.bound, L_FRONT, L_MID, ow);
      if (e != CH_DONE) return e;
      if (threadIdx.x == 0) w.lo = w.hi;  // nothing left to count of this round
      __syncthreads();
    }
    // the additions, in sections of at most as many rows as the working column leaves room for
    uint32_t grown = 0;
    float ents = (float)lr;
    for (uint32_t p0 = 0; p0 < todo;) {
      const uint32_t most =
          (uint32_t)min((unsigned long long)(todo - p0), max(64ull, ((unsigned long long)w.used + 65536) >> sbits));
      const int e = wide_ensure(t, s, w, p, (unsigned long long)most << sbits);
      if (e != CH_DONE) return e;
      wide_process<D>(a, s, t, w, cv, B, p0, p0 + most);
      if (!wide_sync(t, s, w)) return CH_LONG;
      grown += w.d.add[L_FRONT];
      ents += (float)w.d.ents;
      p0 += most;
    }
    if (nl) {
      const int e = wide_ensure(t, s, w, p, lr);
      if (e != CH_DONE) return e;
      wide_longs(s, t, w, p, nl);
      if (threadIdx.x == 0 && t.rank == 0) atomicAdd(s.added, lr);
      if (!wide_sync(t, s, w)) return CH_LONG;
      grown += w.d.add[L_FRONT];
    }
    if (threadIdx.x == 0) {
      w.each = (w.step ? 0.5f : 1.0f) * ents / (float)(todo + nl) + (w.step ? 0.5f * w.each : 0.0f);
      w.step += todo + nl;
    }
    __syncthreads();
    // the rows expected live next time are left out of the next extension
    last = todo + nl;
    const float rest = 1.0f - ((float)last * again + (float)(grown / w.dil)) / (float)k;
    share = rest < 0.25f ? 0.0f : rest;
    if (stop & 2u) return CH_HEAVY;
  }
}

// Stores the finished column (its live rows, in key order up to SORT_RUN of them
// if a warp may still add it) and its pivot, and puts it on the claim list.
__device__ __forceinline__ int wide_finish(const DimArgs& a, const RedState& s, const Team& t, WideState& w, uint64_t* sm,
                           uint64_t piv, uint32_t coef, bool sorted, uint32_t* claim_count) {
  const int lane = threadIdx.x & 31;
  const uint32_t p = a.p;
  unsigned long long roff = 0;
  uint32_t len = 0;
  if (w.step && piv != IDX_NONE) {
    const uint32_t step = (uint32_t)t.size * blockDim.x, first = (uint32_t)t.rank * blockDim.x + threadIdx.x;
    if (const int e = wide_alt(t, s, w, L_MID, w.used)) return e;
    const WideView v = wide_view(t, w);
    const unsigned long long buf = w.list[L_MID][w.cur[L_MID] ^ 1].off;
    wide_scan(t, s, v.toff, v.mask + 1, [&](const uint64_t (&key)[8], const uint32_t (&val)[8]) {
      unsigned m[8], total = 0, base = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        m[u] = __ballot_sync(0xffffffffu, key[u] != IDX_NONE && wide_live(val[u], p));
        total += __popc(m[u]);
      }
      if (!total) return;
      if (lane == 0) base = atomicAdd(&v.c->count, total);
      unsigned long long pos = buf + __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if ((m[u] >> lane) & 1u) {
          s.r_key[pos + __popc(m[u] & ((1u << lane) - 1u))] = key[u];
          s.r_coef[pos + __popc(m[u] & ((1u << lane) - 1u))] = p == 2 ? 1u : val[u] % p;
        }
        pos += __popc(m[u]);
      }
    });
    if (!wide_sync(t, s, w)) return CH_LONG;
    len = w.d.count;
    WideList run;
    if (const int e = wide_alloc(t, s, w, len, &run)) return e;
    roff = run.off;
    if (sorted && len <= SORT_RUN) {
      if (t.rank == 0) {
        uint32_t* sc = (uint32_t*)(sm + SORT_RUN);
        uint32_t n2 = 2;
        while (n2 < len) n2 <<= 1;
        for (uint32_t i = threadIdx.x; i < n2; i += blockDim.x) {
          sm[i] = i < len ? __ldcg(s.r_key + buf + i) : ~0ull;
          sc[i] = i < len ? __ldcg(s.r_coef + buf + i) : 0u;
        }
        __syncthreads();
        block_bitonic(sm, sc, n2);
        for (uint32_t i = threadIdx.x; i < len; i += blockDim.x) {
          s.r_key[roff + i] = sm[i];
          s.r_coef[roff + i] = sc[i];
        }
        __syncthreads();
      }
    } else {
      for (uint32_t i = first; i < len; i += step) {
        s.r_key[roff + i] = __ldcg(s.r_key + buf + i);
        s.r_coef[roff + i] = __ldcg(s.r_coef + buf + i);
      }
    }
    if (!wide_sync(t, s, w)) return CH_LONG;
  }
  if (threadIdx.x == 0 && t.rank == 0) {
    const uint32_t j = w.j;
    if (w.step) {
      s.reduced[j] = !sorted || len > SORT_RUN ? (uint8_t)(s.reduced[j] | 1 | HEAVY | UNSORTED)
                                    : (uint8_t)((s.reduced[j] | 1) & ~UNSORTED);
      atomicAdd(s.steps, (unsigned long long)w.step);
      atomicMax(s.max_chain, w.step);
      if (piv != IDX_NONE) {
        s.r_off[j] = roff;
        s.r_len[j] = len;
      }
    }
    s.piv_key[j] = piv;
    s.piv_coef[j] = coef;
    if (piv != IDX_NONE) s.claim_list[atomicAdd(claim_count, 1u)] = j;
  }
  __syncthreads();
  return CH_DONE;
}

}  // namespace
