// Exclusive scan and LSD radix sort on 64-bit keys (filtration order, Section 2:
// keys pack the diameter rank above the simplex index, so one unsigned sort
// realises "diameter, then index").
//
// Radix sort: 8-bit digits, one pass per digit.  Each pass is
//   (1) tile histograms,
//   (2) for long inputs a per-digit scan over the tiles (for short ones every
//       scatter block adds up the tiles before its own itself),
//   (3) stable scatter: every warp ranks its 32-key steps with
//       __match_any_sync, warps are ordered by a shared-memory prefix, so keys
//       with equal digits keep their relative order (LSD correctness); the
//       tile is put in digit order in shared memory and written out in runs.
// Bits below `low_bit` are not sorted: callers whose keys already come in the
// order of those bits save their passes.  Bound, for long inputs, by the ranking in
// shared memory where many keys share a digit (8.4 million keys: a scatter 73 us, 38
// where digits are spread, with 3 x 8 bytes a key and pass to move; a pass 95 us, 140
// when keys were scattered straight from registers after being ranked twice) and by
// launches for short ones (11000 keys: 0.06 ms in 4 or 5 passes of two launches,
// 0.14 in 7 of three).  Tiles of 2048 keys give 50 blocks at 100000 keys.

#include <atomic>

#include "rips_internal.cuh"

namespace rips {

// ============================================================ scan
namespace {
constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// block-wide exclusive scan of one value per thread; returns total in *total
__device__ uint32_t block_excl_scan(uint32_t v, uint32_t* smem, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t inc = warp_incl_scan(v);
  if (lane == 31) smem[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nw ? smem[lane] : 0;
    uint32_t wi = warp_incl_scan(w);
    if (lane < nw) smem[lane] = wi - w;
    if (lane == nw - 1) smem[32] = wi;
  }
  __syncthreads();
  uint32_t r = smem[warp] + inc - v;
  *total = smem[32];
  __syncthreads();
  return r;
}

__global__ void scan_reduce_kernel(const uint32_t* __restrict__ in, uint32_t n, uint32_t* __restrict__ sums) {
  __shared__ uint32_t sm[33];
  size_t base = (size_t)blockIdx.x * SCAN_TILE;
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    size_t idx = base + (size_t)threadIdx.x * SCAN_ITEMS + i;
    if (idx < n) s += in[idx];
  }
  uint32_t tot;
  block_excl_scan(s, sm, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void scan_sums_kernel(uint32_t* __restrict__ sums, uint32_t nb, uint32_t* __restrict__ total) {
  __shared__ uint32_t sm[33];
  uint32_t carry = 0;
  for (uint32_t base = 0; base < nb; base += blockDim.x) {
    uint32_t idx = base + threadIdx.x;
    uint32_t v = idx < nb ? sums[idx] : 0;
    uint32_t tot;
    uint32_t e = block_excl_scan(v, sm, &tot);
    if (idx < nb) sums[idx] = carry + e;
    carry += tot;
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void scan_apply_kernel(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, uint32_t n,
                                  const uint32_t* __restrict__ sums) {
  __shared__ uint32_t sm[33];
  size_t base = (size_t)blockIdx.x * SCAN_TILE;
  uint32_t v[SCAN_ITEMS];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    size_t idx = base + (size_t)threadIdx.x * SCAN_ITEMS + i;
    v[i] = idx < n ? in[idx] : 0;
    s += v[i];
  }
  uint32_t tot;
  uint32_t e = block_excl_scan(s, sm, &tot) + sums[blockIdx.x];
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    size_t idx = base + (size_t)threadIdx.x * SCAN_ITEMS + i;
    if (idx < n) out[idx] = e;
    e += v[i];
  }
}

// the whole scan by one block, tile after tile (in place allowed: a tile is read before it is written)
__global__ void __launch_bounds__(SCAN_THREADS) scan_one_kernel(const uint32_t* in, uint32_t* out, uint32_t n,
                                                                uint32_t* __restrict__ total) {
  __shared__ uint32_t sm[33];
  uint32_t carry = 0;
  for (uint32_t base = 0; base < n; base += SCAN_TILE) {
    uint32_t v[SCAN_ITEMS];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
      const uint32_t idx = base + threadIdx.x * SCAN_ITEMS + i;
      v[i] = idx < n ? in[idx] : 0;
      s += v[i];
    }
    uint32_t tot;
    uint32_t e = carry + block_excl_scan(s, sm, &tot);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
      const uint32_t idx = base + threadIdx.x * SCAN_ITEMS + i;
      if (idx < n) out[idx] = e;
      e += v[i];
    }
    carry += tot;
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// up to this many values one block scans them (one launch, 2 to 7 us) instead of three kernels (3 launches, 7 us)
constexpr uint32_t SCAN_ONE = 4 * SCAN_TILE;
}  // namespace

size_t scan_temp_bytes(uint32_t n) {
  size_t nb = ((size_t)n + SCAN_TILE - 1) / SCAN_TILE;
  return (nb + 1) * sizeof(uint32_t);
}

cudaError_t launch_exclusive_scan(const uint32_t* in, uint32_t* out, uint32_t n, void* tmp,
                                  uint32_t* d_total, cudaStream_t s) {
  uint32_t nb = (uint32_t)(((size_t)n + SCAN_TILE - 1) / SCAN_TILE);
  if (nb == 0) nb = 1;
  uint32_t* sums = (uint32_t*)tmp;
  if (n <= SCAN_ONE) {
    scan_one_kernel<<<1, SCAN_THREADS, 0, s>>>(in, out, n, d_total);
    note_launch();
    return cudaGetLastError();
  }
  scan_reduce_kernel<<<nb, SCAN_THREADS, 0, s>>>(in, n, sums);
  note_launch();
  scan_sums_kernel<<<1, SCAN_THREADS, 0, s>>>(sums, nb, d_total);
  note_launch();
  scan_apply_kernel<<<nb, SCAN_THREADS, 0, s>>>(in, out, n, sums);
  note_launch();
  return cudaGetLastError();
}

// ============================================================ radix sort
namespace {
constexpr int RS_THREADS = 256;   // 8 warps
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_STEPS = RS_TILE / RS_THREADS;  // 32-key steps per warp
constexpr int RADIX = 256;
// Up to this many tiles a scatter block adds up the counts of the tiles before
// its own (64 rows of 1 KB from L2 at most, about 3 us) instead of a scan launch
// between (about 3 us at any size).
constexpr uint32_t RS_DIRECT_TILES = 64;

__global__ void __launch_bounds__(RS_THREADS) rs_hist_kernel(const uint64_t* __restrict__ keys, uint32_t n, int shift,
                                                             uint32_t* __restrict__ hist, uint32_t dstride,
                                                             uint32_t tstride) {
  __shared__ uint32_t h[RADIX];
  h[threadIdx.x] = 0;
  __syncthreads();
  const size_t base = (size_t)blockIdx.x * RS_TILE;
#pragma unroll
  for (int i = 0; i < RS_STEPS; ++i) {
    const size_t idx = base + i * RS_THREADS + threadIdx.x;
    if (idx < n) atomicAdd(&h[(uint32_t)(keys[idx] >> shift) & 0xFFu], 1u);
  }
  __syncthreads();
  hist[(size_t)threadIdx.x * dstride + (size_t)blockIdx.x * tstride] = h[threadIdx.x];
}

// one block per digit: exclusive scan of hist[digit][0..tiles) and digit total
__global__ void rs_tile_scan_kernel(uint32_t* __restrict__ hist, uint32_t tiles, uint32_t* __restrict__ totals) {
  __shared__ uint32_t sm[33];
  uint32_t* row = hist + (size_t)blockIdx.x * tiles;
  uint32_t carry = 0;
  for (uint32_t b = 0; b < tiles; b += blockDim.x) {
    uint32_t idx = b + threadIdx.x;
    uint32_t v = idx < tiles ? row[idx] : 0;
    uint32_t tot;
    uint32_t e = block_excl_scan(v, sm, &tot);
    if (idx < tiles) row[idx] = carry + e;
    carry += tot;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// DIRECT: hist is [tile][digit] counts; else [digit][tile] prefixes with the digits' totals
template <bool HAS_VALS, bool DIRECT>
__global__ void __launch_bounds__(RS_THREADS) rs_scatter_kernel(
    const uint64_t* __restrict__ keys, uint64_t* __restrict__ keys_out, const uint32_t* __restrict__ vals,
    uint32_t* __restrict__ vals_out, uint32_t n, int shift, const uint32_t* __restrict__ hist, uint32_t tiles,
    const uint32_t* __restrict__ totals) {
  __shared__ uint64_t stage[RS_TILE];
  __shared__ uint32_t stage_v[HAS_VALS ? RS_TILE : 1];
  __shared__ uint32_t delta[RADIX];               // output position minus position in the tile, per digit
  __shared__ uint32_t warp_cnt[RS_WARPS][RADIX];  // per-warp digit counts -> the warp's first position in the tile
  __shared__ uint32_t sm[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, dg = threadIdx.x;  // thread dg owns digit dg
  const unsigned lt_mask = (1u << lane) - 1u;
  const size_t tile0 = (size_t)blockIdx.x * RS_TILE, base = tile0 + (size_t)warp * RS_STEPS * 32;

  uint64_t k[RS_STEPS];
  uint32_t v[HAS_VALS ? RS_STEPS : 1], pos[RS_STEPS];
#pragma unroll
  for (int st = 0; st < RS_STEPS; ++st) {
    const size_t idx = base + st * 32 + lane;
    k[st] = idx < n ? keys[idx] : ~0ull;
    if (HAS_VALS) v[st] = idx < n ? vals[idx] : 0u;
  }
  for (int i = threadIdx.x; i < RS_WARPS * RADIX; i += RS_THREADS) (&warp_cnt[0][0])[i] = 0;
  // this tile's first output position of every digit
  uint32_t mine = 0, all = 0, tot;
  if (DIRECT) {
    for (uint32_t t = 0; t < tiles; ++t) {
      const uint32_t c = hist[(size_t)t * RADIX + dg];
      if (t == blockIdx.x) mine = all;
      all += c;
    }
  } else {
    mine = hist[(size_t)dg * tiles + blockIdx.x];
    all = totals[dg];
  }
  mine += block_excl_scan(all, sm, &tot);  // its barriers also order the clearing of the counts

  // rank of every key among its warp's keys of the same digit
#pragma unroll
  for (int st = 0; st < RS_STEPS; ++st) {
    const bool valid = base + st * 32 + lane < n;
    const uint32_t d = (uint32_t)(k[st] >> shift) & 0xFFu;
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    if (valid) {
      const unsigned peers = __match_any_sync(act, d);
      pos[st] = warp_cnt[warp][d] + __popc(peers & lt_mask);
      __syncwarp(act);
      if ((peers & lt_mask) == 0) warp_cnt[warp][d] += __popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();
  // digit by digit and warp by warp: positions in the tile
  uint32_t cnt = 0;
#pragma unroll
  for (int w = 0; w < RS_WARPS; ++w) cnt += warp_cnt[w][dg];
  uint32_t run = block_excl_scan(cnt, sm, &tot);
  delta[dg] = mine - run;
#pragma unroll
  for (int w = 0; w < RS_WARPS; ++w) {
    const uint32_t c = warp_cnt[w][dg];
    warp_cnt[w][dg] = run;
    run += c;
  }
  __syncthreads();
#pragma unroll
  for (int st = 0; st < RS_STEPS; ++st) {
    if (base + st * 32 + lane < n) {
      const uint32_t at = warp_cnt[warp][(uint32_t)(k[st] >> shift) & 0xFFu] + pos[st];
      stage[at] = k[st];
      if (HAS_VALS) stage_v[at] = v[st];
    }
  }
  __syncthreads();
  const uint32_t valid_n = (uint32_t)(n - tile0 < RS_TILE ? n - tile0 : RS_TILE);
  for (uint32_t i = threadIdx.x; i < valid_n; i += RS_THREADS) {
    const uint64_t key = stage[i];
    const uint32_t out = delta[(uint32_t)(key >> shift) & 0xFFu] + i;
    keys_out[out] = key;
    if (HAS_VALS) vals_out[out] = stage_v[i];
  }
}
}  // namespace

size_t sort_temp_bytes(uint32_t n) {
  size_t tiles = ((size_t)n + RS_TILE - 1) / RS_TILE;
  if (tiles == 0) tiles = 1;
  return (tiles * RADIX + RADIX) * sizeof(uint32_t);
}

// Up to SMALL_SORT keys without values: one block sorts them with a bitonic
// network, in one launch instead of two or three per radix digit.  Without
// values the order of equal keys does not show, so the result is the radix
// sort's.  A thread holds 8 consecutive keys: strides below 8 are exchanged in
// its registers, strides below 256 by shuffles, and only longer ones (15 of the
// 91 steps of 8192 keys) go through shared memory, in two buffers taken in turn
// so that a step has one barrier.  4950 keys: 20 us; 50 with every step in
// shared memory.
constexpr int SMALL_KEYS = 8;

__global__ void __launch_bounds__(SMALL_SORT / SMALL_KEYS) sort_small_kernel(uint64_t* __restrict__ keys, uint32_t n) {
  extern __shared__ uint64_t sbuf[];
  const uint32_t T = blockDim.x, t = threadIdx.x, n2 = T * SMALL_KEYS;
  uint64_t k[SMALL_KEYS];
#pragma unroll
  for (int e = 0; e < SMALL_KEYS; ++e) {  // any assignment will do before the first step: the coalesced one
    const uint32_t i = e * T + t;
    k[e] = i < n ? keys[i] : ~0ull;
  }
  uint64_t* buf = sbuf;
  for (uint32_t size = 2; size <= n2; size <<= 1) {
    for (uint32_t stride = size >> 1; stride >= SMALL_KEYS; stride >>= 1) {
      const uint32_t far = stride / SMALL_KEYS;  // distance in threads; size > stride: one direction a thread
      const bool low = (((t * SMALL_KEYS) & stride) == 0) == (((t * SMALL_KEYS) & size) == 0);
      if (far < 32) {
#pragma unroll
        for (int e = 0; e < SMALL_KEYS; ++e) {
          const uint64_t o = __shfl_xor_sync(0xffffffffu, k[e], far);
          k[e] = (o < k[e]) == low ? o : k[e];
        }
      } else {
#pragma unroll
        for (int e = 0; e < SMALL_KEYS; ++e) buf[e * T + t] = k[e];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < SMALL_KEYS; ++e) {
          const uint64_t o = buf[e * T + (t ^ far)];
          k[e] = (o < k[e]) == low ? o : k[e];
        }
        buf = buf == sbuf ? sbuf + n2 : sbuf;
      }
    }
#pragma unroll
    for (int stride = SMALL_KEYS / 2; stride > 0; stride >>= 1) {
      if ((uint32_t)stride < size) {
#pragma unroll
        for (int e = 0; e < SMALL_KEYS; ++e) {
          if ((e & stride) == 0) {
            const uint64_t x = k[e], y = k[e | stride];
            const bool swap = (x > y) == (((t * SMALL_KEYS + e) & size) == 0);
            k[e] = swap ? y : x;
            k[e | stride] = swap ? x : y;
          }
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < SMALL_KEYS; ++e) {
    const uint32_t i = t * SMALL_KEYS + e;
    if (i < n) keys[i] = k[e];
  }
}

cudaError_t radix_sort_u64(uint64_t* keys, uint64_t* keys_alt, uint32_t* vals, uint32_t* vals_alt, uint32_t n,
                           int low_bit, int key_bits, void* tmp, size_t tmp_bytes, bool* result_in_alt, cudaStream_t s) {
  *result_in_alt = false;
  if (n <= 1 || key_bits <= low_bit) return cudaSuccess;
  if (!vals && n <= SMALL_SORT) {
    uint32_t threads = 32;
    while (threads * SMALL_KEYS < n) threads <<= 1;
    const size_t smem = threads > 32 ? (size_t)threads * SMALL_KEYS * 16 : 0;
    if (smem > 48 * 1024) {
      static std::atomic<bool> opted[64];  // once per device (any thread)
      int dev = 0;
      cudaError_t e = cudaGetDevice(&dev);
      if (e != cudaSuccess) return e;
      if (dev < 0 || dev >= 64 || !opted[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(sort_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(SMALL_SORT * 16));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) opted[dev].store(true, std::memory_order_release);
      }
    }
    sort_small_kernel<<<1, threads, smem, s>>>(keys, n);
    note_launch();
    return cudaGetLastError();
  }
  uint32_t tiles = (uint32_t)(((size_t)n + RS_TILE - 1) / RS_TILE);
  if (tmp_bytes < sort_temp_bytes(n)) return cudaErrorInvalidValue;
  uint32_t* hist = (uint32_t*)tmp;
  uint32_t* totals = hist + (size_t)tiles * RADIX;
  uint64_t* kin = keys;
  uint64_t* kout = keys_alt;
  uint32_t* vin = vals;
  uint32_t* vout = vals_alt;
  bool alt = false;
  const bool direct = tiles <= RS_DIRECT_TILES;
  for (int shift = low_bit; shift < key_bits; shift += 8) {
    rs_hist_kernel<<<tiles, RS_THREADS, 0, s>>>(kin, n, shift, hist, direct ? 1 : tiles, direct ? RADIX : 1);
    note_launch();
    if (direct) {
      if (vals)
        rs_scatter_kernel<true, true><<<tiles, RS_THREADS, 0, s>>>(kin, kout, vin, vout, n, shift, hist, tiles, totals);
      else
        rs_scatter_kernel<false, true><<<tiles, RS_THREADS, 0, s>>>(kin, kout, nullptr, nullptr, n, shift, hist, tiles,
                                                                    totals);
    } else {
      rs_tile_scan_kernel<<<RADIX, 256, 0, s>>>(hist, tiles, totals);
      note_launch();
      if (vals)
        rs_scatter_kernel<true, false><<<tiles, RS_THREADS, 0, s>>>(kin, kout, vin, vout, n, shift, hist, tiles, totals);
      else
        rs_scatter_kernel<false, false><<<tiles, RS_THREADS, 0, s>>>(kin, kout, nullptr, nullptr, n, shift, hist, tiles,
                                                                     totals);
    }
    note_launch();
    uint64_t* t = kin;
    kin = kout;
    kout = t;
    uint32_t* tv = vin;
    vin = vout;
    vout = tv;
    alt = !alt;
  }
  *result_in_alt = alt;
  return cudaGetLastError();
}

}  // namespace rips
