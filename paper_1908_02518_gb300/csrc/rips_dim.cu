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

#include "rips_dim.cuh"
#include "rips_wide_types.cuh"

namespace rips {

// ====================================================================== enumeration

// A warp takes a (d-1)-simplex and 32 candidates of its shortest neighbour list at
// a time, and gathers what it finds in shared memory, up to ENUM_BUF simplices
// that take their place in the list with one atomic.  All warps share that one
// counter: an atomic for every 32 candidates bound the kernel (3-sphere of 144
// points, 13.9 million simplices: 0.50 -> 0.26 ms; 2,048 rotations, 2.2 million
// triangles: 0.147 -> 0.071; 4,096, 17.5 million: 0.96 -> 0.37).
// D = d keeps the vertices in registers and issues a candidate's rank lookups
// together; 0: any d.
constexpr int ENUM_BUF = 128;

template <int D>
__global__ void __launch_bounds__(256) enumerate_kernel(DimArgs a, const uint64_t* __restrict__ pidx,
                                                        const uint32_t* __restrict__ prank, uint32_t np, int pbits,
                                                        uint64_t* __restrict__ out_idx, uint32_t* __restrict__ out_rank,
                                                        unsigned long long* __restrict__ count,
                                                        unsigned long long cap) {
  extern __shared__ uint64_t smem[];
  __shared__ uint64_t buf_idx[WARPS_PER_BLOCK][ENUM_BUF];
  __shared__ uint32_t buf_rank[WARPS_PER_BLOCK][ENUM_BUF];
  Binom B = stage_binom(a, smem);
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int d = D ? D : a.d;  // new simplices are d-simplices, made from (d-1)-simplices
  constexpr int NV = D ? D : MAX_DIM + 2;
  uint64_t* const bi = buf_idx[threadIdx.x >> 5];
  uint32_t* const br = buf_rank[threadIdx.x >> 5];
  int held = 0;  // simplices in the warp's buffer
  auto flush = [&]() {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(count, (unsigned long long)held);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int i = lane; i < held; i += 32)
      if (base + i < cap) {
        out_idx[base + i] = bi[i];
        out_rank[base + i] = br[i];
      }
    __syncwarp();
    held = 0;
  };
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < np; s += warps) {
    const uint64_t g = pidx[s];
    const uint32_t cl = high_part(g, pbits);
    const uint64_t local = g & low_mask(pbits);
    const CV cv = cloud_view(a, cl);
    const uint64_t chi = a.col_bits >= 64 ? 0ull : ((uint64_t)cl << a.col_bits);
    int v[NV];
    int hi = cv.n - 1;
    uint64_t N = local;
    uint32_t beg = 0, end = ~0u;  // the shortest list of a vertex
#pragma unroll
    for (int l = 0; l < NV; ++l)
      if (l < d) {
        const int k = d - l;
        v[l] = k == 1 ? (int)N : max_vertex(B, k, hi, N);
        N -= k == 1 ? N : B(v[l], k);
        hi = v[l] - 1;
        const uint32_t o0 = cv.off[v[l]], o1 = cv.off[v[l] + 1];
        if (o1 - o0 < end - beg) {
          beg = o0;
          end = o1;
        }
      }
    const uint32_t r0 = prank[s];
    const int top = v[0];
    for (uint32_t q0 = beg; q0 < end; q0 += 32) {
      const uint32_t q = q0 + lane;
      const int j = q < end ? (int)cv.nbr[q] : -1;
      bool ok = j > top;
      uint32_t r = r0;
      if (ok) {
        if (D && cv.R) {
#pragma unroll
          for (int l = 0; l < NV; ++l) r = max(r, cv.R[(size_t)v[l] * cv.n + j]);
          ok = r != RANK_INF;
        } else {
          for (int l = 0; l < d; ++l) {
            uint32_t x = RANK_INF;
#pragma unroll
            for (int y = 0; y < NV; ++y)
              if (y == l) x = rank_of(cv, v[y], j);
            if (x == RANK_INF) {
              ok = false;
              break;
            }
            r = max(r, x);
          }
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, ok);
      if (m) {
        if (held + __popc(m) > ENUM_BUF) flush();
        if (ok) {
          const int at = held + __popc(m & lt);
          bi[at] = chi | (local + B(j, d + 1));
          br[at] = r;
        }
        held += __popc(m);
      }
      if (!__all_sync(0xffffffffu, j > top)) break;  // the list went below the top vertex
    }
  }
  if (held) flush();
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

// bars of this dimension and the statistics
__global__ void readout_kernel(DimArgs a, RedState s, const float* __restrict__ rank_value,
                               rips_bar_t* __restrict__ bars, uint32_t* __restrict__ nbars, uint32_t bar_cap,
                               unsigned long long* __restrict__ stats, int st_stride) {
  if (*s.err) return;  // the reduction did not end: no pivots to read, and the call fails or starts it over
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

static cudaError_t prepare(const void* kernel, size_t smem) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> g(g_prep_mu);
  for (const PreparedKernel& pk : g_prepared)
    if (pk.fn == kernel && pk.device == dev && pk.smem >= smem) return cudaSuccess;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  if (smem + fa.sharedSizeBytes > 48 * 1024)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) g_prepared.push_back(PreparedKernel{kernel, dev, smem});
  return e;
}

cudaError_t launch_enumerate(const DimArgs& a, const uint64_t* pidx, const uint32_t* prank, uint32_t np,
                             int prev_col_bits, uint64_t* out_idx, uint32_t* out_rank, unsigned long long* count,
                             unsigned long long cap, cudaStream_t st) {
  if (np == 0) return cudaSuccess;
  size_t sm = binom_smem(a);
  const void* kernel = a.d == 2 ? (const void*)enumerate_kernel<2>
                       : a.d == 3 ? (const void*)enumerate_kernel<3> : (const void*)enumerate_kernel<0>;
  cudaError_t e = prepare(kernel, sm);
  if (e != cudaSuccess) return e;
  DimArgs aa = a;
  void* args[] = {&aa, &pidx, &prank, &np, &prev_col_bits, &out_idx, &out_rank, &count, &cap};
  e = cudaLaunchKernel(kernel, dim3(grid_for_warps(np, a.scan_blocks_per_sm)), dim3(256), args, sm, st);
  note_launch();
  return e;
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

// rips_reduce_d*.cu
const void* reduce_kernel_d0();
const void* reduce_kernel_d1();
const void* reduce_kernel_d2();
const void* reduce_kernel_d3();

static const void* reduce_kernel(int d) {
  return d == 1 ? reduce_kernel_d1() : d == 2 ? reduce_kernel_d2() : d == 3 ? reduce_kernel_d3() : reduce_kernel_d0();
}

size_t wide_ctx_bytes(int blocks) { return (size_t)blocks * sizeof(WideCtx); }

int reduction_blocks(const DimArgs& a, uint32_t ncols) {
  const size_t sm = binom_smem(a);
  const void* kernel = reduce_kernel(a.d);
  if (prepare(kernel, sm) != cudaSuccess) return -1;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, sm) != cudaSuccess)
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
  const void* kernel = reduce_kernel(a.d);
  cudaError_t e = prepare(kernel, sm);
  if (e != cudaSuccess) return e;
  DimArgs aa = a;
  RedState ss = s;
  void* args[] = {&aa, &ss, &ctl};
  e = cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(256), args, sm, st);
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
