// a1 position preparation and a2 counting sort of particles by cell tile.
//
// a1 (Sec. 2.3, s = (x_j - x)/H): an FP64 position is wrapped into [0, L) (periodic box) and split
// into the integer cell c = floor(x/H) and the offset f = x/H - c in [0, 1), stored as FP32.
// a2: particles are grouped by tile of T^3 cells with a counting sort (histogram, exclusive scan,
// scatter), and inside a tile by half-cell slab along x (key tile * 2T + 2 (c_x mod T) + [f_x >= 1/2]),
// which keeps neighbouring cells' particles together in a staged piece; the assignment itself
// accepts any order inside a tile.
// Histogram and scatter use warp-aggregated atomics: consecutive particles of a spatially ordered
// catalogue share a key, and one atomic per distinct key per warp replaces 32. Particles are
// validated on the way (an invalid record is reported and binned as cell 0, offset 0).
#include "internal.cuh"
#include "position.cuh"

namespace pk {

PK_ERR_ACCESSOR(take_err_prepare)

__global__ void k_prepare(const double* __restrict__ pos, int64_t n, int ng, double box, int vec, pk_cellpos* __restrict__ out) {
  const double scale = double(ng) / box;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    bool bad;
    store_rec(out + i, prepare_one(pos + 3 * i, ng, box, scale, &bad), vec);
    if (bad) raise_err(PK_DERR_NONFINITE);
  }
}

// Sort key of a (validated) particle: tile and half-cell slab along x.
__device__ __forceinline__ int bin_key(const pk_cellpos& r, int ntile) {
  const int cx = cell_x(r.cell), tx = cx / kTileCells, ty = cell_y(r.cell) / kTileCells, tz = cell_z(r.cell) / kTileCells;
  const int slab = 2 * (cx - tx * kTileCells) + (r.fx >= 0.5f ? 1 : 0);
  return ((tx * ntile + ty) * ntile + tz) * kSlabs + slab;
}

// Validates a packed particle (coordinates < N, offsets in [0,1)); invalid ones are reported and
// mapped to cell 0 so that every later index stays in bounds.
__device__ __forceinline__ pk_cellpos checked(pk_cellpos r, int ng) {
  const bool ok = cell_x(r.cell) < ng && cell_y(r.cell) < ng && cell_z(r.cell) < ng && (r.cell >> 30) == 0 &&
                  r.fx >= 0.0f && r.fx < 1.0f && r.fy >= 0.0f && r.fy < 1.0f && r.fz >= 0.0f && r.fz < 1.0f;
  if (!ok) {
    raise_err(PK_DERR_CELLRANGE);
    r.cell = 0;
    r.fx = r.fy = r.fz = 0.0f;
  }
  return r;
}

// Warp-aggregated increment of ctr[key]; returns the value this lane would have seen alone.
__device__ __forceinline__ unsigned long long agg_inc(unsigned long long* ctr, int key, unsigned active) {
  const unsigned peers = __match_any_sync(active, key);
  const int leader = __ffs(peers) - 1;
  const int lane = threadIdx.x & 31;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(ctr + key, (unsigned long long)__popc(peers));
  base = __shfl_sync(peers, base, leader);
  return base + __popc(peers & ((1u << lane) - 1u));
}

// The counting pass: each record's place among those of its key (the counter's value before it) goes to rank, so the
// placing pass needs no second atomic, and no key match of the warp: it was bound by the latency of both. h:
// the half-cell shift applied to the records on the way (shift_rec; 0: none).
__global__ void k_tile_hist(const pk_cellpos* __restrict__ p, int64_t n, int ng, int ntile, int h, int vec,
                            unsigned long long* __restrict__ counts, uint32_t* __restrict__ rank) {
  const int64_t stride = gstride();
  const int64_t nround = (n + 31) / 32 * 32;
  for (int64_t i = gtid(); i < nround; i += stride) {
    const bool live = i < n;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (live) {
      pk_cellpos r = load_rec(p + i, vec);
      if (h) r = shift_rec(r, h, ng);
      const unsigned long long k = agg_inc(counts, bin_key(checked(r, ng), ntile), active);
      if (rank) rank[i] = uint32_t(k);
    }
  }
}

// The placing pass: record i goes to the start of its key plus its rank. Without ranks (more than 2^32 - 1 records)
// the place comes from the cursors (cleared by the caller). Four records per thread, loaded before any
// is used. 256^3 particles on N = 256: 153 us before (four 4-byte accesses per record and a second
// atomic), now 99 us (604 MB at 6.1 TB/s).
constexpr int kPlace = 4;
__global__ void __launch_bounds__(256) k_tile_scatter(const pk_cellpos* __restrict__ p, const float* __restrict__ w, int64_t n,
                                                      int ng, int ntile, int h, int vec, const int64_t* __restrict__ sub,
                                                      const uint32_t* __restrict__ rank,
                                                      unsigned long long* __restrict__ cursor, pk_cellpos* __restrict__ out,
                                                      float* __restrict__ wout) {
  if (rank) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x * kPlace;
    for (int64_t i0 = int64_t(blockIdx.x) * blockDim.x * kPlace + threadIdx.x; i0 < n; i0 += stride) {
      pk_cellpos r[kPlace];
      uint32_t q[kPlace];
      float wi[kPlace];
#pragma unroll
      for (int u = 0; u < kPlace; ++u) {
        const int64_t i = i0 + int64_t(u) * blockDim.x;
        if (i < n) {
          r[u] = load_rec(p + i, vec);
          q[u] = rank[i];
          if (wout) wi[u] = w[i];
        }
      }
      int64_t dst[kPlace];
#pragma unroll
      for (int u = 0; u < kPlace; ++u)
        if (i0 + int64_t(u) * blockDim.x < n) {
          if (h) r[u] = shift_rec(r[u], h, ng);
          r[u] = checked(r[u], ng);
          dst[u] = sub[bin_key(r[u], ntile)] + int64_t(q[u]);
        }
#pragma unroll
      for (int u = 0; u < kPlace; ++u)
        if (i0 + int64_t(u) * blockDim.x < n) {
          store_rec(out + dst[u], r[u], vec);
          if (wout) wout[dst[u]] = wi[u];
        }
    }
    return;
  }
  const int64_t stride = gstride();
  const int64_t nround = (n + 31) / 32 * 32;
  for (int64_t i = gtid(); i < nround; i += stride) {
    const bool live = i < n;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (live) {
      pk_cellpos r = load_rec(p + i, vec);
      if (h) r = shift_rec(r, h, ng);
      r = checked(r, ng);
      const int key = bin_key(r, ntile);
      const int64_t dst = sub[key] + int64_t(agg_inc(cursor, key, active));
      store_rec(out + dst, r, vec);
      if (wout) wout[dst] = w[i];
    }
  }
}

// a1 and the counting pass of a2 in one sweep over FP64 positions pos[0 .. cnt) in pinned host memory read over
// the CPU-GPU link: each particle is prepared, written to out[i0 + k]
// and its sort key counted. A block stages its 256 particles' 6 KB of coordinates in shared memory
// with 16-byte loads (when pos is 16-byte aligned), so every byte crosses the link once, in full lines.
constexpr int kPrepBlock = 256;
__global__ void __launch_bounds__(kPrepBlock) k_prepare_hist_host(const double* __restrict__ pos, int64_t i0, int64_t cnt, int ng,
                                                             double box, int ntile, int vec, pk_cellpos* __restrict__ out,
                                                             unsigned long long* __restrict__ counts,
                                                             uint32_t* __restrict__ rank) {
  __shared__ double2 s_pos[kPrepBlock * 3 / 2];
  double* sp = reinterpret_cast<double*>(s_pos);
  const double scale = double(ng) / box;
  for (int64_t base = int64_t(blockIdx.x) * kPrepBlock; base < cnt; base += int64_t(gridDim.x) * kPrepBlock) {
    const int m = int(min(int64_t(kPrepBlock), cnt - base));
    const double* src = pos + 3 * base;
    if (vec) {
      const int nv = (3 * m) / 2;
      for (int v = threadIdx.x; v < nv; v += kPrepBlock) s_pos[v] = reinterpret_cast<const double2*>(src)[v];
      if (((3 * m) & 1) && threadIdx.x == 0) sp[3 * m - 1] = src[3 * m - 1];
    } else {
      for (int v = threadIdx.x; v < 3 * m; v += kPrepBlock) sp[v] = src[v];
    }
    __syncthreads();
    const int k = threadIdx.x;
    const bool live = k < m;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (live) {
      bool bad;
      const pk_cellpos r = prepare_one(sp + 3 * k, ng, box, scale, &bad);
      if (bad) raise_err(PK_DERR_NONFINITE);
      store_rec(out + i0 + base + k, r, true);  // out: the workspace's records, 256-byte aligned
      const unsigned long long q = agg_inc(counts, bin_key(r, ntile), active);
      if (rank) rank[i0 + base + k] = uint32_t(q);
    }
    __syncthreads();
  }
}

// The same from device memory: a thread loads its particle's three coordinates itself (every sector of the warp's 768
// bytes is used, and L1 serves the second and third load), without the staging's shared memory and barriers.
__global__ void __launch_bounds__(kPrepBlock) k_prepare_hist(const double* __restrict__ pos, int64_t i0, int64_t cnt, int ng,
                                                             double box, int ntile, pk_cellpos* __restrict__ out,
                                                             unsigned long long* __restrict__ counts,
                                                             uint32_t* __restrict__ rank) {
  const double scale = double(ng) / box;
  const int64_t nround = (cnt + 31) / 32 * 32;
  for (int64_t k = gtid(); k < nround; k += gstride()) {
    const bool live = k < cnt;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (live) {
      const double x[3] = {__ldg(pos + 3 * k), __ldg(pos + 3 * k + 1), __ldg(pos + 3 * k + 2)};
      bool bad;
      const pk_cellpos r = prepare_one(x, ng, box, scale, &bad);
      if (bad) raise_err(PK_DERR_NONFINITE);
      store_rec(out + i0 + k, r, true);  // out: the workspace's records, 256-byte aligned
      const unsigned long long q = agg_inc(counts, bin_key(r, ntile), active);
      if (rank) rank[i0 + k] = uint32_t(q);
    }
  }
}

// Tile offsets from the slab offsets: offsets[t] = sub[t * kSlabs], t = 0 .. ntiles.
__global__ void k_tile_offsets(const int64_t* __restrict__ sub, int64_t ntiles, int64_t* __restrict__ offsets) {
  for (int64_t t = gtid(); t <= ntiles; t += gstride()) offsets[t] = sub[t * kSlabs];
}

// Batched binning: blockIdx.y = catalogue c of the group, particles r.off[c] .. r.off[c+1]-1 of p,
// key c * ntiles + tile. Sorted output indices count from the group's first particle.
__global__ void k_tile_hist_batch(const pk_cellpos* __restrict__ p, CatRanges r, int ntile, int vec,
                                  unsigned long long* __restrict__ counts) {
  const int c = blockIdx.y;
  const int64_t beg = r.off[c], cnt = r.off[c + 1] - beg;
  const int base = c * ntile * ntile * ntile * kSlabs;
  const int64_t nround = (cnt + 31) / 32 * 32;
  for (int64_t k = gtid(); k < nround; k += gstride()) {
    const bool live = k < cnt;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (live) agg_inc(counts, base + bin_key(checked(load_rec(p + beg + k, vec), r.ng), ntile), active);
  }
}

__global__ void k_tile_scatter_batch(const pk_cellpos* __restrict__ p, CatRanges r, int ntile, int vec,
                                     const int64_t* __restrict__ sub, unsigned long long* __restrict__ cursor,
                                     pk_cellpos* __restrict__ out) {
  const int c = blockIdx.y;
  const int64_t beg = r.off[c], cnt = r.off[c + 1] - beg;
  const int base = c * ntile * ntile * ntile * kSlabs;
  const int64_t nround = (cnt + 31) / 32 * 32;
  for (int64_t k = gtid(); k < nround; k += gstride()) {
    const bool live = k < cnt;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (live) {
      const pk_cellpos rec = checked(load_rec(p + beg + k, vec), r.ng);
      const int key = base + bin_key(rec, ntile);
      store_rec(out + sub[key] + int64_t(agg_inc(cursor, key, active)), rec, true);
    }
  }
}

// Batched binning by tile with shared-memory histograms. Block (x, c) takes particles
// [off[c] + x kBinChunk, ..) of catalogue c: it counts their tiles in shared memory, then adds one
// count per non-empty tile to the global counters (count pass), or reserves one range per non-empty
// tile with a global atomic and places its particles there through shared-memory cursors (place
// pass). Output indices count from the group's first particle, as k_tile_scatter_batch's.
constexpr int kBinChunk = 16384;

__device__ __forceinline__ int tile_of(const pk_cellpos& r, int ntile) {
  return ((cell_x(r.cell) / kTileCells) * ntile + cell_y(r.cell) / kTileCells) * ntile + cell_z(r.cell) / kTileCells;
}

// Records per thread and round of the chunk loops: their loads are issued together, so each thread
// keeps several in flight (one at a time left the kernels waiting on memory at 8 % issue).
constexpr int kBinUnroll = 4;
// The placing pass runs one block of 1024 threads per SM (its shared memory is asked for to that end): 152 chunks of
// 256 KB in flight then fit L2, where the partly written sectors of the chunks' tile runs (some four records
// each) wait for their other half. With four blocks of 512 per SM and 512 KB chunks they were evicted half
// written, and each cost a read and a second write of DRAM. 96 mocks (6e7 particles): 1.81 ms, now
// 0.94 (chunks of 24 K records 1.05, 32 K 1.12, 64 K 1.28). Whole calls, four blocks of 512 against one of 1024: 4 catalogues
// of 5e6 1572 -> 1463 us, 8 of 2e6 1509 -> 1395, 128 of 1e5 1839 -> 1794; small catalogues do not fill L2 either
// way: 512 of 3000 on N = 32 754 and 759 us, 512 of 1000 on N = 16 181 and 184.
constexpr int kPlaceThreads = 1024;
constexpr size_t kPlaceSmem = 120 * 1024;

__global__ void k_tile_count_smem(const pk_cellpos* __restrict__ p, CatRanges r, int ntile, int vec,
                                  unsigned long long* __restrict__ counts) {
  extern __shared__ int s_cnt[];  // [ntiles]
  const int c = blockIdx.y, ntiles = ntile * ntile * ntile;
  const int64_t beg = r.off[c] + int64_t(blockIdx.x) * kBinChunk, end = min(r.off[c + 1], beg + kBinChunk);
  if (beg >= end) return;
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x) s_cnt[t] = 0;
  __syncthreads();
  for (int64_t i0 = beg + threadIdx.x; i0 < end; i0 += int64_t(kBinUnroll) * blockDim.x) {
    pk_cellpos rec[kBinUnroll];
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u) {
      const int64_t i = i0 + int64_t(u) * blockDim.x;
      if (i < end) rec[u] = load_rec(p + i, vec);
    }
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u)
      if (i0 + int64_t(u) * blockDim.x < end) atomicAdd(&s_cnt[tile_of(checked(rec[u], r.ng), ntile)], 1);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x)
    if (s_cnt[t]) atomicAdd(&counts[int64_t(c) * ntiles + t], (unsigned long long)s_cnt[t]);
}

__global__ void __launch_bounds__(kPlaceThreads, 1) k_tile_place_smem(const pk_cellpos* __restrict__ p, CatRanges r, int ntile, int vec, const int64_t* __restrict__ offsets,
                                  unsigned long long* __restrict__ cursor, pk_cellpos* __restrict__ out) {
  extern __shared__ long long s_base[];  // [ntiles] range start, then int cursors [ntiles]
  const int c = blockIdx.y, ntiles = ntile * ntile * ntile;
  int* s_cnt = reinterpret_cast<int*>(s_base + ntiles);
  const int64_t beg = r.off[c] + int64_t(blockIdx.x) * kBinChunk, end = min(r.off[c + 1], beg + kBinChunk);
  if (beg >= end) return;
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x) s_cnt[t] = 0;
  __syncthreads();
  for (int64_t i0 = beg + threadIdx.x; i0 < end; i0 += int64_t(kBinUnroll) * blockDim.x) {
    pk_cellpos rec[kBinUnroll];
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u) {
      const int64_t i = i0 + int64_t(u) * blockDim.x;
      if (i < end) rec[u] = load_rec(p + i, vec);
    }
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u)
      if (i0 + int64_t(u) * blockDim.x < end) atomicAdd(&s_cnt[tile_of(checked(rec[u], r.ng), ntile)], 1);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
    const int k = s_cnt[t];
    if (k) {
      const int64_t key = int64_t(c) * ntiles + t;
      s_base[t] = offsets[key] + (long long)atomicAdd(&cursor[key], (unsigned long long)k);
    }
    s_cnt[t] = 0;
  }
  __syncthreads();
  for (int64_t i0 = beg + threadIdx.x; i0 < end; i0 += int64_t(kBinUnroll) * blockDim.x) {
    pk_cellpos rec[kBinUnroll];
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u) {
      const int64_t i = i0 + int64_t(u) * blockDim.x;
      if (i < end) rec[u] = load_rec_once(p + i, vec);
    }
    int64_t dst[kBinUnroll];
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u) {
      if (i0 + int64_t(u) * blockDim.x < end) {
        rec[u] = checked(rec[u], r.ng);
        const int t = tile_of(rec[u], ntile);
        dst[u] = s_base[t] + atomicAdd(&s_cnt[t], 1);
      }
    }
#pragma unroll
    for (int u = 0; u < kBinUnroll; ++u)
      if (i0 + int64_t(u) * blockDim.x < end) store_rec(out + dst[u], rec[u], true);
  }
}

// Binning of one catalogue by tile only, for the library's own assignment (which takes any order inside a tile):
// k_count_tiles counts a block's chunk of records in shared memory (F64: after preparing them from FP64
// positions, written to cells), one global addition per block and tile; k_scan_tiles turns the counts into
// tile offsets and cursors; k_place_tiles counts its chunk again, reserves a range of every tile with one
// global atomic and places the records through the reserved places in shared memory. No global atomic and
// no key match per record, sixteen times fewer keys than with slabs, and two scan launches less. 32-bit
// counts and places (n < 2^32); one counter per tile in shared memory: up to kTileSmemMax / 4 tiles (N <= 304).
// U: records whose loads a thread issues together. FP64 positions: one where two blocks fit an SM (counters of up to
// 108 KB), two otherwise (256^3 particles on N = 256: 179 us with one, 166 with two; 5e6 on N = 180: 49 and 55).
constexpr int kTileThreads = 1024;
template <bool F64, int U>
__global__ void __launch_bounds__(kTileThreads, F64 && U > 1 ? 1 : 2) k_count_tiles(const void* __restrict__ src, int64_t n, int64_t chunk, int ng,
                                                                 double box, int ntile, int h, int vec,
                                                                 pk_cellpos* __restrict__ cells, uint16_t* __restrict__ tile,
                                                                 unsigned* __restrict__ counts) {
  extern __shared__ unsigned s_tile[];  // [ntiles]
  const int ntiles = ntile * ntile * ntile;
  const int64_t beg = int64_t(blockIdx.x) * chunk, end = min(n, beg + chunk);
  for (int t = threadIdx.x; t < ntiles; t += kTileThreads) s_tile[t] = 0u;
  __syncthreads();
  const double scale = double(ng) / box;
  for (int64_t i0 = beg + threadIdx.x; i0 < end; i0 += U * kTileThreads) {
    double x[F64 ? U : 1][3];
    pk_cellpos r[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * kTileThreads;
      if (i >= end) break;
      if constexpr (F64) {
        const double* p = static_cast<const double*>(src) + 3 * i;
        x[u][0] = __ldg(p);
        x[u][1] = __ldg(p + 1);
        x[u][2] = __ldg(p + 2);
      } else {
        r[u] = load_rec(static_cast<const pk_cellpos*>(src) + i, vec);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * kTileThreads;
      if (i >= end) break;
      if constexpr (F64) {
        bool bad;
        r[u] = prepare_one(x[u], ng, box, scale, &bad);
        if (bad) raise_err(PK_DERR_NONFINITE);
        store_rec(cells + i, r[u], true);
      } else {
        if (h) r[u] = shift_rec(r[u], h, ng);
        r[u] = checked(r[u], ng);
      }
      const int t = tile_of(r[u], ntile);
      tile[i] = uint16_t(t);
      atomicAdd(&s_tile[t], 1u);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ntiles; t += kTileThreads)
    if (s_tile[t]) atomicAdd(&counts[t], s_tile[t]);
}

// offsets[t] and cursor[t]: the records before tile t. A block scans 4096 tiles, four consecutive ones per thread (counts
// 16-byte aligned), after adding up all counts before them itself: at most 14 blocks, so the repeated
// sums are cheaper than a second launch.
constexpr int kScanTiles = 4096;
__global__ void __launch_bounds__(1024) k_scan_tiles(const unsigned* __restrict__ counts, int ntiles, int64_t* __restrict__ offsets,
                                                     unsigned* __restrict__ cursor) {
  __shared__ unsigned warp_sums[32], warp_before[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int base = int(blockIdx.x) * kScanTiles, t = base + 4 * int(threadIdx.x);
  unsigned before = 0;  // counts of the earlier blocks' tiles
  for (int q = 4 * int(threadIdx.x); q < base; q += kScanTiles) {
    const uint4 v = *reinterpret_cast<const uint4*>(counts + q);
    before += v.x + v.y + v.z + v.w;
  }
  unsigned c[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (t + k < ntiles) c[k] = counts[t + k];
  const unsigned sum = c[0] + c[1] + c[2] + c[3];
  unsigned x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
    before += __shfl_xor_sync(0xffffffffu, before, o);
  }
  if (lane == 31) {
    warp_sums[warp] = x;
    warp_before[warp] = before;
  }
  __syncthreads();
  unsigned v = warp_sums[lane];
  before = warp_before[lane];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
    before += __shfl_xor_sync(0xffffffffu, before, o);
  }
  unsigned at = before + x - sum;
  const unsigned warps_before = __shfl_sync(0xffffffffu, v, max(warp - 1, 0));
  if (warp > 0) at += warps_before;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (t + k < ntiles) {
      offsets[t + k] = int64_t(at);
      cursor[t + k] = at;
    }
    at += c[k];
    if (t + k == ntiles - 1) offsets[ntiles] = int64_t(at);
  }
}

// tile: the records' tiles from k_count_tiles (2 bytes read for the count instead of the record again; chunk a
// multiple of 4, so that four tiles are one aligned 8-byte load). trusted: the records were written by
// k_count_tiles<true, U>, valid already.
__global__ void __launch_bounds__(kTileThreads, 1) k_place_tiles(const pk_cellpos* __restrict__ p, const float* __restrict__ w,
                                                                 const uint16_t* __restrict__ tile, int64_t n, int64_t chunk,
                                                                 int ng, int ntiles, int h, int vec, int trusted,
                                                                 unsigned* __restrict__ cursor, pk_cellpos* __restrict__ out,
                                                                 float* __restrict__ wout) {
  extern __shared__ unsigned s_tile[];  // [ntiles]: counts, then the next place of each tile
  const int64_t beg = int64_t(blockIdx.x) * chunk, end = min(n, beg + chunk);
  constexpr int U = 4;  // records in flight per thread
  for (int t = threadIdx.x; t < ntiles; t += kTileThreads) s_tile[t] = 0u;
  __syncthreads();
  for (int64_t i = beg + 4 * int64_t(threadIdx.x); i < end; i += 4 * kTileThreads) {
    if (i + 4 <= end) {
      const ushort4 t = *reinterpret_cast<const ushort4*>(tile + i);
      atomicAdd(&s_tile[t.x], 1u);
      atomicAdd(&s_tile[t.y], 1u);
      atomicAdd(&s_tile[t.z], 1u);
      atomicAdd(&s_tile[t.w], 1u);
    } else {
      for (int64_t q = i; q < end; ++q) atomicAdd(&s_tile[tile[q]], 1u);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ntiles; t += kTileThreads) {
    const unsigned k = s_tile[t];
    if (k) s_tile[t] = atomicAdd(&cursor[t], k);
  }
  __syncthreads();
  for (int64_t i0 = beg + threadIdx.x; i0 < end; i0 += int64_t(U) * kTileThreads) {
    pk_cellpos r[U];
    float wi[U];
    unsigned dst[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * kTileThreads < end) {
        r[u] = load_rec(p + i0 + u * kTileThreads, vec);
        dst[u] = tile[i0 + u * kTileThreads];
        if (wout) wi[u] = w[i0 + u * kTileThreads];
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * kTileThreads < end) dst[u] = atomicAdd(&s_tile[dst[u]], 1u);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * kTileThreads < end) {
        if (h) r[u] = shift_rec(r[u], h, ng);
        store_rec(out + dst[u], trusted ? r[u] : checked(r[u], ng), true);
        if (wout) wout[dst[u]] = wi[u];
      }
  }
}

// Exclusive scan of int64 counts, three phases over blocks of kScanBlock elements.
constexpr int kScanBlock = 1024;

__device__ __forceinline__ long long block_exclusive_scan(long long v, long long* total) {
  __shared__ long long warp_sums[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    long long s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane < nw) warp_sums[lane] = s;
  }
  __syncthreads();
  const long long before = wid > 0 ? warp_sums[wid - 1] : 0;
  if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before + x - v;
}

__global__ void k_scan_blocks(const unsigned long long* __restrict__ in, int64_t n, long long* __restrict__ block_sums) {
  const int64_t i = int64_t(blockIdx.x) * kScanBlock + threadIdx.x;
  long long v = i < n ? (long long)in[i] : 0;
  long long tot;
  block_exclusive_scan(v, &tot);
  if (threadIdx.x == 0) block_sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(long long* __restrict__ block_sums, int nblocks) {
  // one block: sequential chunks of kScanBlock
  long long carry = 0;
  for (int base = 0; base < nblocks; base += kScanBlock) {
    const int i = base + threadIdx.x;
    const long long v = i < nblocks ? block_sums[i] : 0;
    long long tot;
    const long long ex = block_exclusive_scan(v, &tot);
    if (i < nblocks) block_sums[i] = carry + ex;
    carry += tot;
    __syncthreads();
  }
}

__global__ void k_scan_apply(const unsigned long long* __restrict__ in, int64_t n, const long long* __restrict__ block_sums,
                             int64_t* __restrict__ out, int64_t total_slot) {
  const int64_t i = int64_t(blockIdx.x) * kScanBlock + threadIdx.x;
  const long long v = i < n ? (long long)in[i] : 0;
  const long long ex = block_exclusive_scan(v, nullptr);
  if (i < n) out[i] = block_sums[blockIdx.x] + ex;
  if (i == n - 1) out[total_slot] = block_sums[blockIdx.x] + ex + v;
}

// ---- host launchers -----------------------------------------------------------------------------

static int aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 ? 1 : 0; }

cudaError_t launch_prepare(const double* pos, int64_t n, int ng, double box, pk_cellpos* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int threads = 256;
  const int64_t blocks = std::min<int64_t>((n + threads - 1) / threads, int64_t(num_sms()) * 16);
  k_prepare<<<int(blocks), threads, 0, s>>>(pos, n, ng, box, aligned16(out), out); count_launch();
  return cudaGetLastError();
}

size_t scan_scratch_bytes(int64_t n) { return size_t((n + kScanBlock - 1) / kScanBlock) * sizeof(long long); }

cudaError_t launch_exclusive_scan(const unsigned long long* in, int64_t n, int64_t* out, long long* scratch, cudaStream_t s) {
  const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
  k_scan_blocks<<<int(nb), kScanBlock, 0, s>>>(in, n, scratch); count_launch();
  k_scan_sums<<<1, kScanBlock, 0, s>>>(scratch, int(nb)); count_launch();
  k_scan_apply<<<int(nb), kScanBlock, 0, s>>>(in, n, scratch, out, n); count_launch();
  return cudaGetLastError();
}

static cudaError_t launch_tile_offsets(const int64_t* sub, int64_t ntiles, int64_t* offsets, cudaStream_t s) {
  const int threads = 256;
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((ntiles + threads) / threads, int64_t(num_sms()) * 8));
  k_tile_offsets<<<int(blocks), threads, 0, s>>>(sub, ntiles, offsets); count_launch();
  return cudaGetLastError();
}

cudaError_t launch_prepare_hist(const double* pos, int64_t i0, int64_t cnt, int ng, double box, int ntile, pk_cellpos* cells,
                                unsigned long long* counts, uint32_t* rank, bool host, cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  const int64_t blocks = std::min<int64_t>((cnt + kPrepBlock - 1) / kPrepBlock, int64_t(num_sms()) * 16);
  if (host)
    k_prepare_hist_host<<<int(blocks), kPrepBlock, 0, s>>>(pos, i0, cnt, ng, box, ntile, aligned16(pos), cells, counts, rank);
  else
    k_prepare_hist<<<int(blocks), kPrepBlock, 0, s>>>(pos, i0, cnt, ng, box, ntile, cells, counts, rank);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_bin(const pk_cellpos* cells, const float* w, int64_t n, int ng, int ntile, int shift, pk_cellpos* sorted,
                       float* wsorted, int64_t* offsets, unsigned long long* counts, uint32_t* rank, int64_t* sub,
                       long long* scan_scratch, cudaStream_t s) {
  const int64_t nkeys = int64_t(ntile) * ntile * ntile * kSlabs;
  cudaError_t e = cudaMemsetAsync(counts, 0, size_t(nkeys) * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const int threads = 256;
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, int64_t(num_sms()) * 16));
  if (n > 0) {
    k_tile_hist<<<int(blocks), threads, 0, s>>>(cells, n, ng, ntile, shift, aligned16(cells), counts, rank); count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return launch_bin_finish(cells, w, n, ng, ntile, shift, sorted, wsorted, offsets, counts, rank, sub, scan_scratch, s);
}

cudaError_t launch_bin_finish(const pk_cellpos* cells, const float* w, int64_t n, int ng, int ntile, int shift, pk_cellpos* sorted,
                              float* wsorted, int64_t* offsets, unsigned long long* counts, const uint32_t* rank, int64_t* sub,
                              long long* scan_scratch, cudaStream_t s) {
  const int64_t ntiles = int64_t(ntile) * ntile * ntile, nkeys = ntiles * kSlabs;
  const int threads = 256;
  cudaError_t e;
  if ((e = launch_exclusive_scan(counts, nkeys, sub, scan_scratch, s)) != cudaSuccess) return e;
  if ((e = launch_tile_offsets(sub, ntiles, offsets, s)) != cudaSuccess) return e;
  if (n > 0) {
    if (!rank && (e = cudaMemsetAsync(counts, 0, size_t(nkeys) * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    const int64_t per = threads * (rank ? kPlace : 1);
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, int64_t(num_sms()) * 16));
    k_tile_scatter<<<int(blocks), threads, 0, s>>>(cells, w, n, ng, ntile, shift, aligned16(cells) & aligned16(sorted), sub, rank,
                                                   counts, sorted, wsorted); count_launch();
  }
  return cudaGetLastError();
}

// Shared memory of a block is at most 227 KB; the tiles' counters take 4 bytes each. The slab order keeps the pieces of a
// tile compact in the key-cell kernel, which matters to tiles of more than one piece (4608 records); the line at a mean
// population of 2048 keeps it where a uniform catalogue has such tiles. P(k) of PCS on N = 128, FP32, slabs against
// tiles alone: uniform catalogues 341 -> 254 us at a mean of 512, 822 -> 564 at 1900 (and 838 -> 623 at 2200, beyond
// the line); clumps of 10^5 particles within a cell or two 2166 -> 1177 at 512 (slabs crowd few key cells into a
// piece); but clumps spread over whole tiles (a Gaussian of 3.8 cells) 695 -> 786 at 512 and 982 -> 1092 at 1024. FIXED64
// gains on all of them (the last two 1388 -> 1134 and 1571 -> 1246).
constexpr size_t kTileSmemMax = 224 * 1024;
static_assert(kTileSmemMax / sizeof(unsigned) <= 65536, "tile numbers are kept in 16 bits between the passes");
bool bin_by_tile(int64_t n, int ntile) {
  const int64_t ntiles = int64_t(ntile) * ntile * ntile;
  return n > 0 && n <= int64_t(UINT32_MAX) && size_t(ntiles) * sizeof(unsigned) <= kTileSmemMax && n <= 2048 * ntiles;
}

cudaError_t launch_bin_tiles(const void* pos, int fmt, const float* w, int64_t n, int ng, double box, int ntile, int shift,
                             pk_cellpos* cells, pk_cellpos* sorted, float* wsorted, int64_t* offsets, unsigned* scratch,
                             uint16_t* tile, cudaStream_t s) {
  const int ntiles = ntile * ntile * ntile;
  unsigned *counts = scratch, *cursor = scratch + ntiles;
  const bool f64 = fmt == PK_POS_F64_XYZ;
  const size_t smem = size_t(ntiles) * sizeof(unsigned);
  // one block per SM in the placing pass (see kPlaceSmem)
  const size_t psmem = std::max(kPlaceSmem, smem);
  auto* count = !f64 ? k_count_tiles<false, 4> : smem <= 108 * 1024 ? k_count_tiles<true, 1> : k_count_tiles<true, 2>;
  cudaError_t e;
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(count), smem)) != cudaSuccess ||
      (e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_place_tiles), psmem)) != cudaSuccess ||
      (e = cudaMemsetAsync(counts, 0, smem, s)) != cudaSuccess)
    return e;
  // chunks of at most 32 K records in whole waves of one block per SM, at least 2048 records each
  const int64_t sms = num_sms(), waves = (n + sms * 32768 - 1) / (sms * 32768);
  const int64_t chunk = (std::max<int64_t>(2048, (n + sms * waves - 1) / (sms * waves)) + 3) / 4 * 4;
  const int blocks = int((n + chunk - 1) / chunk);
  count<<<blocks, kTileThreads, smem, s>>>(pos, n, chunk, ng, box, ntile, f64 ? 0 : shift, f64 ? 1 : aligned16(pos), cells, tile,
                                           counts);
  count_launch();
  k_scan_tiles<<<(ntiles + kScanTiles - 1) / kScanTiles, 1024, 0, s>>>(counts, ntiles, offsets, cursor); count_launch();
  const pk_cellpos* p = f64 ? cells : static_cast<const pk_cellpos*>(pos);
  k_place_tiles<<<blocks, kTileThreads, psmem, s>>>(p, w, tile, n, chunk, ng, ntiles, f64 ? 0 : shift, aligned16(p), f64 ? 1 : 0,
                                                    cursor, sorted, wsorted); count_launch();
  return cudaGetLastError();
}

cudaError_t launch_bin_batch_tiles(const pk_cellpos* p, const CatRanges& r, int ntile, pk_cellpos* sorted, int64_t* offsets,
                                   unsigned long long* counts, long long* scan_scratch, cudaStream_t s) {
  const int ntiles = ntile * ntile * ntile;
  const int64_t nkeys = int64_t(ntiles) * r.nb;
  cudaError_t e = cudaMemsetAsync(counts, 0, size_t(nkeys) * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  int64_t maxc = 1;
  for (int c = 0; c < r.nb; ++c) maxc = std::max<int64_t>(maxc, r.off[c + 1] - r.off[c]);
  const dim3 blocks(unsigned((maxc + kBinChunk - 1) / kBinChunk), unsigned(r.nb));
  const size_t smem_count = size_t(ntiles) * sizeof(int);
  const size_t smem_place = std::max(kPlaceSmem, size_t(ntiles) * (sizeof(long long) + sizeof(int)));
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_tile_count_smem), smem_count)) != cudaSuccess) return e;
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_tile_place_smem), smem_place)) != cudaSuccess) return e;
  k_tile_count_smem<<<blocks, 512, smem_count, s>>>(p, r, ntile, aligned16(p), counts); count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_exclusive_scan(counts, nkeys, offsets, scan_scratch, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(counts, 0, size_t(nkeys) * sizeof(unsigned long long), s)) != cudaSuccess) return e;
  k_tile_place_smem<<<blocks, kPlaceThreads, smem_place, s>>>(p, r, ntile, aligned16(p), offsets, counts, sorted); count_launch();
  return cudaGetLastError();
}

cudaError_t launch_bin_batch(const pk_cellpos* p, const CatRanges& r, int ng, int ntile, pk_cellpos* sorted, int64_t* offsets,
                             unsigned long long* counts, int64_t* sub, long long* scan_scratch, cudaStream_t s) {
  const int64_t ntiles = int64_t(ntile) * ntile * ntile * r.nb, nkeys = ntiles * kSlabs;
  cudaError_t e = cudaMemsetAsync(counts, 0, size_t(nkeys) * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  int64_t maxc = 1;
  for (int c = 0; c < r.nb; ++c) maxc = std::max<int64_t>(maxc, r.off[c + 1] - r.off[c]);
  const dim3 blocks(unsigned(std::max<int64_t>(1, std::min<int64_t>((maxc + 255) / 256, std::max(1, num_sms() * 16 / r.nb)))),
                    unsigned(r.nb));
  (void)ng;
  k_tile_hist_batch<<<blocks, 256, 0, s>>>(p, r, ntile, aligned16(p), counts); count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_exclusive_scan(counts, nkeys, sub, scan_scratch, s)) != cudaSuccess) return e;
  if ((e = launch_tile_offsets(sub, ntiles, offsets, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(counts, 0, size_t(nkeys) * sizeof(unsigned long long), s)) != cudaSuccess) return e;
  k_tile_scatter_batch<<<blocks, 256, 0, s>>>(p, r, ntile, aligned16(p), sub, counts, sorted); count_launch();
  return cudaGetLastError();
}

}  // namespace pk
