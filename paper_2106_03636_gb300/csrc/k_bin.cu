// k_bin.cu - ingest, per-row statistics, grid and the stable per-row sort.
//
// Steps A1-A4 of the hot path: clusters of a batch of Time Frames are
// decoded to integer (y, zeta), counted per (TF, sector, row), binned into a
// per-row grid of cells (cell = iz * ny + iy) and sorted by
// (TF, sector, row, cell, input index).  The sort is a two-level counting
// sort: tiles of the input scatter into row buckets at offsets from a
// per-(tile,row) prefix (no global atomics), then one CTA per row scatters
// its bucket into cells and restores input order inside each cell, so the
// result is the stable order whatever the atomic interleaving.
#include <algorithm>

#include "o2tpc_kernels.cuh"

namespace o2tpc {

// The stored words of a cluster, as loaded (so that a loop can have several
// clusters' loads in flight before it decodes the first).
struct RawCluster {
  uint32_t a, b, c;  // FIXED: the record; FLOAT: y, z or time, sector | row << 8
};
__device__ inline RawCluster load_raw(const TFDesc& t, int i) {
  RawCluster w;
  if (t.format == 1) {
    const uint32_t* rec = reinterpret_cast<const uint32_t*>(static_cast<const uint8_t*>(t.in0) + 12ll * i);
    w.a = __ldg(rec);
    w.b = __ldg(rec + 1);
    w.c = __ldg(rec + 2);
  } else {
    w.a = __float_as_uint(__ldg(t.y + i));
    w.b = __float_as_uint(t.z ? __ldg(t.z + i) : __ldg(t.time + i));
    w.c = (uint32_t)__ldg(static_cast<const uint8_t*>(t.in0) + i) |
          ((uint32_t)__ldg(static_cast<const uint8_t*>(t.in1) + i) << 8);
  }
  return w;
}

// Decodes a cluster of TF t.  Returns false (and sets the error word) for
// invalid content; the cluster is then filed under row 0 so that indices stay
// in bounds.
__device__ inline bool decode(const TFDesc& t, const RawCluster& w, const GeomConst* __restrict__ G, int& lr, int& yu,
                              int& zu) {
  int s, r;
  bool ok = true;
  if (t.format == 1) {
    ok = decode_fixed(w.a, w.b, w.c, G->npads, s, r, yu, zu);
  } else {
    s = (int)(w.c & 0xFFu);
    r = (int)((w.c >> 8) & 0xFFu);
    float yf = __uint_as_float(w.a), zf = __uint_as_float(w.b);
    if (s >= kNSec || r >= kNRow) { ok = false; s = 0; r = 0; }
    if (!isfinite(yf) || !isfinite(zf)) { ok = false; yf = 0.f; zf = 0.f; }
    float yq = rintf(__fmul_rn(yf, 160.0f));
    float zq;
    if (t.z) {
      const float d = (s < 18) ? __fsub_rn(250.0f, zf) : __fadd_rn(250.0f, zf);
      zq = rintf(__fmul_rn(d, G->kz));
    } else {
      zq = rintf(__fmul_rn(zf, 320.0f));  // drift time (us) -> 1/64 of a 200 ns bin
    }
    if (fabsf(yq) > 1048576.0f || fabsf(zq) > 1073741824.0f) { ok = false; yq = 0.f; zq = 0.f; }
    yu = (int)yq;
    zu = (int)zq;
  }
  lr = s * kNRow + r;
  return ok;
}

// K0: per tile, decode and accumulate per-row count / min / max in shared
// memory; write the tile's 5472-row statistics (SoA: count, zmin, zmax).
__global__ void __launch_bounds__(512) k_ingest_stats(const TFDesc* __restrict__ tfs, const int2* __restrict__ tiles,
                                                      int tileSize, const GeomConst* __restrict__ G,
                                                      int* __restrict__ tileStats, unsigned* __restrict__ err) {
  extern __shared__ int sm[];
  int* s_cnt = sm;
  int* s_min = sm + kRowsPerTF;
  int* s_max = sm + 2 * kRowsPerTF;
  const int tile = blockIdx.x;
  const int2 td = tiles[tile];
  const TFDesc t = tfs[td.x];
  for (int i = threadIdx.x; i < kRowsPerTF; i += blockDim.x) { s_cnt[i] = 0; s_min[i] = INT_MAX; s_max[i] = INT_MIN; }
  __syncthreads();
  const int b = td.y, e = min(t.n, td.y + tileSize);
  bool bad = false;
  constexpr int kU = 4;  // clusters in flight per thread
  for (int i0 = b + threadIdx.x; i0 < e; i0 += kU * 512) {
    RawCluster w[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (i0 + u * 512 < e) w[u] = load_raw(t, i0 + u * 512);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (i0 + u * 512 >= e) continue;
      int lr, yu, zu;
      if (!decode(t, w[u], G, lr, yu, zu)) bad = true;
      atomicAdd(&s_cnt[lr], 1);
      atomicMin(&s_min[lr], zu);
      atomicMax(&s_max[lr], zu);
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, kErrInput);
  int* out = tileStats + (size_t)tile * 3 * kRowsPerTF;
  for (int i = threadIdx.x; i < kRowsPerTF; i += blockDim.x) {
    out[i] = s_cnt[i];
    out[kRowsPerTF + i] = s_min[i];
    out[2 * kRowsPerTF + i] = s_max[i];
  }
}

// Per (TF, row): reduce the tile statistics, and turn each tile's count into
// its exclusive offset inside the row's bucket (tile order = input order).
// A block takes 32 rows of one TF; its 32 warps split the TF's tiles into 32
// consecutive chunks (lane = row, so a warp's loads of one tile are one
// 128-byte line): chunk sums first, their exclusive scan per row in shared
// memory, then each chunk writes its tiles' offsets.
constexpr int kRRRows = 32, kRRChunks = 32;
__global__ void __launch_bounds__(kRRRows * kRRChunks) k_row_reduce(const TFDesc* __restrict__ tfs, int nTF,
                                                                  int* __restrict__ tileStats, int* __restrict__ rowCnt,
                                                                  int* __restrict__ rowMin, int* __restrict__ rowMax) {
  __shared__ int s_sum[kRRChunks][kRRRows + 1], s_min[kRRChunks][kRRRows + 1], s_max[kRRChunks][kRRRows + 1];
  const int blocksPerTF = (kRowsPerTF + kRRRows - 1) / kRRRows;
  const int tf = blockIdx.x / blocksPerTF;
  const int lane = threadIdx.x % kRRRows, q = threadIdx.x / kRRRows;
  const int lr = (blockIdx.x % blocksPerTF) * kRRRows + lane;
  const bool row = tf < nTF && lr < kRowsPerTF;
  const TFDesc t = tfs[min(tf, nTF - 1)];
  const int per = (t.nTiles + kRRChunks - 1) / kRRChunks;
  const int k0 = min(q * per, t.nTiles), k1 = min(k0 + per, t.nTiles);
  int c = 0, mn = INT_MAX, mx = INT_MIN;
  if (row)
    for (int k = k0; k < k1; ++k) {
      const int* ts = tileStats + (size_t)(t.tileBase + k) * 3 * kRowsPerTF;
      c += ts[lr];
      mn = min(mn, ts[kRowsPerTF + lr]);
      mx = max(mx, ts[2 * kRowsPerTF + lr]);
    }
  s_sum[q][lane] = c;
  s_min[q][lane] = mn;
  s_max[q][lane] = mx;
  __syncthreads();
  if (q == 0) {  // per row: exclusive scan of the chunk sums, totals, extremes
    int run = 0, m0 = INT_MAX, m1 = INT_MIN;
    for (int j = 0; j < kRRChunks; ++j) {
      const int v = s_sum[j][lane];
      s_sum[j][lane] = run;
      run += v;
      m0 = min(m0, s_min[j][lane]);
      m1 = max(m1, s_max[j][lane]);
    }
    if (row) {
      const int g = tf * kRowsPerTF + lr;
      rowCnt[g] = run;
      rowMin[g] = m0;
      rowMax[g] = m1;
    }
  }
  __syncthreads();
  if (row) {
    int o = s_sum[q][lane];
    for (int k = k0; k < k1; ++k) {
      int* ts = tileStats + (size_t)(t.tileBase + k) * 3 * kRowsPerTF;
      const int v = ts[lr];
      ts[lr] = o;
      o += v;
    }
  }
}

// Cells, NeighboursFinder blocks and grid of a row.
__device__ inline RowGrid row_grid(int R, int nRows, const int* __restrict__ rowCnt, const int* __restrict__ rowMin,
                                   const int* __restrict__ rowMax, const GeomConst* __restrict__ G) {
  RowGrid g{};
  if (R >= nRows) return g;  // no hits, no cells
  const int n = rowCnt[R];
  g.ny = cells_y(G->npads[(R % kRowsPerTF) % kNRow]);
  g.nz = 1;
  g.cz = 1;
  g.count = n;
  if (n > 0) {
    g.nz = min(max((n + kHitsPerCell * g.ny - 1) / (kHitsPerCell * g.ny), 1), kMaxNz);
    g.cz = cell_height(rowMin[R], rowMax[R], g.nz);
    g.zmin = rowMin[R];
  }
  return g;
}

// Grid of every row and the three row-level exclusive scans (hits, cells,
// NeighboursFinder blocks) in two launches of one thread per row: the sums of
// every block of kGridRows rows, then each block adds up the sums before it
// and scans its own rows.  totals[0..2] = hits, cells, NF blocks; sums:
// 3 * grid_blocks(nRows) ints.  (One CTA over all rows, each thread walking
// its run of rows twice, took 31 us for one Time Frame and 286 us for eight.)
constexpr int kGridRows = 256;
__global__ void __launch_bounds__(kGridRows) k_grid_sums(int nRows, const int* __restrict__ rowCnt,
                                                         const int* __restrict__ rowMin,
                                                         const int* __restrict__ rowMax,
                                                         const GeomConst* __restrict__ G, int nfBlock,
                                                         int* __restrict__ sums) {
  __shared__ int ws[3][kGridRows / 32];
  const RowGrid g = row_grid(blockIdx.x * kGridRows + threadIdx.x, nRows, rowCnt, rowMin, rowMax, G);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int v[3] = {g.count, g.ny * g.nz, (g.count + nfBlock - 1) / nfBlock};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int x = __reduce_add_sync(0xffffffffu, v[q]);
    if (lane == 0) ws[q][w] = x;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    int s = 0;
    for (int k = 0; k < kGridRows / 32; ++k) s += ws[threadIdx.x][k];
    sums[threadIdx.x * gridDim.x + blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(kGridRows) k_grid(int nRows, const int* __restrict__ rowCnt, const int* __restrict__ rowMin,
                                                    const int* __restrict__ rowMax, const GeomConst* __restrict__ G,
                                                    RowGrid* __restrict__ grid, int* __restrict__ nfBlockStart,
                                                    int* __restrict__ nfBlockRow, int nfBlock,
                                                    const int* __restrict__ sums,
                                                    int* __restrict__ totals) {
  __shared__ int ws[3][kGridRows / 32], base[3][kGridRows / 32];
  const int R = blockIdx.x * kGridRows + threadIdx.x;
  RowGrid g = row_grid(R, nRows, rowCnt, rowMin, rowMax, G);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int v[3] = {g.count, g.ny * g.nz, (g.count + nfBlock - 1) / nfBlock};
  int x[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int b = 0;  // of the blocks before
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += kGridRows) b += sums[q * gridDim.x + k];
    b = __reduce_add_sync(0xffffffffu, b);
    x[q] = v[q];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x[q], o);
      if (lane >= o) x[q] += y;
    }
    if (lane == 31) {
      ws[q][w] = x[q];
      base[q][w] = b;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    x[q] -= v[q];
    for (int k = 0; k < kGridRows / 32; ++k) x[q] += base[q][k] + (k < w ? ws[q][k] : 0);
  }
  if (R < nRows) {
    g.start = x[0];
    g.cellBase = x[1];
    grid[R] = g;
    nfBlockStart[R] = x[2];
    if (nfBlockRow)
      for (int b = 0; b < v[2]; ++b) nfBlockRow[x[2] + b] = R;
    if (R == nRows - 1) {
      totals[0] = x[0] + v[0];
      totals[1] = x[1] + v[1];
      totals[2] = x[2] + v[2];
      nfBlockStart[nRows] = x[2] + v[2];
    }
  }
}

__global__ void k_cell_sentinel(int* __restrict__ cellStart, const int* __restrict__ totals) {
  cellStart[totals[1]] = totals[0];
}

// K3a: scatter each tile's clusters into its row bucket at
// rowStart + (tile offset within the row) + (unordered rank inside the tile).
// Records: {y_u, zeta_u, batch input index, cell}.  Persistent: one CTA per
// SM takes the tiles in turn, so that only one tile per SM is open at a time
// and the partly written 32-byte sectors of its 5472 row segments stay in L2
// until they fill (with one CTA per tile the whole grid's open sectors
// outgrew L2 on a 128-orbit TF).  Each thread keeps the loads of its next kU
// clusters in flight while it files the current ones, and the row table (drift
// origin, cell size and count, 12 bytes a row) is held in shared memory with
// the slot counters.
// 1 ms frame 0.46 -> 0.40 ms, 32 orbits 1.56 -> 1.40 ms, 240 k clusters 24.5 ->
// 19 us.
#ifndef O2TPC_SCATTER_THREADS
#define O2TPC_SCATTER_THREADS 1024
#endif
#ifndef O2TPC_SCATTER_UNROLL
#define O2TPC_SCATTER_UNROLL 4
#endif
constexpr int kScatterT = O2TPC_SCATTER_THREADS, kScatterU = O2TPC_SCATTER_UNROLL;
constexpr size_t kScatterSmem = 4 * kRowsPerTF * sizeof(int);
__global__ void __launch_bounds__(kScatterT) k_row_scatter(const TFDesc* __restrict__ tfs, const int2* __restrict__ tiles,
                                                           int nTiles, int tileSize, const GeomConst* __restrict__ G,
                                                           const int* __restrict__ tileStats,
                                                           const RowGrid* __restrict__ grid, int4* __restrict__ bucket) {
  extern __shared__ int sm[];
  int *s_cur = sm, *s_zmin = sm + kRowsPerTF, *s_cz = sm + 2 * kRowsPerTF, *s_nz = sm + 3 * kRowsPerTF;
  __shared__ int s_npads[kNRow];
  for (int r = threadIdx.x; r < kNRow; r += kScatterT) s_npads[r] = G->npads[r];
  int tfHeld = -1;
  for (int tile = blockIdx.x; tile < nTiles; tile += gridDim.x) {
    const int2 td = tiles[tile];
    const TFDesc t = tfs[td.x];
    const int b = td.y, e = min(t.n, td.y + tileSize);
    if (b >= e) continue;  // an unused tile slot (block-uniform)
    const int Rbase = td.x * kRowsPerTF;
    const int* ts = tileStats + (size_t)tile * 3 * kRowsPerTF;
    RawCluster next[kScatterU];
    auto fetch = [&](int i0) {
#pragma unroll
      for (int u = 0; u < kScatterU; ++u)
        if (i0 + u * kScatterT < e) next[u] = load_raw(t, i0 + u * kScatterT);
    };
    fetch(b + threadIdx.x);
    __syncthreads();  // the previous tile's tables are no longer in use
    for (int i = threadIdx.x; i < kRowsPerTF; i += kScatterT) {
      const RowGrid g = grid[Rbase + i];
      s_cur[i] = g.start + ts[i];
      if (td.x != tfHeld) {
        s_zmin[i] = g.zmin;
        s_cz[i] = g.cz;
        s_nz[i] = g.nz;
      }
    }
    tfHeld = td.x;
    __syncthreads();
    for (int i0 = b + threadIdx.x; i0 < e; i0 += kScatterT * kScatterU) {
      RawCluster now[kScatterU];
#pragma unroll
      for (int u = 0; u < kScatterU; ++u) now[u] = next[u];
      fetch(i0 + kScatterT * kScatterU);
#pragma unroll
      for (int u = 0; u < kScatterU; ++u) {
        const int i = i0 + u * kScatterT;
        if (i < e) {
          int lr, yu, zu;
          decode(t, now[u], G, lr, yu, zu);
          RowGrid g;
          g.zmin = s_zmin[lr];
          g.cz = s_cz[lr];
          g.nz = s_nz[lr];
          const int npads = s_npads[lr % kNRow];
          g.ny = cells_y(npads);
          const int iy = cell_iy(g, npads, yu);
          const int iz = cell_iz_floor(zu, g);  // zu >= zmin of its row: 0..nz-1
          const int slot = atomicAdd(&s_cur[lr], 1);
          bucket[slot] = make_int4(yu, zu, t.inBase + i, iz * g.ny + iy);
        }
      }
    }
  }
}

// K3b: one CTA per row.  Counting sort of the row's bucket by cell into the
// final arrays, then input order restored inside every cell (insertion sort
// by input index).  Cell counters live in shared memory when the row has at
// most smemCells cells.  smemCells is sized for rows of 2.5 times the average
// (launch_cell_sort), so that more CTAs share an SM than with room for the
// largest (47.5 KB): 1 ms frame 0.62 -> 0.41 ms, 32 orbits 2.08 -> 1.63 ms, 3
// collisions 112 -> 56 us.  Rows of more cells count in the global scratch;
// those of more than farCells, which only frames with few filled rows have, are
// left to k_cell_sort_large.
constexpr int kSmemCells = 12160;  // at most: 47.5 KB, so that with the kernel's own 144 bytes a CTA stays within 48 KB
constexpr int kLargeCells = 11520;  // with k_cell_sort_large's list and statics within 48 KB too
constexpr int kRegSort = 8;

__device__ inline void sort_row(const RowGrid& g, int* cnt, const int4* __restrict__ bucket,
                                int* __restrict__ cellStart, int2* __restrict__ syz, int* __restrict__ sorig) {
  __shared__ int s_carry;
  const int nc = g.ny * g.nz;
  for (int c = threadIdx.x; c < nc; c += blockDim.x) cnt[c] = 0;
  __syncthreads();
  const int4* bk = bucket + g.start;
  for (int i = threadIdx.x; i < g.count; i += blockDim.x) atomicAdd(&cnt[bk[i].w], 1);
  __syncthreads();
  // exclusive scan of the cell counts, in chunks of blockDim
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  for (int c0 = 0; c0 < nc; c0 += blockDim.x) {
    int c = c0 + threadIdx.x;
    int v = (c < nc) ? cnt[c] : 0;
    // warp + block scan (up to 1024 threads)
    __shared__ int ws[32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    int wo = 0;
    for (int k = 0; k < w; ++k) wo += ws[k];
    int excl = s_carry + wo + x - v;
    __syncthreads();
    if (c < nc) {
      cnt[c] = excl;
      cellStart[g.cellBase + c] = g.start + excl;
    }
    if (threadIdx.x == blockDim.x - 1) s_carry = excl + v;
    __syncthreads();
  }
  // scatter (unordered inside a cell)
  for (int i = threadIdx.x; i < g.count; i += blockDim.x) {
    int4 rec = bk[i];
    int pos = g.start + atomicAdd(&cnt[rec.w], 1);
    syz[pos] = make_int2(rec.x, rec.y);
    sorig[pos] = rec.z;
  }
  __syncthreads();
  // restore input order inside each cell: a cell of at most kRegSort hits is
  // loaded at once and sorted in registers (odd-even transposition network);
  // a larger one by insertion in place
  for (int c = threadIdx.x; c < nc; c += blockDim.x) {
    int b = cellStart[g.cellBase + c];
    int e = (c + 1 < nc) ? cellStart[g.cellBase + c + 1] : g.start + g.count;
    const int m = e - b;
    if (m <= 1) continue;
    if (m <= kRegSort) {
      int ko[kRegSort];
      int2 kv[kRegSort];
#pragma unroll
      for (int j = 0; j < kRegSort; ++j) {
        ko[j] = (j < m) ? sorig[b + j] : INT_MAX;  // input indices are unique and < INT_MAX
        kv[j] = (j < m) ? syz[b + j] : make_int2(0, 0);
      }
#pragma unroll
      for (int rd = 0; rd < kRegSort; ++rd) {
#pragma unroll
        for (int j = rd & 1; j + 1 < kRegSort; j += 2) {
          if (ko[j] > ko[j + 1]) {
            const int tk = ko[j];
            ko[j] = ko[j + 1];
            ko[j + 1] = tk;
            const int2 tv = kv[j];
            kv[j] = kv[j + 1];
            kv[j + 1] = tv;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kRegSort; ++j) {
        if (j < m) {
          sorig[b + j] = ko[j];
          syz[b + j] = kv[j];
        }
      }
      continue;
    }
    for (int i = b + 1; i < e; ++i) {
      int ko = sorig[i];
      int2 kv = syz[i];
      int j = i - 1;
      while (j >= b && sorig[j] > ko) {
        sorig[j + 1] = sorig[j];
        syz[j + 1] = syz[j];
        --j;
      }
      sorig[j + 1] = ko;
      syz[j + 1] = kv;
    }
  }
}

template <int kT>
__global__ void __launch_bounds__(kT) k_cell_sort(const RowGrid* __restrict__ grid, const int4* __restrict__ bucket,
                                                   int* __restrict__ cellStart, int2* __restrict__ syz,
                                                   int* __restrict__ sorig, int* __restrict__ gscratch,
                                                   int smemCells, int farCells) {
  extern __shared__ int s_cnt[];
  const RowGrid g = grid[blockIdx.x];
  const int nc = g.ny * g.nz;
  if (g.count == 0) {
    for (int c = threadIdx.x; c < nc; c += blockDim.x) cellStart[g.cellBase + c] = g.start;
    return;
  }
  if (nc > farCells) return;
  sort_row(g, nc <= smemCells ? s_cnt : gscratch + g.cellBase, bucket, cellStart, syz, sorig);
}

// The rows of more than minCells cells, by resident CTAs of 512 threads with
// the largest counters: each looks for them among every gridDim.x-th row, a row
// a thread.  One sector filled, 2.1 M clusters in 152 rows: sort 0.39 -> 0.19 ms
// (CTAs of 128 threads that count in the global scratch, one an SM, before),
// 4.2 M 0.88 -> 0.38 ms.
template <int kT>
__global__ void __launch_bounds__(kT) k_cell_sort_large(int nRows, const RowGrid* __restrict__ grid,
                                                         const int4* __restrict__ bucket, int* __restrict__ cellStart,
                                                         int2* __restrict__ syz, int* __restrict__ sorig,
                                                         int* __restrict__ gscratch, int minCells) {
  extern __shared__ int s_cnt[];
  __shared__ int s_rows[kT], s_n;
  for (int r0 = blockIdx.x; r0 < nRows; r0 += kT * gridDim.x) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const long long r = r0 + (long long)threadIdx.x * gridDim.x;
    if (r < nRows && grid[r].count > 0 && grid[r].ny * grid[r].nz > minCells) s_rows[atomicAdd(&s_n, 1)] = (int)r;
    __syncthreads();
    for (int k = 0; k < s_n; ++k) {
      const RowGrid g = grid[s_rows[k]];
      sort_row(g, g.ny * g.nz <= kLargeCells ? s_cnt : gscratch + g.cellBase, bucket, cellStart, syz, sorig);
      __syncthreads();  // the counters are no longer in use
    }
    __syncthreads();  // nor the list
  }
}

// K3c: the drift-ordered view of every row (ZRow), one CTA per row, from the
// sorted hits.  Bins of at least 0.5 cm, at most one per hit.  The sorted order
// runs through the cell rows in drift order, so a chunk of cell rows is a
// contiguous run of hits whose bins are a contiguous run too (its first bin
// may be shared with the chunk before, whose hits come first): every chunk is
// counted, scanned and scattered by itself in shared memory, its output range
// is its input range, and the writes stay inside it.  Bound by memory: 8
// bytes read (twice, the second time from L2), 10 + 2 per bin written per hit.
constexpr int kZThreads = 256;
__global__ void __launch_bounds__(kZThreads) k_zorder(const RowGrid* __restrict__ grid, const int* __restrict__ rowMax,
                                                      const int* __restrict__ cellStart, const int2* __restrict__ syz,
                                                      ZRow* __restrict__ zrow, int4* __restrict__ bucket) {
  __shared__ int s_cnt[kZBins + 1];
  __shared__ int s_warp[kZThreads / 32];
  const RowGrid g = grid[blockIdx.x];
  ZRow z{};
  z.start = g.start;
  z.count = g.count;
  z.cellBase = g.cellBase;
  z.cz = g.cz;
  z.flags = g.nz << kZnz;
  if (g.count == 0) {
    if (threadIdx.x == 0) zrow[blockIdx.x] = z;
    return;
  }
  const float range = (float)((unsigned)rowMax[blockIdx.x] - (unsigned)g.zmin) + 1.f;
  z.zmin = g.zmin;
  z.nzb = drift_bins(range, g.count, g.nz);
  z.zinv = (float)z.nzb / range;
  // expected hits of a whole row in a window (plus the bins' own width)
  // against ~10 in the cells that cover it
  const float perUnit = (float)g.count / range, binw = range / (float)z.nzb;
  if (perUnit * (2 * kWinZ + binw) > 20.f) z.flags |= kZNFCells;
  if (perUnit * (140.f + binw) > 12.f) z.flags |= kZFollowCells;
  if (threadIdx.x == 0) zrow[blockIdx.x] = z;
  char* mem = reinterpret_cast<char*>(bucket) + 16ll * g.start;
  int2* yz = reinterpret_cast<int2*>(mem);
  short* idx = reinterpret_cast<short*>(mem + 8ll * g.count);
  unsigned short* bins16 = reinterpret_cast<unsigned short*>(mem + 12ll * g.count);
  int* bins32 = reinterpret_cast<int*>(mem + 12ll * g.count);
  // A row whose view neither searches: its hits are better taken in sorted order,
  // so that the lanes of a warp search the same cells (one sector filled,
  // NeighboursFinder: 2.1 M clusters 17.7 ms in drift order, 16.7 so; 4.2 M 110 and
  // 103).
  const bool unsearched = (z.flags & (kZNFCells | kZFollowCells)) == (kZNFCells | kZFollowCells);
  bool far = false;  // this thread met an index distance beyond 16 bits
  const float perCellRow = (float)g.cz * z.zinv * 1.0001f + 1.f;
  const int izPer = max(1, (int)((float)(kZBins - 8) / perCellRow));
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int bL = -1;  // last bin of the chunks before
  for (int iz0 = 0; iz0 < g.nz && !unsearched; iz0 += izPer) {
    const int iz1 = min(iz0 + izPer, g.nz);
    const int hb = cellStart[g.cellBase + iz0 * g.ny];
    const int he = iz1 < g.nz ? cellStart[g.cellBase + iz1 * g.ny] : g.start + g.count;
    const int bR = iz1 < g.nz ? z_bin(g.zmin + iz1 * g.cz - 1, g.zmin, z.zinv, z.nzb) : z.nzb - 1;
    const int nb = min(bR - bL, kZBins);  // counters 1..nb for bins bL + 1..bR, counter 0 for the shared bin bL
    for (int c = threadIdx.x; c <= nb; c += kZThreads) s_cnt[c] = 0;
    __syncthreads();
    for (int h = hb + threadIdx.x; h < he; h += kZThreads) {
      const int b = z_bin(syz[h].y, g.zmin, z.zinv, z.nzb);
      atomicAdd(&s_cnt[min(max(b - bL, 0), nb)], 1);
    }
    __syncthreads();
    // exclusive scan of the nb + 1 counters: a run per thread
    const int per = (nb + kZThreads) / kZThreads;
    const int c0 = min(threadIdx.x * per, nb + 1), c1 = min(c0 + per, nb + 1);
    int s = 0;
    for (int c = c0; c < c1; ++c) s += s_cnt[c];
    int x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    int off = x - s;
    for (int k = 0; k < w; ++k) off += s_warp[k];
    const int base = hb - g.start;
    for (int c = c0; c < c1; ++c) {
      const int v = s_cnt[c];
      s_cnt[c] = off;
      if (c > 0) {
        if (g.count <= kZShortRow) bins16[bL + c] = (unsigned short)(base + off);
        else bins32[bL + c] = base + off;
      }
      off += v;
    }
    __syncthreads();
    for (int h = hb + threadIdx.x; h < he; h += kZThreads) {
      const int2 p = syz[h];
      const int b = z_bin(p.y, g.zmin, z.zinv, z.nzb);
      const int pos = base + atomicAdd(&s_cnt[min(max(b - bL, 0), nb)], 1);
      yz[pos] = p;
      const int d = h - g.start - pos;
      idx[pos] = (short)d;
      far = far || d != (int)(short)d;
    }
    __syncthreads();
    bL = bR;
  }
  // the view becomes the sorted order itself (distance 0 throughout, which the
  // row's own hits are taken from), and the searches into this row take the cells
  if (__syncthreads_or(far || unsearched)) {
    for (int h = threadIdx.x; h < g.count; h += kZThreads) {
      yz[h] = syz[g.start + h];
      idx[h] = 0;
    }
    if (threadIdx.x == 0) zrow[blockIdx.x].flags = z.flags | kZNFCells | kZFollowCells;
  }
}

// ------------------------------------------------------------- launchers
void launch_zorder(int nRows, const RowGrid* grid, const int* rowMax, const int* cellStart, const int2* syz,
                   ZRow* zrow, int4* bucket, cudaStream_t st) {
  if (nRows > 0) {
    k_zorder<<<nRows, kZThreads, 0, st>>>(grid, rowMax, cellStart, syz, zrow, bucket);
    ++g_launch_count;
  }
}

void launch_ingest_stats(const TFDesc* tfs, const int2* tiles, int nTiles, int tileSize, const GeomConst* G,
                         int* tileStats, unsigned* err, cudaStream_t st) {
  size_t smem = 3 * kRowsPerTF * sizeof(int);
  cudaFuncSetAttribute(k_ingest_stats, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (nTiles > 0) {
    k_ingest_stats<<<nTiles, 512, smem, st>>>(tfs, tiles, tileSize, G, tileStats, err);
    ++g_launch_count;
  }
}

void launch_row_reduce(const TFDesc* tfs, int nTF, int* tileStats, int* rowCnt, int* rowMin, int* rowMax,
                       cudaStream_t st) {
  if (nTF <= 0) return;
  const int blocksPerTF = (kRowsPerTF + kRRRows - 1) / kRRRows;
  k_row_reduce<<<nTF * blocksPerTF, kRRRows * kRRChunks, 0, st>>>(tfs, nTF, tileStats, rowCnt, rowMin, rowMax);
  ++g_launch_count;
}

void launch_grid(int nRows, const int* rowCnt, const int* rowMin, const int* rowMax, const GeomConst* G,
                 RowGrid* grid, int* nfBlockStart, int* nfBlockRow, int nfBlock, int* totals, cudaStream_t st) {
  if (nRows <= 0) return;
  int* sums = totals + 4;
  const int nb = grid_blocks(nRows);
  k_grid_sums<<<nb, kGridRows, 0, st>>>(nRows, rowCnt, rowMin, rowMax, G, nfBlock, sums);
  k_grid<<<nb, kGridRows, 0, st>>>(nRows, rowCnt, rowMin, rowMax, G, grid, nfBlockStart, nfBlockRow, nfBlock, sums,
                               totals);
  g_launch_count += 2;
}

int grid_blocks(int nRows) { return (nRows + kGridRows - 1) / kGridRows; }

// Tiles: their number bounds the parallelism of the ingest and of the scatter
// (a CTA takes tiles in turn), each costs 64 KB of row statistics written and
// read.  Four tiles per SM, of 8192 to 65536 clusters: with 65536 throughout,
// 1.3 M clusters gave 20 tiles to 152 SMs (ingest 84, scatter 131 us), and the
// 310 tiles of 20 M clusters left the scatter's last round nearly empty.
int ingest_tile(long long n) {
  static const int sms = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 148;
  }();
  const long long t = (n + 4ll * sms - 1) / (4ll * sms);
  return (int)std::min<long long>(std::max<long long>((t + 255) / 256 * 256, kTileMin), kTileMax);
}

// CTAs per SM of the persistent row scatter
#ifndef O2TPC_SCATTER_CTAS_PER_SM
#define O2TPC_SCATTER_CTAS_PER_SM 1
#endif

void launch_row_scatter(const TFDesc* tfs, const int2* tiles, int nTiles, int tileSize, const GeomConst* G,
                        const int* tileStats, const RowGrid* grid, int4* bucket, cudaStream_t st) {
  if (nTiles > 0) {
    int dev = 0, nSM = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nSM, cudaDevAttrMultiProcessorCount, dev);
    const int nb = nSM > 0 ? std::min(nTiles, nSM * O2TPC_SCATTER_CTAS_PER_SM) : nTiles;
    cudaFuncSetAttribute(k_row_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScatterSmem);
    k_row_scatter<<<nb, kScatterT, kScatterSmem, st>>>(tfs, tiles, nTiles, tileSize, G, tileStats, grid, bucket);
    ++g_launch_count;
  }
}

// No shape asked for: by the hits of an average row.  Short rows idle large
// CTAs in every barrier; of long rows, fewer at once stay in L2 between
// the two reads.  Sort of 3 collisions (240 a row) 96 / 109 / 131 us with
// 128 / 256 / 512 threads, 10 collisions (750) 217 / 225 / 248 us, 1 ms frame
// (3700) 1.13 / 1.06 / 1.08 ms, 16 orbits (5400) 2.25 / 1.95 / 1.96, 48 orbits
// (16 k) 7.66 / 7.12 / 6.09, 96 orbits (32 k) 13.6 / 12.2 / 11.5.
int cell_sort_threads(int n, int nRows, int asked) {
  if (asked != 0) return asked;
  const int perRow = n / std::max(nRows, 1);
  return perRow < 1000 ? 128 : perRow < 8000 ? 256 : 512;
}

void launch_cell_sort(int n, int nRows, const RowGrid* grid, const int4* bucket, int* cellStart, int2* syz, int* sorig,
                      int* gscratch, const int* totals, cudaStream_t st, int threadsPerRow) {
  if (nRows > 0) {
    threadsPerRow = cell_sort_threads(n, nRows, threadsPerRow);
    const long long want = 5ll * n / (2ll * kHitsPerCell * nRows) + 128;
    const int cells = (int)std::min<long long>(std::max<long long>(want, 512), kSmemCells);
    const size_t smem = sizeof(int) * cells;
    // Rows of four times the counters of a TF that holds all n clusters (ten
    // times its average) are k_cell_sort_large's; its launch (2-3 us) is left out
    // where a single filled sector would not have them.  (All rows past the
    // counters there: one sector the same, but a graph with room for 64 TFs given
    // one of 20 M clusters 10.23 -> 10.35 ms, eight of 0.7 M 1 % slower.)
    const int farCells = (int)std::min<long long>(
        std::max<long long>(5ll * n / (2ll * kHitsPerCell * kRowsPerTF) + 128, 512) * 4, INT_MAX);
    const bool large = n / (kNRow * kHitsPerCell) > farCells;
    auto sort = [&](auto kernel, int threads) {
      kernel<<<nRows, threads, smem, st>>>(grid, bucket, cellStart, syz, sorig, gscratch, cells,
                                           large ? farCells : INT_MAX);
      ++g_launch_count;
    };
    if (threadsPerRow == 128) sort(k_cell_sort<128>, 128);
    else if (threadsPerRow == 512) sort(k_cell_sort<512>, 512);
    else sort(k_cell_sort<256>, 256);
    if (large) {
      constexpr int kT = 512;
      static const int ctas = [] {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cell_sort_large<kT>, kT, sizeof(int) * kLargeCells);
        return std::max(sms, 1) * std::max(per, 1);
      }();
      k_cell_sort_large<kT><<<std::min(ctas, nRows), kT, sizeof(int) * kLargeCells, st>>>(
          nRows, grid, bucket, cellStart, syz, sorig, gscratch, farCells);
      ++g_launch_count;
    }
  }
  k_cell_sentinel<<<1, 1, 0, st>>>(cellStart, totals);
  ++g_launch_count;
}

}  // namespace o2tpc
