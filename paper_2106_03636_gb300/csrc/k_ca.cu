// k_ca.cu - cellular-automaton seeding: NeighboursFinder, NeighboursCleaner,
// StartHitsFinder, plus the device-wide scan used for ordered compaction.
//
// All decisions here are integer: the straightness metric of a hit h with an
// upper neighbour u (row r+1) and a lower neighbour d (row r-1) is
//   D = 2077 (2 y_h - y_u - y_d)^2 + 1536 (2 z_h - z_u - z_d)^2
// (a 2-dof chi2 scaled by 6 sigma_y^2 * 6 sigma_z^2 in integer units; it fits
// in 31 bits inside the windows), accepted when D <= 16 * 1536 * 2077, and
// the winner is the lexicographic minimum of (D, u, d), which no enumeration
// order can change.
#include "o2tpc_kernels.cuh"

namespace o2tpc {

#ifndef O2TPC_NF_CAND
#define O2TPC_NF_CAND 6
#endif
constexpr int kNFCand = O2TPC_NF_CAND;  // candidates per side held in registers by the NeighboursFinder

// Candidate residuals of one side, packed: (y_h - y_c + 1024) << 16 |
// (z_h - z_c + 1024).  Inside the windows both halves stay in [776, 1272], so
// the sum of an up and a down residual adds the halves without carries and
// unpacks to (2 y_h - y_u - y_d + 2048, 2 z_h - z_u - z_d + 2048).
__device__ inline unsigned pack_res(int dy, int dz) { return ((unsigned)(dy + 1024) << 16) | (unsigned)(dz + 1024); }

// Appends the in-window candidates of one side (cells [iy0, iy1] of cell
// rows iz0..iz1 of row g, visited in ascending sorted index) to the register
// slots: the newest goes to slot kNFCand-1, older ones move down, so slots
// [kNFCand - n, kNFCand) hold them in ascending index order.  Returns the
// number found (more than kNFCand: the caller takes the general path).
// pts[c - base] holds the coordinates of sorted hit c (the block's staged
// slab, or the global array with base 0).
__device__ inline int nf_collect(const RowGrid& g, int iy0, int iy1, int iz0, int iz1,
                                 const int* __restrict__ cellStart, const int2* pts, int base, int2 hh,
                                 int (&idx)[kNFCand], unsigned (&res)[kNFCand]) {
  int n = 0;
  for (int iz = iz0; iz <= iz1; ++iz) {
    const int a = __ldg(cellStart + g.cellBase + iz * g.ny + iy0);
    const int b = __ldg(cellStart + g.cellBase + iz * g.ny + iy1 + 1);
    for (int c = a; c < b; ++c) {
      const int2 p = pts[c - base];
      const int dy = hh.x - p.x, dz = hh.y - p.y;
      if (abs(dy) > kWinY || abs(dz) > kWinZ) continue;
#pragma unroll
      for (int q = 0; q < kNFCand - 1; ++q) {
        idx[q] = idx[q + 1];
        res[q] = res[q + 1];
      }
      idx[kNFCand - 1] = c;
      res[kNFCand - 1] = pack_res(dy, dz);
      ++n;
    }
  }
  return n;
}

// One hit's best pair in the cell rectangles of the adjacent rows; su / sd:
// coordinates of sorted hit c at su[c - bu0] / sd[c - bd0] (a staged slab, or
// the global array with offset 0).
__device__ inline void nf_cells(const RowGrid& gu, const RowGrid& gd, int uy0, int uy1, int uz0, int uz1, int dy0,
                                int dy1, int dz0, int dz1, const int* __restrict__ cellStart,
                                const int2* __restrict__ syz, const int2* su, int bu0, const int2* sd, int bd0, int2 hh,
                                int& bu, int& bd) {
  const int yh = hh.x, zh = hh.y;
  int ui[kNFCand] = {}, di[kNFCand] = {};
  unsigned ur[kNFCand] = {}, dr[kNFCand] = {};
  const int nu = nf_collect(gu, uy0, uy1, uz0, uz1, cellStart, su, bu0, hh, ui, ur);
  const int nd = nu > 0 ? nf_collect(gd, dy0, dy1, dz0, dz1, cellStart, sd, bd0, hh, di, dr) : 0;
  // bestD starts one above the cut, so "D < bestD" also applies the cut
  int bestD = kMaxMetric + 1;
  // pairs in ascending (u, d): a strict "<" keeps the first minimum,
  // which is the lexicographic minimum of (D, u, d).  Slots [a0, kNFCand)
  // of both sides: the last four when both sides fit there (the common
  // case), else all of them.
  auto pair_scan = [&](const int a0) {
#pragma unroll
    for (int a = a0; a < kNFCand; ++a)
#pragma unroll
      for (int b = a0; b < kNFCand; ++b) {
        const unsigned sres = ur[a] + dr[b];
        const int ey = (int)(sres >> 16) - 2048, ez = (int)(sres & 0xFFFFu) - 2048;
        const int D = kWeightY * ey * ey + kWeightZ * ez * ez;
        if (a >= kNFCand - nu && b >= kNFCand - nd && D < bestD) {
          bestD = D;
          bu = ui[a];
          bd = di[b];
        }
      }
  };
  constexpr int kNFSmall = kNFCand < 4 ? kNFCand : 4;
  if (nu <= kNFSmall && nd <= kNFSmall) {
    pair_scan(kNFCand - kNFSmall);
  } else if (nu <= kNFCand && nd <= kNFCand) {
    pair_scan(0);
  } else {
    const int y2 = 2 * yh, z2 = 2 * zh;
    for (int izu = uz0; izu <= uz1; ++izu) {
      const int ua = __ldg(cellStart + gu.cellBase + izu * gu.ny + uy0);
      const int ub = __ldg(cellStart + gu.cellBase + izu * gu.ny + uy1 + 1);
      for (int u = ua; u < ub; ++u) {
        const int2 pu = __ldg(syz + u);
        if (abs(pu.x - yh) > kWinY || abs(pu.y - zh) > kWinZ) continue;
        for (int izd = dz0; izd <= dz1; ++izd) {
          const int da = __ldg(cellStart + gd.cellBase + izd * gd.ny + dy0);
          const int db = __ldg(cellStart + gd.cellBase + izd * gd.ny + dy1 + 1);
          for (int d = da; d < db; ++d) {
            const int2 pd = __ldg(syz + d);
            if (abs(pd.x - yh) > kWinY || abs(pd.y - zh) > kWinZ) continue;
            const int ey = y2 - pu.x - pd.x, ez = z2 - pu.y - pd.y;
            const int D = kWeightY * ey * ey + kWeightZ * ez * ez;
            if (D < bestD) {  // (u, d) visited in ascending order
              bestD = D;
              bu = u;
              bd = d;
            }
          }
        }
      }
    }
  }
}

// One hit's best pair in the drift-ordered views of the adjacent rows,
// candidates at positions [ua, ub) and [da, db).  The candidates of a side are
// tested into a bit mask (no branch, loads independent), the one or two that
// pass are fetched again: the lanes of a warp then differ only in short loops.
// Sides of at most four candidates each (the common case) go through all 16
// pairs in registers.  Equal metrics go to the smaller sorted up, then down
// index.
__device__ inline void nf_view(const ZView& V, const ZRow& gu, const ZRow& gd, int ua, int ub, int da, int db, int2 hh,
                               int& bu, int& bd) {
  const int2* pu = V.yz(gu);
  const int2* pd = V.yz(gd);
  auto inside = [&](int2 c) {
    return (unsigned)(hh.x - c.x + kWinY) <= 2u * kWinY && (unsigned)(hh.y - c.y + kWinZ) <= 2u * kWinZ;
  };
  auto metric = [&](int2 u, int2 d) {
    const int ey = (hh.x - u.x) + (hh.x - d.x), ez = (hh.y - u.y) + (hh.y - d.y);
    return kWeightY * ey * ey + kWeightZ * ez * ez;
  };
  int bestD = kMaxMetric + 1, pbu = -1, pbd = -1;
  auto take = [&](int D, int u, int d) {
    bool better = D < bestD;
    if (D == bestD && pbu >= 0) {
      const int a = V.idx(gu, u), b = V.idx(gu, pbu);
      better = a < b || (a == b && V.idx(gd, d) < V.idx(gd, pbd));
    }
    if (better) {
      bestD = D;
      pbu = u;
      pbd = d;
    }
  };
  if (ub - ua <= 32 && db - da <= 32) {
    auto mask = [&](const int2* p, int m) {
      unsigned k = 0;
#pragma unroll 4
      for (int i = 0; i < m; ++i) k |= inside(__ldg(p + i)) ? 1u << i : 0u;
      return k;
    };
    pu += ua;
    pd += da;
    const unsigned mu = mask(pu, ub - ua);
    if (!mu) return;
    const unsigned md = mask(pd, db - da);
    if (!md) return;
    if (__popc(mu) <= 4 && __popc(md) <= 4) {
      // residuals of the four slots; an empty slot's y residual (700) puts
      // every pair with it past the cut (700 - 240 = 460: 2077 * 460^2 > cut)
      int uy[4], uz[4], dy[4], dz[4];
      unsigned uPos = 0, dPos = 0, m = mu;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        uy[a] = 700;
        uz[a] = 0;
        if (m) {
          const int i = __ffs(m) - 1;
          m &= m - 1;
          const int2 c = __ldg(pu + i);
          uy[a] = hh.x - c.x;
          uz[a] = hh.y - c.y;
          uPos |= (unsigned)i << (8 * a);
        }
      }
      m = md;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        dy[b] = 700;
        dz[b] = 0;
        if (m) {
          const int i = __ffs(m) - 1;
          m &= m - 1;
          const int2 c = __ldg(pd + i);
          dy[b] = hh.x - c.x;
          dz[b] = hh.y - c.y;
          dPos |= (unsigned)i << (8 * b);
        }
      }
      unsigned D[16], best = ~0u;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const unsigned ey = (unsigned)(uy[k >> 2] + dy[k & 3]), ez = (unsigned)(uz[k >> 2] + dz[k & 3]);
        D[k] = (unsigned)kWeightY * ey * ey + (unsigned)kWeightZ * ez * ez;
        best = min(best, D[k]);
      }
      if (best > (unsigned)kMaxMetric) return;
      unsigned eq = 0;
#pragma unroll
      for (int k = 0; k < 16; ++k) eq |= D[k] == best ? 1u << k : 0u;
      bestD = (int)best;
      do {  // one pair, or several of the same metric
        const int k = __ffs(eq) - 1;
        eq &= eq - 1;
        const int u = (int)((uPos >> (8 * (k >> 2))) & 255u), d = (int)((dPos >> (8 * (k & 3))) & 255u);
        if (pbu < 0) {
          pbu = ua + u;
          pbd = da + d;
        } else {
          take(bestD, ua + u, da + d);
        }
      } while (eq);
    } else {
      for (unsigned m = mu; m; m &= m - 1) {
        const int u = __ffs(m) - 1;
        const int2 cu = __ldg(pu + u);
        for (unsigned n = md; n; n &= n - 1) {
          const int d = __ffs(n) - 1;
          take(metric(cu, __ldg(pd + d)), ua + u, da + d);
        }
      }
    }
  } else {
    for (int u = ua; u < ub; ++u) {
      const int2 cu = __ldg(pu + u);
      if (!inside(cu)) continue;
      for (int d = da; d < db; ++d) {
        const int2 cd = __ldg(pd + d);
        if (inside(cd)) take(metric(cu, cd), u, d);
      }
    }
  }
  if (pbu >= 0) {
    bu = V.idx(gu, pbu);
    bd = V.idx(gd, pbd);
  }
}

// Threads of the NeighboursFinder kernels resident on an SM: 40 registers a
// thread with some 190 bytes of spills, for twelve warps a scheduler.  They
// wait for candidates more than they compute: 1 ms frame (20.3 M clusters) 0.90
// ms with 64 registers, 0.80 with 48, 0.75 with 40, 0.77 with 32; across a
// missing row (10 collisions) 0.21 -> 0.18 ms.
constexpr int kNFResident = 1536;

// K4: one thread per hit in the drift order of its row; blocks of kB hits
// tile the rows (nfBlockRow, built for the same block size, names a block's
// row).  The hits of a warp are neighbours in drift, so their candidates on an
// adjacent row are one run of 40-50 hits and every lane's share of it is about
// equal: 8 candidates a side to test, against 11 in the cells with the second
// cell row scanned by the few lanes that reach it.  A hit next to a row flagged dense takes the cells.
// Against the search in the cells: 1 ms frame (20.3 M clusters) 1.80 -> 0.94
// ms, 32 orbits (59 M) 6.02 -> 3.63 ms (0.75 and 2.75 with kNFResident); the views
// cost 0.20 and 0.62 ms.
template <int kB>
__global__ void __launch_bounds__(kB, kNFResident / kB) k_neighbours_view(const RowGrid* __restrict__ grid,
                                                        const int* __restrict__ nfBlockStart,
                                                        const int* __restrict__ nfBlockRow, int nRows,
                                                        const int* __restrict__ cellStart,
                                                        const int2* __restrict__ syz, const GeomConst* __restrict__ G,
                                                        ZView zv, int* __restrict__ upRaw, int* __restrict__ dnRaw) {
  if ((int)blockIdx.x >= nfBlockStart[nRows]) return;  // launched with an upper bound of blocks
  const int R = nfBlockRow[blockIdx.x];
  const ZRow g = zv.rows[R];
  const int q = (blockIdx.x - nfBlockStart[R]) * kB + threadIdx.x;
  if (q >= g.count) return;
  const int r = (R % kRowsPerTF) % kNRow;
  if (r < 1 || r > kNRow - 2) {  // rows 0 and 151 get no links
    upRaw[g.start + q] = -1;
    dnRaw[g.start + q] = -1;
    return;
  }
  const int2 hh = zv.yz(g)[q];
  const int h = zv.idx(g, q);
  const ZRow gu = zv.rows[R + 1], gd = zv.rows[R - 1];
  int bu = -1, bd = -1;
  if ((gu.flags | gd.flags) & kZNFCells) {
    const RowGrid cu = grid[R + 1], cd = grid[R - 1];
    int uy0, uy1, uz0, uz1, dy0, dy1, dz0, dz1;
    if (cell_range(cu, G->npads[r + 1], hh.x - kWinY, hh.x + kWinY, hh.y - kWinZ, hh.y + kWinZ, uy0, uy1, uz0, uz1) &&
        cell_range(cd, G->npads[r - 1], hh.x - kWinY, hh.x + kWinY, hh.y - kWinZ, hh.y + kWinZ, dy0, dy1, dz0, dz1))
      nf_cells(cu, cd, uy0, uy1, uz0, uz1, dy0, dy1, dz0, dz1, cellStart, syz, syz, 0, syz, 0, hh, bu, bd);
  } else {
    int ua, ub, da, db;
    if (z_range(zv, gu, hh.y - kWinZ, hh.y + kWinZ, ua, ub) && z_range(zv, gd, hh.y - kWinZ, hh.y + kWinZ, da, db))
      nf_view(zv, gu, gd, ua, ub, da, db, hh, bu, bd);
  }
  upRaw[h] = bu;
  dnRaw[h] = bd;
}

// --- staging of the adjacent rows' candidate slabs (TMA bulk copy)
constexpr int kSlab = 1024;            // staged hits per side (8 KB)
constexpr int kSlabWaitLimit = 1 << 22;  // mbarrier polls before giving up on a copy

__device__ inline unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Injected fault (o2tpc_config.debug_inject bit 0): the barrier is armed for
// the slab bytes but no copy is issued, and the waits give up after this many
// polls - a wait that runs out with nothing in flight.
constexpr int kSlabWaitInjected = 64;

// Waits (bounded) for phase 0 of the mbarrier; false if it did not complete.
__device__ inline bool slab_wait(unsigned bar, int limit) {
  for (int i = 0; i < limit; ++i) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// K4, staged form (o2tpc_config.nf_staged): one thread per hit in sorted
// order, the candidate cells from shared memory: a block's
// hits are consecutive in (cell, input) order, so they lie in the cell rows
// between those of its first and last hit, and their candidates in the cell
// rows of each adjacent pad row that this drift range (widened by the window)
// reaches - every cell across the row, one contiguous range of the sorted
// coordinates.  Thread 0 issues one TMA bulk copy per side as soon as it knows
// the range, completing on an mbarrier; the threads set up their windows
// meanwhile and wait just before scanning.  A side whose range exceeds kSlab
// hits (or a copy that does not complete within the wait limit, flagged in
// err) reads global memory instead.
template <int kB>
__global__ void __launch_bounds__(kB) k_neighbours_staged(const RowGrid* __restrict__ grid,
                                                   const int* __restrict__ nfBlockStart, int nRows,
                                                   const int* __restrict__ cellStart, const int2* __restrict__ syz,
                                                   const GeomConst* __restrict__ G, int* __restrict__ upRaw,
                                                   int* __restrict__ dnRaw, unsigned* __restrict__ err,
                                                   unsigned inject) {
  if ((int)blockIdx.x >= nfBlockStart[nRows]) return;  // launched with an upper bound of blocks
  __shared__ __align__(16) int2 s_slab[2][kSlab];
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ int s_row, s_base[2], s_use[2];
  const unsigned bar = smem_addr(&s_bar);
  if (threadIdx.x == 0) {
    const int R0 = upper_bound_i32(nfBlockStart, nRows + 1, blockIdx.x) - 1;
    s_row = R0;
    s_use[0] = s_use[1] = 0;
    const int r0 = (R0 % kRowsPerTF) % kNRow;
    if (r0 >= 1 && r0 <= kNRow - 2) {
      const RowGrid g0 = grid[R0];
      const int hf = g0.start + (blockIdx.x - nfBlockStart[R0]) * kB;
      const int hl = min(hf + kB, g0.start + g0.count) - 1;
      // drift range of the block's cell rows
      const int izf = cell_iz_floor(syz[hf].y, g0), izl = cell_iz_floor(syz[hl].y, g0);
      const long long zlo = (long long)g0.zmin + (long long)izf * g0.cz - kWinZ;
      const long long zhi = (long long)g0.zmin + (long long)(izl + 1) * g0.cz - 1 + kWinZ;
      unsigned bytes = 0;
      for (int side = 0; side < 2; ++side) {
        const RowGrid g2 = grid[side == 0 ? R0 + 1 : R0 - 1];
        s_base[side] = 0;
        if (g2.count == 0) continue;
        const int zl = (int)max(zlo, (long long)INT_MIN + 1), zh = (int)min(zhi, (long long)INT_MAX - 1);
        int iza = cell_iz_floor(zl, g2), izb = cell_iz_floor(zh, g2);
        if (iza < 0) iza = 0;
        if (izb > g2.nz - 1) izb = g2.nz - 1;
        if (iza > izb) continue;
        const int a = cellStart[g2.cellBase + iza * g2.ny], b = cellStart[g2.cellBase + (izb + 1) * g2.ny];
        const int a0 = a & ~1, b0 = (b + 1) & ~1;  // 16-byte aligned range (syz has one int2 of padding)
        if (b0 - a0 > kSlab || b0 <= a0) continue;
        s_use[side] = b0 - a0;
        s_base[side] = a0;
        bytes += (unsigned)(b0 - a0) * 8u;
      }
      if (bytes) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        for (int side = 0; side < 2; ++side)
          if (s_use[side] && !(inject & 1u))
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_addr(&s_slab[side][0])),
                "l"(syz + s_base[side]), "r"((unsigned)s_use[side] * 8u), "r"(bar)
                : "memory");
      }
    }
  }
  __syncthreads();
  const int R = s_row;
  const RowGrid g = grid[R];
  const int h = g.start + (blockIdx.x - nfBlockStart[R]) * kB + threadIdx.x;
  const bool valid = h < g.start + g.count;
  const int r = (R % kRowsPerTF) % kNRow;
  if (r < 1 || r > kNRow - 2) {  // rows 0 and 151 get no links (no copy was issued)
    if (valid) {
      upRaw[h] = -1;
      dnRaw[h] = -1;
    }
    return;
  }
  const bool staged = s_use[0] || s_use[1];
  const int waitLimit = (inject & 1u) ? kSlabWaitInjected : kSlabWaitLimit;
  bool slabOk = true;
  int bu = -1, bd = -1;
  if (valid) {
    const RowGrid gu = grid[R + 1], gd = grid[R - 1];
    const int npu = G->npads[r + 1], npd = G->npads[r - 1];
    const int2 hh = syz[h];
    const int yh = hh.x, zh = hh.y;
    int uy0, uy1, uz0, uz1, dy0, dy1, dz0, dz1;
    const bool inWin = cell_range(gu, npu, yh - kWinY, yh + kWinY, zh - kWinZ, zh + kWinZ, uy0, uy1, uz0, uz1) &&
                       cell_range(gd, npd, yh - kWinY, yh + kWinY, zh - kWinZ, zh + kWinZ, dy0, dy1, dz0, dz1);
    if (staged) {
      slabOk = slab_wait(bar, waitLimit);
      if (!slabOk) atomicOr(err, kErrTimeout);
    }
    const int2* su = (staged && slabOk && s_use[0]) ? s_slab[0] : syz;
    const int bu0 = (staged && slabOk && s_use[0]) ? s_base[0] : 0;
    const int2* sd = (staged && slabOk && s_use[1]) ? s_slab[1] : syz;
    const int bd0 = (staged && slabOk && s_use[1]) ? s_base[1] : 0;
    if (inWin)
      nf_cells(gu, gd, uy0, uy1, uz0, uz1, dy0, dy1, dz0, dz1, cellStart, syz, su, bu0, sd, bd0, hh, bu, bd);
  }
  if (valid) {
    upRaw[h] = bu;
    dnRaw[h] = bd;
  }
  // a copy that did not complete in time must land before the block's shared
  // memory is released: thread 0 waits once more (the copies are at most 16 KB
  // of device memory, microseconds against a limit of seconds; with the
  // injected fault nothing was issued, so nothing can land later)
  if (staged && threadIdx.x == 0) slab_wait(bar, waitLimit);
}

// K4b (row step 2, optional): a hit with no accepted pair on the adjacent
// rows may link across one missing row - up on row r + a, down on row r - b,
// (a, b) in {(2,1), (1,2), (2,2)} - with the residual (a + b) h - b u - a d,
// whose variance is f = (a + b)^2 + a^2 + b^2 times a cluster's, so the
// metric D = 2077 e_y^2 + 1536 e_zeta^2 scaled by 6 / f is the same 2-dof
// chi2 (accepted if 6 D <= kMaxMetric f); windows scale with the row
// distance.  The best pair minimises D / f (compared exactly as
// D1 f2 < D2 f1 in 64 bits), ties to the smaller u, then d.
struct GapBest {
  long long D = -1, f = 1;
  int u = -1, d = -1;  // sorted indices
  __device__ void offer(long long Dn, long long fn, int un, int dn) {
    if (6 * Dn > (long long)kMaxMetric * fn) return;
    if (u < 0 || Dn * f < D * fn || (Dn * f == D * fn && (un < u || (un == u && dn < d)))) {
      D = Dn;
      f = fn;
      u = un;
      d = dn;
    }
  }
};

// One (a, b) in the cell rectangles of the two rows.
__device__ inline void gap_cells(const RowGrid& gu, const RowGrid& gd, int npu, int npd, int a, int b, int2 hh,
                                 const int* __restrict__ cellStart, const int2* __restrict__ syz, GapBest& best) {
  const int yh = hh.x, zh = hh.y;
  int uy0, uy1, uz0, uz1, dy0, dy1, dz0, dz1;
  if (!cell_range(gu, npu, yh - a * kWinY, yh + a * kWinY, zh - a * kWinZ, zh + a * kWinZ, uy0, uy1, uz0, uz1)) return;
  if (!cell_range(gd, npd, yh - b * kWinY, yh + b * kWinY, zh - b * kWinZ, zh + b * kWinZ, dy0, dy1, dz0, dz1)) return;
  const long long f = (long long)((a + b) * (a + b) + a * a + b * b);
  for (int izu = uz0; izu <= uz1; ++izu) {
    const int ua = __ldg(cellStart + gu.cellBase + izu * gu.ny + uy0);
    const int ub = __ldg(cellStart + gu.cellBase + izu * gu.ny + uy1 + 1);
    for (int u = ua; u < ub; ++u) {
      const int2 pu = __ldg(syz + u);
      if (abs(pu.x - yh) > a * kWinY || abs(pu.y - zh) > a * kWinZ) continue;
      for (int izd = dz0; izd <= dz1; ++izd) {
        const int da = __ldg(cellStart + gd.cellBase + izd * gd.ny + dy0);
        const int db = __ldg(cellStart + gd.cellBase + izd * gd.ny + dy1 + 1);
        for (int d = da; d < db; ++d) {
          const int2 pd = __ldg(syz + d);
          if (abs(pd.x - yh) > b * kWinY || abs(pd.y - zh) > b * kWinZ) continue;
          const long long ey = (long long)(a + b) * yh - (long long)b * pu.x - (long long)a * pd.x;
          const long long ez = (long long)(a + b) * zh - (long long)b * pu.y - (long long)a * pd.y;
          best.offer((long long)kWeightY * ey * ey + (long long)kWeightZ * ez * ez, f, u, d);
        }
      }
    }
  }
}

// One (a, b) in the drift-ordered views: the candidates of each side into a
// bit mask, then the pairs of those inside.
__device__ inline void gap_view(const ZView& V, const ZRow& gu, const ZRow& gd, int a, int b, int2 hh, GapBest& best) {
  int ua, ub, da, db;
  if (!z_range(V, gu, hh.y - a * kWinZ, hh.y + a * kWinZ, ua, ub)) return;
  if (!z_range(V, gd, hh.y - b * kWinZ, hh.y + b * kWinZ, da, db)) return;
  const int2 *pu = V.yz(gu), *pd = V.yz(gd);
  const int f = (a + b) * (a + b) + a * a + b * b;
  auto inside = [&](int2 c, int w) {
    return (unsigned)(hh.x - c.x + w * kWinY) <= 2u * w * kWinY && (unsigned)(hh.y - c.y + w * kWinZ) <= 2u * w * kWinZ;
  };
  // 32 candidates of a side at a time (a window of 8 cm holds 12-20)
  for (int u0 = ua; u0 < ub; u0 += 32) {
    unsigned mu = 0;
#pragma unroll 4
    for (int i = 0; i < min(32, ub - u0); ++i) mu |= inside(__ldg(pu + u0 + i), a) ? 1u << i : 0u;
    if (!mu) continue;
    for (int d0 = da; d0 < db; d0 += 32) {
      unsigned md = 0;
#pragma unroll 4
      for (int i = 0; i < min(32, db - d0); ++i) md |= inside(__ldg(pd + d0 + i), b) ? 1u << i : 0u;
      if (!md) continue;
      for (unsigned m = mu; m; m &= m - 1) {
        const int u = u0 + __ffs(m) - 1;
        const int2 cu = __ldg(pu + u);
        const int ryu = b * (hh.x - cu.x), rzu = b * (hh.y - cu.y);
        for (unsigned k = md; k; k &= k - 1) {
          const int d = d0 + __ffs(k) - 1;
          const int2 cd = __ldg(pd + d);
          const int ey = ryu + a * (hh.x - cd.x), ez = rzu + a * (hh.y - cd.y);
          // past the cut for every f (<= 24): 6 * 2077 * 320^2 and 6 * 1536 * 370^2 > kMaxMetric * 24
          if (abs(ey) > 320 || abs(ez) > 370) continue;
          const long long D = (long long)(kWeightY * ey * ey) + (long long)(kWeightZ * ez * ez);
          if (6 * D <= (long long)kMaxMetric * f) best.offer(D, f, V.idx(gu, u), V.idx(gd, d));
        }
      }
    }
  }
}

// Blocks of kGapBlock hits of a row in drift order (as k_neighbours_view);
// the hits that found no adjacent-row pair are gathered first, so that whole
// warps work.  Rows flagged dense take the cells.
// 10 collisions of a 1 ms frame with 5 % of the clusters lost: 1.36 -> 0.21 ms.
template <int kB>
__global__ void __launch_bounds__(kB, kNFResident / kB) k_neighbours_gap(const int* __restrict__ nfBlockStart,
                                                       const int* __restrict__ nfBlockRow, int nRows,
                                                       const RowGrid* __restrict__ grid,
                                                       const int* __restrict__ cellStart,
                                                       const int2* __restrict__ syz, const GeomConst* __restrict__ G,
                                                       ZView zv, int* __restrict__ upRaw, int* __restrict__ dnRaw) {
  if ((int)blockIdx.x >= nfBlockStart[nRows]) return;  // launched with an upper bound of blocks
  __shared__ int s_pos[kB], s_cnt[kB / 32];
  const int R = nfBlockRow[blockIdx.x];
  const int r = (R % kRowsPerTF) % kNRow;
  if (r < 1 || r > kNRow - 2) return;
  const ZRow g = zv.rows[R];
  const int q = (blockIdx.x - nfBlockStart[R]) * kB + threadIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool free = q < g.count && upRaw[zv.idx(g, q)] < 0;
  const unsigned m = __ballot_sync(0xffffffffu, free);
  if (lane == 0) s_cnt[w] = __popc(m);
  __syncthreads();
  int before = __popc(m & ((1u << lane) - 1u)), total = 0;
  for (int k = 0; k < kB / 32; ++k) {
    if (k < w) before += s_cnt[k];
    total += s_cnt[k];
  }
  if (free) s_pos[before] = q;
  __syncthreads();
  if ((int)threadIdx.x >= total) return;
  const int p = s_pos[threadIdx.x];
  const int2 hh = zv.yz(g)[p];
  GapBest best;
  constexpr int kSteps[3][2] = {{2, 1}, {1, 2}, {2, 2}};
#pragma unroll 1
  for (int s = 0; s < 3; ++s) {
    const int a = kSteps[s][0], b = kSteps[s][1];
    if (r + a > kNRow - 1 || r - b < 0) continue;
    const ZRow gu = zv.rows[R + a], gd = zv.rows[R - b];
    if ((gu.flags | gd.flags) & kZNFCells)
      gap_cells(grid[R + a], grid[R - b], G->npads[r + a], G->npads[r - b], a, b, hh, cellStart, syz, best);
    else
      gap_view(zv, gu, gd, a, b, hh, best);
  }
  if (best.u >= 0) {
    const int h = zv.idx(g, p);
    upRaw[h] = best.u;
    dnRaw[h] = best.d;
  }
}

// K5 + K6a: reciprocity filter on the raw (snapshot) links and the chain-head
// flag: dn < 0, up >= 0, up[up] >= 0 (chains of at least three hits).
__global__ void k_clean(const int* __restrict__ nDev, const int* __restrict__ upRaw, const int* __restrict__ dnRaw,
                        int* __restrict__ up, int* __restrict__ dn, int* __restrict__ startFlag) {
  int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= *nDev) return;
  int u = upRaw[h], d = dnRaw[h];
  int uc = (u >= 0 && dnRaw[u] == h) ? u : -1;
  int dc = (d >= 0 && upRaw[d] == h) ? d : -1;
  up[h] = uc;
  dn[h] = dc;
  int flag = 0;
  if (dc < 0 && uc >= 0) {
    int uu = upRaw[uc];
    int uuc = (uu >= 0 && dnRaw[uu] == uc) ? uu : -1;
    flag = uuc >= 0;
  }
  startFlag[h] = flag;
}

// --------------------------------------------------------------- scans
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ inline int warp_incl(int x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// inclusive block scan for blockDim == 1024; returns the exclusive prefix
__device__ inline int block_excl(int v, int* total) {
  __shared__ int ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = warp_incl(v);
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) ws[lane] = warp_incl(ws[lane]);
  __syncthreads();
  int incl = x + (w > 0 ? ws[w - 1] : 0);
  if (total) *total = ws[31];
  __syncthreads();
  return incl - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const int* __restrict__ in, int nHost,
                                                            const int* __restrict__ nDev, int* __restrict__ sums) {
  const int n = nDev ? *nDev : nHost;
  long long base = (long long)blockIdx.x * kScanTile;
  int s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    long long i = base + (long long)k * kScanThreads + threadIdx.x;
    if (i < n) s += in[i];
  }
  int tot;
  block_excl(s, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_mid(int* __restrict__ sums, int nb) {
  int per = (nb + kScanThreads - 1) / kScanThreads;
  int b = threadIdx.x * per, e = min(nb, b + per);
  int s = 0;
  for (int i = b; i < e; ++i) s += sums[i];
  int off = block_excl(s, nullptr);
  for (int i = b; i < e; ++i) {
    int v = sums[i];
    sums[i] = off;
    off += v;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const int* __restrict__ in, int nHost,
                                                             const int* __restrict__ nDev, const int* __restrict__ sums,
                                                             int* __restrict__ out) {
  const int n = nDev ? *nDev : nHost;
  long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
  int v[kScanItems];
  int s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    long long i = base + k;
    v[k] = (i < n) ? in[i] : 0;
    s += v[k];
  }
  int tot;
  int off = block_excl(s, &tot) + sums[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    long long i = base + k;
    if (i < n) out[i] = off;
    off += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = off;
}

// out[0..m] = exclusive scan of in[0..m-1], out[m] = total, m = *nDev <= n
// (the grid covers n; tiles past m add zeros), or m = n when nDev is null;
// out may alias in.
// scratch: >= scan_scratch_ints(n) ints.
int scan_scratch_ints(long long n) { return (int)((n + kScanTile - 1) / kScanTile) + 1; }

__global__ void k_store_zero_at(int* __restrict__ out, int nHost, const int* __restrict__ nDev) {
  out[nDev ? *nDev : nHost] = 0;
}

// Short scans by one CTA in one launch, tile after tile (the next tile's
// values loaded ahead).  A tile takes about 1 us, the three launches of the
// tiled scan about 9 us: the line lies at eight tiles.
constexpr int kScanOneMax = 8 * kScanTile;
__global__ void __launch_bounds__(kScanThreads) k_scan_one(const int* __restrict__ in, int nHost,
                                                           const int* __restrict__ nDev, int* __restrict__ out) {
  const int n = nDev ? *nDev : nHost;
  int carry = 0, next[kScanItems];
  auto fetch = [&](int base) {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      const int i = base + threadIdx.x * kScanItems + k;
      next[k] = i < n ? in[i] : 0;
    }
  };
  fetch(0);
  for (int base = 0; base < n; base += kScanTile) {
    int v[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      v[k] = next[k];
      s += v[k];
    }
    if (base + kScanTile < n) fetch(base + kScanTile);
    int tot;
    int off = carry + block_excl(s, &tot);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      const int i = base + threadIdx.x * kScanItems + k;
      if (i < n) out[i] = off;
      off += v[k];
    }
    carry += tot;
  }
  if (threadIdx.x == 0) out[n] = carry;
}

void scan_exclusive(const int* in, int* out, int n, const int* nDev, int* scratch, cudaStream_t st) {
  int nb = (n + kScanTile - 1) / kScanTile;
  if (nb == 0) {
    k_store_zero_at<<<1, 1, 0, st>>>(out, n, nDev);
    ++g_launch_count;
    return;
  }
  if (n <= kScanOneMax) {
    k_scan_one<<<1, kScanThreads, 0, st>>>(in, n, nDev, out);
    ++g_launch_count;
    return;
  }
  k_scan_sums<<<nb, kScanThreads, 0, st>>>(in, n, nDev, scratch);
  ++g_launch_count;
  k_scan_mid<<<1, kScanThreads, 0, st>>>(scratch, nb);
  ++g_launch_count;
  k_scan_apply<<<nb, kScanThreads, 0, st>>>(in, n, nDev, scratch, out);
  ++g_launch_count;
}

// ---- processing order by length
// A block orders its kOrderChunk consecutive items longest first (a counting
// sort in shared memory).
constexpr int kOrderChunk = 1024, kOrderBins = 256;
__global__ void __launch_bounds__(kOrderChunk) k_length_order(const int* __restrict__ nDev, const int* __restrict__ a,
                                                              int diff, int* __restrict__ perm) {
  __shared__ int hist[kOrderBins];
  const int n = *nDev, base = blockIdx.x * kOrderChunk, i = base + threadIdx.x;
  if (base >= n) return;
  for (int b = threadIdx.x; b < kOrderBins; b += kOrderChunk) hist[b] = 0;
  __syncthreads();
  int bin = -1, rank = 0;
  if (i < n) {
    const int len = diff ? a[i + 1] - a[i] : a[i];
    bin = kOrderBins - 1 - min(max(len, 0), kOrderBins - 1);
    rank = atomicAdd(&hist[bin], 1);
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // exclusive scan of the bins
    constexpr int per = kOrderBins / 32;
    int v[per], sum = 0;
#pragma unroll
    for (int q = 0; q < per; ++q) {
      v[q] = hist[threadIdx.x * per + q];
      sum += v[q];
    }
    int x = warp_incl(sum) - sum;
#pragma unroll
    for (int q = 0; q < per; ++q) {
      hist[threadIdx.x * per + q] = x;
      x += v[q];
    }
  }
  __syncthreads();
  if (bin >= 0) perm[base + hist[bin] + rank] = i;
}

void launch_length_order(int n, const int* nDev, const int* a, bool diff, int* perm, cudaStream_t st) {
  if (n <= 0) return;
  k_length_order<<<(n + kOrderChunk - 1) / kOrderChunk, kOrderChunk, 0, st>>>(nDev, a, diff ? 1 : 0, perm);
  ++g_launch_count;
}

// *dst = min(arr[*idx], cap) (a count read off the end of a scan), flagging
// an overflow; optionally also writes the count at base[*dst] (CSR end).
__global__ void k_count_at(const int* __restrict__ arr, const int* __restrict__ idx, int* __restrict__ dst, int cap,
                           int* __restrict__ overflow, const int* __restrict__ arr2, int* __restrict__ dst2, int cap2,
                           int* __restrict__ endBase) {
  int v = arr[*idx];
  if (v > cap) {
    v = cap;
    *overflow = 1;
  }
  *dst = v;
  if (arr2) {
    int v2 = arr2[*idx];
    if (v2 > cap2) {
      v2 = cap2;
      *overflow = 1;
    }
    *dst2 = v2;
    if (endBase) endBase[v] = v2;
  }
}

// first entry of a sorted list that is >= each TF's first sorted hit
__global__ void k_tf_ranges(int nTF, const RowGrid* __restrict__ grid, const int* __restrict__ list,
                            const int* __restrict__ nListDev, int* __restrict__ tfBegin) {
  int tf = blockIdx.x * blockDim.x + threadIdx.x;
  if (tf > nTF) return;
  const int nList = *nListDev;
  int key = (tf == nTF) ? INT_MAX : grid[tf * kRowsPerTF].start;
  int lo = 0, hi = nList;
  while (lo < hi) {
    int m = (lo + hi) >> 1;
    if (list[m] < key) lo = m + 1;
    else hi = m;
  }
  tfBegin[tf] = (tf == nTF) ? nList : lo;
}

// out[i] = first index of the sorted list with list[j] >= keys[i]
__global__ void k_lower_bounds(const int* __restrict__ list, const int* __restrict__ nListDev,
                               const int* __restrict__ keys, int nKeys, int* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nKeys) return;
  const int nList = *nListDev;
  const int key = keys[i];
  int lo = 0, hi = nList;
  while (lo < hi) {
    int m = (lo + hi) >> 1;
    if (list[m] < key) lo = m + 1;
    else hi = m;
  }
  out[i] = lo;
}

// ------------------------------------------------------------- launchers
void launch_lower_bounds(const int* list, const int* nListDev, const int* keys, int nKeys, int* out,
                         cudaStream_t st) {
  if (nKeys > 0) {
    k_lower_bounds<<<(nKeys + 127) / 128, 128, 0, st>>>(list, nListDev, keys, nKeys, out);
    ++g_launch_count;
  }
}

void launch_neighbours(int nfBlocks, int hitsPerBlock, bool stage, const RowGrid* grid, const int* nfBlockStart,
                       const int* nfBlockRow, int nRows, const int* cellStart, const int2* syz, const GeomConst* G,
                       ZView zv, int* upRaw, int* dnRaw, unsigned* err, cudaStream_t st, unsigned inject) {
  if (nfBlocks > 0) {
#define O2TPC_NF(B)                                                                                                  \
  if (stage)                                                                                                         \
    k_neighbours_staged<B><<<nfBlocks, B, 0, st>>>(grid, nfBlockStart, nRows, cellStart, syz, G, upRaw, dnRaw, err,  \
                                                   inject);                                                          \
  else                                                                                                               \
    k_neighbours_view<B><<<nfBlocks, B, 0, st>>>(grid, nfBlockStart, nfBlockRow, nRows, cellStart, syz, G, zv, upRaw, dnRaw)
    if (hitsPerBlock == 64) {
      O2TPC_NF(64);
    } else if (hitsPerBlock == 256) {
      O2TPC_NF(256);
    } else {
      O2TPC_NF(128);
    }
#undef O2TPC_NF
    ++g_launch_count;
  }
}

void launch_neighbours_gap(int nfBlocks, int hitsPerBlock, const int* nfBlockStart, const int* nfBlockRow,
                           const RowGrid* grid, int nRows, const int* cellStart, const int2* syz, const GeomConst* G, ZView zv, int* upRaw, int* dnRaw,
                           cudaStream_t st) {
  if (nfBlocks > 0) {
#define O2TPC_GAP(B) \
  k_neighbours_gap<B><<<nfBlocks, B, 0, st>>>(nfBlockStart, nfBlockRow, nRows, grid, cellStart, syz, G, zv, upRaw, dnRaw)
    if (hitsPerBlock == 64) O2TPC_GAP(64);
    else if (hitsPerBlock == 256) O2TPC_GAP(256);
    else O2TPC_GAP(128);
#undef O2TPC_GAP
    ++g_launch_count;
  }
}

void launch_clean(int n, const int* nDev, const int* upRaw, const int* dnRaw, int* up, int* dn, int* startFlag,
                  cudaStream_t st) {
  if (n > 0) {
    k_clean<<<(n + 255) / 256, 256, 0, st>>>(nDev, upRaw, dnRaw, up, dn, startFlag);
    ++g_launch_count;
  }
}


// ---- ordered compaction with warp ballots
// Flags are taken in tiles of kBallotTile (1024 threads x 4 chunks).  Pass 1
// counts each tile's set flags with one ballot and popcount per warp and
// chunk; the tile counts are scanned; pass 2 writes every flagged index at
// tile offset + earlier chunks + earlier warps (a 32-entry shuffle scan) +
// its rank among the set lanes of its warp (popcount of the lower lanes).
// Only one int per tile is scanned instead of one per flag.
constexpr int kBallotTile = 4096;

__global__ void __launch_bounds__(1024) k_ballot_counts(const int* __restrict__ flag, const int* __restrict__ nDev,
                                                        int* __restrict__ tileCnt) {
  __shared__ int ws[32];
  const int n = *nDev, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int c = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = blockIdx.x * kBallotTile + k * 1024 + threadIdx.x;
    c += __popc(__ballot_sync(0xffffffffu, i < n && flag[i] != 0));
  }
  if (lane == 0) ws[w] = c;
  __syncthreads();
  if (w == 0) {
    int v = ws[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) tileCnt[blockIdx.x] = v;
  }
}

__global__ void __launch_bounds__(1024) k_ballot_compact(const int* __restrict__ flag, const int* __restrict__ nDev,
                                                         const int* __restrict__ tileOff, int* __restrict__ out,
                                                         int cap, int* __restrict__ overflow) {
  __shared__ int ws[32], s_tot;
  const int n = *nDev, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int carry = tileOff[blockIdx.x];
  for (int k = 0; k < 4; ++k) {
    const int i = blockIdx.x * kBallotTile + k * 1024 + threadIdx.x;
    const bool f = i < n && flag[i] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) ws[w] = __popc(m);
    __syncthreads();
    if (w == 0) {  // exclusive scan of the 32 warp counts
      const int v = ws[lane];
      int x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      ws[lane] = x - v;
      if (lane == 31) s_tot = x;
    }
    __syncthreads();
    if (f) {
      const int p = carry + ws[w] + __popc(m & ((1u << lane) - 1u));
      if (p < cap) out[p] = i;
      else *overflow = 1;
    }
    carry += s_tot;
    __syncthreads();
  }
}

// *dst = min(total, cap) with total = tileOff[number of tiles of *nDev]
__global__ void k_ballot_total(const int* __restrict__ tileOff, const int* __restrict__ nDev, int* __restrict__ dst,
                               int cap, int* __restrict__ overflow) {
  int v = tileOff[(*nDev + kBallotTile - 1) / kBallotTile];
  if (v > cap) {
    v = cap;
    *overflow = 1;
  }
  *dst = v;
}

int ballot_tiles(long long n) { return (int)((n + kBallotTile - 1) / kBallotTile); }

void launch_ballot_count(int n, const int* nDev, const int* flag, int* tileCnt, int* tileOff, int* count, int cap,
                         int* overflow, int* scratch, cudaStream_t st) {
  const int nt = ballot_tiles(n);
  if (nt > 0) {
    k_ballot_counts<<<nt, 1024, 0, st>>>(flag, nDev, tileCnt);
    ++g_launch_count;
  }
  // tiles past *nDev count zero; the scan runs over all nt
  scan_exclusive(tileCnt, tileOff, nt, nullptr, scratch, st);
  k_ballot_total<<<1, 1, 0, st>>>(tileOff, nDev, count, cap, overflow);
  ++g_launch_count;
}

void launch_ballot_compact(int n, const int* nDev, const int* flag, const int* tileOff, int* out, int cap,
                           int* overflow, cudaStream_t st) {
  const int nt = ballot_tiles(n);
  if (nt > 0) {
    k_ballot_compact<<<nt, 1024, 0, st>>>(flag, nDev, tileOff, out, cap, overflow);
    ++g_launch_count;
  }
}

__global__ void k_iota(int* __restrict__ out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = i;
}

__global__ void k_stream_tail() {}

void launch_stream_tail(cudaStream_t st) {
  k_stream_tail<<<1, 32, 0, st>>>();
  ++g_launch_count;
}

void launch_iota(int* out, int n, cudaStream_t st) {
  if (n > 0) {
    k_iota<<<(n + 255) / 256, 256, 0, st>>>(out, n);
    ++g_launch_count;
  }
}

void launch_count_at(const int* arr, const int* idx, int* dst, int cap, int* overflow, cudaStream_t st,
                     const int* arr2, int* dst2, int cap2, int* endBase) {
  k_count_at<<<1, 1, 0, st>>>(arr, idx, dst, cap, overflow, arr2, dst2, cap2, endBase);
  ++g_launch_count;
}

void launch_tf_ranges(int nTF, const RowGrid* grid, const int* list, const int* nListDev, int* tfBegin,
                      cudaStream_t st) {
  k_tf_ranges<<<(nTF + 1 + 63) / 64, 64, 0, st>>>(nTF, grid, list, nListDev, tfBegin);
  ++g_launch_count;
}

}  // namespace o2tpc
