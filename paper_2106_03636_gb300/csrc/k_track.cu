// k_track.cu - TrackletConstructor, TrackletSelector and the sector-track fits.
//
// A tracklet starts at a chain head: the chain's hits are fitted with the
// FP32 Kalman filter, the track is followed outward row by row (best hit in a
// +-3 sigma window, chi2 <= 18, stop after 4 rows without a hit or at
// |sin phi| > 0.95), then refitted inward from its top hit and followed below
// the chain start.  The selector gives every hit to the longest tracklet
// holding it (ties: the earlier start) through a 64-bit atomicMax of
// (nHits << 32 | ~id), which makes the result independent of thread order,
// splits tracklets at gaps of more than 4 rows and keeps segments of >= 10
// owned hits as sector tracks, each refitted outward and inward.
#include <algorithm>

#include "o2tpc_kernels.cuh"

namespace o2tpc {

// Hit coordinates in cm relative to per-fit origins (yref, zref in integer
// units): the fits then work on small magnitudes, where single precision keeps
// its digits.
__device__ inline float hit_y(int yu, int yref) { return (float)(yu - yref) * 0.00625f; }
__device__ inline float hit_z(int zu, int zref, float zunit) { return (float)(zu - zref) * zunit; }

// Row (batch-global) holding sorted hit h.
__device__ inline int find_row(const RowGrid* __restrict__ grid, int nRows, int h) {
  int lo = 0, hi = nRows;
  while (lo < hi) {
    int m = (lo + hi) >> 1;
    if (grid[m].start <= h) lo = m + 1;
    else hi = m;
  }
  return lo - 1;
}

// Row of hit h linked up from a hit on row R: R + 1, or R + 2 when the link
// crosses a missing row (only with row step 2; without it no row is read).
__device__ inline int link_row(const RowGrid* __restrict__ grid, int R, int h, int rowStep2) {
  if (!rowStep2) return R + 1;
  const RowGrid g = grid[R + 1];
  return h < g.start + g.count ? R + 1 : R + 2;
}

__device__ inline int clamp_i(float v) { return (int)fminf(fmaxf(v, -1.0e9f), 1.0e9f); }

__device__ inline void reset_cov(KState<float>& s, int angErr) {
#pragma unroll
  for (int i = 0; i < 15; ++i) s.C[i] = 0.f;
  kf_meas_cov<float>(s, angErr);
  s.C[5] = 0.04f;
  s.C[9] = 0.25f;
  s.C[14] = 400.f;
}

// Stores a state with y back in absolute cm (yref in units).
__device__ inline void store_state(float* dst, const KState<float>& s, int yref) {
  dst[0] = s.x;
#pragma unroll
  for (int i = 0; i < 5; ++i) dst[1 + i] = s.p[i];
  dst[1] = s.p[0] + (float)yref * 0.00625f;
#pragma unroll
  for (int i = 0; i < 15; ++i) dst[6 + i] = s.C[i];
}
// Stores a state as it is (y relative to the fit's origin): the hand-over
// between the passes of the tracklet constructor.
__device__ inline void store_raw(float* dst, const KState<float>& s) {
  dst[0] = s.x;
#pragma unroll
  for (int i = 0; i < 5; ++i) dst[1 + i] = s.p[i];
#pragma unroll
  for (int i = 0; i < 15; ++i) dst[6 + i] = s.C[i];
}
__device__ inline void load_state(KState<float>& s, const float* src) {
  s.x = src[0];
#pragma unroll
  for (int i = 0; i < 5; ++i) s.p[i] = src[1 + i];
#pragma unroll
  for (int i = 0; i < 15; ++i) s.C[i] = src[6 + i];
}

// K7: the TrackletConstructor in four passes, one persistent kernel each:
// (a) chain fit, (b) outward following, (c) inward refit of the attached
// hits, (d) inward following below the chain start.  Within a pass every
// lane runs the same loop body (transport, then either the next known hit or
// a row search, then the update), so a warp stays converged; lanes take the
// next tracklet from a global counter as soon as theirs is done.  Between the
// passes a tracklet's state waits in tb.state (21 floats), its hit count in
// tb.nasc and its row base in tb.rbase; tb.nhits is written by the last pass
// (0: dropped).  Results do not depend on which thread builds which tracklet.

// Lanes with want = true take consecutive work items from *counter, one
// atomic per warp; returns this lane's item (meaningful where want).  All 32
// lanes must call it.
__device__ inline int warp_take(int* counter, bool want) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(full, want);
  int base = 0;
  if (m) {
    const int leader = __ffs(m) - 1;
    if (lane == leader) base = atomicAdd(counter, __popc(m));
    base = __shfl_sync(full, base, leader);
  }
  return base + __popc(m & ((1u << lane) - 1u));
}

// (a) chain fit: seed from the first and third chain hits, then one update
// per chain hit.  A transport failure drops the tracklet.  With enough
// tracklets to fill the GPU a first kernel follows the links alone and lists the
// hits, so that the fits can be taken in order of length: the chains' lengths
// differ so much that a warp of consecutive ones has 9 of 32 lanes active.
// Below kChainOrdered tracklets (about an eighth of the GPU's threads) the time
// is one chain's latency, and the fit follows the links itself.
// 1 ms frame (664 k tracklets) 0.57 -> 0.34 ms + 0.15 for the walk and the order,
// 32 orbits 1.57 -> 0.89 + 0.5.
// One CTA per SM as the least for the fits (here, the refits, the sector fits, the
// merger's pairs): they are bound by their chains of arithmetic, so registers
// (72-96 against 68-72) count for more than warps; 16 orbits: chain and refit
// 1.73 -> 1.68 ms, sector fits 0.65 -> 0.63 ms; with 64 registers 1.80 and 0.68.
constexpr int kChainOrdered = 40000;

__global__ void __launch_bounds__(256) k_tl_walk(const int* __restrict__ nTlDev, const int* __restrict__ starts,
                                                 const int* __restrict__ up, TrackletBufs tb) {
  const int k = blockIdx.x * 256 + threadIdx.x, nTl = *nTlDev;
  if (k >= nTl) return;
  if (nTl < kChainOrdered) {
    tb.nasc[k] = 0;
    return;
  }
  int* H = tb.hits + (size_t)k * kMaxTlHits;
  int n = 0;
  for (int h = starts[k]; h >= 0 && n < kMaxTlHits; h = up[h]) H[n++] = h;
  tb.nasc[k] = n;
}

__global__ void __launch_bounds__(128, 1) k_tl_chain(const int* __restrict__ nTlDev, int* __restrict__ counter,
                                                  const int* __restrict__ perm, const int* __restrict__ starts,
                                                  const int* __restrict__ up, const RowGrid* __restrict__ grid,
                                                  int nRows, const int2* __restrict__ syz,
                                                  const GeomConst* __restrict__ G, TrackletBufs tb) {
  const float zunit = G->zunit, bzc = G->bzc;
  const int rs2 = G->rowStep2;
  const int nTl = *nTlDev;
  const bool walked = nTl >= kChainOrdered;
  for (int k; take_ordered(counter, walked ? perm : nullptr, nTl, k);) {
    if (k < 0) continue;
    const int h0 = starts[k];
    const int R0 = find_row(grid, nRows, h0);
    const int r0 = (R0 % kRowsPerTF) % kNRow;
    int* H = tb.hits + (size_t)k * kMaxTlHits;
    uint8_t* Rw = tb.rows + (size_t)k * kMaxTlHits;
    const int len = walked ? tb.nasc[k] : kMaxTlHits;
    // the hit after the n-th, which is h: from the list, or by the link
    auto link = [&](int n, int h) { return walked ? (n + 1 < len ? H[n + 1] : -1) : up[h]; };
    const int2 a0 = syz[h0];
    const int zref = a0.y;
    int yref = a0.x;
    tb.zref[k] = zref;
    tb.rbase[k] = R0 - r0;
    const int h1 = link(0, h0);
    const int R1 = link_row(grid, R0, h1, rs2);
    const int h2 = link(1, h1);
    const int R2 = link_row(grid, R1, h2, rs2);
    const int2 a2 = syz[h2];
    const float x0 = G->rowx[r0];
    const float dx = (float)(R2 - R0) * G->pitch, dy = hit_y(a2.x, yref) - hit_y(a0.x, yref);
    const float tphi = dy / dx;
    const float s0 = tphi / sqrtf(1.f + tphi * tphi);
    const float t0 = (hit_z(a2.y, zref, zunit) - hit_z(a0.y, zref, zunit)) / sqrtf(dx * dx + dy * dy);
    KState<float> st;
    kf_reset<float>(st, x0, hit_y(a0.x, yref), hit_z(a0.y, zref, zunit), s0, t0, 0.f);
    kf_meas_cov<float>(st, G->angErr);
    H[0] = h0;
    Rw[0] = (uint8_t)r0;
    int nc = 1, hit = h1, prev = r0, Rh = R1;
    int2 hn = syz[h1];
    int next = h2;
    bool dropped = false;
    while (hit >= 0 && nc < kMaxTlHits) {
      const int row = r0 + (Rh - R0);
      // the next hit's coordinates and link, in flight during this hit's step
      const int2 hp = hn;
      int after = -1;
      if (next >= 0) {
        hn = syz[next];
        after = link(nc + 1, next);
      }
      if (kf_prop_row<float, kF1Rounded>(st, prev, row, G, bzc) != 0) {
        dropped = true;
        break;
      }
      recentre_y(st.p[0], yref, hp.x);
      kf_update<float>(st, hit_y(hp.x, yref), hit_z(hp.y, zref, zunit), nullptr, G->angErr);
      if (!walked) H[nc] = hit;
      Rw[nc] = (uint8_t)row;
      ++nc;
      prev = row;
      hit = next;
      next = after;
      if (hit >= 0) Rh = link_row(grid, Rh, hit, rs2);
    }
    tb.nasc[k] = dropped ? 0 : nc;
    tb.yref[k] = yref;
    if (dropped) tb.nhits[k] = 0;
    else store_raw(tb.state + (size_t)k * 21, st);
  }
}

// (c) inward refit from the top hit through every attached hit; a hit whose
// transport fails is skipped.  One thread per tracklet, the tracklets in
// order of their length; hits are loaded one step ahead.
// 1 ms frame (664 k tracklets): 0.64 -> 0.49 ms, 32 orbits 1.85 -> 1.43 ms (27 of
// 32 lanes active, 20 in plain order; now 65 % issue-active).
__global__ void __launch_bounds__(128, 1) k_tl_refit(const int* __restrict__ nTlDev, int* __restrict__ counter,
                                                            const int* __restrict__ perm, const int2* __restrict__ syz,
                                                            const GeomConst* __restrict__ G, TrackletBufs tb) {
  const float zunit = G->zunit, bzc = G->bzc;
  const int nTl = *nTlDev;
  for (int k; take_ordered(counter, perm, nTl, k);) {
    if (k < 0) continue;
    const int na = tb.nasc[k];
    if (na == 0) continue;
    const int* H = tb.hits + (size_t)k * kMaxTlHits;
    const uint8_t* Rw = tb.rows + (size_t)k * kMaxTlHits;
    const int zref = tb.zref[k];
    int yref = tb.yref[k];
    // from the top hit, with the direction that the outward pass left and a
    // fresh covariance
    KState<float> st;
    float* S = tb.state + (size_t)k * 21;
    const int2 top = syz[H[na - 1]];
    int srow = Rw[na - 1];
    st.x = G->rowx[srow];
    st.p[0] = hit_y(top.x, yref);
    st.p[1] = hit_z(top.y, zref, zunit);
    st.p[2] = S[3];
    st.p[3] = S[4];
    st.p[4] = S[5];
    reset_cov(st, G->angErr);
    int2 hn = na > 1 ? syz[H[na - 2]] : top;
    int rn = na > 1 ? Rw[na - 2] : 0;
    for (int i = na - 2; i >= 0; --i) {
      const int2 hp = hn;
      const int row = rn;
      if (i > 0) {
        hn = syz[H[i - 1]];
        rn = Rw[i - 1];
      }
      if (kf_prop_row<float, kF1Rounded>(st, srow, row, G, bzc) != 0) continue;
      srow = row;
      recentre_y(st.p[0], yref, hp.x);
      kf_update<float>(st, hit_y(hp.x, yref), hit_z(hp.y, zref, zunit), nullptr, G->angErr);
    }
    tb.yref[k] = yref;
    store_raw(S, st);
  }
}

// --------------------------------------------- following (passes b, d)
// From the row after the chain's top (b, outward) or below its start (d,
// inward), one pad row per step: transport, search the +-3 sigma window of
// the prediction, update with the best hit; stop after kMaxMiss rows without
// a hit, at the row range end, on a transport failure or when |sin phi| >
// kSinFollow.  The state after the last accepted hit is kept (shared memory)
// and is the pass's result.
//
// One persistent kernel per direction, written as one loop in which every
// iteration is one row step of every busy lane: a lane whose tracklet ends
// takes the next one (one atomic per warp for all such lanes), so the
// transport and the update run converged whatever the tracklets' lengths.
// The row search comes in two forms that pick the same hit:
// * per lane: each lane scans the candidates of its own window, in the row's
//   drift-ordered view;
// * warp-cooperative: the candidate cells of all lanes' windows on this step
//   are laid out one after another and scanned 32 at a time by the whole warp
//   (a lane finds the owner of candidate q by a binary search over the
//   warp's exclusive candidate offsets; per owner the smallest key wins).
// Both score a candidate by the same explicitly rounded expression and keep
// the smallest (chi2 bits << 32 | hit) - chi2 >= 0, so its bit pattern orders
// like its value - which is the rule "smallest chi2, then the smaller
// sorted index".

struct SearchPar {
  float y, z, wy, wz, isy2, isz2;
  int yref, zref;
};

// Window of a row search: its parameters and drift range; false: unusable, no
// candidate can pass.  The range only has to cover the window: one unit of
// slack on each side absorbs the rounding of the float products.
__device__ inline bool search_window(const KState<float>& s, int yref, int zref, float izunit, int angErr,
                                     SearchPar& P, int& zlo, int& zhi) {
  float vy, vz;
  meas_var<float>(angErr, s, vy, vz);
  const float sy2 = s.C[0] + vy, sz2 = s.C[2] + vz;
  const float wy = 3.f * sqrtf(sy2), wz = 3.f * sqrtf(sz2);
  if (!(wy < 1e4f) || !(wz < 1e4f) || !isfinite(s.p[0]) || !isfinite(s.p[1])) return false;
  zlo = zref + clamp_i(floorf((s.p[1] - wz) * izunit)) - 1;
  zhi = zref + clamp_i(ceilf((s.p[1] + wz) * izunit)) + 1;
  P.y = s.p[0];
  P.z = s.p[1];
  P.wy = wy;
  P.wz = wz;
  P.isy2 = 1.f / sy2;
  P.isz2 = 1.f / sz2;
  P.yref = yref;
  P.zref = zref;
  return true;
}
// The window's y range in units, with the same slack.
__device__ inline void window_y(const SearchPar& P, int& ylo, int& yhi) {
  ylo = P.yref + clamp_i(floorf((P.y - P.wy) * 160.f)) - 1;
  yhi = P.yref + clamp_i(ceilf((P.y + P.wy) * 160.f)) + 1;
}

constexpr unsigned long long kNoHit = ~0ull;

// Key of candidate hit h at p against window P, or kNoHit if it fails the
// window or the chi2 cut.  Every operation is rounded explicitly, so the key
// is the same number wherever this is inlined.
__device__ inline unsigned long long cand_key(int h, int2 p, const SearchPar& P, float zunit) {
  const float dy = __fsub_rn(__fmul_rn((float)(p.x - P.yref), 0.00625f), P.y);
  const float dz = __fsub_rn(__fmul_rn((float)(p.y - P.zref), zunit), P.z);
  if (fabsf(dy) > P.wy || fabsf(dz) > P.wz) return kNoHit;
  const float chi = __fadd_rn(__fmul_rn(__fmul_rn(dy, dy), P.isy2), __fmul_rn(__fmul_rn(dz, dz), P.isz2));
  if (chi > kChi2Follow) return kNoHit;
  return ((unsigned long long)__float_as_uint(chi) << 32) | (unsigned)h;
}

// Best hit of a search: its place in the row's view (cells: its sorted index),
// -1 for none, and its coordinates.
struct BestHit {
  int pos;
  int2 p;
};

// Per-lane search through the cells [iy0, iy1] of rows [iz0, iz1] (rows so
// dense that the cells hold fewer candidates than the drift window).
__device__ inline BestHit cell_search(const RowGrid& g, int iy0, int iy1, int iz0, int iz1,
                                      const int* __restrict__ cellStart, const int2* __restrict__ syz,
                                      const SearchPar& P, float zunit) {
  unsigned long long best = kNoHit;
  BestHit B{-1, make_int2(0, 0)};
  for (int iz = iz0; iz <= iz1; ++iz) {
    const int cb = g.cellBase + iz * g.ny;
    const int a = __ldg(cellStart + cb + iy0);
    const int b = __ldg(cellStart + cb + iy1 + 1);
    for (int h = a; h < b; ++h) {
      const int2 p = __ldg(syz + h);
      const unsigned long long key = cand_key(h, p, P, zunit);
      if (key < best) {
        best = key;
        B.pos = h;
        B.p = p;
      }
    }
  }
  return B;
}

// Per-lane search through positions [a, b) of a row's drift-ordered view:
// four candidates loaded at once (a window holds 3-4 on average), so a row
// step waits for one load and not for one per candidate.  Equal chi2 (rare)
// goes to the smaller sorted index.
__device__ inline BestHit z_search(const ZView& V, const ZRow& g, int a, int b, const SearchPar& P, float zunit) {
  const int2* yz = V.yz(g);
  unsigned best = ~0u;
  bool tie = false;
  BestHit B{-1, make_int2(0, 0)};
  for (int h = a; h < b; h += 4) {
    int2 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = __ldg(yz + min(h + u, b - 1));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      // as cand_key, without branches
      const float dy = __fsub_rn(__fmul_rn((float)(q[u].x - P.yref), 0.00625f), P.y);
      const float dz = __fsub_rn(__fmul_rn((float)(q[u].y - P.zref), zunit), P.z);
      const float chi = __fadd_rn(__fmul_rn(__fmul_rn(dy, dy), P.isy2), __fmul_rn(__fmul_rn(dz, dz), P.isz2));
      const bool ok = (h + u < b) & (fabsf(dy) <= P.wy) & (fabsf(dz) <= P.wz) & (chi <= kChi2Follow);
      const unsigned c = ok ? __float_as_uint(chi) : ~0u;
      tie |= ok & (c == best);
      const bool take = c < best;
      best = take ? c : best;
      B.pos = take ? h + u : B.pos;
      B.p.x = take ? q[u].x : B.p.x;
      B.p.y = take ? q[u].y : B.p.y;
    }
  }
  if (tie) {
    for (int h = a; h < b; ++h) {
      const int2 q = __ldg(yz + h);
      if ((unsigned)(cand_key(0, q, P, zunit) >> 32) == best && V.idx(g, h) < V.idx(g, B.pos)) {
        B.pos = h;
        B.p = q;
      }
    }
  }
  return B;
}

// Warp-cooperative search.  Lane l searches cell rows [iz0, iz0 + nseg) x
// columns [iy0, iy1] of its window sp[l] when nseg > 0; returns its best key.
// All 32 lanes must call it.  sp / sbest: this warp's 32 slots.
__device__ inline unsigned long long coop_search(int nseg, int cellBase, int ny, int iy0, int iy1, int iz0,
                                                 const int* __restrict__ cellStart, const int2* __restrict__ syz,
                                                 const SearchPar* sp, unsigned long long* sbest, float zunit) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  sbest[lane] = kNoHit;
  const int maxseg = (int)__reduce_max_sync(full, (unsigned)nseg);
  __syncwarp();
  for (int j = 0; j < maxseg; ++j) {
    int a = 0, c = 0;
    if (j < nseg) {
      const int cb = cellBase + (iz0 + j) * ny;
      a = __ldg(cellStart + cb + iy0);
      c = __ldg(cellStart + cb + iy1 + 1) - a;
    }
    int inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(full, inc, o);
      if (lane >= o) inc += v;
    }
    const int total = __shfl_sync(full, inc, 31);
    const int exc = inc - c;
    for (int base = 0; base < total; base += 32) {
      const int q = base + lane;
      // owner: the last lane whose candidates start at or before q
      int own = 0, eown = 0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int e = __shfl_sync(full, exc, own + step);
        if (e <= q) {
          own += step;
          eown = e;
        }
      }
      const int aown = __shfl_sync(full, a, own);
      unsigned long long key = kNoHit;
      if (q < total) {
        const int h = aown + (q - eown);
        key = cand_key(h, __ldg(syz + h), sp[own], zunit);
      } else {
        own = 32;  // past the end: a run of its own
      }
      // minimum over each run of equal owners (the runs are contiguous)
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_down_sync(full, key, o);
        const int ow = __shfl_down_sync(full, own, o);
        if (lane + o < 32 && ow == own && v < key) key = v;
      }
      const int prevOwn = __shfl_up_sync(full, own, 1);
      if (own < 32 && (lane == 0 || prevOwn != own) && key < sbest[own]) sbest[own] = key;
      __syncwarp();
    }
  }
  __syncwarp();
  return sbest[lane];
}

// (b) kDir = +1: outward following above the chain; its result is the
// inward refit's starting point: the direction parameters of the last
// accepted state (position: the top hit; fresh covariance).  (d) kDir = -1:
// inward following below the chain start; the state kept is the one at the
// innermost accepted hit.
// This form searches warp-cooperatively (O2TPC_FLAG_COOP_SEARCH).
template <int kDir>
__global__ void __launch_bounds__(128, 7) k_tl_follow_coop(const int* __restrict__ nTlDev, int* __restrict__ counter,
                                                     const RowGrid* __restrict__ grid,
                                                     const int* __restrict__ cellStart,
                                                     const int2* __restrict__ syz,
                                                     const GeomConst* __restrict__ G, TrackletBufs tb) {
  __shared__ float s_last[21][128];
  __shared__ SearchPar s_par[128];
  __shared__ unsigned long long s_best[128];
  const unsigned full = 0xffffffffu;
  const int wb = threadIdx.x & ~31;
  const float zunit = G->zunit, izunit = G->kz, bzc = G->bzc;
  const int nTl = *nTlDev;
  auto save_last = [&](const KState<float>& q) {
    s_last[0][threadIdx.x] = q.x;
#pragma unroll
    for (int j = 0; j < 5; ++j) s_last[1 + j][threadIdx.x] = q.p[j];
#pragma unroll
    for (int j = 0; j < 15; ++j) s_last[6 + j][threadIdx.x] = q.C[j];
  };
  bool have = false, exhausted = false;
  int k = 0, r = 0, n = 0, misses = 0, srow = 0, yref = 0, yrefLast = 0, zref = 0, Rs = 0;
  KState<float> st;
  // ends the lane's tracklet with the state after its last accepted hit
  auto finish = [&]() {
    st.x = s_last[0][threadIdx.x];
#pragma unroll
    for (int j = 0; j < 5; ++j) st.p[j] = s_last[1 + j][threadIdx.x];
#pragma unroll
    for (int j = 0; j < 15; ++j) st.C[j] = s_last[6 + j][threadIdx.x];
    yref = yrefLast;
    float* S = tb.state + (size_t)k * 21;
    if (kDir > 0) {
      const int2 p = syz[tb.hits[(size_t)k * kMaxTlHits + n - 1]];  // the top hit
      recentre_y(st.p[0], yref, p.x);
      st.p[0] = hit_y(p.x, yref);
      st.p[1] = hit_z(p.y, zref, zunit);
      reset_cov(st, G->angErr);
      tb.nasc[k] = n;
      tb.yref[k] = yref;
      store_raw(S, st);
    } else {
      tb.nhits[k] = n;
      store_state(S, st, yref);
    }
    have = false;
  };
  for (;;) {
    // lanes without a tracklet take the next ones
    const bool want = !have && !exhausted;
    const int kk = warp_take(counter, want);
    {
      if (want) {
        k = kk;
        if (k >= nTl) {
          exhausted = true;
        } else {
          const int na = tb.nasc[k];
          if (na > 0) {
            const uint8_t* Rw = tb.rows + (size_t)k * kMaxTlHits;
            Rs = tb.rbase[k];
            zref = tb.zref[k];
            yref = tb.yref[k];
            load_state(st, tb.state + (size_t)k * 21);
            n = na;
            r = (kDir > 0) ? Rw[na - 1] + 1 : Rw[0] - 1;
            misses = 0;
            srow = row_of_x(st.x);
            save_last(st);
            yrefLast = yref;
            have = true;
          }
        }
      }
    }
    if (__ballot_sync(full, have) == 0) {
      if (__all_sync(full, exhausted)) break;
      continue;
    }
    // one row step of every busy lane: transport, then the window
    int nseg = 0, cellBase = 0, ny = 0, iy0 = 0, iy1 = 0, iz0 = 0, iz1 = 0;
    SearchPar P;
    if (have) {
      if ((kDir > 0) ? (r >= kNRow) : (r < 0)) {
        finish();
      } else if (kf_prop_row<float, kF1Fused>(st, srow, r, G, bzc) != 0 || fabsf(st.p[2]) > kSinFollow) {
        finish();
      } else {
        srow = r;
        const RowGrid g = grid[Rs + r];
        int ylo, yhi, zlo, zhi;
        if (g.count > 0 && search_window(st, yref, zref, izunit, G->angErr, P, zlo, zhi)) {
          window_y(P, ylo, yhi);
          if (cell_range(g, G->npads[r], ylo, yhi, zlo, zhi, iy0, iy1, iz0, iz1)) nseg = iz1 - iz0 + 1;
          cellBase = g.cellBase;
          ny = g.ny;
        }
      }
    }
    if (nseg > 0) s_par[threadIdx.x] = P;
    __syncwarp();
    const unsigned long long best =
        coop_search(nseg, cellBase, ny, iy0, iy1, iz0, cellStart, syz, s_par + wb, s_best + wb, zunit);
    if (have) {
      if (best != kNoHit) {
        const int hit = (int)(unsigned)(best & 0xffffffffull);
        const int2 hp = syz[hit];
        recentre_y(st.p[0], yref, hp.x);
        kf_update<float>(st, hit_y(hp.x, yref), hit_z(hp.y, zref, zunit), nullptr, G->angErr);
        tb.hits[(size_t)k * kMaxTlHits + n] = hit;
        tb.rows[(size_t)k * kMaxTlHits + n] = (uint8_t)r;
        ++n;
        save_last(st);
        yrefLast = yref;
        misses = 0;
        r += kDir;
      } else if (++misses >= kMaxMiss) {
        finish();
      } else {
        r += kDir;
      }
    }
  }
}

// The same passes with the per-lane search in the drift-ordered views (rows
// flagged dense: in the cells, whose place is in the view's row table: with the
// cells' own table as one more dependent load a sector of 2.1 M clusters took
// 0.77 + 1.24 ms, now 0.74 + 1.23).  Bound by the latency of the dependent chain of a row
// step (row table -> bin starts -> candidates -> update) and by its ~450
// instructions.  Only what the next reader needs survives a step: the
// direction parameters and the row of the last accepted state (with kKeep the
// whole state, for inspection), so nothing is copied per accepted hit.
// Measured against the search in the cells with the state copied per hit:
// 1 ms frame (20.3 M clusters) 2.26 + 1.73 -> 1.51 + 1.26 ms, 32 orbits (59 M)
// 6.87 + 5.19 -> 4.45 + 3.75 ms, 3 collisions (1.3 M, one tracklet a lane)
// 0.58 + 0.55 -> 0.38 + 0.44 ms.
// The list index of the hit is loaded off the step's chain (beside the
// update).  Loading the next row's bin starts ahead (prefetch to L1 or L2) cost
// 6 %.  Blocks of 128 per SM the kernel is compiled for: 7 (72 registers)
// measured 1.58 + 1.32 ms, 8 1.73 + 1.42, 6 1.59 + 1.36.
#ifndef O2TPC_FOLLOW_MIN_BLOCKS
#define O2TPC_FOLLOW_MIN_BLOCKS 7
#endif

// Tracklets a warp reserves at a time: 1 (an atomic for every refill) measured 1.54 +
// 1.27 ms on the 1 ms frame, 8 1.51 + 1.26, 32 1.67 + 1.46 (the tracklets in
// flight, and what they touch, spread out: L2 hits 47 -> 38 %).
constexpr int kFollowBatch = 8;

template <int kDir, bool kKeep>
__global__ void __launch_bounds__(128, O2TPC_FOLLOW_MIN_BLOCKS)
    k_tl_follow(const int* __restrict__ nTlDev, int* __restrict__ counter, const int* __restrict__ cellStart,
                const int2* __restrict__ syz, const GeomConst* __restrict__ G,
                ZView zv, TrackletBufs tb) {
  constexpr bool kWhole = kKeep && kDir < 0;
  __shared__ float s_last[kWhole ? 20 : 1][128];
  const unsigned full = 0xffffffffu;
  const float zunit = G->zunit, izunit = G->kz, bzc = G->bzc;
  const int angErr = G->angErr;
  const int nTl = *nTlDev;
  const int lane = threadIdx.x & 31;
  int batch = 0, batchEnd = 0;
  bool have = false, exhausted = false;
  int k = 0, r = 0, n = 0, misses = 0, srow = 0, yref = 0, yrefLast = 0, zref = 0, Rs = 0, lastRow = 0;
  float last2 = 0.f, last3 = 0.f, last4 = 0.f;
  KState<float> st;
  auto save_last = [&]() {
    last2 = st.p[2];
    last3 = st.p[3];
    last4 = st.p[4];
    lastRow = srow;
    yrefLast = yref;
    if (kWhole) {
#pragma unroll
      for (int j = 0; j < 5; ++j) s_last[j % (kWhole ? 20 : 1)][threadIdx.x] = st.p[j];
#pragma unroll
      for (int j = 0; j < 15; ++j) s_last[(5 + j) % (kWhole ? 20 : 1)][threadIdx.x] = st.C[j];
    }
  };
  // ends the lane's tracklet with the state after its last accepted hit
  auto finish = [&]() {
    float* S = tb.state + (size_t)k * 21;
    if (kDir > 0) {
      tb.nasc[k] = n;
      tb.yref[k] = yrefLast;
    } else {
      tb.nhits[k] = n;
      S[0] = G->rowx[lastRow];
    }
    S[3] = last2;
    S[4] = last3;
    S[5] = last4;
    if (kWhole) {
      S[1] = s_last[0][threadIdx.x] + (float)yrefLast * 0.00625f;
      S[2] = s_last[1 % (kWhole ? 20 : 1)][threadIdx.x];
#pragma unroll
      for (int j = 0; j < 15; ++j) S[6 + j] = s_last[(5 + j) % (kWhole ? 20 : 1)][threadIdx.x];
    }
    have = false;
  };
  for (;;) {
    // lanes without a tracklet take the next ones (the warp reserves a few at a
    // time); their loads depend on the index alone
    const bool want = !have && !exhausted;
    const unsigned wants = __ballot_sync(full, want);
    if (wants) {
      const int cnt = __popc(wants), rank = __popc(wants & ((1u << lane) - 1u)), left = batchEnd - batch;
      int kk = batch + rank;
      batch += cnt;
      if (cnt > left) {
        const int take = max(cnt - left, kFollowBatch);
        int nb = 0;
        if (lane == 0) nb = atomicAdd(counter, take);
        nb = __shfl_sync(full, nb, 0);
        if (rank >= left) kk = nb + rank - left;
        batch = nb + cnt - left;
        batchEnd = nb + take;
      }
      if (want) {
        k = kk;
        if (k >= nTl) {
          exhausted = true;
        } else {
          const int na = tb.nasc[k];
          const int row0 = tb.rows[(size_t)k * kMaxTlHits];
          Rs = tb.rbase[k];
          zref = tb.zref[k];
          yref = tb.yref[k];
          load_state(st, tb.state + (size_t)k * 21);
          if (na > 0) {
            n = na;
            misses = 0;
            srow = row_of_x(st.x);
            // the chain's last fitted hit is its top; the refit may have skipped the lowest
            r = (kDir > 0) ? srow + 1 : row0 - 1;
            save_last();
            have = true;
          }
        }
      }
    }
    if (__ballot_sync(full, have) == 0) {
      if (__all_sync(full, exhausted)) break;
      continue;
    }
    // one row step of every busy lane: transport, then the window
    BestHit best{-1, make_int2(0, 0)};
    ZRow gv{};  // the row of best.pos; count 0: best.pos is the sorted index
    if (have) {
      if ((kDir > 0) ? (r >= kNRow) : (r < 0)) {
        finish();
      } else if (kf_prop_row<float, kF1Fused>(st, srow, r, G, bzc) != 0 || fabsf(st.p[2]) > kSinFollow) {
        finish();
      } else {
        srow = r;
        const ZRow g = zv.rows[Rs + r];
        SearchPar P;
        int zlo, zhi;
        if (g.count > 0 && search_window(st, yref, zref, izunit, angErr, P, zlo, zhi)) {
          if (g.flags & kZFollowCells) {
            RowGrid gc;
            gc.count = g.count;
            // (not with g: two more registers over the step cost every row 3 %)
            asm volatile("ld.global.nc.v2.s32 {%0, %1}, [%2];"
                         : "=r"(gc.cellBase), "=r"(gc.cz)
                         : "l"(&zv.rows[Rs + r].cellBase));
            gc.ny = cells_y(G->npads[r]);
            gc.nz = g.flags >> kZnz;
            gc.zmin = g.zmin;
            int ylo, yhi, iy0, iy1, iz0, iz1;
            window_y(P, ylo, yhi);
            if (cell_range(gc, G->npads[r], ylo, yhi, zlo, zhi, iy0, iy1, iz0, iz1))
              best = cell_search(gc, iy0, iy1, iz0, iz1, cellStart, syz, P, zunit);
          } else {
            int a, b;
            if (z_range(zv, g, zlo, zhi, a, b)) {
              best = z_search(zv, g, a, b, P, zunit);
              gv.start = g.start;
              gv.count = g.count;
            }
          }
        }
      }
    }
    if (have) {
      if (best.pos >= 0) {
        const int hit = gv.count ? zv.idx(gv, best.pos) : best.pos;  // in flight during the update
        recentre_y(st.p[0], yref, best.p.x);
        kf_update<float>(st, hit_y(best.p.x, yref), hit_z(best.p.y, zref, zunit), nullptr, angErr);
        tb.rows[(size_t)k * kMaxTlHits + n] = (uint8_t)r;
        tb.hits[(size_t)k * kMaxTlHits + n] = hit;
        ++n;
        save_last();
        misses = 0;
        r += kDir;
      } else if (++misses >= kMaxMiss) {
        finish();
      } else {
        r += kDir;
      }
    }
  }
}

// Ownership keys.  Only tracklets of the same sector can share a hit, so the
// tie-break id is the tracklet's index within its sector (same order as the
// index within the TF): (nHits << 24 | 2^24-1-id) in 32 bits, or the 64-bit
// (nHits << 32 | 2^32-1-id) when a sector holds 2^24 tracklets or more.
__device__ inline unsigned own_key32(int nh, int lid) { return ((unsigned)nh << 24) | (0xFFFFFFu - (unsigned)lid); }
__device__ inline unsigned long long own_key64(int nh, int lid) {
  return ((unsigned long long)(unsigned)nh << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)lid);
}

// First tracklet of every (TF, sector) (start hits are sorted by hit index);
// *wide = 1 when a sector holds 2^24 tracklets or more.
__global__ void k_sector_ranges(int nSec, const RowGrid* __restrict__ grid, const int* __restrict__ starts,
                                const int* __restrict__ nTlDev, int* __restrict__ secBegin, int* __restrict__ wide) {
  const int ts = blockIdx.x * blockDim.x + threadIdx.x;
  if (ts > nSec) return;
  const int nTl = *nTlDev;
  auto lower = [&](int key) {
    int lo = 0, hi = nTl;
    while (lo < hi) {
      const int m = (lo + hi) >> 1;
      if (starts[m] < key) lo = m + 1;
      else hi = m;
    }
    return lo;
  };
  const int b = (ts == nSec) ? nTl : lower(grid[ts * kNRow].start);
  secBegin[ts] = b;
  if (ts < nSec) {
    const int e = (ts + 1 == nSec) ? nTl : lower(grid[(ts + 1) * kNRow].start);
    if (e - b >= (1 << 24)) atomicOr(wide, 1);
  }
}

struct OwnCtx {
  const int* secBegin;
  const int* wide;
  void* w;  // unsigned[n] or unsigned long long[n]
};

// Key of tracklet k.
struct TlKey {
  bool wide;
  unsigned k32;
  unsigned long long k64;
};
__device__ inline TlKey tl_key(const OwnCtx& o, const TrackletBufs& tb, int k, int nh) {
  const int lid = k - o.secBegin[tb.rbase[k] / kNRow];
  TlKey t;
  t.wide = *o.wide != 0;
  t.k32 = own_key32(nh, lid);
  t.k64 = own_key64(nh, lid);
  return t;
}

// Slots [0, 8) of a tracklet's hit list from a 16-byte aligned address (a
// tracklet's 152 slots start on 608-byte boundaries).  Slots past the
// tracklet's hits hold stale values that the callers mask.
__device__ inline void load_hits8(const int* H, int (&hh)[8]) {
  const int4 a = reinterpret_cast<const int4*>(H)[0], b = reinterpret_cast<const int4*>(H)[1];
  hh[0] = a.x; hh[1] = a.y; hh[2] = a.z; hh[3] = a.w;
  hh[4] = b.x; hh[5] = b.y; hh[6] = b.z; hh[7] = b.w;
}

// K8a: hit ownership (atomicMax of the key, no answer waited for: looking a
// word up first, to skip the atomic where a larger key stands, cost more than
// the atomics it saved: 1 ms frame 0.44 -> 0.28 ms, 32 orbits 1.34 -> 0.87 without).  8 hits per step
// (two 16-byte loads; the 152 slots are a multiple of 8).
__global__ void k_ownership(const int* __restrict__ nTlDev, OwnCtx o, TrackletBufs tb) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= *nTlDev) return;
  const int nh = tb.nhits[k];
  if (nh < kMinHits) return;
  const TlKey key = tl_key(o, tb, k, nh);
  const int* H = tb.hits + (size_t)k * kMaxTlHits;
  for (int i = 0; i < nh; i += 8) {
    int hh[8];
    load_hits8(H + i, hh);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (i + u >= nh) continue;
      if (key.wide) atomicMax(static_cast<unsigned long long*>(o.w) + hh[u], key.k64);
      else atomicMax(static_cast<unsigned*>(o.w) + hh[u], key.k32);
    }
  }
}

// Segments: a tracklet's owned hits in row order (its inward hits backwards,
// then its chain and outward hits), split at gaps of more than kMaxMiss rows;
// segments of >= kMinHits are kept.  A warp takes a group of consecutive
// tracklets, loads what it needs of each at once, and works on one after the
// other with a lane per hit, the next one's lists on their way: lists, rows and
// results are read and written as whole lines, 32 random words in flight.
// (With a thread per tracklet the write pass ran with 6.5 of 32 lanes active.)
// Count and write with the coordinate gather, against a thread per tracklet, with groups
// of 32 (groups of 8 take another tenth off): 1 ms frame 0.30 + 0.55 -> 0.31 + 0.32 ms, one
// sector's frame 39 + 57 -> 8 + 8 us, 32 orbits 0.76 + 1.44 -> 0.95 + 1.35 ms.  128 orbits:
// 3.0 + 5.7 -> 4.6 + 6.1 ms with groups of 8.
constexpr int kSegWords = kOwnWords;

// Slot of the tracklet's j-th hit in row order (nd of its nh hits are inward).
__device__ inline int slot_of(int j, int nh, int nd) { return j < nd ? nh - 1 - j : j - nd; }

// Of the owned hits `own` of 32 consecutive places (lane = place): those that
// begin a segment.  prevRow: row of the last owned hit before (a large negative
// number if there is none), moved on.
__device__ inline unsigned segment_starts(unsigned own, int row, int& prevRow) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned before = own & ((1u << lane) - 1u);
  const int pl = __shfl_sync(full, row, before ? 31 - __clz(before) : 0);
  const int pr = before ? pl : prevRow;
  const unsigned st = __ballot_sync(full, ((own >> lane) & 1u) && row - pr - 1 > kMaxMiss);
  if (own) prevRow = __shfl_sync(full, row, 31 - __clz(own));
  return st;
}

// A tracklet's hits and rows in row order, five places a lane.
struct TlPlaces {
  int hit[kSegWords], row[kSegWords];
  __device__ void load(const TrackletBufs& tb, int k, int nh, int nd) {
    const int lane = threadIdx.x & 31;
    const int* H = tb.hits + (size_t)k * kMaxTlHits;
    const uint8_t* Rw = tb.rows + (size_t)k * kMaxTlHits;
#pragma unroll
    for (int c = 0; c < kSegWords; ++c) {
      const int j = c * 32 + lane;
      hit[c] = -1;
      row[c] = 0;
      if (j < nh) {
        const int i = slot_of(j, nh, nd);
        hit[c] = H[i];
        row[c] = Rw[i];
      }
    }
  }
};

// CTAs an SM of the two passes: all resident, so that the tracklets in flight are
// one run of consecutive ones; fewer from kSegMany tracklets on, where the words
// and coordinates of that run no longer stay in L2.  (Grids of 12 CTAs an SM and
// groups of 32 ran over the TF twice: selection of 16 orbits (1.1 M tracklets) 1.88 ->
// 1.67 ms, 96 orbits (6.4 M) 13.1 -> 11.6 ms, with 7 and 4 CTAs 10.2; of 16
// orbits with 7 and 4 1.70 ms.)
constexpr int kSegCountCtas = 10, kSegWriteCtas = 6, kSegCountMany = 7, kSegWriteMany = 4, kSegMany = 3000000;

// Consecutive tracklets a warp takes at once: 8 (selection of 16 orbits 1.92 ms
// with 32, 1.69 with 8, 1.79 with 2), fewer when there are too few for every warp
// of the grid.
constexpr int kSegGroup = 8;
__device__ inline int segment_group(int nTl) {
  const int warps = gridDim.x * (blockDim.x >> 5);
  return min(kSegGroup, max(1, (nTl + warps - 1) / warps));
}

// K8b: count pass; also keeps the ownership bits (in row order) for the write
// pass, which then reads no ownership words.
__global__ void __launch_bounds__(128, kSegCountCtas) k_segments_count(const int* __restrict__ nTlDev, OwnCtx o,
                                                        TrackletBufs tb, int* __restrict__ nSeg, int* __restrict__ nSegHits,
                                                        unsigned* __restrict__ ownBits) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, nTl = *nTlDev;
  const int group = segment_group(nTl), warps = gridDim.x * (blockDim.x >> 5);
  const bool wide = *o.wide != 0;
  for (int k0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * group; k0 < nTl; k0 += warps * group) {
    const int kl = k0 + lane;
    const bool mineTl = lane < group && kl < nTl;
    // of this lane's tracklet
    const int nhl = mineTl ? tb.nhits[kl] : 0;
    int ndl = 0, lidl = 0;
    if (nhl >= kMinHits) {
      ndl = nhl - tb.nasc[kl];
      lidl = kl - o.secBegin[tb.rbase[kl] / kNRow];
    }
    int csl = 0, chl = 0;
    unsigned todo = __ballot_sync(full, nhl >= kMinHits);
    TlPlaces next;
    auto fetch = [&]() {
      const int src = todo ? __ffs(todo) - 1 : 0;
      const int nh = __shfl_sync(full, nhl, src), nd = __shfl_sync(full, ndl, src);
      if (todo) next.load(tb, k0 + src, nh, nd);
    };
    fetch();
    while (todo) {
      const int src = __ffs(todo) - 1, k = k0 + src;
      todo &= todo - 1;
      const TlPlaces T = next;
      const int nh = __shfl_sync(full, nhl, src), lid = __shfl_sync(full, lidl, src);
      bool mine[kSegWords];
      if (wide) {
        const unsigned long long key = own_key64(nh, lid);
#pragma unroll
        for (int c = 0; c < kSegWords; ++c)
          mine[c] = T.hit[c] >= 0 && static_cast<const unsigned long long*>(o.w)[T.hit[c]] == key;
      } else {
        const unsigned key = own_key32(nh, lid);
#pragma unroll
        for (int c = 0; c < kSegWords; ++c)
          mine[c] = T.hit[c] >= 0 && static_cast<const unsigned*>(o.w)[T.hit[c]] == key;
      }
      fetch();
      int cs = 0, ch = 0, m = 0, prevRow = -1000;
#pragma unroll
      for (int c = 0; c < kSegWords; ++c) {
        const unsigned own = __ballot_sync(full, mine[c]);
        if (lane == c) ownBits[(size_t)k * kSegWords + c] = own;
        if (!own) continue;
        unsigned rest = own;
        for (unsigned st = segment_starts(own, T.row[c], prevRow); st; st &= st - 1) {
          const unsigned lower = (st & -st) - 1u;  // places before the start
          m += __popc(rest & lower);
          if (m >= kMinHits) {
            ++cs;
            ch += m;
          }
          m = 0;
          rest &= ~lower;
        }
        m += __popc(rest);
      }
      if (m >= kMinHits) {
        ++cs;
        ch += m;
      }
      if (lane == src) {
        csl = cs;
        chl = ch;
      }
    }
    if (mineTl) {
      nSeg[kl] = csl;
      nSegHits[kl] = chl;
    }
  }
}

// K8c: write the sector tracks of each tracklet (ids in tracklet order) and
// gather the coordinates and input indices of their hits for the fits.  A
// tracklet has at most 27 segments, kept or not (they lie 6 rows apart): a lane
// each for their table entries.
__global__ void __launch_bounds__(128, kSegWriteCtas) k_segments_write(const int* __restrict__ nTlDev, TrackletBufs tb,
                                                        const unsigned* __restrict__ ownBits,
                                                        const int* __restrict__ segPos,
                                                        const int* __restrict__ segHitPos,
                                                        const int2* __restrict__ syz,
                                                        const int* __restrict__ sorig, SectorTrackBufs sb, int capSt,
                                                        int capHits) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, nTl = *nTlDev;
  const int group = segment_group(nTl), warps = gridDim.x * (blockDim.x >> 5);
  for (int k0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * group; k0 < nTl; k0 += warps * group) {
    const int kl = k0 + lane;
    const bool mineTl = lane < group && kl < nTl;
    const int idl = mineTl ? segPos[kl] : 0;
    const bool some = mineTl && segPos[kl + 1] > idl;
    int nhl = 0, ndl = 0, tsl = 0, hol = 0;
    unsigned ownl[kSegWords] = {};
    if (some) {
      nhl = tb.nhits[kl];
      ndl = nhl - tb.nasc[kl];
      tsl = tb.rbase[kl] / kNRow;
      hol = segHitPos[kl];
#pragma unroll
      for (int c = 0; c < kSegWords; ++c) ownl[c] = ownBits[(size_t)kl * kSegWords + c];
    }
    unsigned todo = __ballot_sync(full, some);
    TlPlaces next;
    auto fetch = [&]() {
      const int src = todo ? __ffs(todo) - 1 : 0;
      const int nh = __shfl_sync(full, nhl, src), nd = __shfl_sync(full, ndl, src);
      if (todo) next.load(tb, k0 + src, nh, nd);
    };
    fetch();
    while (todo) {
      const int src = __ffs(todo) - 1, k = k0 + src;
      todo &= todo - 1;
      const TlPlaces T = next;
      unsigned own[kSegWords];
      int2 yz[kSegWords];
      int orig[kSegWords];
#pragma unroll
      for (int c = 0; c < kSegWords; ++c) {
        own[c] = __shfl_sync(full, ownl[c], src);
        if ((own[c] >> lane) & 1u) {
          yz[c] = syz[T.hit[c]];
          orig[c] = sorig[T.hit[c]];
        }
      }
      fetch();
      // lane q: hits of segment q and owned hits before it
      unsigned start[kSegWords];
      int seg = -1, total = 0, prevRow = -1000, rankl = 0;
#pragma unroll
      for (int c = 0; c < kSegWords; ++c) {
        start[c] = own[c] ? segment_starts(own[c], T.row[c], prevRow) : 0u;
        for (unsigned st = start[c]; st; st &= st - 1) {
          ++seg;
          const int before = total + __popc(own[c] & ((st & -st) - 1u));
          if (lane == seg) rankl = before;
        }
        total += __popc(own[c]);
      }
      const int nextRank = __shfl_down_sync(full, rankl, 1);
      const int len = lane > seg ? 0 : (lane == seg ? total : nextRank) - rankl;
      const bool keep = len >= kMinHits;
      const unsigned kept = __ballot_sync(full, keep);
      // output slots of the kept ones and their table entries
      int ho = keep ? len : 0;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(full, ho, d);
        if (lane >= d) ho += y;
      }
      ho += __shfl_sync(full, hol, src) - (keep ? len : 0);
      const int ts = __shfl_sync(full, tsl, src);
      const int id = __shfl_sync(full, idl, src) + __popc(kept & ((1u << lane) - 1u));
      if (keep && id < capSt) {
        sb.tl[id] = k;
        sb.tf[id] = ts / kNSec;
        sb.sector[id] = ts % kNSec;
        sb.off[id] = min(ho, capHits);
      }
      // the hits: a place's segment is the last one that starts at or before it
      int segBefore = -1, rankBefore = 0;
#pragma unroll
      for (int c = 0; c < kSegWords; ++c) {
        const unsigned below = (1u << lane) - 1u;
        const int q = max(segBefore + __popc(start[c] & (below | (1u << lane))), 0);
        const int dst = __shfl_sync(full, ho, q), first = __shfl_sync(full, rankl, q), idq = __shfl_sync(full, id, q);
        const int r = rankBefore + __popc(own[c] & below) - first;  // place in the segment
        if (((own[c] >> lane) & 1u) && ((kept >> q) & 1u)) {
          const int at = dst + r;
          if (at < capHits) {
            sb.hits[at] = T.hit[c];
            sb.rows[at] = (uint8_t)T.row[c];
            sb.yz[at] = yz[c];
            sb.orig[at] = orig[c];
          }
          if (r == 0 && idq < capSt) sb.zref[idq] = yz[c].y;
        }
        segBefore += __popc(start[c]);
        rankBefore += __popc(own[c]);
      }
    }
  }
}

// The sector tracks' fits, one thread per track, the tracks in order of
// their length; hits are loaded one step ahead.
// Alone with few tracks (one collision of a sector) 164 -> 110 us: its time is the
// chain of steps; 32 orbits 0.99 ms as in a global order by length, without its
// scattered results.
__global__ void __launch_bounds__(128, 1) k_sector_fit(const int* __restrict__ nStDev, int* __restrict__ counter,
                                                              const int* __restrict__ perm, TrackletBufs tb, const GeomConst* __restrict__ G,
                                                              SectorTrackBufs sb) {
  const float zunit = G->zunit, bzc = G->bzc;
  const int nSt = *nStDev;
  for (int id; take_ordered(counter, perm, nSt, id);) {
    if (id < 0) continue;
    const int b = sb.off[id], m = sb.off[id + 1] - b;
    const int2* P = sb.yz + b;
    const uint8_t* Rw = sb.rows + b;
    const int zref = sb.zref[id];
    KState<float> sd;
    load_state(sd, tb.state + (size_t)sb.tl[id] * 21);
    const float xa = G->rowx[Rw[0]];
    {
      KState<float> tmp = sd;
      if (kf_prop_row<float>(tmp, row_of_x(sd.x), Rw[0], G, bzc) == 0) sd = tmp;
    }
    KState<float> t;
    int2 p = P[0];
    int yref = p.x;
    kf_reset<float>(t, xa, hit_y(p.x, yref), hit_z(p.y, zref, zunit), sd.p[2], sd.p[3], sd.p[4]);
    kf_meas_cov<float>(t, G->angErr);
    int srow = Rw[0], zcur = zref;
    int2 pn = P[1];  // a sector track has at least kMinHits hits
    int rn = Rw[1];
    for (int i = 1; i < m; ++i) {
      p = pn;
      const int row = rn;
      if (i + 1 < m) {
        pn = P[i + 1];
        rn = Rw[i + 1];
      }
      if (kf_prop_row<float, kF1Fused>(t, srow, row, G, bzc) != 0) continue;
      srow = row;
      recentre_y(t.p[0], yref, p.x);
      recentre_z(t.p[1], zcur, p.y, zunit);
      kf_update<float>(t, hit_y(p.x, yref), 0.f, nullptr, G->angErr);
    }
    t.p[1] += (float)(zcur - zref) * zunit;
    store_state(sb.out + (size_t)id * 21, t, yref);
    KState<float> u;
    p = P[m - 1];
    yref = p.x;
    kf_reset<float>(u, G->rowx[Rw[m - 1]], hit_y(p.x, yref), hit_z(p.y, zref, zunit), t.p[2], t.p[3], t.p[4]);
    kf_meas_cov<float>(u, G->angErr);
    srow = Rw[m - 1];
    zcur = p.y;
    u.p[1] = 0.f;
    pn = P[m - 2];
    rn = Rw[m - 2];
    for (int i = m - 2; i >= 0; --i) {
      p = pn;
      const int row = rn;
      if (i > 0) {
        pn = P[i - 1];
        rn = Rw[i - 1];
      }
      if (kf_prop_row<float, kF1Rounded>(u, srow, row, G, bzc) != 0) continue;
      srow = row;
      recentre_y(u.p[0], yref, p.x);
      recentre_z(u.p[1], zcur, p.y, zunit);
      kf_update<float>(u, hit_y(p.x, yref), 0.f, nullptr, G->angErr);
    }
    u.p[1] += (float)(zcur - zref) * zunit;
    store_state(sb.in + (size_t)id * 21, u, yref);
  }
}

// ------------------------------------------------------------- launchers
namespace {
struct PassGrid {
  int sms = 0, chain = 0, out = 0, refit = 0, in = 0, fit = 0;
};
PassGrid pass_grid() {
  static PassGrid g;
  if (g.sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g.sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g.chain, k_tl_chain, 128, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g.out, k_tl_follow<1, false>, 128, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g.refit, k_tl_refit, 128, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g.fit, k_sector_fit, 128, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g.in, k_tl_follow<-1, false>, 128, 0);
  }
  return g;
}
}  // namespace

void launch_tracklets(int nTl, const int* nTlDev, int* workCounter, const int* starts, const int* up,
                      const RowGrid* grid, int nRows, const int* cellStart, const int2* syz, const GeomConst* G,
                      ZView zv, TrackletBufs tb, int* perm, cudaStream_t st, cudaEvent_t* passEnd, bool coopSearch,
                      bool keepState) {
  auto mark = [&](int i) {
    if (passEnd) cudaEventRecord(passEnd[i], st);
  };
  cudaMemsetAsync(workCounter, 0, kWorkCounters * sizeof(int), st);
  if (nTl <= 0) {
    for (int i = 0; i < 4; ++i) mark(i);
    return;
  }
  const PassGrid g = pass_grid();
  auto blocks = [&](int perSm) { return std::min((nTl + 127) / 128, g.sms * std::max(perSm, 1)); };
  k_tl_walk<<<(nTl + 255) / 256, 256, 0, st>>>(nTlDev, starts, up, tb);
  launch_length_order(nTl, nTlDev, tb.nasc, false, perm, st);
  k_tl_chain<<<blocks(g.chain), 128, 0, st>>>(nTlDev, workCounter, perm, starts, up, grid, nRows, syz, G, tb);
  mark(0);
  if (coopSearch) {
    k_tl_follow_coop<1><<<blocks(g.out), 128, 0, st>>>(nTlDev, workCounter + 1, grid, cellStart, syz, G, tb);
  } else {
    k_tl_follow<1, false><<<blocks(g.out), 128, 0, st>>>(nTlDev, workCounter + 1, cellStart, syz, G, zv, tb);
  }
  mark(1);
  launch_length_order(nTl, nTlDev, tb.nasc, false, perm, st);
  k_tl_refit<<<blocks(g.refit), 128, 0, st>>>(nTlDev, workCounter + 2, perm, syz, G, tb);
  mark(2);
  if (coopSearch) {
    k_tl_follow_coop<-1><<<blocks(g.in), 128, 0, st>>>(nTlDev, workCounter + 3, grid, cellStart, syz, G, tb);
  } else if (keepState) {
    k_tl_follow<-1, true><<<blocks(g.in), 128, 0, st>>>(nTlDev, workCounter + 3, cellStart, syz, G, zv, tb);
  } else {
    k_tl_follow<-1, false><<<blocks(g.in), 128, 0, st>>>(nTlDev, workCounter + 3, cellStart, syz, G, zv, tb);
  }
  mark(3);
  g_launch_count += 5;
}

void launch_ownership(int nTl, const int* nTlDev, int nSec, const RowGrid* grid, const int* starts, TrackletBufs tb,
                      void* w, int* secBegin, int* wide, cudaStream_t st) {
  cudaMemsetAsync(wide, 0, sizeof(int), st);
  k_sector_ranges<<<(nSec + 1 + 127) / 128, 128, 0, st>>>(nSec, grid, starts, nTlDev, secBegin, wide);
  ++g_launch_count;
  if (nTl > 0) {
    k_ownership<<<(nTl + 127) / 128, 128, 0, st>>>(nTlDev, OwnCtx{secBegin, wide, w}, tb);
    ++g_launch_count;
  }
}

namespace {
int segment_blocks(int nTl, int perSM, int perSMMany) {
  return std::min((nTl + 3) / 4, pass_grid().sms * (nTl < kSegMany ? perSM : perSMMany));
}
}  // namespace

void launch_segments_count(int nTl, const int* nTlDev, const int* secBegin, const int* wide, const void* w,
                           TrackletBufs tb, int* nSeg, int* nSegHits, unsigned* ownBits, cudaStream_t st) {
  if (nTl > 0) {
    k_segments_count<<<segment_blocks(nTl, kSegCountCtas, kSegCountMany), 128, 0, st>>>(
        nTlDev, OwnCtx{secBegin, wide, const_cast<void*>(w)}, tb, nSeg, nSegHits, ownBits);
    ++g_launch_count;
  }
}

void launch_segments_write(int nTl, const int* nTlDev, TrackletBufs tb, const unsigned* ownBits, const int* segPos,
                           const int* segHitPos, const int2* syz, const int* sorig, SectorTrackBufs sb, int capSt,
                           int capHits, cudaStream_t st) {
  if (nTl > 0) {
    k_segments_write<<<segment_blocks(nTl, kSegWriteCtas, kSegWriteMany), 128, 0, st>>>(
        nTlDev, tb, ownBits, segPos, segHitPos, syz, sorig, sb, capSt, capHits);
    ++g_launch_count;
  }
}

void launch_sector_fit(int nSt, const int* nStDev, int* counter, int* perm, const TrackletBufs tb, const GeomConst* G,
                       SectorTrackBufs sb, cudaStream_t st) {
  if (nSt > 0) {
    const PassGrid g = pass_grid();
    const int nb = std::min((nSt + 127) / 128, g.sms * std::max(g.fit, 1));
    launch_length_order(nSt, nStDev, sb.off, true, perm, st);
    k_sector_fit<<<nb, 128, 0, st>>>(nStDev, counter, perm, tb, G, sb);
    ++g_launch_count;
  }
}

}  // namespace o2tpc
