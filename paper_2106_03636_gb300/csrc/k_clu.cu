// TPC clusterizer (Sec. 2.2: the raw ADC values are turned into hits before
// tracking) on the device, behind o2tpc_clusterize.
//
// Readings (the paper gives no algorithm): zero-suppressed digits sorted by
// (sector, row, time bin, pad); a peak is a digit with ADC >= 3 larger than
// each of its up to eight pad/time neighbours in the same row that come
// before it in that order and not smaller than each that comes after it; a
// peak's cluster is the 3 x 3 cells around it: Q = sum of ADC, centre of
// gravity of the cell centres (pad p spans [p, p + 1), bin t spans
// [t, t + 1)) in 1/64 units rounded half up in integers; one 12-byte record
// (u32 time64, u16 pad64, u16 min(Q, 65535), u8 row, u8 sector, u16 0) per
// peak, in the order of the peaks.  Exact integer arithmetic throughout.
//
// Tiles of 3072 digits and a halo of 272 on each side are staged in shared
// memory as 64-bit keys and ADC values: a (row, time bin) holds at most 256
// digits, so the neighbours one bin earlier or later lie within 258 places.
// Every digit is held against its neighbours in its own time bin, the adjacent
// ones; the third or so that pass go into an ordered queue, and the queue is
// worked off with all lanes busy: two searches in shared memory find the
// neighbours in the other bins.  (A digit at a time through all tests, with
// the few lanes that get past the first ones holding the warp, ran 4x longer.)
// Pass 1 checks the input and counts the peaks of each tile; the counts are
// scanned; pass 2 repeats the tile and writes the records.  Repeating costs a
// second read of 9 bytes a digit; it keeps the scratch at two ints per tile,
// where keys and flags of every digit (16 bytes, allocated on each call) were
// written and read back before.
// 20 collisions (84 M digits, 8.5 M clusters): a call 7.15 -> 1.84 ms, its
// kernels 3.47 -> 1.42 ms (0.61 and 0.80 ms the two passes, latency of the
// shared-memory searches).
#include <cstdint>

#include "o2tpc.h"
#include "o2tpc_internal.cuh"
#include "o2tpc_kernels.cuh"

namespace o2tpc {

namespace {

constexpr int kPeakMin = 3;
constexpr int kCluThreads = 256;
constexpr int kCluPer = 12;                       // digits a thread, four consecutive ones at a time
constexpr int kCluTile = kCluPer * kCluThreads;   // 3072: 43 KB of shared memory, five tiles per SM
constexpr int kCluHalo = 272;                     // >= 258, a multiple of 16
constexpr int kCluSpan = kCluTile + 2 * kCluHalo;

__device__ inline unsigned long long dkey(unsigned s, unsigned r, unsigned t, unsigned p) {
  return ((unsigned long long)(s * kNRow + r) << 40) | ((unsigned long long)t << 8) | (unsigned long long)p;
}

struct CluIn {
  long long n;
  const uint8_t *sector, *row, *pad;
  const uint32_t* time;
  const uint16_t* adc;
  int wide;  // 1: every array on a 16-byte boundary
};

}  // namespace

// Pass 1 (kWrite false): peaks of each tile into tileCnt, the error word.
// Pass 2 (kWrite true): the records, tile b's from tileOff[b] on.
template <bool kWrite>
__global__ void __launch_bounds__(kCluThreads) k_clu_tile(CluIn d, int* __restrict__ tileCnt,
                                                          const int* __restrict__ tileOff, uint8_t* __restrict__ out,
                                                          unsigned* __restrict__ err) {
  __shared__ __align__(16) unsigned long long s_key[kCluSpan];
  __shared__ __align__(16) uint16_t s_adc[kCluSpan];
  __shared__ uint16_t s_queue[kCluTile];
  __shared__ int s_cnt[kCluPer][kCluThreads / 32];
  __shared__ int s_warp[kCluThreads / 32], s_total;
  const long long base = (long long)blockIdx.x * kCluTile - kCluHalo;  // digit of span index 0
  const int lo = base < 0 ? (int)-base : 0;                            // span indices of digits: [lo, hi)
  const int hi = (int)min((long long)kCluSpan, d.n - base);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  bool bad = false;
  auto keyed = [&](unsigned s, unsigned r, unsigned t, unsigned p) {
    if (s >= (unsigned)kNSec || r >= (unsigned)kNRow || t >= (1u << 24)) {
      bad = true;
      s = r = t = 0;
    }
    return dkey(s, r, t, p);
  };
  for (int i = 4 * threadIdx.x; i < kCluSpan; i += 4 * kCluThreads) {
    const long long g = base + i;
    if (d.wide && i >= lo && i + 4 <= hi) {  // lo is 0 or the halo: a multiple of 4
      const unsigned vs = *reinterpret_cast<const unsigned*>(d.sector + g);
      const unsigned vr = *reinterpret_cast<const unsigned*>(d.row + g);
      const unsigned vp = *reinterpret_cast<const unsigned*>(d.pad + g);
      const uint4 vt = *reinterpret_cast<const uint4*>(d.time + g);
      *reinterpret_cast<uint2*>(s_adc + i) = *reinterpret_cast<const uint2*>(d.adc + g);
      const unsigned t[4] = {vt.x, vt.y, vt.z, vt.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        s_key[i + k] = keyed((vs >> (8 * k)) & 255u, (vr >> (8 * k)) & 255u, t[k], (vp >> (8 * k)) & 255u);
    } else {
      for (int k = 0; k < 4; ++k) {
        const int q = i + k;
        if (q < lo || q >= hi) continue;
        s_key[q] = keyed(d.sector[g + k], d.row[g + k], d.time[g + k], d.pad[g + k]);
        s_adc[q] = d.adc[g + k];
      }
    }
  }
  __syncthreads();
  // digits that beat their neighbours in the same time bin, in order
  const int end = min(kCluHalo + kCluTile, hi);
  unsigned cand = 0;  // bit j: span index halo + j * threads + thread
  int mine[kCluPer];
#pragma unroll
  for (int j = 0; j < kCluPer; ++j) {
    const int i = kCluHalo + j * kCluThreads + threadIdx.x;
    bool ok = false;
    if (i < end) {
      const unsigned long long ki = s_key[i];
      const unsigned a = s_adc[i];
      ok = a >= (unsigned)kPeakMin;
      if (i > lo) {
        const unsigned long long kb = s_key[i - 1];
        if (kb >= ki) bad = true;  // not strictly ascending
        if (kb + 1 == ki && (ki & 255u) != 0) ok = ok && a > s_adc[i - 1];
      }
      if (i + 1 < hi && s_key[i + 1] == ki + 1 && (ki & 255u) != 255u) ok = ok && a >= s_adc[i + 1];
    }
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    if (ok) cand |= 1u << j;
    mine[j] = __popc(m & ((1u << lane) - 1u));
    if (lane == 0) s_cnt[j][w] = __popc(m);
  }
  const int anyBad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    int run = 0;
    for (int j = 0; j < kCluPer; ++j)
      for (int k = 0; k < kCluThreads / 32; ++k) {
        const int v = s_cnt[j][k];
        s_cnt[j][k] = run;
        run += v;
      }
    s_total = run;
    if (!kWrite && anyBad) atomicOr(err, kErrInput);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kCluPer; ++j)
    if (cand & (1u << j)) s_queue[s_cnt[j][w] + mine[j]] = (uint16_t)(kCluHalo + j * kCluThreads + threadIdx.x);
  __syncthreads();
  // first span index in [a, b) with a key >= k
  auto lower = [&](int a, int b, unsigned long long k) {
    while (a < b) {
      const int m = (a + b) >> 1;
      if (s_key[m] < k) a = m + 1;
      else b = m;
    }
    return a;
  };
  const int total = s_total;
  int done = kWrite ? tileOff[blockIdx.x] : 0;
  for (int q0 = 0; q0 < total; q0 += kCluThreads) {
    const int q = q0 + threadIdx.x;
    bool peak = false;
    long long Q = 0, SP = 0, ST = 0;
    unsigned long long ki = 0;
    if (q < total) {
      const int i = s_queue[q];
      ki = s_key[i];
      const unsigned a = s_adc[i];
      const int p = (int)(ki & 0xff);
      const long long t = (long long)((ki >> 8) & 0xffffffffull);
      const int p0 = p > 0 ? 1 : 0, p1 = p < 255 ? 1 : 0;
      auto add = [&](unsigned b, int pb, long long tb) {
        Q += b;
        SP += (long long)b * (64 * pb + 32);
        ST += (long long)b * (64 * tb + 32);
      };
      peak = true;
      if (kWrite) {
        add(a, p, t);
        if (p0 && i > lo && s_key[i - 1] + 1 == ki) add(s_adc[i - 1], p - 1, t);
        if (p1 && i + 1 < hi && s_key[i + 1] == ki + 1) add(s_adc[i + 1], p + 1, t);
      }
      if (t > 0) {
        const unsigned long long k0 = ki - 256 - p0, k1 = ki - 256 + p1;
        for (int j = lower(max(lo, i - kCluHalo), i, k0); j < i; ++j) {
          const unsigned long long kj = s_key[j];
          if (kj > k1) break;
          const unsigned b = s_adc[j];
          if (!(a > b)) peak = false;
          if (kWrite) add(b, (int)(kj & 0xff), t - 1);
        }
      }
      {
        const unsigned long long k0 = ki + 256 - p0, k1 = ki + 256 + p1;
        for (int j = lower(i + 1, min(hi, i + kCluHalo), k0); j < hi; ++j) {
          const unsigned long long kj = s_key[j];
          if (kj > k1) break;
          const unsigned b = s_adc[j];
          if (!(a >= b)) peak = false;
          if (kWrite) add(b, (int)(kj & 0xff), t + 1);
        }
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, peak);
    if (!kWrite) {
      done += __popc(m);  // of this warp
      continue;
    }
    __syncthreads();  // the counts of the round before are read
    if (lane == 0) s_warp[w] = __popc(m);
    __syncthreads();
    int pos = done + __popc(m & ((1u << lane) - 1u));
    for (int k = 0; k < kCluThreads / 32; ++k) {
      const int v = s_warp[k];
      if (k < w) pos += v;
      done += v;
    }
    if (peak) {
      const unsigned t64 = (unsigned)((2 * ST + Q) / (2 * Q));
      const unsigned p64 = (unsigned)((2 * SP + Q) / (2 * Q));
      const unsigned ch = Q > 65535 ? 65535u : (unsigned)Q;
      const unsigned rr = (unsigned)(ki >> 40);
      uint32_t* r = reinterpret_cast<uint32_t*>(out + 12 * (size_t)pos);  // 12-byte records: 4-byte aligned
      r[0] = t64;
      r[1] = (p64 & 0xffffu) | (ch << 16);
      r[2] = (rr % kNRow) | ((rr / kNRow) << 8);
    }
  }
  if (!kWrite) {
    if (lane == 0) s_warp[w] = done;
    __syncthreads();
    if (threadIdx.x == 0) {
      int s = 0;
      for (int k = 0; k < kCluThreads / 32; ++k) s += s_warp[k];
      tileCnt[blockIdx.x] = s;
    }
  }
}

// Whether two ranges of bytes share any.
static bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return x < y + nb && y < x + na;
}

}  // namespace o2tpc

using namespace o2tpc;

extern "C" int o2tpc_clusterize(const o2tpc_digits* d, void* records, uint64_t cap, uint64_t* n_clusters,
                                void* stream) {
  if (!d || !n_clusters || (d->n > 0 && (!d->sector || !d->row || !d->pad || !d->time || !d->adc)) ||
      (cap > 0 && !records) || (reinterpret_cast<uintptr_t>(records) & 3))
    return O2TPC_EINVAL;
  *n_clusters = 0;
  if (d->n >= (1ull << 31)) return O2TPC_ETOOBIG;
  const long long n = (long long)d->n;
  if (n == 0) return O2TPC_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int nt = (int)((n + kCluTile - 1) / kCluTile);
  const size_t scanInts = (size_t)scan_scratch_ints(nt + 8) + 64;
  const size_t ints = 2 * ((size_t)nt + 1) + scanInts + 4;
  int* base = nullptr;
  if (cudaMallocAsync(reinterpret_cast<void**>(&base), sizeof(int) * ints, st) != cudaSuccess) {
    cudaGetLastError();
    return O2TPC_ENOMEM;
  }
  int* tileCnt = base;
  int* tileOff = tileCnt + nt + 1;
  int* scratch = tileOff + nt + 1;
  unsigned* err = reinterpret_cast<unsigned*>(scratch + scanInts);
  CluIn in{n, d->sector, d->row, d->pad, d->time, d->adc, 0};
  const uintptr_t all = reinterpret_cast<uintptr_t>(d->sector) | reinterpret_cast<uintptr_t>(d->row) |
                        reinterpret_cast<uintptr_t>(d->pad) | reinterpret_cast<uintptr_t>(d->time) |
                        reinterpret_cast<uintptr_t>(d->adc);
  in.wide = (all & 15) == 0;
  int rc = O2TPC_OK;
  do {
    int total = 0;
    unsigned herr = 0;
    if (cudaMemsetAsync(err, 0, sizeof(unsigned), st) != cudaSuccess) { rc = O2TPC_ECUDA; break; }
    k_clu_tile<false><<<nt, kCluThreads, 0, st>>>(in, tileCnt, nullptr, nullptr, err);
    scan_exclusive(tileCnt, tileOff, nt, nullptr, scratch, st);
    if (cudaMemcpyAsync(&total, tileOff + nt, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&herr, err, sizeof(unsigned), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      rc = O2TPC_ECUDA;
      break;
    }
    if (herr & kErrInput) { rc = O2TPC_EINVAL; break; }
    *n_clusters = (uint64_t)total;
    if ((uint64_t)total > cap) { rc = O2TPC_ETOOBIG; break; }
    if (total > 0) {
      // pass 2 reads the digits again: records that are to take their place are
      // written beside them first
      const size_t bytes = 12 * (size_t)total, m = (size_t)n;
      uint8_t *dst = static_cast<uint8_t*>(records), *beside = nullptr;
      if (overlap(dst, bytes, d->sector, m) || overlap(dst, bytes, d->row, m) || overlap(dst, bytes, d->pad, m) ||
          overlap(dst, bytes, d->time, 4 * m) || overlap(dst, bytes, d->adc, 2 * m)) {
        if (cudaMallocAsync(reinterpret_cast<void**>(&beside), bytes, st) != cudaSuccess) {
          cudaGetLastError();
          rc = O2TPC_ENOMEM;
          break;
        }
      }
      k_clu_tile<true><<<nt, kCluThreads, 0, st>>>(in, nullptr, tileOff, beside ? beside : dst, nullptr);
      if (beside) {
        if (cudaMemcpyAsync(dst, beside, bytes, cudaMemcpyDeviceToDevice, st) != cudaSuccess) rc = O2TPC_ECUDA;
        cudaFreeAsync(beside, st);
      }
    }
    if (cudaGetLastError() != cudaSuccess) rc = O2TPC_ECUDA;
  } while (false);
  cudaFreeAsync(base, st);
  if (cudaStreamSynchronize(st) != cudaSuccess && rc == O2TPC_OK) rc = O2TPC_ECUDA;
  return rc;
}
