// Host decoder of the compressed Time Frame written by csrc/k_ctf.cu: the
// reader side of the format (Sec. 2.2: the compressed TF is what is stored;
// decoding it must give back exactly the kept clusters).  Plain host code, no
// device work: a consumer of stored TFs needs no GPU.
//
// Format (see k_ctf.cu): header (magic 'O2CT', version 1, kept tracks, their
// clusters, other clusters, 10 streams), per stream (symbols, chunks,
// 256 frequencies summing to 4096, chunk sizes), then the chunk payloads.
// Each chunk holds at most 4096 symbols: a 32-bit rANS state (little endian)
// followed by the renormalisation bytes in decoding order.  The ten streams
// are byte planes of the per-cluster fields (sector delta mod 36, row delta
// mod 256, y residual lo/hi, zeta residual bytes 0-3) and of the per-track
// cluster counts (lo/hi); residuals are zigzag-mapped, against the straight
// line through the two previous clusters of the same sector segment of a
// track (rows ascending) or else against the previous cluster.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>
#include <thread>
#include <utility>
#include <vector>

#include "o2tpc.h"

namespace {

constexpr uint32_t kMagic = 0x5443324Fu;
constexpr int kStreams = 10;
constexpr uint32_t kScaleBits = 12, kM = 1u << kScaleBits, kL = 1u << 23;
constexpr int64_t kChunk = 4096;
constexpr int kRows = 152;

uint32_t rd32(const uint8_t* p) {
  return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
}

// One coded stream: its table, its symbols and where its chunks lie.
struct Stream {
  // per state slot: symbol << 24 | frequency << 12 | slot - cumulative start, for
  // streams of a whole group of chunks at least
  std::vector<uint32_t> slot;
  uint32_t f[256], c[257];
  bool wide = false;           // a frequency of 4096, which the slots cannot hold
  uint64_t nsym = 0, nch = 0;
  const uint8_t* sizes = nullptr;  // chunk sizes in the header
  std::vector<uint64_t> at;        // first payload byte of each chunk
  std::vector<uint8_t> out;
};

// Chunk ch as the format defines it, every byte checked.
bool decode_chunk(const Stream& s, const uint8_t* blob, uint64_t ch, uint8_t* out, const uint8_t* __restrict__ sym) {
  const uint8_t* __restrict__ q = blob + s.at[ch];
  const uint64_t nb = rd32(s.sizes + 4 * ch), a = ch * kChunk;
  const uint64_t m = s.nsym - a < (uint64_t)kChunk ? s.nsym - a : (uint64_t)kChunk;
  // the bytes written alias none of what is read
  const uint32_t *__restrict__ f = s.f, *__restrict__ c = s.c;
  uint8_t* __restrict__ o = out + a;
  uint32_t x = rd32(q);
  uint64_t r = 4;
  for (uint64_t i = 0; i < m; ++i) {
    const uint32_t sl = x & (kM - 1);
    const uint8_t v = sym[sl];
    o[i] = v;
    x = f[v] * (x >> kScaleBits) + sl - c[v];
    while (x < kL) {
      if (r >= nb) return false;
      x = (x << 8) | q[r++];
    }
  }
  return r == nb && x == kL;
}

// Up to four chunks from ch on.  Full chunks of which the bytes that any state
// can read (two a symbol) lie inside the blob are decoded together: four
// independent states, and no branch on whether a byte is due.  What such a
// chunk ends with tells whether it kept to its size; states outside the coder's range (an
// odd blob) and all other chunks take decode_chunk.
bool decode_group(const Stream& s, const uint8_t* blob, uint64_t bytes, uint64_t ch, uint64_t n, uint8_t* out,
                  const uint8_t* sym) {
  bool done = false;
  if (n == 4 && !s.slot.empty() && (ch + 4) * kChunk <= s.nsym && s.at[ch + 3] + 4 + 2 * kChunk + 1 <= bytes) {
    const uint8_t* q[4];
    uint32_t x[4], low = 0;
    uint8_t* o[4];
    for (int k = 0; k < 4; ++k) {
      q[k] = blob + s.at[ch + k];
      x[k] = rd32(q[k]);
      low |= x[k] < kL;
      q[k] += 4;
      o[k] = out + (ch + k) * kChunk;
    }
    const uint32_t* slot = s.slot.data();
    for (int64_t i = 0; i < kChunk; ++i)
      for (int k = 0; k < 4; ++k) {
        const uint32_t e = slot[x[k] & (kM - 1)];
        o[k][i] = (uint8_t)(e >> 24);
        uint32_t y = ((e >> 12) & 0xfffu) * (x[k] >> kScaleBits) + (e & 0xfffu);
        for (int t = 0; t < 2; ++t) {
          const uint32_t due = y < kL;
          y = due ? (y << 8) | *q[k] : y;
          q[k] += due;
        }
        low |= y < kL;
        x[k] = y;
      }
    if (!low) {
      for (int k = 0; k < 4; ++k)
        if (q[k] != blob + s.at[ch + k] + rd32(s.sizes + 4 * (ch + k)) || x[k] != kL) return false;
      done = true;
    }
  }
  for (uint64_t k = 0; k < n && !done; ++k)
    if (!decode_chunk(s, blob, ch + k, out, sym)) return false;
  return true;
}

long long floor_div(long long a, long long b) {  // b > 0
  long long q = a / b;
  if (a % b != 0 && a < 0) --q;
  return q;
}

}  // namespace

namespace {

// The streams' tables and chunk places; false: not a compressed TF.
bool read_headers(const uint8_t* blob, uint64_t bytes, uint64_t nSeq, uint64_t nTrk, Stream* st) {
  uint64_t pos = 24;
  for (int k = 0; k < kStreams; ++k) {
    Stream& s = st[k];
    if (pos + 8 + 512 > bytes) return false;
    s.nsym = rd32(blob + pos);
    s.nch = rd32(blob + pos + 4);
    const uint8_t* f = blob + pos + 8;
    s.c[0] = 0;
    for (int v = 0; v < 256; ++v) {
      s.f[v] = (uint32_t)f[2 * v] | ((uint32_t)f[2 * v + 1] << 8);
      s.c[v + 1] = s.c[v] + s.f[v];
      s.wide |= s.f[v] >= kM;
    }
    s.sizes = blob + pos + 8 + 512;
    pos += 8 + 512 + 4 * s.nch;
    if (pos > bytes || s.nch != (s.nsym + kChunk - 1) / kChunk || (s.nsym > 0 && s.c[256] != kM)) return false;
    if (s.nsym != (k < 8 ? nSeq : nTrk)) return false;
  }
  for (int k = 0; k < kStreams; ++k) {  // the payloads follow the last header, and end the blob
    Stream& s = st[k];
    s.at.resize(s.nch);
    for (uint64_t ch = 0; ch < s.nch; ++ch) {
      const uint64_t nb = rd32(s.sizes + 4 * ch);
      s.at[ch] = pos;
      pos += nb;
      if (nb < 4 || pos > bytes) return false;
    }
  }
  return pos == bytes;
}

// All streams.  Chunks are independent: blocks of four go to up to eight threads,
// of at least 32 blocks (half a million symbols, 1-2 ms) each; smaller blobs
// stay on the caller's.  1.7 M clusters on 8 cores: 82 -> 18 ms with the
// four-state loop and the division-free rebuild.
bool decode_streams(const uint8_t* blob, uint64_t bytes, Stream* st) {
  std::vector<uint8_t> sym((size_t)kStreams * kM);
  std::vector<std::pair<int, uint64_t>> units;
  for (int k = 0; k < kStreams; ++k) {
    Stream& s = st[k];
    s.out.resize(s.nsym);
    if (!s.nsym) continue;
    for (int v = 0; v < 256; ++v)  // c[256] = 4096
      if (s.f[v]) std::memset(sym.data() + (size_t)k * kM + s.c[v], v, s.f[v]);
    // (16 KB a stream: with a table for every stream a blob of 30 clusters took 61
    // us, of 10 000 545; now 26 and 451)
    if (!s.wide && s.nsym >= 4 * (uint64_t)kChunk) {
      s.slot.resize(kM);
      for (int v = 0; v < 256; ++v)
        for (uint32_t q = s.c[v]; q < s.c[v + 1]; ++q) s.slot[q] = ((uint32_t)v << 24) | (s.f[v] << 12) | (q - s.c[v]);
    }
    for (uint64_t ch = 0; ch < s.nch; ch += 4) units.emplace_back(k, ch);
  }
  std::atomic<size_t> next{0};
  std::atomic<bool> ok{true};
  auto work = [&]() {
    for (;;) {
      const size_t u = next.fetch_add(1);
      if (u >= units.size() || !ok.load(std::memory_order_relaxed)) return;
      Stream& s = st[units[u].first];
      const uint64_t ch = units[u].second, n = s.nch - ch < 4 ? s.nch - ch : 4;
      if (!decode_group(s, blob, bytes, ch, n, s.out.data(), sym.data() + (size_t)units[u].first * kM)) ok = false;
    }
  };
  const size_t cores = std::max(1u, std::thread::hardware_concurrency());
  const size_t want = std::min<size_t>(std::min<size_t>(cores, 8), units.size() / 32);
  std::vector<std::thread> helpers;
  try {
    for (size_t k = 1; k < want; ++k) helpers.emplace_back(work);
  } catch (...) {  // fewer threads then
  }
  work();
  for (auto& h : helpers) h.join();
  return ok;
}

// The cluster sequence from its byte planes; false: a row that does not exist.
bool rebuild(const Stream* st, uint64_t nSeq, uint64_t nTrk, uint64_t nFree, int32_t* sec, int32_t* row, int32_t* y,
             int32_t* z, uint32_t* len) {
  const uint8_t *p0 = st[0].out.data(), *p1 = st[1].out.data(), *p2 = st[2].out.data(), *p3 = st[3].out.data();
  const uint8_t *p4 = st[4].out.data(), *p5 = st[5].out.data(), *p6 = st[6].out.data(), *p7 = st[7].out.data();
  // the previous cluster, and of the one before what the line needs
  int32_t s1 = 0, r1 = 0, y1 = 0, z1 = 0, s0 = -1, r0 = 0, y0 = 0, z0 = 0;
  int32_t top = 0;
  uint64_t o = 0;
  for (uint64_t t = 0; t <= nTrk; ++t) {
    const uint64_t m = t < nTrk ? len[t] : nFree;
    for (uint64_t q = 0; q < m; ++q, ++o) {
      const int32_t s = (s1 + p0[o]) % 36;
      const int32_t r = (r1 + p1[o]) & 0xff;
      const uint16_t zy = (uint16_t)(p2[o] | (p3[o] << 8));
      const uint32_t zz = (uint32_t)p4[o] | ((uint32_t)p5[o] << 8) | ((uint32_t)p6[o] << 16) | ((uint32_t)p7[o] << 24);
      const int32_t ry = (int16_t)((zy >> 1) ^ (uint16_t)(0u - (zy & 1u)));
      const int32_t rz = (int32_t)((zz >> 1) ^ (0u - (zz & 1u)));
      // the straight line through the two previous clusters of the track's
      // current sector segment, else the previous cluster
      long long predY = y1, predZ = z1;
      if (t < nTrk && q >= 2 && s0 == s && s1 == s && r0 < r1 && r1 < r) {
        const long long dy = (long long)(y1 - y0) * (r - r1), dz = (long long)(z1 - z0) * (r - r1);
        if (r1 - r0 == 1) {  // nearly always
          predY += dy;
          predZ += dz;
        } else {
          predY += floor_div(dy, r1 - r0);
          predZ += floor_div(dz, r1 - r0);
        }
      }
      s0 = s1;
      r0 = r1;
      y0 = y1;
      z0 = z1;
      s1 = s;
      r1 = r;
      y1 = (int32_t)(int16_t)(uint16_t)(uint64_t)(predY + ry);
      z1 = (int32_t)(uint32_t)(uint64_t)(predZ + rz);
      sec[o] = s;
      row[o] = r;
      y[o] = y1;
      z[o] = z1;
      top = r > top ? r : top;
    }
  }
  return nSeq == 0 || top < kRows;
}

}  // namespace

extern "C" int o2tpc_ctf_decode(const uint8_t* blob, uint64_t bytes, o2tpc_ctf_clusters* out) {
  if (!blob || !out) return O2TPC_EINVAL;
  std::memset(out, 0, sizeof(*out));
  if (bytes < 24 || rd32(blob) != kMagic || rd32(blob + 4) != 1 || rd32(blob + 20) != (uint32_t)kStreams)
    return O2TPC_EINVAL;
  const uint64_t nTrk = rd32(blob + 8), nTc = rd32(blob + 12), nFree = rd32(blob + 16), nSeq = nTc + nFree;
  int32_t *sec = nullptr, *row = nullptr, *y = nullptr, *z = nullptr;
  uint32_t* len = nullptr;
  int rc = O2TPC_OK;
  try {
    std::vector<Stream> st(kStreams);
    if (!read_headers(blob, bytes, nSeq, nTrk, st.data()) || !decode_streams(blob, bytes, st.data()))
      return O2TPC_EINVAL;
    sec = static_cast<int32_t*>(std::malloc(4 * (nSeq + 1)));
    row = static_cast<int32_t*>(std::malloc(4 * (nSeq + 1)));
    y = static_cast<int32_t*>(std::malloc(4 * (nSeq + 1)));
    z = static_cast<int32_t*>(std::malloc(4 * (nSeq + 1)));
    len = static_cast<uint32_t*>(std::malloc(4 * (nTrk + 1)));
    if (!sec || !row || !y || !z || !len) {
      rc = O2TPC_ENOMEM;
    } else {
      uint64_t sum = 0;
      for (uint64_t t = 0; t < nTrk; ++t) {
        len[t] = (uint32_t)st[8].out[t] | ((uint32_t)st[9].out[t] << 8);
        sum += len[t];
      }
      if (sum != nTc || !rebuild(st.data(), nSeq, nTrk, nFree, sec, row, y, z, len)) rc = O2TPC_EINVAL;
    }
  } catch (...) {  // std::bad_alloc
    rc = O2TPC_ENOMEM;
  }
  if (rc != O2TPC_OK) {
    std::free(sec), std::free(row), std::free(y), std::free(z), std::free(len);
    return rc;
  }
  out->n = nSeq;
  out->n_tracks = nTrk;
  out->sector = sec;
  out->row = row;
  out->y = y;
  out->zeta = z;
  out->track_len = len;
  return O2TPC_OK;
}

extern "C" void o2tpc_ctf_free(o2tpc_ctf_clusters* c) {
  if (!c) return;
  std::free(const_cast<int32_t*>(c->sector));
  std::free(const_cast<int32_t*>(c->row));
  std::free(const_cast<int32_t*>(c->y));
  std::free(const_cast<int32_t*>(c->zeta));
  std::free(const_cast<uint32_t*>(c->track_len));
  std::memset(c, 0, sizeof(*c));
}

extern "C" int o2tpc_ctf_records(const o2tpc_ctf_clusters* c, void* records) {
  if (!c || (c->n > 0 && !records)) return O2TPC_EINVAL;
  // pads per row: floor(2 x_r tan(10 deg) / 0.4 cm), x_r = 85 + r 160/151 cm
  int npads[kRows];
  for (int r = 0; r < kRows; ++r)
    npads[r] = (int)std::floor(2.0 * (85.0 + r * 160.0 / 151.0) * std::tan(10.0 * 3.14159265358979323846 / 180.0) / 0.4);
  uint8_t* o = static_cast<uint8_t*>(records);
  for (uint64_t i = 0; i < c->n; ++i, o += 12) {
    const int r = c->row[i];
    const long long pad64 = (long long)c->y[i] + 32ll * npads[r];
    const long long t64 = c->zeta[i];
    if (r < 0 || r >= kRows || c->sector[i] < 0 || c->sector[i] >= 36 || pad64 < 0 || pad64 > 0xffff || t64 < 0 ||
        t64 >= (1ll << 30))
      return O2TPC_EINVAL;
    // little endian; charges are not stored
    const uint32_t w[3] = {(uint32_t)t64, (uint32_t)pad64, (uint32_t)r | ((uint32_t)c->sector[i] << 8)};
    std::memcpy(o, w, 12);
  }
  return O2TPC_OK;
}
