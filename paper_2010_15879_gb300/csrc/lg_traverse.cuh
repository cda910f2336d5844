// Graph kernels with the Log(Graph) decoder fused in (Sections 3.7.2-3.7.3 for
// the access path, Section 7.1.2 for BFS and PageRank).
//
// PageRank sweeps are in lg_pull.cuh.  The other pull sweeps (bottom-up BFS,
// batched personalized PageRank) are one launch with two kinds of CTA:
//   * heavy CTAs walk the heavy-vertex schedule built at encode time: vertices
//     of degree > heavy_min split into items of <= heavy_seg fields, one warp per
//     item, lane i decoding field i of each 32-field chunk with 4 chunks in
//     flight (gap-coded IDs by a warp prefix sum from the item's carry);
//   * tile CTAs take 64 to 512 consecutive stored labels each (tile_map):
//     1. offsets x_v of the tile (packed fields, CSR row_ptr, or an
//        Elias-Fano block decode: from the sample at or below the tile's first
//        vertex on, every thread lists the ones of its words);
//     2. per vertex: degree and field width from the offsets and the
//        neighborhood header;
//     3. light vertices (degree <= heavy_min) are split over the threads in
//        contiguous runs of nearly equal field counts, each thread decoding
//        its run with a sequential bit reader (one 32-byte sector per 256 bits,
//        a shift and a mask per field, a running sum for gap-coded IDs, four
//        gathers in flight).
// A BFS's vertices split into several items are finished by the item that
// arrives last, those of personalized PageRank by a small second kernel.
// Push steps and neighbor queries decode one random vertex per warp.
#pragma once

#include <algorithm>

#include "lg_internal.h"
#include "lg_window.cuh"

namespace lg {

constexpr int TV = LG_TILE_V;  // vertices per tile
constexpr int TNT = 256;       // threads per tile CTA
// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t udiv_small(uint64_t a, uint32_t b) {
  return a < 0x100000000ull ? (uint64_t)((uint32_t)a / b) : a / b;
}

template <typename M> __device__ __forceinline__ M atomic_or_mask(M* p, M m);
template <> __device__ __forceinline__ uint16_t atomic_or_mask<uint16_t>(uint16_t* p, uint16_t m) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  uint32_t* w = reinterpret_cast<uint32_t*>(a & ~(uintptr_t)3);
  const uint32_t sh = (uint32_t)(a & 2) * 8u;
  return (uint16_t)(atomicOr(w, (uint32_t)m << sh) >> sh);
}
template <> __device__ __forceinline__ uint32_t atomic_or_mask<uint32_t>(uint32_t* p, uint32_t m) {
  return atomicOr(p, m);
}
template <> __device__ __forceinline__ uint64_t atomic_or_mask<uint64_t>(uint64_t* p, uint64_t m) {
  return (uint64_t)atomicOr(reinterpret_cast<unsigned long long*>(p), (unsigned long long)m);
}

// reads and clears a mask
template <typename M> __device__ __forceinline__ M atomic_take_mask(M* p);
template <> __device__ __forceinline__ uint16_t atomic_take_mask<uint16_t>(uint16_t* p) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  const uint32_t sh = (uint32_t)(a & 2) * 8u;
  return (uint16_t)(atomicAnd(reinterpret_cast<uint32_t*>(a & ~(uintptr_t)3), ~(0xffffu << sh)) >> sh);
}
template <> __device__ __forceinline__ uint32_t atomic_take_mask<uint32_t>(uint32_t* p) { return atomicExch(p, 0u); }
template <> __device__ __forceinline__ uint64_t atomic_take_mask<uint64_t>(uint64_t* p) {
  return (uint64_t)atomicExch(reinterpret_cast<unsigned long long*>(p), 0ull);
}

// depth of v for every source in bitsv: row s of the S x n array, or row
// rows[s] when the caller keeps one separate row per source (a source that
// joined a running sweep at level row_base[s] counts depths from there)
template <typename M>
__device__ __forceinline__ void write_depths(const BfsArgs& a, uint64_t n, uint64_t v, M bitsv, uint32_t d) {
  uint64_t b = (uint64_t)bitsv;
  while (b) {
    const int s = __ffsll((long long)b) - 1;
    b &= b - 1;
    if (a.rows) a.rows[s][a.row_perm ? (uint64_t)a.row_perm[v] : v] = d - a.row_base[s];
    else if (a.vmajor) a.depth[v * a.S + s] = d;
    else a.depth[(uint64_t)s * n + v] = d;
  }
}

// ---------------------------------------------------------------------------
// offsets of a tile: xs[i] = x_{v0+i}, i = 0..cnt (cnt+1 values)
// ---------------------------------------------------------------------------
struct TileScratch {
  uint32_t red[TNT / 32];
};

template <int OFF>
__device__ __forceinline__ void tile_offsets(const GView& g, uint64_t v0, int cnt, uint64_t* xs, TileScratch& ts);

template <>
__device__ __forceinline__ void tile_offsets<OFF_PACKED>(const GView& g, uint64_t v0, int cnt, uint64_t* xs,
                                                         TileScratch&) {
  for (int i = threadIdx.x; i <= cnt; i += TNT) xs[i] = ext64(g.O, (v0 + i) * g.w_O, g.w_O);
}

template <>
__device__ __forceinline__ void tile_offsets<OFF_ROWPTR>(const GView& g, uint64_t v0, int cnt, uint64_t* xs,
                                                         TileScratch&) {
  for (int i = threadIdx.x; i <= cnt; i += TNT) xs[i] = __ldg(g.O + v0 + i);
}

// Elias-Fano block decode (Section 4.3): ones number v0 .. v0+cnt of the high
// vector, starting from the sample at or below v0.  A thread lists the ones of
// its word: some twelve, while a search of the words' ranks for every one took
// a hundred instructions each.
template <>
__device__ __forceinline__ void tile_offsets<OFF_EF>(const GView& g, uint64_t v0, int cnt, uint64_t* xs,
                                                     TileScratch& ts) {
  const uint64_t k = v0 >> g.sample_log2;
  const uint64_t p0 = __ldg(g.ef_samples + k);
  const uint64_t skip = v0 - (k << g.sample_log2);
  const uint64_t need_end = skip + (uint64_t)cnt + 1;
  uint64_t wbase = (p0 >> 5) & ~3ull, carry = 0;
  auto list = [&](uint32_t w, uint64_t wi, int64_t i) {  // the word's first one is that of vertex v0 + i
    for (; w && i <= cnt; i++, w &= w - 1u)
      if (i >= 0) xs[i] = wi * 32u + (uint32_t)__ffs((int)w) - 1u;
  };
  uint32_t total;
  {
    const uint64_t wi = wbase + threadIdx.x;
    uint32_t w = wi < g.ef_high_words32 && wi >= (p0 >> 5) ? __ldg(g.ef_high32 + wi) : 0u;
    if (wi == (p0 >> 5)) w &= 0xffffffffu << ((uint32_t)p0 & 31u);
    const uint32_t pre = block_excl_scan<uint32_t, TNT>((uint32_t)__popc(w), total, ts.red);
    list(w, wi, (int64_t)pre - (int64_t)skip);
  }
  // hubs spread a tile over thousands of words: four per thread from here on
  for (carry = total, wbase += TNT; carry < need_end && wbase < g.ef_high_words32; carry += total, wbase += 4 * TNT) {
    const uint64_t wi = wbase + 4u * threadIdx.x;  // the array is padded to 16 bytes with zeros
    const uint4 y = wi < g.ef_high_words32 ? ldg128(g.ef_high32 + wi) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t c0 = __popc(y.x), c1 = c0 + __popc(y.y), c2 = c1 + __popc(y.z);
    const uint32_t pre = block_excl_scan<uint32_t, TNT>(c2 + __popc(y.w), total, ts.red);
    const int64_t i = (int64_t)(carry + pre) - (int64_t)skip;
    list(y.x, wi, i);
    list(y.y, wi + 1, i + c0);
    list(y.z, wi + 2, i + c1);
    list(y.w, wi + 3, i + c2);
  }
  __syncthreads();
  for (int i = threadIdx.x; i <= cnt; i += TNT) {
    const uint64_t lo = g.ef_l ? ext64(g.ef_low, (v0 + i) * g.ef_l, g.ef_l) : 0u;
    xs[i] = ((xs[i] - (v0 + i)) << g.ef_l) | lo;
  }
}

// ---------------------------------------------------------------------------
// random-access offsets x_v, x_{v+1}; called by all 32 lanes of a warp
// ---------------------------------------------------------------------------
template <int OFF>
__device__ __forceinline__ void offset_pair(const GView& g, uint64_t v, uint64_t& x0, uint64_t& x1);

template <>
__device__ __forceinline__ void offset_pair<OFF_PACKED>(const GView& g, uint64_t v, uint64_t& x0, uint64_t& x1) {
  x0 = ext64(g.O, v * g.w_O, g.w_O);
  x1 = ext64(g.O, (v + 1) * g.w_O, g.w_O);
}
template <>
__device__ __forceinline__ void offset_pair<OFF_ROWPTR>(const GView& g, uint64_t v, uint64_t& x0, uint64_t& x1) {
  x0 = __ldg(g.O + v);
  x1 = __ldg(g.O + v + 1);
}
// Warp select of ones number v and v+1 (Section 4.1: O_v = select_O(v)), from
// the sample at or below v.  32 words hold the 512 ones of an ordinary sample
// block; a hub among its vertices spreads it (degree >> l zeros), so later
// steps take 128 words.
template <>
__device__ __forceinline__ void offset_pair<OFF_EF>(const GView& g, uint64_t v, uint64_t& x0, uint64_t& x1) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t k = v >> g.sample_log2;
  const uint64_t p0 = __ldg(g.ef_samples + k);
  const uint64_t lo0 = g.ef_l ? ext64(g.ef_low, v * g.ef_l, g.ef_l) : 0;
  const uint64_t lo1 = g.ef_l ? ext64(g.ef_low, (v + 1) * g.ef_l, g.ef_l) : 0;
  const uint64_t rem = v - (k << g.sample_log2);
  uint64_t carry = 0;
  uint64_t pos[2] = {0, 0};
  uint32_t found = 0;
  // a lane's words wi .. wi + 3 of the high vector
  auto step = [&](const uint32_t (&w)[4], uint64_t wi) {
    const uint32_t c = __popc(w[0]) + __popc(w[1]) + __popc(w[2]) + __popc(w[3]);
    const uint32_t incl = warp_incl_scan<uint32_t>(c);
#pragma unroll
    for (int t = 0; t < 2; t++) {
      const uint64_t at = carry + incl - c;
      const bool here = !(found >> t & 1u) && at <= rem + t && rem + t < carry + incl;
      const uint32_t b = __ballot_sync(LG_FULL_MASK, here);
      uint64_t p = 0;
      if (here) {
        uint32_t r = (uint32_t)(rem + t - at), q = 0, x = w[0];
#pragma unroll
        for (int z = 1; z < 4; z++)
          if (r >= (uint32_t)__popc(x) && q == (uint32_t)(z - 1)) { r -= __popc(x); x = w[z]; q = z; }
        p = (wi + q) * 32u + select_in_u32(x, r);
      }
      if (b) {
        pos[t] = __shfl_sync(LG_FULL_MASK, p, __ffs((int)b) - 1);
        found |= 1u << t;
      }
    }
    carry += __shfl_sync(LG_FULL_MASK, incl, 31);
  };
  uint64_t wbase = (p0 >> 5) & ~3ull;
  {
    const uint64_t wi = wbase + lane;
    uint32_t w[4] = {wi < g.ef_high_words32 && wi >= (p0 >> 5) ? __ldg(g.ef_high32 + wi) : 0u, 0u, 0u, 0u};
    if (wi == (p0 >> 5)) w[0] &= 0xffffffffu << ((uint32_t)p0 & 31u);
    step(w, wi);
  }
  for (wbase += 32; found != 3u && wbase < g.ef_high_words32; wbase += 128) {
    const uint64_t wi = wbase + 4u * lane;  // the array is padded to 16 bytes with zeros
    const uint4 y = wi < g.ef_high_words32 ? ldg128(g.ef_high32 + wi) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t w[4] = {y.x, y.y, y.z, y.w};
    step(w, wi);
  }
  x0 = ((pos[0] - v) << g.ef_l) | lo0;
  x1 = ((pos[1] - (v + 1)) << g.ef_l) | lo1;
}

// ---------------------------------------------------------------------------
// neighborhood geometry from consecutive offsets (Section 3.7.3: d_v from
// O[v+1] - O[v]; in the local modes from the bit length and the header)
//   start: bit of the first field; w: field width (IDs, or gaps for LOCAL_GAP)
// ---------------------------------------------------------------------------
template <int IDM>
__device__ __forceinline__ uint32_t vhead(const GView& g, uint64_t x0) {  // the header of a neighborhood, if it has one
  return IDM == ID_LOCAL || IDM == ID_LOCAL_GAP ? ext32(g.A32, x0, g.H) : 0u;
}
template <int IDM>
__device__ __forceinline__ void vgeo(const GView& g, uint64_t x0, uint64_t x1, uint32_t head, uint64_t& start,
                                     uint32_t& deg, uint32_t& w) {
  if (IDM == ID_GLOBAL) {
    start = x0 * g.r; deg = (uint32_t)(x1 - x0); w = g.s;
  } else if (IDM == ID_CSR32) {
    start = x0 * 32u; deg = (uint32_t)(x1 - x0); w = 32;
  } else if (IDM == ID_LOCAL) {
    w = head;
    deg = w ? (uint32_t)udiv_small(x1 - x0 - g.H, w) : 0u;
    start = x0 + g.H;
  } else {
    w = head;
    const uint64_t len = x1 - x0;
    deg = len == g.H ? 0u : (w == 0 ? 1u : 1u + (uint32_t)udiv_small(len - g.H - g.s, w));
    start = x0 + g.H;
  }
}
template <int IDM>
__device__ __forceinline__ void vgeo(const GView& g, uint64_t x0, uint64_t x1, uint64_t& start, uint32_t& deg,
                                     uint32_t& w) {
  vgeo<IDM>(g, x0, x1, vhead<IDM>(g, x0), start, deg, w);
}

// First schedule item of heavy vertex v (a warp; the items are in vertex order).
__device__ __forceinline__ uint64_t first_item(const GView& g, uint64_t v) {
  uint64_t lo = 0, hi = g.n_items;  // the first item whose vertex is not below v
  while (lo < hi) {
    const uint64_t step = (hi - lo + 31) / 32, at = lo + (threadIdx.x & 31u) * step;
    const uint32_t c = __popc(__ballot_sync(LG_FULL_MASK, at < hi && (uint64_t)g.items[at].v < v));
    const uint64_t next = c ? lo + (uint64_t)(c - 1) * step + 1 : lo;
    hi = min(hi, lo + (uint64_t)c * step);
    lo = next;
  }
  return lo;
}

// Geometry of one random vertex, by a warp.  In DM order the leading vertices'
// Elias-Fano blocks are long (their first 512 vertices hold a tenth or more of
// the arcs, thousands of words to scan: 24 us on R-MAT 2^20), so those are
// looked up in the schedule, which lists them in order (four steps of 32
// probes at most).
template <int IDM, int OFF>
__device__ __forceinline__ void vertex_geo(const GView& g, uint64_t v, uint64_t& start, uint32_t& d, uint32_t& w) {
  if (OFF == OFF_EF && v < g.heavy_prefix) {
    const HeavyItem* h = g.items + first_item(g, v);
    start = h->bit;
    d = h->deg;
    w = h->w;
    return;
  }
  uint64_t x0, x1;
  offset_pair<OFF>(g, v, x0, x1);
  vgeo<IDM>(g, x0, x1, start, d, w);
}

// sequential decoder for one neighborhood (light path)
template <int IDM>
struct SeqDec {
  BitReader br;
  uint32_t w, s, omega, id;
  bool first;
  __device__ __forceinline__ void init(const GView& g, uint64_t start, uint32_t width, uint64_t pol) {
    br.init(g.A32, start, pol);
    w = width; s = g.s; omega = g.omega; id = 0; first = true;
  }
  __device__ __forceinline__ uint32_t next() {
    if (IDM == ID_GLOBAL) {
      const uint32_t v = br.get(s);
      if (omega) br.skip(omega);
      return v;
    } else if (IDM == ID_CSR32) {
      return br.get(32);
    } else if (IDM == ID_LOCAL) {
      return br.get(w);
    } else {
      id = first ? br.get(s) : id + br.get(w);
      first = false;
      return id;
    }
  }
};

// value of field i for the warp path (not yet prefix-summed for gaps)
template <int IDM>
__device__ __forceinline__ uint32_t field_at(const GView& g, uint64_t start, uint32_t w, uint64_t i) {
  if (IDM == ID_GLOBAL) return ext32(g.A32, start + i * g.r, g.s);
  if (IDM == ID_CSR32) return __ldg(g.A32 + (start >> 5) + i);
  if (IDM == ID_LOCAL) return ext32(g.A32, start + i * w, w);
  // the first field holds the absolute ID in s bits, the others gaps in w bits
  const uint64_t p = i == 0 ? start : start + g.s + (i - 1) * (uint64_t)w;
  return ext32(g.A32, p, i == 0 ? g.s : w);
}
__device__ __forceinline__ uint32_t weight_at(const GView& g, uint64_t start, uint64_t i) {
  return ext32(g.A32, start + i * g.r + g.s, g.omega);
}

// Lane-parallel decode of U chunks of 32 fields starting at field `base`
// (fields >= f1 read as 0).  Gap-coded IDs are prefix-summed across the warp
// with `carry` = the absolute ID before field `base`; carry is advanced.  All
// field loads of the U chunks are independent, so they are in flight together.
template <int IDM, int U>
__device__ __forceinline__ void warp_ids(const GView& g, uint64_t start, uint32_t w, uint32_t base, uint32_t f1,
                                         uint32_t& carry, uint32_t (&val)[U]) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int u = 0; u < U; u++) {
    const uint32_t idx = base + 32u * u + lane;
    val[u] = idx < f1 ? field_at<IDM>(g, start, w, idx) : 0u;
  }
  if (IDM == ID_LOCAL_GAP) {
#pragma unroll
    for (int u = 0; u < U; u++) {
      val[u] = warp_incl_scan<uint32_t>(val[u]) + carry;
      carry = __shfl_sync(LG_FULL_MASK, val[u], 31);
    }
  }
}

constexpr int HEAVY_U = 4;  // chunks of 32 fields in flight per warp

}  // namespace lg

#include "lg_pull.cuh"

namespace lg {

// ---------------------------------------------------------------------------
// tile phases shared by the pull kernels
// ---------------------------------------------------------------------------
struct TileSmem {
  uint64_t xs[TV + 1];     // offsets
  uint64_t st[TV];         // first-field bit of each vertex
  uint32_t deg[TV];
  uint32_t fpre[TV + 1];   // field prefix over the compacted light list
  uint16_t clist[TV];      // compacted light vertices (local index)
  uint8_t wid[TV];
  uint32_t nlight, nfields;
  uint64_t red64[TNT / 32];
  TileScratch ts;
};

// Phase 2: geometry of each vertex; light vertices (0 < degree <= heavy_min)
// that `keep(i)` accepts form the compacted, field-prefix-summed list.
// Heavier vertices are left to the heavy schedule.
template <int IDM, typename Keep>
__device__ __forceinline__ void tile_classify(const GView& g, TileSmem& sm, int cnt, Keep keep) {
  uint32_t lc = 0, lf = 0;
  bool light[TV / TNT];
#pragma unroll
  for (int q = 0; q < TV / TNT; q++) {
    const int i = threadIdx.x * (TV / TNT) + q;
    light[q] = false;
    if (i < cnt) {
      uint64_t start; uint32_t d, w;
      vgeo<IDM>(g, sm.xs[i], sm.xs[i + 1], start, d, w);
      sm.st[i] = start; sm.deg[i] = d; sm.wid[i] = (uint8_t)w;
      if (d > 0 && d <= g.heavy_min && keep(i)) { light[q] = true; lc++; lf += d; }
    }
  }
  uint64_t total;
  const uint64_t pre = block_excl_scan<uint64_t, TNT>(((uint64_t)lc << 32) | lf, total, sm.red64);
  uint32_t ci = (uint32_t)(pre >> 32), cf = (uint32_t)pre;
#pragma unroll
  for (int q = 0; q < TV / TNT; q++) {
    const int i = threadIdx.x * (TV / TNT) + q;
    if (light[q]) {
      sm.clist[ci] = (uint16_t)i;
      sm.fpre[ci] = cf;
      ci++;
      cf += sm.deg[i];
    }
  }
  if (threadIdx.x == 0) {
    sm.nlight = (uint32_t)(total >> 32);
    sm.nfields = (uint32_t)total;
    sm.fpre[sm.nlight] = (uint32_t)total;
  }
  __syncthreads();
}

// range of compacted light vertices owned by this thread (balanced by fields)
__device__ __forceinline__ void light_range(const TileSmem& sm, uint32_t& jb, uint32_t& je) {
  const uint64_t F = sm.nfields;
  const uint32_t flo = (uint32_t)((F * threadIdx.x) / TNT);
  const uint32_t fhi = (uint32_t)((F * (threadIdx.x + 1)) / TNT);
  const uint32_t nl = sm.nlight;
  uint32_t a = 0, b = nl;
  while (a < b) { const uint32_t m = (a + b) >> 1; if (sm.fpre[m] < flo) a = m + 1; else b = m; }
  jb = a;
  b = nl;
  while (a < b) { const uint32_t m = (a + b) >> 1; if (sm.fpre[m] < fhi) a = m + 1; else b = m; }
  je = a;
}

// number of CTAs that work on the heavy schedule (one item per warp)
__host__ __device__ inline unsigned heavy_blocks(uint64_t n_items) {
  return (unsigned)((n_items + (TNT / 32) - 1) / (TNT / 32));
}

// A tile of 512 vertices of 256 arcs gives each thread 512 fields, four at a
// time: 130 us for a BFS level, 490 us for a personalized PageRank sweep, even
// on a graph of 62,000 vertices (measured), and a warp per 4,096-field item 30
// to 60 us.  On large graphs other CTAs fill that time; below 2^22 vertices
// the DM-ordered vertices of more than 32 arcs go in tiles of 64 to 512, as many
// as keep a tile's fields (at most heavy_min a vertex) a small part of the
// arcs: 1 / 450 where every degree is near the largest, down to 1 / 1800 where
// few are and the large tiles all start first.  Small tiles spend their time on
// offsets and scans, large ones end late; BFS from 16 sources at 64 / 128 / 256
// / 512, us (taken: *): R-MAT 2^18 577* 696 821 1118, 2^20 1017* 1043 1191 1622,
// 3 M vertices 1713 1705* 1942 2528; community 0.7 M 702* 757 866 1074; 400,000
// vertices of degree 160 608 549 474* 513, 1.5 M of 40 1703 1355 1202 1165*,
// 1 M of 250 1779 1483 1241 1239*.  The others go in tiles small enough for
// about four CTAs per SM, and when items are few a whole CTA takes one
// (gap-coded items cannot be entered mid-way).
inline TileMap tile_map(const GView& g, bool gap) {
  TileMap m;
  const bool small = g.n < (1ull << 22);
  // 1 / 4 .. 1: mean degree over the largest
  const double even = std::max(0.25, (double)g.arcs / ((double)g.n * std::max(g.max_degree, 1u)));
  const double vertices = (double)g.arcs * even / 450.0 / std::max(std::min(g.max_degree, g.heavy_min), 1u);
  m.ta = 64;
  while (m.ta < TV && 2.0 * m.ta <= vertices) m.ta *= 2;
  m.tb = TV;
  if (small)
    while (m.tb > 64 && g.n / m.tb < 4 * 152) m.tb /= 2;
  m.a = g.heavy_prefix & ~(uint64_t)((small ? 64 : TV) - 1);
  m.b = small && g.mid_prefix > m.a ? (g.mid_prefix + TV - 1) & ~(uint64_t)(TV - 1) : m.a;
  m.na = (uint32_t)((std::min(g.n, m.b) - std::min(g.n, m.a) + m.ta - 1) / m.ta);
  m.shared = !gap && g.n_items < 152 * 16;
  m.hb = m.shared ? (uint32_t)g.n_items : heavy_blocks(g.n_items);
  return m;
}
inline unsigned tile_map_grid(const GView& g, const TileMap& m) {
  return m.hb + m.na + (g.n > m.b ? (unsigned)((g.n - m.b + m.tb - 1) / m.tb) : 0u);
}
__device__ __forceinline__ void tile_of(const GView& g, const TileMap& m, uint64_t& v0, int& cnt) {
  const uint32_t t = blockIdx.x - m.hb;
  v0 = t < m.na ? m.a + (uint64_t)t * m.ta : m.b + (uint64_t)(t - m.na) * m.tb;
  cnt = t < m.na ? (int)min((uint64_t)m.ta, min(g.n, m.b) - v0) : (int)min((uint64_t)m.tb, g.n - v0);
}

// ===========================================================================
// PageRank: r_0 (the sweeps are in lg_pull.cuh).  Also zeroes the ticket and
// part counters of the sweeps and, with Elias-Fano offsets, notes where each
// warp tile's first one is in the high vector (`aux`), so that a sweep's tiles
// need no select whatever the sample rate.
// ===========================================================================
template <int IDM, int OFF>
__global__ void __launch_bounds__(TNT) k_pr_init(GView g, PrArgs a, uint32_t tile0) {
  __shared__ uint64_t xs[TV + 1];
  __shared__ TileScratch ts;
  const uint64_t gt = (uint64_t)blockIdx.x * TNT + threadIdx.x, gs = (uint64_t)gridDim.x * TNT;
  for (uint64_t i = gt; i < a.nsync; i += gs) a.sync[i] = 0;
  // vertices of tiles that hold none but heavy ones
  for (uint64_t i = gt; i < g.n_items && tile0; i += gs) {
    const HeavyItem h = g.items[i];
    if (h.f0 == 0) a.contrib_out[h.v] = (a.personal < 0 ? a.r0_all : ((int64_t)h.v == a.personal ? 1.0f : 0.0f)) / (float)h.deg;
  }
  const uint64_t v0 = ((uint64_t)blockIdx.x + tile0) * TV;
  if (v0 >= g.n) return;
  const int cnt = (int)min((uint64_t)TV, g.n - v0);
  tile_offsets<OFF>(g, v0, cnt, xs, ts);
  __syncthreads();
  for (int i = threadIdx.x; i < cnt; i += TNT) {
    uint64_t start; uint32_t d, w;
    vgeo<IDM>(g, xs[i], xs[i + 1], start, d, w);
    const uint64_t v = v0 + i;
    const float r0 = a.personal < 0 ? a.r0_all : ((int64_t)v == a.personal ? 1.0f : 0.0f);
    a.contrib_out[v] = d ? r0 / (float)d : 0.0f;
    if (OFF == OFF_EF && v >= a.tile_a) {
      const bool small = v < a.tile_b;
      const uint64_t k = small ? v - a.tile_a : v - a.tile_b, nv = small ? a.tile_nv : PW_TV;
      if (k % nv == 0) a.aux[k / nv + (small ? 0 : (a.tile_b - a.tile_a) / a.tile_nv)] = (xs[i] >> g.ef_l) + v;
    }
  }
}

// ===========================================================================
// Personalized PageRank, PPR_K requests per sweep (serving engine).  Slot k
// iterates r_t[v] = (1-d_k)[v == s_k] + d_k * sum_{u in N_v} r_{t-1}[u] / d_u;
// tile CTAs and heavy items as described at the top, with PPR_K sums per
// vertex and one 32-byte gather per arc for all slots.
// ===========================================================================
__device__ __forceinline__ void ppr_finish(const PprArgs& a, uint64_t v, uint32_t d, const float (&sum)[PPR_K]) {
  float out[PPR_K];
#pragma unroll
  for (int k = 0; k < PPR_K; k++) {
    const bool act = (a.active >> k) & 1u;
    const float r = ((uint64_t)a.src[k] == v ? 1.0f - a.damp[k] : 0.0f) + a.damp[k] * sum[k];
    out[k] = (act && d) ? r / (float)d : 0.0f;
    if (act && ((a.last >> k) & 1u)) a.result[k][a.result_perm ? (uint64_t)a.result_perm[v] : v] = r;
  }
  float4* o = reinterpret_cast<float4*>(a.cout + v * PPR_K);
  __stcs(o, make_float4(out[0], out[1], out[2], out[3]));
  __stcs(o + 1, make_float4(out[4], out[5], out[6], out[7]));
}

// half h of the slots (4 of them) for vertex v, written by one lane of a pair
__device__ __forceinline__ void ppr_finish_half(const PprArgs& a, uint64_t v, uint32_t d, const float4& sum, int h) {
  const float sv[4] = {sum.x, sum.y, sum.z, sum.w};
  float out[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int k = h * 4 + q;
    const bool act = (a.active >> k) & 1u;
    const float r = ((uint64_t)a.src[k] == v ? 1.0f - a.damp[k] : 0.0f) + a.damp[k] * sv[q];
    out[q] = (act && d) ? r / (float)d : 0.0f;
    if (act && ((a.last >> k) & 1u)) a.result[k][a.result_perm ? (uint64_t)a.result_perm[v] : v] = r;
  }
  __stcs(reinterpret_cast<float4*>(a.cout + v * PPR_K + h * 4), make_float4(out[0], out[1], out[2], out[3]));
}

// one 16-byte half row of slot contributions; rows of the first `hot`
// vertices (the hubs, after DM relabeling) stay in L2, the rest stream through
__device__ __forceinline__ float4 gather_row(const float* ch, uint32_t u, uint32_t hot, uint64_t keep, uint64_t stream) {
  return ldg_gather4(ch + (uint64_t)u * PPR_K, u < hot ? keep : stream);
}

__device__ __forceinline__ void add4(float4& s, const float4& x) {
  s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
}

// range of compacted light vertices owned by lane pair `p` of `np` pairs
__device__ __forceinline__ void light_range_of(const TileSmem& sm, uint32_t p, uint32_t np, uint32_t& jb,
                                               uint32_t& je) {
  const uint64_t F = sm.nfields;
  const uint32_t flo = (uint32_t)((F * p) / np);
  const uint32_t fhi = (uint32_t)((F * (p + 1)) / np);
  const uint32_t nl = sm.nlight;
  uint32_t lo = 0, hi = nl;
  while (lo < hi) { const uint32_t m = (lo + hi) >> 1; if (sm.fpre[m] < flo) lo = m + 1; else hi = m; }
  jb = lo;
  hi = nl;
  while (lo < hi) { const uint32_t m = (lo + hi) >> 1; if (sm.fpre[m] < fhi) lo = m + 1; else hi = m; }
  je = lo;
}

// Light vertices are decoded by lane PAIRS: both lanes of a pair walk the
// same run of neighborhoods, lane h gathering the 16-byte half h of each
// neighbor's 32-byte slot row, so a pair's two loads of one arc coalesce into
// one sector and every thread keeps four arcs in flight.
template <int IDM, int OFF>
__global__ void __launch_bounds__(TNT, 4) k_ppr_pull(GView g, PprArgs a, TileMap tm) {
  __shared__ TileSmem sm;
  const float* __restrict__ c = a.cin;
  const int lane = threadIdx.x & 31;
  const uint64_t pstream = policy_stream(), pkeep = policy_keep();
  if (blockIdx.x < tm.hb) {
    // heavy item: lane pairs again -- the pair (2i, 2i+1) gathers both halves
    // of field i of each 16-field round; Kahan-compensated lane sums
    const uint32_t wid = threadIdx.x >> 5, step = tm.shared ? 64 * (TNT / 32) : 64;
    const uint64_t it = tm.shared ? blockIdx.x : (uint64_t)blockIdx.x * (TNT / 32) + wid;
    if (it >= g.n_items) return;
    const HeavyItem hv = g.items[it];
    const uint32_t f1 = hv.f0 + hv.nf;
    const int h = lane & 1;
    const float* ch = c + h * 4;
    uint32_t carry = hv.carry;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), comp = acc;
    for (uint32_t base = hv.f0 + (tm.shared ? 64 * wid : 0); base < f1; base += step) {
      uint32_t id[2];
      warp_ids<IDM, 2>(g, hv.bit, hv.w, base, f1, carry, id);
      float4 x[4];
#pragma unroll
      for (int u = 0; u < 2; u++) {
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const uint32_t from = (uint32_t)(r * 16 + (lane >> 1));
          const uint32_t fid = __shfl_sync(LG_FULL_MASK, id[u], from);
          x[u * 2 + r] = (base + 32u * u + from < f1) ? gather_row(ch, fid, a.hot, pkeep, pstream)
                                                      : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; q++) {
        float* ap = &acc.x;
        float* cp = &comp.x;
        const float* xp = &x[q].x;
#pragma unroll
        for (int e = 0; e < 4; e++) {
          const float y = xp[e] - cp[e];
          const float t = ap[e] + y;
          cp[e] = (t - ap[e]) - y;
          ap[e] = t;
        }
      }
    }
    // sum the 16 lanes of each parity (offsets 16, 8, 4, 2 keep the parity)
#pragma unroll
    for (int o = 16; o >= 2; o >>= 1) {
      acc.x += __shfl_xor_sync(LG_FULL_MASK, acc.x, o);
      acc.y += __shfl_xor_sync(LG_FULL_MASK, acc.y, o);
      acc.z += __shfl_xor_sync(LG_FULL_MASK, acc.z, o);
      acc.w += __shfl_xor_sync(LG_FULL_MASK, acc.w, o);
    }
    if (tm.shared) {  // the warps' sums in warp order
      __shared__ float4 wsum[TNT / 32][2];
      if (lane < 2) wsum[wid][h] = acc;
      __syncthreads();
      if (wid == 0 && lane < 2)
        for (int k = 1; k < TNT / 32; k++) add4(acc, wsum[k][h]);
    }
    if (lane < 2 && (!tm.shared || wid == 0)) {
      if (hv.nitems == 1) {
        ppr_finish_half(a, hv.v, hv.deg, acc, h);
      } else {
        float* pp = a.part + it * PPR_K + h * 4;
        pp[0] = acc.x; pp[1] = acc.y; pp[2] = acc.z; pp[3] = acc.w;
      }
    }
    return;
  }
  uint64_t v0;
  int cnt;
  tile_of(g, tm, v0, cnt);
  if (v0 + cnt <= g.heavy_prefix) return;  // all in the schedule
  tile_offsets<OFF>(g, v0, cnt, sm.xs, sm.ts);
  __syncthreads();
  tile_classify<IDM>(g, sm, cnt, [](int) { return true; });
  const float zero[PPR_K] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int i = threadIdx.x; i < cnt; i += TNT)
    if (sm.deg[i] == 0) ppr_finish(a, v0 + i, 0, zero);
  const int h = threadIdx.x & 1;
  const float* ch = c + h * 4;
  if (IDM == ID_LOCAL_GAP) {
    // gap-coded IDs cannot start mid-neighborhood: runs of whole vertices
    uint32_t jb, je;
    light_range_of(sm, threadIdx.x >> 1, TNT / 2, jb, je);
    for (uint32_t j = jb; j < je; j++) {
      const int i = sm.clist[j];
      const uint32_t d = sm.deg[i];
      SeqDec<IDM> dec;
      dec.init(g, sm.st[i], sm.wid[i], pstream);
      float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
      uint32_t k = 0;
      for (; k + 4 <= d; k += 4) {
        const uint32_t u0 = dec.next(), u1 = dec.next(), u2 = dec.next(), u3 = dec.next();
        const float4 x0 = ldg_gather4(ch + (uint64_t)u0 * PPR_K, u0 < a.hot ? pkeep : pstream);
        const float4 x1 = ldg_gather4(ch + (uint64_t)u1 * PPR_K, u1 < a.hot ? pkeep : pstream);
        const float4 x2 = ldg_gather4(ch + (uint64_t)u2 * PPR_K, u2 < a.hot ? pkeep : pstream);
        const float4 x3 = ldg_gather4(ch + (uint64_t)u3 * PPR_K, u3 < a.hot ? pkeep : pstream);
        add4(s0, x0); add4(s1, x1); add4(s0, x2); add4(s1, x3);
      }
      for (; k < d; k++) add4(s0, gather_row(ch, dec.next(), a.hot, pkeep, pstream));
      add4(s0, s1);
      ppr_finish_half(a, v0 + i, d, s0, h);
    }
    return;
  }
  // Fields-balanced light phase: pair w takes fields [F*w/NW, F*(w+1)/NW) of
  // the tile's compacted light fields, starting mid-neighborhood if need be.
  // A vertex's sum over the range that contains its first field goes to
  // vsum[j]; a pair that entered its first vertex mid-way leaves that partial
  // in carry[w].  A uniform phase then adds, per vertex, vsum and the carries
  // of the following pairs in pair order (deterministic) and finishes it.
  __shared__ float4 vsum[TV][2];
  __shared__ float4 carry[TNT / 2][2];
  constexpr uint32_t NW = TNT / 2;
  const uint32_t w = threadIdx.x >> 1;
  const uint32_t F = sm.nfields, nl = sm.nlight;
  const uint32_t flo = (uint32_t)((uint64_t)F * w / NW), fhi = (uint32_t)((uint64_t)F * (w + 1) / NW);
  carry[w][h] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (flo < fhi) {
    uint32_t lo = 0, hi = nl - 1;  // the vertex holding field flo: last j with fpre[j] <= flo
    while (lo < hi) {
      const uint32_t m = (lo + hi + 1) >> 1;
      if (sm.fpre[m] <= flo) lo = m; else hi = m - 1;
    }
    uint32_t j = lo, f = flo;
    bool head = sm.fpre[j] < flo;
    while (f < fhi) {
      const int i = sm.clist[j];
      const uint32_t vend = min(sm.fpre[j + 1], fhi);
      const uint32_t off = f - sm.fpre[j];
      const uint32_t fw = IDM == ID_GLOBAL ? g.r : (IDM == ID_CSR32 ? 32u : (uint32_t)sm.wid[i]);
      SeqDec<IDM> dec;
      dec.init(g, sm.st[i] + (uint64_t)off * fw, sm.wid[i], pstream);
      float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
      const uint32_t d = vend - f;
      uint32_t k = 0;
      for (; k + 4 <= d; k += 4) {  // four arcs in flight
        const uint32_t u0 = dec.next(), u1 = dec.next(), u2 = dec.next(), u3 = dec.next();
        const float4 x0 = ldg_gather4(ch + (uint64_t)u0 * PPR_K, u0 < a.hot ? pkeep : pstream);
        const float4 x1 = ldg_gather4(ch + (uint64_t)u1 * PPR_K, u1 < a.hot ? pkeep : pstream);
        const float4 x2 = ldg_gather4(ch + (uint64_t)u2 * PPR_K, u2 < a.hot ? pkeep : pstream);
        const float4 x3 = ldg_gather4(ch + (uint64_t)u3 * PPR_K, u3 < a.hot ? pkeep : pstream);
        add4(s0, x0); add4(s1, x1); add4(s0, x2); add4(s1, x3);
      }
      for (; k < d; k++) add4(s0, gather_row(ch, dec.next(), a.hot, pkeep, pstream));
      add4(s0, s1);
      if (head) carry[w][h] = s0;
      else vsum[j][h] = s0;
      head = false;
      f = vend;
      j++;
    }
  }
  __syncthreads();
  for (uint32_t t = threadIdx.x; t < nl * 2; t += TNT) {
    const uint32_t j = t >> 1;
    const int hh = (int)(t & 1);
    const uint32_t fs = sm.fpre[j], fe = sm.fpre[j + 1];
    float4 sum = vsum[j][hh];
    // pairs after the owner whose ranges start inside this vertex
    uint32_t q = (uint32_t)((uint64_t)fs * NW / (F ? F : 1));
    while (q + 1 < NW && (uint32_t)((uint64_t)F * (q + 1) / NW) <= fs) q++;
    while (q > 0 && (uint32_t)((uint64_t)F * q / NW) > fs) q--;
    for (q = q + 1; q < NW && (uint32_t)((uint64_t)F * q / NW) < fe; q++) add4(sum, carry[q][hh]);
    const int i = sm.clist[j];
    ppr_finish_half(a, v0 + i, sm.deg[i], sum, hh);
  }
}

// a slot joins: its column of `cin` is all zero (the slot was idle for a
// whole sweep, or the array is fresh); r_0 = e_src gives cin[src] = 1 / d_src
template <int IDM, int OFF>
__global__ void __launch_bounds__(32) k_ppr_join(GView g, float* cin, uint32_t slot, uint32_t src) {
  uint64_t start;
  uint32_t d, w;
  vertex_geo<IDM, OFF>(g, src, start, d, w);
  if (threadIdx.x == 0) cin[(uint64_t)src * PPR_K + slot] = d ? 1.0f / (float)d : 0.0f;
}

// ===========================================================================
// BFS (multi-source, bit-parallel): bit s of a mask is source s
// ===========================================================================
template <typename M>
__device__ __forceinline__ void bfs_finish(const GView& g, const BfsArgs& a, uint64_t v, M need, M found,
                                           uint32_t* qbuf, uint32_t* qn, uint32_t* pairs) {
  M* vis = reinterpret_cast<M*>(a.vis);
  M* fout = reinterpret_cast<M*>(a.front_out);
  const M nb = (M)(found & need);
  fout[v] = nb;
  if (nb) {
    vis[v] = (M)(vis[v] | nb);
    write_depths<M>(a, g.n, v, nb, a.level + 1);
    if (qbuf) {
      qbuf[atomicAdd(qn, 1u)] = (uint32_t)v;
      atomicAdd(pairs, (uint32_t)__popcll((unsigned long long)nb));
    } else {
      a.queue_out[atomicAdd(&a.counters[0], 1u)] = (uint32_t)v;
      atomicAdd(&a.counters[1], (uint32_t)__popcll((unsigned long long)nb));
    }
  }
}

template <int IDM, int OFF, typename M>
__global__ void __launch_bounds__(TNT, IDM == ID_LOCAL_GAP ? 6 : 5) k_bfs_pull(GView g, BfsArgs a, TileMap tm) {
  __shared__ TileSmem sm;
  __shared__ M need_sm[TV];
  __shared__ uint32_t qbuf[TV];
  __shared__ uint32_t qn, newpairs, qbase;
  const M* vis = reinterpret_cast<const M*>(a.vis);
  const M* __restrict__ fin = reinterpret_cast<const M*>(a.front_in);
  M* fout = reinterpret_cast<M*>(a.front_out);
  const M all = (M)a.all_mask;
  const int lane = threadIdx.x & 31;
  const uint64_t pstream = policy_stream(), pkeep = policy_keep();
  if (blockIdx.x < tm.hb) {
    const uint32_t wid = threadIdx.x >> 5, step = tm.shared ? 32 * HEAVY_U * (TNT / 32) : 32 * HEAVY_U;
    const uint64_t it = tm.shared ? blockIdx.x : (uint64_t)blockIdx.x * (TNT / 32) + wid;
    if (it >= g.n_items) return;
    const HeavyItem h = g.items[it];
    const M need = (M)(all & (M)~vis[h.v]);
    if (need == 0) {
      if (h.f0 == 0 && lane == 0 && (!tm.shared || wid == 0)) fout[h.v] = 0;
      return;
    }
    const uint32_t f1 = h.f0 + h.nf;
    uint32_t carry = h.carry;
    M acc = 0;
    for (uint32_t base = h.f0 + (tm.shared ? 32 * HEAVY_U * wid : 0); base < f1; base += step) {
      uint32_t id[HEAVY_U];
      warp_ids<IDM, HEAVY_U>(g, h.bit, h.w, base, f1, carry, id);
      M x[HEAVY_U];
#pragma unroll
      for (int u = 0; u < HEAVY_U; u++) x[u] = (base + 32u * u + lane < f1) ? ldg_gather(fin + id[u], id[u] < a.hot ? pkeep : pstream) : (M)0;
#pragma unroll
      for (int u = 0; u < HEAVY_U; u++) acc |= x[u];
      acc = warp_or<M>(acc);
      if ((M)(acc & need) == need) break;
    }
    if (tm.shared) {
      __shared__ M wacc[TNT / 32];
      if (lane == 0) wacc[wid] = acc;
      __syncthreads();
      if (threadIdx.x == 0)
        for (int k = 1; k < TNT / 32; k++) acc |= wacc[k];
    }
    if (lane == 0 && (!tm.shared || wid == 0)) {
      bool last = true;
      if (h.nitems > 1) {  // the item that arrives last finishes the vertex
        M* p = reinterpret_cast<M*>(a.hacc) + h.slot;
        atomic_or_mask<M>(p, acc);
        __threadfence();
        last = atomicInc(a.hcnt + h.slot, h.nitems - 1) == h.nitems - 1;  // wraps to 0 for the next level
        if (last) {
          __threadfence();
          acc = atomic_take_mask<M>(p);
        }
      }
      if (last) bfs_finish<M>(g, a, h.v, need, acc, nullptr, nullptr, nullptr);
    }
    return;
  }
  if (threadIdx.x == 0) { qn = 0; newpairs = 0; }
  uint64_t v0;
  int cnt;
  tile_of(g, tm, v0, cnt);
  if (v0 + cnt <= g.heavy_prefix) return;  // all in the schedule
  for (int i = threadIdx.x; i < cnt; i += TNT) need_sm[i] = (M)(all & (M)~vis[v0 + i]);
  tile_offsets<OFF>(g, v0, cnt, sm.xs, sm.ts);
  __syncthreads();
  tile_classify<IDM>(g, sm, cnt, [&](int i) { return need_sm[i] != 0; });

  for (int i = threadIdx.x; i < cnt; i += TNT)
    if (sm.deg[i] == 0 || (sm.deg[i] <= g.heavy_min && need_sm[i] == 0)) fout[v0 + i] = 0;

  if (IDM == ID_LOCAL_GAP) {
    // gap-coded IDs: runs of whole vertices (no mid-neighborhood start)
    uint32_t jb, je;
    light_range(sm, jb, je);
    for (uint32_t j = jb; j < je; j++) {
      const int i = sm.clist[j];
      const uint32_t d = sm.deg[i];
      const M need = need_sm[i];
      SeqDec<IDM> dec;
      dec.init(g, sm.st[i], sm.wid[i], pstream);
      M acc = 0;
      uint32_t k = 0;
      for (; k + 4 <= d; k += 4) {  // early exit once every unvisited source is found
        const uint32_t u0 = dec.next(), u1 = dec.next(), u2 = dec.next(), u3 = dec.next();
        acc |= (M)(ldg_gather(fin + u0, u0 < a.hot ? pkeep : pstream) | ldg_gather(fin + u1, u1 < a.hot ? pkeep : pstream) | ldg_gather(fin + u2, u2 < a.hot ? pkeep : pstream) |
                   ldg_gather(fin + u3, u3 < a.hot ? pkeep : pstream));
        if ((M)(acc & need) == need) break;
      }
      if ((M)(acc & need) != need)
        for (; k < d; k++) {
          const uint32_t u = dec.next();
          acc |= ldg_gather(fin + u, u < a.hot ? pkeep : pstream);
        }
      bfs_finish<M>(g, a, v0 + i, need, acc, qbuf, &qn, &newpairs);
    }
  } else {
    // fields-balanced (as in k_ppr_pull): partial ORs of a vertex split over
    // threads are combined exactly in a uniform phase
    __shared__ M vor[TV];
    __shared__ M carry[TNT];
    const uint32_t F = sm.nfields, nl = sm.nlight;
    const uint32_t flo = (uint32_t)((uint64_t)F * threadIdx.x / TNT);
    const uint32_t fhi = (uint32_t)((uint64_t)F * (threadIdx.x + 1) / TNT);
    carry[threadIdx.x] = 0;
    if (flo < fhi) {
      uint32_t lo = 0, hi = nl - 1;
      while (lo < hi) {
        const uint32_t m = (lo + hi + 1) >> 1;
        if (sm.fpre[m] <= flo) lo = m; else hi = m - 1;
      }
      uint32_t j = lo, f = flo;
      M* ps = sm.fpre[j] < flo ? &carry[threadIdx.x] : &vor[j];
      while (f < fhi) {
        const int i = sm.clist[j];
        const M need = need_sm[i];
        const uint32_t vend = min(sm.fpre[j + 1], fhi);
        const uint32_t fw = IDM == ID_GLOBAL ? g.r : (IDM == ID_CSR32 ? 32u : (uint32_t)sm.wid[i]);
        SeqDec<IDM> dec;
        dec.init(g, sm.st[i] + (uint64_t)(f - sm.fpre[j]) * fw, sm.wid[i], pstream);
        const uint32_t d = vend - f;
        M acc = 0;
        uint32_t k = 0;
        for (; k + 4 <= d; k += 4) {
          const uint32_t u0 = dec.next(), u1 = dec.next(), u2 = dec.next(), u3 = dec.next();
          acc |= (M)(ldg_gather(fin + u0, u0 < a.hot ? pkeep : pstream) | ldg_gather(fin + u1, u1 < a.hot ? pkeep : pstream) | ldg_gather(fin + u2, u2 < a.hot ? pkeep : pstream) |
                     ldg_gather(fin + u3, u3 < a.hot ? pkeep : pstream));
          if ((M)(acc & need) == need) break;
        }
        if ((M)(acc & need) != need)
          for (; k < d; k++) {
          const uint32_t u = dec.next();
          acc |= ldg_gather(fin + u, u < a.hot ? pkeep : pstream);
        }
        *ps = acc;
        f = vend;
        j++;
        ps = &vor[j];
      }
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < nl; j += TNT) {
      const uint32_t fs = sm.fpre[j], fe = sm.fpre[j + 1];
      M acc = vor[j];
      uint32_t q = (uint32_t)((uint64_t)fs * TNT / (F ? F : 1));
      while (q + 1 < TNT && (uint32_t)((uint64_t)F * (q + 1) / TNT) <= fs) q++;
      while (q > 0 && (uint32_t)((uint64_t)F * q / TNT) > fs) q--;
      for (q = q + 1; q < TNT && (uint32_t)((uint64_t)F * q / TNT) < fe; q++) acc |= carry[q];
      const int i = sm.clist[j];
      bfs_finish<M>(g, a, v0 + i, need_sm[i], acc, qbuf, &qn, &newpairs);
    }
  }

  __syncthreads();
  if (threadIdx.x == 0 && qn) {
    qbase = atomicAdd(&a.counters[0], qn);
    atomicAdd(&a.counters[1], newpairs);
  }
  __syncthreads();
  for (uint32_t t = threadIdx.x; t < qn; t += TNT) a.queue_out[qbase + t] = qbuf[t];
}

// top-down step over fields [f0, f1) of a frontier vertex with source mask m:
// every neighbor not yet visited by some of m's sources joins the next
// frontier for them (a warp, 32 * HEAVY_U fields per step)
template <int IDM, typename M>
__device__ __forceinline__ void push_fields(const GView& g, const BfsArgs& a, M m, uint64_t start, uint32_t w,
                                            uint32_t f0, uint32_t f1, uint32_t carry, uint32_t& pairs) {
  M* vis = reinterpret_cast<M*>(a.vis);
  M* fout = reinterpret_cast<M*>(a.front_out);
  const int lane = threadIdx.x & 31;
  const uint32_t nd = a.level + 1;
  for (uint32_t base = f0; base < f1; base += 32 * HEAVY_U) {
    uint32_t id[HEAVY_U];
    warp_ids<IDM, HEAVY_U>(g, start, w, base, f1, carry, id);
    M cur[HEAVY_U];
#pragma unroll
    for (int u = 0; u < HEAVY_U; u++) cur[u] = (base + 32u * u + lane < f1) ? vis[id[u]] : (M)~(M)0;
#pragma unroll
    for (int u = 0; u < HEAVY_U; u++) {
      const uint32_t u_id = id[u];
      bool app = false;
      M nb = (M)(m & (M)~cur[u]);
      if (nb) {
        const M old = atomic_or_mask<M>(vis + u_id, nb);
        nb = (M)(nb & (M)~old);
        if (nb) {
          const M oldf = atomic_or_mask<M>(fout + u_id, nb);
          app = (oldf == 0);
          write_depths<M>(a, g.n, u_id, nb, nd);
          pairs += __popcll((unsigned long long)nb);
        }
      }
      const uint32_t bal = __ballot_sync(LG_FULL_MASK, app);
      if (bal) {
        uint32_t basepos = 0;
        if (lane == 0) basepos = atomicAdd(&a.counters[0], (uint32_t)__popc(bal));
        basepos = __shfl_sync(LG_FULL_MASK, basepos, 0);
        if (app) a.queue_out[basepos + __popc(bal & lane_lt_mask())] = u_id;
      }
    }
  }
}

// Top-down step.  Blocks [0, hb) take the heavy-vertex schedule, a warp per
// item (or a block per item, when items are few), working when the item's
// vertex is in the frontier (a hub's arcs are spread over as many warps as it
// has items); the other blocks take the frontier queue, a warp per vertex of
// degree <= heavy_min.
template <int IDM, int OFF, typename M>
__global__ void __launch_bounds__(256) k_bfs_push(GView g, BfsArgs a, unsigned hb, uint32_t shared) {
  const M* __restrict__ fin = reinterpret_cast<const M*>(a.front_in);
  const int lane = threadIdx.x & 31;
  uint32_t pairs = 0;
  if (blockIdx.x < hb) {
    const uint32_t wid = threadIdx.x >> 5;
    const uint64_t it = shared ? blockIdx.x : (uint64_t)blockIdx.x * (blockDim.x >> 5) + wid;
    if (it < g.n_items) {
      const HeavyItem h = g.items[it];
      const M m = fin[h.v];
      uint32_t f0 = h.f0, f1 = h.f0 + h.nf;
      if (shared) {  // this warp's eighth
        const uint32_t part = (h.nf + 7) / 8;
        f0 = min(f1, f0 + wid * part);
        f1 = min(f1, f0 + part);
      }
      if (m) push_fields<IDM, M>(g, a, m, h.bit, h.w, f0, f1, h.carry, pairs);
    }
  } else {
    const uint64_t warps = (uint64_t)(gridDim.x - hb) * (blockDim.x >> 5);
    for (uint64_t q = (uint64_t)(blockIdx.x - hb) * (blockDim.x >> 5) + (threadIdx.x >> 5); q < a.queue_in_len;
         q += warps) {
      const uint32_t v = a.queue_in[q];
      if (v < g.heavy_prefix) continue;  // in the heavy schedule
      const M m = fin[v];
      uint64_t x0, x1, start;
      uint32_t d, w;
      offset_pair<OFF>(g, v, x0, x1);
      vgeo<IDM>(g, x0, x1, start, d, w);
      if (d > g.heavy_min && g.n_items) continue;  // in the heavy schedule
      push_fields<IDM, M>(g, a, m, start, w, 0, d, 0, pairs);
    }
  }
  pairs = warp_sum<uint32_t>(pairs);
  if (lane == 0 && pairs) atomicAdd(&a.counters[1], pairs);
}

// ===========================================================================
// neighbor queries (getNeighbors of Listing 3)
// ===========================================================================
// Degrees, a warp per query, and the largest.  With a.scan the block that
// finishes last turns them into offsets (a scan of its own took three launches).
template <int IDM, int OFF>
__global__ void __launch_bounds__(256) k_nbr_degrees(GView g, NbrArgs a) {
  const int lane = threadIdx.x & 31;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  uint32_t most = 0;
  for (uint64_t q = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < a.k; q += warps) {
    const uint32_t vo = a.vertices[q];
    if (vo >= g.n) {
      if (lane == 0) { set_err(&a.stat->err, DERR_QUERY); a.out_offsets[q] = 0; }
      continue;
    }
    const uint64_t v = g.perm ? (uint64_t)g.perm[vo] : vo;
    uint64_t start;
    uint32_t d, w;
    vertex_geo<IDM, OFF>(g, v, start, d, w);
    most = max(most, d);
    if (lane == 0) a.out_offsets[q] = d;
  }
  if (lane == 0 && most) atomicMax(&a.stat->max_degree, most);
  if (!a.scan) return;
  __shared__ uint64_t tmp[8];
  __shared__ uint32_t last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&a.stat->arrived, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  uint64_t carry = 0;
  for (uint64_t base = 0; base < a.k; base += 256 * 4) {
    uint64_t x[4], sum = 0, total;
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const uint64_t i = base + 4 * threadIdx.x + e;
      x[e] = i < a.k ? __ldcg(a.out_offsets + i) : 0;
      sum += x[e];
    }
    uint64_t pre = block_excl_scan<uint64_t, 256>(sum, total, tmp) + carry;
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const uint64_t i = base + 4 * threadIdx.x + e;
      if (i < a.k) a.out_offsets[i] = pre;
      pre += x[e];
    }
    carry += total;
  }
  if (threadIdx.x == 0) {
    a.out_offsets[a.k] = carry;
    a.stat->total = carry;
  }
}

// One row of a query, written as original IDs.  Field idx of the row has ID id.
template <int IDM>
__device__ __forceinline__ uint32_t nbr_weight(const GView& g, uint64_t start, uint32_t idx) {
  if (IDM == ID_GLOBAL && g.omega) return weight_at(g, start, idx);
  if (IDM == ID_CSR32 && g.W32) return __ldg(g.W32 + (start >> 5) + idx);
  return 0u;
}

// Ascending order of a warp's 32 R keys, key R lane + r in x[r], by a bitonic
// network: compare-exchanges inside a lane's registers and by shuffles.  VALS:
// y moves along.
template <bool VALS>
__device__ __forceinline__ void exchange(uint32_t& a, uint32_t& b, uint32_t& va, uint32_t& vb, bool up) {
  if (VALS) {
    const bool swap = up ? a > b : a < b;
    const uint32_t ta = swap ? b : a, tb = swap ? a : b, sa = swap ? vb : va, sb = swap ? va : vb;
    a = ta; b = tb; va = sa; vb = sb;
  } else {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = up ? lo : hi;
    b = up ? hi : lo;
  }
}
template <int R, bool VALS>
__device__ __forceinline__ void warp_sort(uint32_t (&x)[R], uint32_t (&y)[R]) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int k = 2; k <= R; k *= 2) {
#pragma unroll
    for (int j = k / 2; j > 0; j /= 2) {
#pragma unroll
      for (int r = 0; r < R; r++)
        if ((r & j) == 0) exchange<VALS>(x[r], x[r | j], y[r], y[r | j], k < R ? (r & k) == 0 : (lane & 1u) == 0);
    }
  }
#pragma unroll 1
  for (uint32_t k = 2; k <= 32; k *= 2) {  // runs of k lanes
    const bool up = (lane & k) == 0;
#pragma unroll 1
    for (uint32_t m = k / 2; m > 0; m /= 2) {
      const bool low = ((lane & m) == 0) == up;
#pragma unroll
      for (int r = 0; r < R; r++) {
        const uint32_t o = __shfl_xor_sync(LG_FULL_MASK, x[r], m);
        if (VALS) {
          const uint32_t ov = __shfl_xor_sync(LG_FULL_MASK, y[r], m);
          const bool take = low ? o < x[r] : o > x[r];
          x[r] = take ? o : x[r];
          y[r] = take ? ov : y[r];
        } else {
          x[r] = low ? min(x[r], o) : max(x[r], o);
        }
      }
    }
#pragma unroll
    for (int j = R / 2; j > 0; j /= 2) {
#pragma unroll
      for (int r = 0; r < R; r++)
        if ((r & j) == 0) exchange<VALS>(x[r], x[r | j], y[r], y[r | j], up);
    }
  }
}

// Rows, decoded and (a.sort: on relabeled graphs) put in ascending order.  A
// CTA takes a.per queries, 8 or, where rows are long, fewer (launch_nbr_rows): a
// warp decodes a row of up to 256 neighbors into registers and sorts it there
// (1, 2, 4 or 8 keys a lane); the CTA then takes its longer rows together,
// sorting up to NBR_SORT of them with a bitonic network in shared memory.
// Longer rows are left unsorted (the caller sorts them).  A hub's row does not
// rest on one warp, and a batch needs one launch where the decode and the
// size-class sort took eight and a wait.  All rows of 400,000 vertices of degree
// 160: 1.34 ms with those, 2.25 with each ID ranked among its row's, 1.34 so.
constexpr uint32_t NBR_WARP = 256;  // neighbors of a row that a warp takes

// a row of up to 32 R neighbors, id[u] that of field 32 u + lane, to out
template <int IDM, int R>
__device__ __forceinline__ void nbr_row(const GView& g, const NbrArgs& a, const uint32_t (&id)[NBR_WARP / 32],
                                        uint64_t start, uint32_t d, uint64_t o, uint32_t* mine) {
  const uint32_t lane = threadIdx.x & 31u;
  // with weights the field moves along: in the key's low 8 bits if the IDs leave them
  const bool packed = a.sort && a.out_weights && g.n <= 1ull << 24, beside = a.sort && a.out_weights && !packed;
  uint32_t x[R], y[R];
#pragma unroll
  for (int r = 0; r < R; r++) {
    y[r] = 32u * r + lane;
    x[r] = y[r] < d ? (packed ? id[r] << 8 | y[r] : id[r]) : 0xffffffffu;
  }
  if (a.sort) {
    if (beside) warp_sort<R, true>(x, y);
    else warp_sort<R, false>(x, y);
    // sorted by lane; out in order
#pragma unroll
    for (int r = 0; r < R; r++) mine[R * lane + r] = x[r];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; r++) x[r] = mine[32 * r + lane];
    if (packed) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        y[r] = x[r] & 255u;
        x[r] >>= 8;
      }
    }
    if (beside) {
      __syncwarp();
#pragma unroll
      for (int r = 0; r < R; r++) mine[R * lane + r] = y[r];
      __syncwarp();
#pragma unroll
      for (int r = 0; r < R; r++) y[r] = mine[32 * r + lane];
    }
  }
#pragma unroll
  for (int r = 0; r < R; r++) {
    if (32u * r + lane < d) {
      a.out_ids[o + 32u * r + lane] = x[r];
      if (a.out_weights) a.out_weights[o + 32u * r + lane] = nbr_weight<IDM>(g, start, y[r]);
    }
  }
}

template <int IDM, int OFF>
__global__ void __launch_bounds__(256) k_nbr_rows(GView g, NbrArgs a) {
  __shared__ __align__(16) uint32_t sk[NBR_SORT];
  __shared__ uint32_t sv[NBR_SORT];
  __shared__ uint32_t big[8], nbig;
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) nbig = 0;
  __syncthreads();
  const uint64_t q0 = (uint64_t)blockIdx.x * a.per;
  if (wid < a.per && q0 + wid < a.k) {
    const uint32_t vo = a.vertices[q0 + wid];
    uint64_t start;
    uint32_t d, w, carry = 0;
    vertex_geo<IDM, OFF>(g, g.perm ? (uint64_t)g.perm[vo] : vo, start, d, w);
    if (d > NBR_WARP) {
      if (lane == 0) big[atomicAdd(&nbig, 1u)] = wid;
    } else if (d) {
      constexpr int U = NBR_WARP / 32;
      const uint64_t o = a.out_offsets[q0 + wid];
      uint32_t id[U];
      if (d <= 32) {
        uint32_t one[1];
        warp_ids<IDM, 1>(g, start, w, 0, d, carry, one);
        id[0] = one[0];
      } else {
        warp_ids<IDM, U>(g, start, w, 0, d, carry, id);
      }
      if (g.inv_perm) {
#pragma unroll
        for (int u = 0; u < U; u++)
          if (32u * u + lane < d) id[u] = g.inv_perm[id[u]];
      }
      uint32_t* mine = sk + wid * NBR_WARP;
      if (d <= 32) nbr_row<IDM, 1>(g, a, id, start, d, o, mine);
      else if (d <= 64) nbr_row<IDM, 2>(g, a, id, start, d, o, mine);
      else if (d <= 128) nbr_row<IDM, 4>(g, a, id, start, d, o, mine);
      else nbr_row<IDM, 8>(g, a, id, start, d, o, mine);
    }
  }
  __syncthreads();
  for (uint32_t b = 0; b < nbig; b++) {
    const uint64_t q = q0 + big[b], o = a.out_offsets[q];
    const uint32_t vo = a.vertices[q];
    const uint64_t v = g.perm ? (uint64_t)g.perm[vo] : vo;
    uint64_t start;
    uint32_t d, w;
    vertex_geo<IDM, OFF>(g, v, start, d, w);
    const bool inside = a.sort && d <= NBR_SORT;
    auto put = [&](uint32_t idx, uint32_t id) {
      if (g.inv_perm) id = g.inv_perm[id];
      const uint32_t wt = a.out_weights ? nbr_weight<IDM>(g, start, idx) : 0u;
      if (inside) {
        sk[idx] = id;
        sv[idx] = wt;
      } else {
        a.out_ids[o + idx] = id;
        if (a.out_weights) a.out_weights[o + idx] = wt;
      }
    };
    // gap-coded rows by their schedule items (which hold the ID before them), or
    // whole if they are in none; the others in steps of all warps
    const bool items = IDM == ID_LOCAL_GAP && d > g.heavy_min;
    const uint64_t i0 = items ? first_item(g, v) : 0;
    const uint32_t parts = IDM == ID_LOCAL_GAP ? (items ? g.items[i0].nitems : 1u) : 8u;
    for (uint32_t k = wid; k < parts; k += 8) {
      uint32_t f0 = 0, f1 = d, step = 128, carry = 0;
      if (IDM != ID_LOCAL_GAP) {
        f0 = 128 * k;
        step = 128 * 8;
      } else if (items) {
        const HeavyItem h = g.items[i0 + k];
        f0 = h.f0;
        f1 = h.f0 + h.nf;
        carry = h.carry;
      }
      for (uint32_t base = f0; base < f1; base += step) {
        uint32_t id[4];
        warp_ids<IDM, 4>(g, start, w, base, f1, carry, id);
#pragma unroll
        for (int u = 0; u < 4; u++)
          if (base + 32u * u + lane < f1) put(base + 32u * u + lane, id[u]);
      }
    }
    if (inside) {
      uint32_t P = 512;
      while (P < d) P <<= 1;
      for (uint32_t i = d + threadIdx.x; i < P; i += 256) sk[i] = 0xffffffffu;
      __syncthreads();
      for (uint32_t k = 2; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j; j >>= 1) {
          for (uint32_t t = threadIdx.x; t < P / 2; t += 256) {
            const uint32_t x = 2 * t - (t & (j - 1)), y = x + j;
            const uint32_t kx = sk[x], ky = sk[y];
            if ((kx > ky) == ((x & k) == 0)) {
              sk[x] = ky;
              sk[y] = kx;
              if (a.out_weights) {
                const uint32_t z = sv[x];
                sv[x] = sv[y];
                sv[y] = z;
              }
            }
          }
          __syncthreads();
        }
      }
      for (uint32_t i = threadIdx.x; i < d; i += 256) {
        a.out_ids[o + i] = sk[i];
        if (a.out_weights) a.out_weights[o + i] = sv[i];
      }
    }
    __syncthreads();
  }
}

// ===========================================================================
// Whole-graph decode (lg_decode): every neighborhood (Section 3.7.2's access
// applied to all vertices) written to a CSR in stored order.
//
// Global IDs (and CSR-32) keep their records in arc order, so record j is
// col[j] and the offsets x_v are the row offsets: one launch writes row_ptr
// from the offsets (a tile decode per 512 vertices) and maps records to IDs,
// consecutive threads on consecutive records (coalesced stream reads and
// coalesced writes, no vertex lookup).  Local IDs: one
// kernel, described above k_dec_local.
// ===========================================================================
template <int IDM, int U>
__device__ __forceinline__ void dec_fields(const GView& g, const DecArgs& a, uint64_t start, uint32_t w, uint32_t f0,
                                           uint32_t f1, uint32_t carry, uint64_t o) {
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t base = f0; base < f1; base += 32u * U) {
    uint32_t id[U];
    warp_ids<IDM, U>(g, start, w, base, f1, carry, id);
#pragma unroll
    for (int u = 0; u < U; u++) {
      const uint32_t idx = base + 32u * u + lane;
      if (idx < f1) __stcs(a.ids + o + idx, id[u]);
    }
  }
}

constexpr uint32_t DEC_FLAT_CH = 512;                      // records per warp chunk (flat decode)
constexpr uint32_t DEC_FLAT_WORDS = DEC_FLAT_CH * 64 / 32 + 4;  // stream words of a chunk of <= 64-bit records

// Flat decode of global-ID records (or CSR-32 IDs), one launch, one block per
// tile of TV vertices: the block writes the tile's row_ptr entries from the
// offsets, then decodes its share of the records (arcs / tiles, rounded up to
// whole chunks) chunk by chunk, a warp per chunk of DEC_FLAT_CH records: the
// chunk's stream words come into shared memory with 16-byte loads (a chunk
// starts on a 16-byte boundary: DEC_FLAT_CH * r bits is a multiple of 128),
// then lane l extracts records l, l + 32, ... with a funnel shift and writes
// them coalesced.
template <int IDM, int OFF>
__global__ void __launch_bounds__(256) k_dec_flat(GView g, DecArgs a, uint64_t per_block) {
  __shared__ __align__(16) uint32_t fw[TNT / 32][DEC_FLAT_WORDS];
  {
    __shared__ uint64_t xs[TV + 1];
    __shared__ TileScratch ts;
    const uint64_t v0 = (uint64_t)blockIdx.x * TV;
    const int cnt = (int)min((uint64_t)TV, g.n - v0);
    tile_offsets<OFF>(g, v0, cnt, xs, ts);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += TNT) a.row_out[v0 + i] = xs[i];
    if (v0 + (uint64_t)cnt == g.n && threadIdx.x == 0) a.row_out[g.n] = xs[cnt];
  }
  const uint64_t arcs = g.arcs;
  const uint64_t jb = (uint64_t)blockIdx.x * per_block, je = min(arcs, jb + per_block);
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const bool want_w = a.weights != nullptr;
  if constexpr (IDM == ID_CSR32) {
    for (uint64_t j = jb + threadIdx.x; j < je; j += TNT) {
      __stcs(a.ids + j, __ldcs(g.A32 + j));
      if (want_w) __stcs(a.weights + j, g.W32 ? __ldcs(g.W32 + j) : 0u);
    }
  } else {
    const uint32_t r = g.r, s = g.s;
    const uint32_t ms = mask_lo(s), mw = mask_lo(g.omega);
    uint32_t* sw = fw[wid];
    for (uint64_t c = jb + (uint64_t)wid * DEC_FLAT_CH; c < je; c += (uint64_t)(TNT / 32) * DEC_FLAT_CH) {
      const uint32_t nrec = (uint32_t)min((uint64_t)DEC_FLAT_CH, je - c);
      const uint64_t w0 = c * r / 32;  // a multiple of 4: c is a multiple of DEC_FLAT_CH
      const uint32_t nw = (nrec * r + 31) / 32 + 1;  // the chunk's words and the one after
      const uint4* src = reinterpret_cast<const uint4*>(g.A32 + w0);
      for (uint32_t q = lane; q * 4 < nw; q += 32) reinterpret_cast<uint4*>(sw)[q] = __ldcs(src + q);
      __syncwarp();
      for (uint32_t t = lane; t < nrec; t += 32) {
        const uint32_t p = t * r;
        const uint32_t x0 = sw[p >> 5], x1 = sw[(p >> 5) + 1];
        __stcs(a.ids + c + t, __funnelshift_r(x0, x1, p & 31u) & ms);
        if (want_w) {
          uint32_t wt = 0;
          if (g.omega) {
            const uint32_t q = p + s;
            wt = __funnelshift_r(sw[q >> 5], sw[(q >> 5) + 1], q & 31u) & mw;
          }
          __stcs(a.weights + c + t, wt);
        }
      }
      __syncwarp();
    }
  }
}

// ---------------------------------------------------------------------------
// Local-ID decode: one launch writes row_ptr and every row (a graph that is mostly
// heavy has its heavy items in a second one, see k_dec_heavy).
//
// Blocks take a ticket when they start: tickets below the tile count are tile
// CTAs (tiles in start order), the rest are heavy-schedule CTAs, a warp per
// item.  A tile CTA decodes its offsets together; then each warp has its own
// vertices (see dec_tiles) as in the pull sweep: geometry, and the arcs counted.  The
// CTA publishes its arc count, finds the arcs of all earlier tiles by a
// decoupled look-back over their published counts (a tile waits only on tiles
// that started before it) while its warps' first windows are on their way, and
// writes its row offsets, flagged ready for the heavy items.  The warps then
// decode window by window -- 256 fields, 8 consecutive ones per lane, the next
// window's words in flight -- and write a window's IDs coalesced by way of
// shared memory.
//
// What bounds it is instructions and the blocks' start: 2.6 warp instructions
// a field, 3.3 with a serial reader per lane and vertex.  4 M vertices, 94 M arcs in
// local-gap IDs: 438 us before, 307 now, of which the offsets, the geometry and
// the look-back take half (18 us a block, overlapped by the SM's other three).
// ---------------------------------------------------------------------------
constexpr uint64_t DEC_AGG = 1ull << 62, DEC_INCL = 2ull << 62, DEC_VAL = (1ull << 62) - 1;
static_assert(DEC_WARPS == TNT / 32, "a warp tile per warp");

struct DecSmem {
  PrWarp w[DEC_WARPS];
  uint32_t hdeg[DEC_WARPS][PW_TV];  // degrees of the warp tile's heavy vertices
  union {
    uint64_t xs[DEC_WARPS * PW_TV + 1];               // the tile's offsets, until the geometry is known
    __align__(16) uint32_t out[DEC_WARPS][PW_WF];     // a window's IDs
  };
  TileScratch ts;
  uint64_t sums[DEC_WARPS];  // arcs of each warp tile, then of those before it
  uint64_t base;             // arcs of all earlier tiles
  uint32_t ticket, ok;
};

// flag and count of a tile are one word: nothing else is read on its account
__device__ __forceinline__ uint64_t ld_relaxed_u64(const unsigned long long* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u64(unsigned long long* p, uint64_t v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t dec_clock_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Arcs of all tiles before tile b (warp 0 of the tile CTA; the result in lane 0).
// Returns false if a wait ran out.
__device__ __forceinline__ bool dec_lookback(const DecArgs& a, uint64_t b, uint64_t& base) {
  const uint32_t lane = threadIdx.x & 31u;
  base = 0;
  int64_t p = (int64_t)b - 1 - (int64_t)lane;  // lane 0 reads the nearest predecessor
  const uint64_t t0 = dec_clock_ns();
  uint64_t spins = 0;
  while (true) {
    const uint64_t v = p >= 0 ? ld_relaxed_u64(a.tile_status + p) : DEC_INCL;  // nothing before tile 0
    const uint64_t flag = v >> 62;
    const uint32_t incl = __ballot_sync(LG_FULL_MASK, flag == 2);
    const uint32_t stop = incl ? (uint32_t)(__ffs(incl) - 1) : 31u;  // nearest inclusive prefix
    const uint32_t unready = __ballot_sync(LG_FULL_MASK, flag == 0 && lane <= stop);
    if (unready) {
      if (++spins > (a.wait_ns >> 5) + 1024 || ((spins & 63u) == 0 && dec_clock_ns() - t0 > a.wait_ns)) return false;
      __nanosleep(32);
      continue;
    }
    base += warp_sum<uint64_t>(lane <= stop ? (v & DEC_VAL) : 0ull);
    if (incl) return true;
    p -= 32;
  }
}

template <int IDM, int OFF, bool RUNS>
__global__ void __launch_bounds__(TNT, 4) k_dec_local(GView g, DecArgs a) {
  DecSmem& sm = *reinterpret_cast<DecSmem*>(dyn_smem);
  const uint64_t ntiles = a.tiles, va = a.tiles_a * dec_tile(a.nv_a);  // from vertex va on tiles of a.nv per warp
  if (threadIdx.x == 0) sm.ticket = atomicAdd(a.ticket, 1u);
  __syncthreads();
  const uint64_t b = sm.ticket;
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (b >= ntiles) {
    // heavy items, a warp each; the row start comes from the tile that owns the vertex
    const uint64_t it = (b - ntiles) * (TNT / 32) + wid;
    if (it >= g.n_items) return;
    const HeavyItem h = g.items[it];
    uint64_t o = 0;
    bool ok = true;
    if (lane == 0) {
      const uint32_t* ready =
          a.tile_ready + (h.v < va ? h.v / dec_tile(a.nv_a) : a.tiles_a + (h.v - va) / dec_tile(a.nv));
      const uint64_t t0 = dec_clock_ns();
      uint64_t spins = 0;
      while (ld_acquire_u32(ready) == 0) {
        if (++spins > (a.wait_ns >> 5) + 1024 || ((spins & 63u) == 0 && dec_clock_ns() - t0 > a.wait_ns)) {
          ok = false;
          break;
        }
        __nanosleep(64);
      }
      if (ok) o = __ldcg(a.row_ptr + h.v);
      else atomicOr(a.err, DERR_INTERNAL);
    }
    if (!__shfl_sync(LG_FULL_MASK, ok ? 1u : 0u, 0)) return;
    o = __shfl_sync(LG_FULL_MASK, o, 0);
    dec_fields<IDM, HEAVY_U>(g, a, h.bit, h.w, h.f0, h.f0 + h.nf, h.carry, o);
    return;
  }
  // ---- the tile's offsets, then each warp's own vertices
  const uint32_t nv = b < a.tiles_a ? a.nv_a : a.nv;
  const uint64_t v0 = b < a.tiles_a ? b * dec_tile(a.nv_a) : va + (b - a.tiles_a) * dec_tile(a.nv);
  const uint32_t cnt = (uint32_t)min((uint64_t)dec_tile(nv), g.n - v0);
  tile_offsets<OFF>(g, v0, (int)cnt, sm.xs, sm.ts);
  __syncthreads();
  PrWarp& W = sm.w[wid];
  const uint32_t i0 = min(cnt, wid * nv), i1 = min(cnt, i0 + nv);
  uint64_t ap[PW_VPL], total = 0;  // arcs of the warp tile before each owned vertex, and in all
  LightTile T;
  {
    uint64_t x[PW_VPL];
    uint32_t deg[PW_VPL];
#pragma unroll
    for (int q = 0; q < PW_VPL; q++) x[q] = sm.xs[min(i1, i0 + lane + 32u * q)];
    light_geometry<IDM>(g, v0 + i0, v0 + i1, x, sm.xs[i1], W, T, [&](int q, uint32_t d, uint32_t h) {
      deg[q] = d;
      if (h != ~0u) sm.hdeg[wid][h] = d;
    });
    __syncwarp();
#pragma unroll
    for (int q = 0; q < PW_VPL; q++) {
      const uint64_t incl = T.NH ? warp_incl_scan<uint64_t>(deg[q]) : warp_incl_scan<uint32_t>(deg[q]);
      ap[q] = total + incl - deg[q];
      total += __shfl_sync(LG_FULL_MASK, incl, 31);
    }
  }
  if (lane == 0) sm.sums[wid] = total;
  // ---- the first window is on its way while the CTA finds the arcs before its tile
  const uint64_t pol = policy_stream();
  int jb = -1, ja = -1;  // the light vertices open before and after the window
  Window cur, nxt;
  nxt.f0 = nxt.nf = nxt.fcur = 0;
  nxt.h = 0;
  nxt.fend = T.NH ? W.info[PW_TV - 1] & ((1u << 19) - 1u) : T.F;
  nxt.rbit = T.tb + T.first;
  nxt.at = nxt.ro = 0;
  uint32_t gcarry = 0, buf = 0, hseen = 0;
  bool more = next_window(T, W, PW_WF, nxt);
  if (more) ja = open_window<IDM>(g, T, nxt, 0, -1, pol, W);
  __syncthreads();
  if (wid == 0) {
    const uint64_t mine = lane < DEC_WARPS ? sm.sums[lane] : 0;
    const uint64_t incl = warp_incl_scan<uint64_t>(mine), all = __shfl_sync(LG_FULL_MASK, incl, 31);
    if (lane < DEC_WARPS) sm.sums[lane] = incl - mine;
    if (lane == 0) st_release_u64(a.tile_status + b, (b == 0 ? DEC_INCL : DEC_AGG) | all);
    uint64_t before = 0;
    const bool ok = b == 0 || dec_lookback(a, b, before);
    if (lane == 0) {
      if (!ok) atomicOr(a.err, DERR_INTERNAL);
      if (b > 0) st_release_u64(a.tile_status + b, DEC_INCL | (before + all));
      sm.base = before;
      sm.ok = ok;
      if (v0 + cnt == g.n) a.row_out[g.n] = before + all;
    }
  }
  __syncthreads();
  if (!sm.ok) {
    stage_wait<0>();
    return;
  }
  uint64_t base = sm.base + sm.sums[wid];  // arcs before the warp tile; later also its heavy ones passed
#pragma unroll
  for (int q = 0; q < PW_VPL; q++)
    if (i0 + lane + 32u * q < i1) a.row_out[v0 + i0 + lane + 32u * q] = base + ap[q];
  if (g.n_items) {  // heavy items read their row's start
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      st_release_u32(a.tile_ready + b, 1u);
    }
  }
  // ---- windows
  const uint32_t k0 = PW_E * lane;
  uint32_t* out = sm.out[wid];
  auto rows_to = [&](const Window& w) {  // light field f of the tile goes to base + f
    for (; hseen < w.h; hseen++) base += sm.hdeg[wid][hseen];
    return base + w.f0;
  };
  uint64_t dst = 0, dst_next = more ? rows_to(nxt) : 0;
  for (; more; buf ^= 1u) {
    cur = nxt;
    dst = dst_next;
    const int jc = ja;
    more = next_window(T, W, PW_WF, nxt);
    if (more) {
      dst_next = rows_to(nxt);
      ja = open_window<IDM>(g, T, nxt, buf ^ 1u, jc, pol, W);
      stage_wait<1>();
    } else {
      stage_wait<0>();
    }
    const uint32_t hb = (W.heads[buf][lane >> 2] >> (8u * (lane & 3u))) & 255u;
    const int c = (int)__popc(hb);
    const int je = jb + warp_incl_scan<int>(c) - c;
    jb = jc;
    uint32_t id[PW_E];
    decode_window<IDM, RUNS>(g, cur, hb, je, W, gcarry, id);
    uint4* o4 = reinterpret_cast<uint4*>(out + k0);
    o4[0] = make_uint4(id[0], id[1], id[2], id[3]);
    o4[1] = make_uint4(id[4], id[5], id[6], id[7]);
    __syncwarp();
#pragma unroll
    for (uint32_t u = 0; u < PW_G; u++)
      if (lane + 32u * u < cur.nf) __stcs(a.ids + dst + lane + 32u * u, out[lane + 32u * u]);
    __syncwarp();  // the stage, the heads and the IDs may be overwritten
  }
}

// The heavy items of a graph that is mostly heavy (DecArgs::heavy_after), a warp
// each, once the rows' offsets are written: they need none of the tiles' shared
// memory, which leaves an SM 32 warps (400,000 vertices of degree 300, local IDs
// in DM order: 539 us with the tiles, 346 so; R-MAT 2^19 of degree 90 in local-gap
// IDs 454 and 288).
template <int IDM>
__global__ void __launch_bounds__(TNT) k_dec_heavy(GView g, DecArgs a) {
  const uint64_t it = (uint64_t)blockIdx.x * (TNT / 32) + (threadIdx.x >> 5);
  if (it >= g.n_items || __ldcg(a.err)) return;  // a tile that gave up left its offsets unwritten
  const HeavyItem h = g.items[it];
  dec_fields<IDM, HEAVY_U>(g, a, h.bit, h.w, h.f0, h.f0 + h.nf, h.carry, a.row_ptr[h.v]);
}

// ===========================================================================
// heavy-vertex schedule, built once per graph from the encoded arrays
// ===========================================================================
__device__ __forceinline__ uint32_t items_of(const GView& g, uint32_t d) {
  return d > g.heavy_min ? (d + g.heavy_seg - 1) / g.heavy_seg : 0u;
}

template <int IDM, int OFF>
__global__ void __launch_bounds__(TNT) k_plan_count(GView g, PlanArgs p) {
  __shared__ TileSmem sm;
  const uint64_t v0 = (uint64_t)blockIdx.x * TV;
  const int cnt = (int)min((uint64_t)TV, g.n - v0);
  tile_offsets<OFF>(g, v0, cnt, sm.xs, sm.ts);
  __syncthreads();
  uint64_t mine = 0, top = 0, heavy = 0;
  uint32_t mid = 0;
  for (int i = threadIdx.x; i < cnt; i += TNT) {
    uint64_t start; uint32_t d, w;
    vgeo<IDM>(g, sm.xs[i], sm.xs[i + 1], start, d, w);
    const uint32_t k = items_of(g, d);
    mine += ((uint64_t)k << 32) | (k > 1 ? 1u : 0u);
    if (d > 32) mid = (uint32_t)(v0 + i) + 1u;
    if (v0 + i < PW_TOP) top += d;
    if (k) heavy += d;
  }
  if (p.mid) {
    mid = __reduce_max_sync(LG_FULL_MASK, mid);
    if ((threadIdx.x & 31) == 0 && mid) atomicMax(p.mid, mid);
  }
  if (v0 < PW_TOP) {
    top = warp_sum<uint64_t>(top);
    if ((threadIdx.x & 31) == 0 && top) atomicAdd(p.top, (unsigned long long)top);
  }
  uint64_t total;
  block_excl_scan<uint64_t, TNT>(mine, total, sm.red64);
  if (threadIdx.x == 0) {
    p.tile_count[blockIdx.x] = (uint32_t)(total >> 32);
    p.multi_count[blockIdx.x] = (uint32_t)total;
  }
  if (total) {  // the same in every thread
    uint64_t arcs;
    block_excl_scan<uint64_t, TNT>(heavy, arcs, sm.red64);
    if (threadIdx.x == 0) atomicAdd(p.heavy, (unsigned long long)arcs);
  }
}

template <int IDM, int OFF>
__global__ void __launch_bounds__(TNT) k_plan_fill(GView g, PlanArgs p) {
  __shared__ TileSmem sm;
  const uint64_t v0 = (uint64_t)blockIdx.x * TV;
  const int cnt = (int)min((uint64_t)TV, g.n - v0);
  tile_offsets<OFF>(g, v0, cnt, sm.xs, sm.ts);
  __syncthreads();
  uint64_t st_[TV / TNT];
  uint32_t d_[TV / TNT], w_[TV / TNT];
  uint64_t mine = 0;
#pragma unroll
  for (int q = 0; q < TV / TNT; q++) {
    const int i = threadIdx.x * (TV / TNT) + q;
    d_[q] = 0;
    if (i < cnt) vgeo<IDM>(g, sm.xs[i], sm.xs[i + 1], st_[q], d_[q], w_[q]);
    const uint32_t k = items_of(g, d_[q]);
    mine += ((uint64_t)k << 32) | (k > 1 ? 1u : 0u);
  }
  uint64_t total;
  const uint64_t pre = block_excl_scan<uint64_t, TNT>(mine, total, sm.red64);
  uint64_t it = p.tile_off[blockIdx.x] + (pre >> 32);
  uint64_t slot = p.multi_off[blockIdx.x] - p.multi_off[0] + (uint32_t)pre;
#pragma unroll
  for (int q = 0; q < TV / TNT; q++) {
    const uint32_t k = items_of(g, d_[q]);
    if (k == 0) continue;
    const uint64_t first = it;
    for (uint32_t j = 0; j < k; j++) {
      HeavyItem h;
      h.bit = st_[q];
      h.v = (uint32_t)(v0 + threadIdx.x * (TV / TNT) + q);
      h.f0 = j * g.heavy_seg;
      h.nf = min(g.heavy_seg, d_[q] - h.f0);
      h.carry = 0;
      h.deg = d_[q];
      h.first = (uint32_t)first;
      h.nitems = k;
      h.w = w_[q];
      h.slot = k > 1 ? (uint32_t)slot : 0xffffffffu;
      p.items[it++] = h;
    }
    if (k > 1) p.multi[slot++] = (uint32_t)first;
  }
}

// per item of a split vertex: the sum of its values (for gap-coded IDs the
// first item's sum is its last ID, later items' sums are sums of differences)
template <int IDM, int OFF>
__global__ void __launch_bounds__(256) k_plan_carry(GView g, PlanArgs p) {
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t it = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < g.n_items; it += warps) {
    const HeavyItem h = g.items[it];
    if (h.nitems == 1) continue;
    uint32_t carry = 0;
    const uint32_t f1 = h.f0 + h.nf;
    for (uint32_t base = h.f0; base < f1; base += 32 * HEAVY_U) {
      uint32_t id[HEAVY_U];
      warp_ids<IDM, HEAVY_U>(g, h.bit, h.w, base, f1, carry, id);
    }
    if ((threadIdx.x & 31) == 0) p.segsum[it] = carry;
  }
}

// ===========================================================================
// launchers
// ===========================================================================
inline unsigned tiles_of(uint64_t n) { return (unsigned)((n + TV - 1) / TV); }

// Grid of the kernels whose tiles start at tile0 and whose threads fill the
// labels before them from the schedule: a block per tile, and enough of them
// for the items.  (400,000 vertices of degree 300 in degree order leave one
// tile, whose block then walked 400,000 items alone: 740 us.)
inline unsigned schedule_tiles_grid(const GView& g, uint32_t tile0) {
  const unsigned items = tile0 ? grid_for(g.n_items, TNT, 152 * 8) : 1u;
  return std::max(items, tiles_of(g.n) - tile0);
}

// the sweep for a graph (see decode_window on relabeled ones) and plan
template <int IDM, int OFF>
auto pr_pull_kernel(const GView& g, const PrArgs& a) {
  if constexpr (IDM == ID_LOCAL || IDM == ID_LOCAL_GAP) {
    if (g.perm) return a.tabn ? k_pr_pull<IDM, OFF, true, true> : k_pr_pull<IDM, OFF, false, true>;
  }
  return a.tabn ? k_pr_pull<IDM, OFF, true, false> : k_pr_pull<IDM, OFF, false, false>;
}
template <int IDM, int OFF>
cudaError_t launch_pr_init(const GView& g, const PrArgs& a, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(pr_pull_kernel<IDM, OFF>(g, a),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PW_SMEM);
  if (e != cudaSuccess) return e;
  const uint32_t tile0 = (uint32_t)(g.heavy_prefix / TV);
  k_pr_init<IDM, OFF><<<schedule_tiles_grid(g, tile0), TNT, 0, st>>>(g, a, tile0);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_pr_pull(const GView& g, const PrArgs& a, cudaStream_t st) {
  const uint64_t units = g.n_items + (g.n - a.tile_a) / a.tile_nv + 1;
  // the shared memory beside the table is the warps' (PrWarp)
  const unsigned grid = (unsigned)std::min<uint64_t>(units, PW_SMS);
  const size_t smem = PW_WARPS * sizeof(PrWarp) + (size_t)a.tabn * 4;
  pr_pull_kernel<IDM, OFF>(g, a)<<<grid, PW_NT, smem, st>>>(g, a);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_bfs_pull(const GView& g, const BfsArgs& a, int mb, cudaStream_t st) {
  const TileMap tm = tile_map(g, IDM == ID_LOCAL_GAP);
  const unsigned grid = tile_map_grid(g, tm);
  if (grid == 0) return cudaSuccess;
  if (mb == 2) { k_bfs_pull<IDM, OFF, uint16_t><<<grid, TNT, 0, st>>>(g, a, tm); count_launch(); }
  else if (mb == 4) { k_bfs_pull<IDM, OFF, uint32_t><<<grid, TNT, 0, st>>>(g, a, tm); count_launch(); }
  else { k_bfs_pull<IDM, OFF, uint64_t><<<grid, TNT, 0, st>>>(g, a, tm); count_launch(); }
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_bfs_push(const GView& g, const BfsArgs& a, int mb, cudaStream_t st) {
  if (a.queue_in_len == 0) return cudaSuccess;
  const TileMap tm = tile_map(g, IDM == ID_LOCAL_GAP);
  const unsigned grid = tm.hb + grid_for(a.queue_in_len, 8, 152 * 16);
  if (mb == 2) { k_bfs_push<IDM, OFF, uint16_t><<<grid, 256, 0, st>>>(g, a, tm.hb, tm.shared); count_launch(); }
  else if (mb == 4) { k_bfs_push<IDM, OFF, uint32_t><<<grid, 256, 0, st>>>(g, a, tm.hb, tm.shared); count_launch(); }
  else { k_bfs_push<IDM, OFF, uint64_t><<<grid, 256, 0, st>>>(g, a, tm.hb, tm.shared); count_launch(); }
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_nbr_degrees(const GView& g, const NbrArgs& a, cudaStream_t st) {
  if (a.k == 0) return cudaSuccess;
  k_nbr_degrees<IDM, OFF><<<grid_for(a.k, 8, 152 * 16), 256, 0, st>>>(g, a);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_nbr_rows(const GView& g, const NbrArgs& a, cudaStream_t st) {
  if (a.k == 0) return cudaSuccess;
  NbrArgs b = a;
  // A warp's row needs no CTA to itself: beside other work a server's lookups
  // take an eighth of the room so (2,190 requests/s; 2,000 with a CTA per query).
  // Where most rows take a whole CTA, there are four per SM before they share.
  b.per = g.arcs <= NBR_WARP * g.n ? 8 : (uint32_t)std::min<uint64_t>(8, (a.k + 152 * 4 - 1) / (152 * 4));
  k_nbr_rows<IDM, OFF><<<(unsigned)((a.k + b.per - 1) / b.per), 256, 0, st>>>(g, b);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_plan_count(const GView& g, const PlanArgs& p, cudaStream_t st) {
  k_plan_count<IDM, OFF><<<tiles_of(g.n), TNT, 0, st>>>(g, p);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_plan_fill(const GView& g, const PlanArgs& p, cudaStream_t st) {
  k_plan_fill<IDM, OFF><<<tiles_of(g.n), TNT, 0, st>>>(g, p);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_plan_carry(const GView& g, const PlanArgs& p, cudaStream_t st) {
  if (g.n_items == 0) return cudaSuccess;
  k_plan_carry<IDM, OFF><<<grid_for(g.n_items, 8, 152 * 16), 256, 0, st>>>(g, p);
  count_launch();
  return cudaGetLastError();
}

template <int IDM, int OFF>
cudaError_t launch_ppr_pull(const GView& g, const PprArgs& a, cudaStream_t st) {
  const TileMap tm = tile_map(g, IDM == ID_LOCAL_GAP);
  k_ppr_pull<IDM, OFF><<<tile_map_grid(g, tm), TNT, 0, st>>>(g, a, tm);
  count_launch();
  return cudaGetLastError();
}
template <int IDM, int OFF>
cudaError_t launch_ppr_join(const GView& g, float* cin, uint32_t slot, uint32_t src, cudaStream_t st) {
  k_ppr_join<IDM, OFF><<<1, 32, 0, st>>>(g, cin, slot, src);
  count_launch();
  return cudaGetLastError();
}

template <int IDM, int OFF>
cudaError_t launch_dec_all(const GView& g, const DecArgs& a, cudaStream_t st) {
  if (g.n == 0) return cudaSuccess;
  if constexpr (IDM == ID_GLOBAL || IDM == ID_CSR32) {
    const uint64_t tiles = tiles_of(g.n);
    const uint64_t unit = (uint64_t)(TNT / 32) * DEC_FLAT_CH;
    const uint64_t per_block = (g.arcs + tiles - 1) / tiles;
    k_dec_flat<IDM, OFF><<<(unsigned)tiles, 256, 0, st>>>(g, a, (per_block + unit - 1) / unit * unit);
  } else {
    const auto tiles_kernel = g.perm ? k_dec_local<IDM, OFF, true> : k_dec_local<IDM, OFF, false>;
    const cudaError_t e = cudaFuncSetAttribute(tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(DecSmem));
    if (e != cudaSuccess) return e;
    if (a.heavy_after && g.n_items) {
      GView tiles = g;
      tiles.n_items = 0;
      tiles_kernel<<<(unsigned)a.tiles, TNT, sizeof(DecSmem), st>>>(tiles, a);
      count_launch();
      k_dec_heavy<IDM><<<heavy_blocks(g.n_items), TNT, 0, st>>>(g, a);
    } else {
      tiles_kernel<<<(unsigned)a.tiles + heavy_blocks(g.n_items), TNT, sizeof(DecSmem), st>>>(g, a);
    }
  }
  count_launch();
  return cudaGetLastError();
}

template <int IDM, int OFF>
const TravOps* make_ops() {
  static const TravOps ops = {
      &launch_pr_init<IDM, OFF>,    &launch_pr_pull<IDM, OFF>,     &launch_bfs_pull<IDM, OFF>,
      &launch_bfs_push<IDM, OFF>,   &launch_nbr_degrees<IDM, OFF>, &launch_nbr_rows<IDM, OFF>,
      // the schedule is built while the offsets are still at hand in plain form (GView::O)
      &launch_plan_count<IDM, OFF_ROWPTR>, &launch_plan_fill<IDM, OFF_ROWPTR>, &launch_plan_carry<IDM, OFF>,
      &launch_ppr_pull<IDM, OFF>,   &launch_ppr_join<IDM, OFF>,   &launch_dec_all<IDM, OFF>,
  };
  return &ops;
}

}  // namespace lg
