// Pull PageRank with the decoder fused in (Sections 3.7.2 and 7.1.2).
//
// One launch per iteration, one CTA of 24 warps per SM, no block barrier after
// the prologue: every warp takes work by itself -- heavy-schedule items and
// warp tiles of up to 128 consecutive vertices.
//
// What bounds it: one 4-byte gather of r[u] / d_u per arc.  An SM's L1 looks
// up one line per clock, so gathers that leave the SM cannot pass 274-297 G/s
// on this GPU (152 SMs, measured with 32 distinct lines per request), while
// shared memory answers 1,515 G/s.  The CTA therefore keeps the contributions
// of the first `tabn` stored labels in shared memory where that pays (pr_plan):
// in DM order these are the hubs.  The rest of the design serves the
// gathers: the stream comes in once, by 16-byte loads, a window of 256 fields
// at a time, and every lane takes 8 fields of the window whatever vertices
// they belong to, so its eight gathers are in flight together and no lane
// waits for a longer vertex.  Consecutive fields per lane keep the rest cheap:
// most of a vertex is summed inside a lane, and one segmented scan per window
// joins the lanes.
//
// Measured per sweep, before (tile CTAs of 512 vertices, each thread a serial
// reader; heavy items by warp) and now: R-MAT 2^16 60 -> 17 us, R-MAT 2^18 in
// DM order 376 -> 40 us, 2^22 597 -> 355 us, 2^24 1.75 -> 1.61 ms (not
// relabeled 3.63 -> 2.10), 2^26 8.95 -> 7.08 ms (297 G arcs/s); community 2^24
// in local-gap IDs 1.99 -> 1.90 ms, in global IDs 1.93 -> 1.55 ms.
#pragma once

#include "lg_internal.h"
#include "lg_window.cuh"

namespace lg {

constexpr int PW_NT = 768;                // threads per CTA, one CTA per SM (80 registers: no spills)
constexpr int PW_WARPS = PW_NT / 32;
constexpr int PW_SMS = 152;
constexpr int PW_VPL = 4;                 // vertices per lane of a warp tile
constexpr uint32_t PW_TV = 32 * PW_VPL;   // vertices of a warp tile, at most
constexpr uint32_t PW_STAGE = 344;        // stream words a window may need (see window_fields)
constexpr uint32_t PW_POS_BITS = 26;      // bit positions inside a run of light fields
constexpr uint32_t PW_POSM = (1u << PW_POS_BITS) - 1u;
constexpr uint32_t PW_HEAVY_MAX = 4096;   // largest light degree (128 * 4096 fields of <= 38 bits < 2^26 bits)
// Shared memory of a CTA with a table of contributions.  Measured: with a
// carve-out of 132 or 228 KB the L1 serves scattered gathers at half its rate
// (142 G/s), with 100 and 164 at 291 and with 196 at 274.  So the table stops
// where the CTA fills 163 KB; without one the warps alone take 90 KB.
constexpr size_t PW_SMEM = 163 * 1024;
constexpr uint32_t PW_TOP = 16384;        // labels whose share of the arcs decides on the table

// Fields of a window whose records take r bits: 256 records of <= 40 bits
// (GLOBAL), or 256 local fields of <= 32 bits with a header of <= 6 bits each
// and <= 127 empty headers, fit PW_STAGE words from a 16-byte boundary.
__device__ __forceinline__ uint32_t window_fields(uint32_t r) { return r <= 40 ? PW_WF : PW_WF / 2; }

struct PrWarp {
  // stream words of two windows: one is decoded while the next is on its way
  // (before that stage[0] holds the tile's Elias-Fano positions)
  __align__(16) uint32_t stage[2][PW_STAGE];
  uint32_t heads[2][PW_G];  // bit f: field f of the window is the first of its vertex
  // From the front, per light vertex of the tile in order: where its fields are
  // (local modes), its sum.  From the back, per heavy vertex in order: (upper
  // bits of the stream bit after it) << 19 | light fields before it, and the
  // lower 32 bits of that stream bit; positions count from LightTile::tb.
  uint32_t info[PW_TV];
  float vsum[PW_TV];
};

// ---------------------------------------------------------------------------
// offsets of a warp tile of nv vertices: x[q] = x_v for v = v0 + lane + 32 q,
// xe = x of the vertex after the tile (x_n at the end; vertices past the tile
// give xe too).  Elias-Fano: p0 is the position of one number v0 in the high
// vector, pos holds nv + 1 words.
// ---------------------------------------------------------------------------
template <int OFF>
__device__ __forceinline__ void warp_offsets(const GView& g, uint64_t v0, uint32_t nv, uint64_t p0, uint32_t* pos,
                                             uint64_t (&x)[PW_VPL], uint64_t& xe) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t ve = min(g.n, v0 + nv);
  if (OFF == OFF_PACKED) {
#pragma unroll
    for (int q = 0; q < PW_VPL; q++) x[q] = ext64(g.O, min(ve, v0 + lane + 32u * q) * g.w_O, g.w_O);
    xe = ext64(g.O, ve * g.w_O, g.w_O);
  } else if (OFF == OFF_ROWPTR) {
#pragma unroll
    for (int q = 0; q < PW_VPL; q++) x[q] = __ldg(g.O + min(ve, v0 + lane + 32u * q));
    xe = __ldg(g.O + ve);
  } else {
    // Elias-Fano (Section 4.3): ones number v0 .. ve of the high vector, 1024
    // bits per step; a lane lists the ones of its word
    const uint32_t need = (uint32_t)(ve - v0) + 1;
    const uint64_t w0 = p0 >> 5;
    uint32_t carry = 0;
    for (uint64_t wb = w0; carry < need && wb < g.ef_high_words32; wb += 32) {
      const uint64_t wi = wb + lane;
      uint32_t w = wi < g.ef_high_words32 ? __ldg(g.ef_high32 + wi) : 0u;
      if (wb == w0 && lane == 0) w &= 0xffffffffu << ((uint32_t)p0 & 31u);
      const uint32_t c = __popc(w);
      const uint32_t incl = warp_incl_scan<uint32_t>(c);
      uint32_t r = carry + incl - c;  // rank of the word's first one
      carry += __shfl_sync(LG_FULL_MASK, incl, 31);
      const uint32_t at = (uint32_t)(wi - w0) * 32u;
      for (; w && r < need; r++, w &= w - 1u) pos[r] = at + (uint32_t)__ffs((int)w) - 1u;
    }
    __syncwarp();
    const uint64_t b0 = w0 * 32u;
#pragma unroll
    for (int q = 0; q <= PW_VPL; q++) {
      const uint64_t v = q < PW_VPL ? min(ve, v0 + lane + 32u * q) : ve;
      const uint64_t lo = g.ef_l ? ext64(g.ef_low, v * g.ef_l, g.ef_l) : 0;
      const uint64_t y = ((b0 + pos[(uint32_t)(v - v0)] - v) << g.ef_l) | lo;
      if (q < PW_VPL) x[q < PW_VPL ? q : 0] = y; else xe = y;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// PageRank
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pr_finish(const GView& g, const PrArgs& a, uint64_t v, uint32_t d, float sum) {
  const float base = a.personal < 0 ? a.base_all : ((int64_t)v == a.personal ? a.base_all : 0.0f);
  const float r = base + a.damp * sum;
  __stcs(a.contrib_out + v, d ? r / (float)d : 0.0f);  // streamed: read again only next iteration
  if (a.last) __stcs(a.ranks_out + (g.inv_perm ? (uint64_t)g.inv_perm[v] : v), r);
}

template <bool TAB>
struct PrGather {
  const float* c;
  const float* tab;   // TAB: shared-memory copy of c[0 .. tabn)
  uint32_t tabn, hot;
  uint64_t pstream, pkeep;
  // Eight gathers, one L2 policy for them (IDs ascend along a neighborhood).
  // Beside a table, whose shared memory leaves the L1 92 KB, gathers pass the
  // L1 by (R-MAT 2^24 1.665 -> 1.611 ms); without one they are quicker through
  // it (1.81 against 2.99 ms: it catches the hubs).
  __device__ __forceinline__ void operator()(const uint32_t (&id)[PW_E], float (&val)[PW_E]) const {
    const uint64_t pol = id[0] < hot ? pkeep : pstream;
#pragma unroll
    for (int e = 0; e < PW_E; e++) {
      if (TAB) val[e] = id[e] < tabn ? tab[id[e]] : ldcg_gather(c + id[e], pol);
      else val[e] = ldg_gather(c + id[e], pol);
    }
  }
};

// sum of the contributions of one heavy item's fields: a window of 256 fields at
// a time, eight values of a lane added as a tree, those sums Kahan-compensated.
// A window's values are added while the next one's gathers are in flight (items
// of 300 fields in local-gap IDs 0.574 -> 0.554 ms a sweep, others equal).
template <int IDM, class Gather>
__device__ __forceinline__ float pr_item(const GView& g, const HeavyItem& h, const Gather& G, PrWarp& W) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t w = IDM == ID_GLOBAL ? g.r : (IDM == ID_CSR32 ? 32u : h.w);  // bits from field to field
  const uint32_t mask = mask_lo(IDM == ID_GLOBAL ? g.s : w);                   // of an ID (or gap)
  const uint32_t wf = window_fields(w);
  const uint32_t f0 = h.f0, f1 = h.f0 + h.nf;
  // gap mode: the first field holds s bits, field i > 0 starts at bit + s - w + i * w
  const uint64_t origin = IDM == ID_LOCAL_GAP ? h.bit + g.s - w : h.bit;
  auto first_word = [&](uint32_t base) {
    return (((IDM == ID_LOCAL_GAP && base == 0) ? h.bit : origin + (uint64_t)base * w) >> 5) & ~3ull;
  };
  auto issue = [&](uint32_t base, uint32_t b) {
    const uint64_t w0 = first_word(base), b1 = origin + (uint64_t)(base + min(wf, f1 - base)) * w;
    stage_issue<3>(W.stage[b], g.A32, w0, (uint32_t)(((b1 + 31) >> 5) + 1 - w0), G.pstream);
  };
  uint32_t carry = h.carry, b = 0;
  float acc = 0.f, comp = 0.f;
  float xp[PW_G] = {};  // the window before: summed while this one's gathers are in flight
  const auto add = [&] {
    const float y = (((xp[0] + xp[1]) + (xp[2] + xp[3])) + ((xp[4] + xp[5]) + (xp[6] + xp[7]))) - comp;
    const float t = acc + y;
    comp = (t - acc) - y;
    acc = t;
  };
  issue(f0, 0);
  for (uint32_t base = f0; base < f1; base += wf, b ^= 1u) {
    const uint32_t nf = min(wf, f1 - base);
    if (base + wf < f1) {
      issue(base + wf, b ^ 1u);
      stage_wait<1>();
    } else {
      stage_wait<0>();
    }
    // unguarded: positions past the item's end stay inside the warp's memory
    const uint32_t at0 = sh_bit0(W.stage[b]) - (uint32_t)(first_word(base) * 32u);
    uint32_t id[PW_G], p = at0 + (uint32_t)(origin + (uint64_t)base * w) + lane * w;
#pragma unroll
    for (int u = 0; u < PW_G; u++, p += 32u * w) id[u] = sh_bits(p) & mask;
    if (IDM == ID_LOCAL_GAP && base + lane == 0) id[0] = sh_bits(at0 + (uint32_t)h.bit) & mask_lo(g.s);
    const bool whole = nf == PW_WF;
    if (!whole) {
#pragma unroll
      for (int u = 0; u < PW_G; u++) id[u] = 32u * u + lane < nf ? id[u] : 0u;
    }
    if (IDM == ID_LOCAL_GAP) {
#pragma unroll
      for (int u = 0; u < PW_G; u++) {
        id[u] = warp_incl_scan<uint32_t>(id[u]) + carry;
        carry = __shfl_sync(LG_FULL_MASK, id[u], 31);
      }
    }
    float x[PW_G];
    G(id, x);
    if (!whole) {
#pragma unroll
      for (int u = 0; u < PW_G; u++) x[u] = 32u * u + lane < nf ? x[u] : 0.f;
    }
    add();
#pragma unroll
    for (int u = 0; u < PW_G; u++) xp[u] = x[u];
    __syncwarp();  // the stage may be overwritten
  }
  add();
  return warp_sum<float>(acc);
}

// ---------------------------------------------------------------------------
// Warp tile: lane l owns the vertices v0 + l + 32 q, q < 4.  Its light
// neighborhoods (degree <= heavy_min) are fields 0 .. F - 1 of the tile.
// ---------------------------------------------------------------------------
constexpr uint32_t PW_HEAVY = 8191;               // in the place of a heavy vertex's degree
constexpr uint32_t PW_NOFIELD = (1u << 19) - 1u;  // in the place of the first field of a vertex without light fields

struct LightTile {
  uint32_t pk[PW_VPL];  // per owned vertex: first light field << 13 | degree
  uint64_t tb;          // stream bit that positions count from (a 16-byte boundary)
  uint32_t first;       // first bit of the tile, from tb
  uint32_t F, NH;       // light fields, heavy vertices
};

// info of a light vertex (local modes): width << 26 | base, its field f of the
// tile is at bit (base + f * width) mod 2^26; gap mode: the fields after the
// first, which holds s bits and begins s - width bits before that formula
//
// x: the offsets of the owned vertices, xe of ve.  seen(q, d, h): owned vertex
// q has degree d, h its number among the tile's heavy vertices (or ~0).
template <int IDM, class Seen>
__device__ __forceinline__ void light_geometry(const GView& g, uint64_t v0, uint64_t ve, const uint64_t (&x)[PW_VPL],
                                               uint64_t xe, PrWarp& W, LightTile& T, Seen seen) {
  const uint32_t lane = threadIdx.x & 31u, lt = lane_lt_mask();
  constexpr bool FLAT = IDM == ID_GLOBAL || IDM == ID_CSR32;
  const uint32_t rw = FLAT ? (IDM == ID_GLOBAL ? g.r : 32u) : 1u;  // stream bits per unit of an offset
  const uint64_t first = __shfl_sync(LG_FULL_MASK, x[0], 0) * rw;
  T.tb = first & ~127ull;
  T.first = (uint32_t)(first - T.tb);
  T.F = 0;
  T.NH = 0;
  uint32_t NL = 0, head[PW_VPL];  // the headers' loads go out together
#pragma unroll
  for (int q = 0; q < PW_VPL; q++) head[q] = v0 + lane + 32u * q < ve ? vhead<IDM>(g, x[q]) : 0u;
#pragma unroll
  for (int q = 0; q < PW_VPL; q++) {
    uint64_t x1 = __shfl_down_sync(LG_FULL_MASK, x[q], 1);
    const uint64_t nx = q + 1 < PW_VPL ? __shfl_sync(LG_FULL_MASK, x[q + 1 < PW_VPL ? q + 1 : q], 0) : xe;
    if (lane == 31) x1 = nx;
    uint64_t start = 0;
    uint32_t d = 0, w = 0;
    if (v0 + lane + 32u * q < ve) vgeo<IDM>(g, x[q], x1, head[q], start, d, w);
    const bool heavy = d > g.heavy_min, light = d > 0 && !heavy;
    const uint32_t lf = heavy ? 0u : d;
    const uint32_t incl = warp_incl_scan<uint32_t>(lf);
    const uint32_t fp = T.F + incl - lf;
    T.F += __shfl_sync(LG_FULL_MASK, incl, 31);
    T.pk[q] = ((light ? fp : PW_NOFIELD) << 13) | (heavy ? PW_HEAVY : d);
    const uint32_t hm = __ballot_sync(LG_FULL_MASK, heavy);
    if (!FLAT) {
      const uint32_t lm = __ballot_sync(LG_FULL_MASK, light);
      if (light) {
        const uint32_t st = (uint32_t)(start - T.tb) + (IDM == ID_LOCAL_GAP ? g.s - w : 0u);
        W.info[NL + __popc(lm & lt)] = (w << PW_POS_BITS) | ((st - fp * w) & PW_POSM);
      }
      NL += __popc(lm);
    }
    if (heavy) {
      const uint32_t h = PW_TV - 1 - (T.NH + __popc(hm & lt));
      const uint64_t after = x1 * rw - T.tb;
      W.info[h] = ((uint32_t)(after >> 32) << 19) | fp;
      W.vsum[h] = __uint_as_float((uint32_t)after);
    }
    seen(q, d, heavy ? T.NH + __popc(hm & lt) : ~0u);
    T.NH += __popc(hm);
  }
  __syncwarp();
}

template <int IDM, int OFF>
__device__ __forceinline__ void light_tile(const GView& g, uint64_t v0, uint32_t nv, uint64_t p0, PrWarp& W,
                                           LightTile& T) {
  uint64_t x[PW_VPL], xe;
  warp_offsets<OFF>(g, v0, nv, p0, W.stage[0], x, xe);
  light_geometry<IDM>(g, v0, min(g.n, v0 + nv), x, xe, W, T, [](int, uint32_t, uint32_t) {});
}

// A window: fields [f0, f0 + nf) of the tile, inside one run of light fields
// with contiguous stream bits (a heavy vertex ends a run).
struct Window {
  uint32_t f0, nf;
  uint32_t fcur, fend, h;  // its run: fields [fcur, fend), ended by heavy vertex h of the tile
  uint64_t rbit;           // stream bit of the run's first field
  uint32_t at, ro;         // FLAT: shared-memory bit of field f0; local modes: shared-memory bit of
                           // the tile's bit ro (mod 2^26)
};
// the window after fields [.., w.f0 + w.nf), false at the tile's end
__device__ __forceinline__ bool next_window(const LightTile& T, const PrWarp& W, uint32_t wf, Window& w) {
  w.f0 += w.nf;
  while (w.f0 == w.fend) {
    if (w.h == T.NH) return false;
    const uint32_t hv = W.info[PW_TV - 1 - w.h];
    w.rbit = T.tb + (((uint64_t)(hv >> 19) << 32) | __float_as_uint(W.vsum[PW_TV - 1 - w.h]));
    w.fcur = w.fend;
    w.h++;
    w.fend = w.h < T.NH ? W.info[PW_TV - 1 - w.h] & ((1u << 19) - 1u) : T.F;
  }
  w.nf = min(wf, w.fend - w.f0);
  return true;
}
// Heads of a window and its copy into stage b.  j: the light vertex open before
// it; returns the one open at its end.
template <int IDM>
__device__ __forceinline__ int open_window(const GView& g, const LightTile& T, Window& w, uint32_t b, int j,
                                           uint64_t pol, PrWarp& W) {
  const uint32_t lane = threadIdx.x & 31u;
  if (lane < PW_G) W.heads[b][lane] = 0;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < PW_VPL; q++) {
    const uint32_t k = (T.pk[q] >> 13) - w.f0;
    if (k < w.nf) atomicOr(&W.heads[b][k >> 5], 1u << (k & 31u));
  }
  __syncwarp();
  const int jn = j + (int)__reduce_add_sync(LG_FULL_MASK, lane < PW_G ? __popc(W.heads[b][lane]) : 0u);
  if (IDM == ID_GLOBAL || IDM == ID_CSR32) {
    const uint32_t rw = IDM == ID_GLOBAL ? g.r : 32u;
    const uint64_t b0 = w.rbit + (uint64_t)(w.f0 - w.fcur) * rw;
    const uint64_t w0 = (b0 >> 5) & ~3ull;
    w.at = sh_bit0(W.stage[b]) + (uint32_t)(b0 - w0 * 32u);
    stage_issue<3>(W.stage[b], g.A32, w0, (uint32_t)(((b0 + w.nf * rw + 31) >> 5) + 1 - w0), pol);
  } else {
    const uint64_t rb = w.rbit & ~127ull;
    w.ro = (uint32_t)(rb - T.tb);
    // first and last bit, from rb: of the vertices that hold the first and the last field
    const uint32_t head = W.heads[b][0] & 1u;
    const uint32_t ia = W.info[j + (int)head], ib = W.info[jn];
    const uint32_t wa = ia >> PW_POS_BITS, wb = ib >> PW_POS_BITS;
    const uint32_t bs = (ia + w.f0 * wa - w.ro - (IDM == ID_LOCAL_GAP && head ? g.s - wa : 0u)) & PW_POSM;
    const uint32_t be = ((ib + (w.f0 + w.nf - 1) * wb - w.ro) & PW_POSM) + wb;
    const uint32_t w0 = (bs >> 5) & ~3u;
    w.at = sh_bit0(W.stage[b]) - w0 * 32u;
    stage_issue<3>(W.stage[b], g.A32, (rb >> 5) + w0, ((be + 31) >> 5) + 1 - w0, pol);
  }
  return jn;
}

// IDs of the lane's 8 consecutive fields of a window: hb their head bits, je
// the light vertex that is open before them.  RUNS: windows in which no lane
// enters a second vertex are decoded in their own way.
template <int IDM, bool RUNS>
__device__ __forceinline__ void decode_window(const GView& g, const Window& wd, uint32_t hb, int je, const PrWarp& W,
                                              uint32_t& gcarry, uint32_t (&id)[PW_E]) {
  const uint32_t lane = threadIdx.x & 31u, k0 = PW_E * lane;
  if (IDM == ID_GLOBAL || IDM == ID_CSR32) {  // unguarded: positions past the window stay inside the warp's memory
    const uint32_t rw = IDM == ID_GLOBAL ? g.r : 32u, mask = mask_lo(IDM == ID_GLOBAL ? g.s : 32u);
    uint32_t p = wd.at + min(k0, wd.nf) * rw;
#pragma unroll
    for (int e = 0; e < PW_E; e++, p += rw) id[e] = sh_bits(p) & mask;
    return;
  }
  const uint32_t rel = wd.ro;
  uint32_t v = 0;
  if (RUNS && wd.nf == PW_WF && !__any_sync(LG_FULL_MASK, (hb & (hb - 1u)) != 0)) {
    // The fields before the lane's head h follow each other at one width, those
    // from it on at another: one vertex's info each, and no multiplication per
    // field.  Local-gap IDs in DM order, ms a sweep: 1.5 M vertices of degree 40
    // 0.302 -> 0.291, community 2^24 1.92 -> 1.87, R-MAT 2^16 0.043 -> 0.039.
    // Sweeps of graphs that are not relabeled, whose windows mix short and long
    // vertices, lose 3 % to the two paths and keep the other.
    const uint32_t h = hb ? (uint32_t)__ffs((int)hb) - 1u : (uint32_t)PW_E;
    const uint32_t ia = W.info[max(je, 0)], ib = W.info[je + (hb != 0)];  // je is -1 only if the first field is a head
    const uint32_t wa = ia >> PW_POS_BITS, wb = ib >> PW_POS_BITS, ma = mask_lo(wa), mb = mask_lo(wb);
    const uint32_t ph = ((ib + (wd.f0 + k0 + h) * wb - rel) & PW_POSM) + wd.at;
    uint32_t pa = ((ia + (wd.f0 + k0) * wa - rel) & PW_POSM) + wd.at, pb = ph - h * wb;
    // a first field is an absolute ID of s bits
    const uint32_t first = IDM == ID_LOCAL_GAP ? sh_bits(hb ? ph - (g.s - wb) : pa) & mask_lo(g.s) : 0u;
#pragma unroll
    for (int e = 0; e < PW_E; e++, pa += wa, pb += wb) {
      const bool after = e >= h;
      const uint32_t x = sh_bits(after ? pb : pa) & (after ? mb : ma);
      v = IDM == ID_LOCAL_GAP ? (e == h ? first : v + x) : x;
      id[e] = v;
    }
  } else {
    // A field's place comes from its vertex's info alone, so that no lane waits
    // for one that enters a vertex there (a step per entered vertex: 4 % more
    // instructions in a whole-graph decode).
    const uint32_t n8 = k0 < wd.nf ? wd.nf - k0 : 0u;
    int j = je;  // -1 only before the tile's first field
#pragma unroll
    for (int e = 0; e < PW_E; e++) {
      const bool head = (hb >> e) & 1u;
      j += head;
      const uint32_t i = e < n8 ? W.info[j] : 0u, w = i >> PW_POS_BITS;
      const uint32_t bits = IDM == ID_LOCAL_GAP && head ? g.s : w;  // a first field is an absolute ID of s bits
      const uint32_t p = (i + (wd.f0 + k0 + e) * w - rel) & PW_POSM;
      const uint32_t x = e < n8 ? sh_bits(p + wd.at - (bits - w)) & mask_lo(bits) : 0u;
      v = IDM == ID_LOCAL_GAP && !head ? v + x : x;
      id[e] = v;
    }
  }
  if (IDM == ID_LOCAL_GAP) {
    // fields before the lane's first head continue the neighborhood of the lane before
    const uint32_t before = __ballot_sync(LG_FULL_MASK, hb != 0) & (lane_lt_mask() | (1u << lane));
    const int seg = 31 - __clz((int)(before | 1u));
    uint32_t y = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(LG_FULL_MASK, y, o);
      if ((int)lane - o >= seg) y += z;
    }
    if (!before) y += gcarry;
    uint32_t in = __shfl_up_sync(LG_FULL_MASK, y, 1);
    if (lane == 0) in = gcarry;
    gcarry = __shfl_sync(LG_FULL_MASK, y, 31);
#pragma unroll
    for (int e = 0; e < PW_E; e++)
      if ((hb & ((2u << e) - 1u)) == 0) id[e] += in;
  }
}

template <int IDM, int OFF, bool RUNS, class Gather>
__device__ __forceinline__ void pr_tile(const GView& g, const PrArgs& a, uint64_t v0, uint32_t nv, uint64_t p0,
                                        const Gather& G, PrWarp& W) {
  const uint32_t lane = threadIdx.x & 31u, lt = lane_lt_mask(), k0 = PW_E * lane;
  const uint32_t wf = window_fields(IDM == ID_GLOBAL ? g.r : 32u);
  LightTile T;
  light_tile<IDM, OFF>(g, v0, nv, p0, W, T);
  float open = 0.f;     // sum so far of the light vertex open before the window
  uint32_t gcarry = 0;  // gap mode: the ID of the field before
  int jb = -1, ja = -1;  // the light vertices open before and after the window
  Window cur, nxt;
  nxt.f0 = nxt.nf = nxt.fcur = 0;
  nxt.h = 0;
  nxt.fend = T.NH ? W.info[PW_TV - 1] & ((1u << 19) - 1u) : T.F;
  nxt.rbit = T.tb + T.first;
  nxt.at = nxt.ro = 0;
  uint32_t b = 0;
  bool more = next_window(T, W, wf, nxt);
  if (more) ja = open_window<IDM>(g, T, nxt, 0, -1, G.pstream, W);
  for (; more; b ^= 1u) {
    cur = nxt;
    const int jc = ja;
    more = next_window(T, W, wf, nxt);
    if (more) {
      ja = open_window<IDM>(g, T, nxt, b ^ 1u, jc, G.pstream, W);
      stage_wait<1>();
    } else {
      stage_wait<0>();
    }
    const uint32_t hb = (W.heads[b][lane >> 2] >> (8u * (lane & 3u))) & 255u;
    const int c = (int)__popc(hb);
    const int je = jb + warp_incl_scan<int>(c) - c;
    jb = jc;
    uint32_t id[PW_E];
    decode_window<IDM, RUNS>(g, cur, hb, je, W, gcarry, id);
    const bool whole = cur.nf == PW_WF;
    if (!whole) {
#pragma unroll
      for (int e = 0; e < PW_E; e++) id[e] = k0 + e < cur.nf ? id[e] : 0u;
    }
    float val[PW_E];
    G(id, val);
    if (!whole) {
#pragma unroll
      for (int e = 0; e < PW_E; e++) val[e] = k0 + e < cur.nf ? val[e] : 0.f;
    }
    open = join_window(val, hb, je, open, W.vsum);
    __syncwarp();  // the stage and the heads may be overwritten
  }
  if (lane == 0 && jb >= 0) W.vsum[jb] = open;
  __syncwarp();
  uint32_t NL = 0;
#pragma unroll
  for (int q = 0; q < PW_VPL; q++) {
    const uint64_t v = v0 + lane + 32u * q;
    const uint32_t d = T.pk[q] & 8191u;
    const bool light = d > 0 && d < PW_HEAVY;
    const uint32_t lm = __ballot_sync(LG_FULL_MASK, light);
    if (v < min(g.n, v0 + nv) && d < PW_HEAVY) pr_finish(g, a, v, d, light ? W.vsum[NL + __popc(lm & lt)] : 0.f);
    NL += __popc(lm);
  }
  __syncwarp();
}

// Work units, large ones first: the small tiles (PrArgs::tile_a to tile_b), the
// heavy items, tiles of 128 vertices.  Warp w of CTA b starts with ticket
// w * grid + b and goes on with the shared counter.  That is one word, and a
// graph of many short items would ask more of it than it gives (400,000 items
// of 300 fields, 0.54 ms a sweep: 0.8 G tickets/s; 0.47 with 8 to a ticket), so
// a ticket may stand for k items (PrArgs::items, a power of two).
__device__ __forceinline__ uint32_t first_unit(uint32_t ticket, uint32_t n1, uint32_t n2, uint32_t k) {
  if (ticket < n1) return ticket;
  const uint32_t q = ticket - n1, q2 = (n2 + k - 1) >> (31 - __clz(k));
  return q < q2 ? n1 + q * k : n1 + n2 + (q - q2);
}
// the unit after t belongs to the same ticket
__device__ __forceinline__ bool same_ticket(uint32_t t, uint32_t n1, uint32_t n2, uint32_t k) {
  return t - n1 + 1 < n2 && ((t - n1 + 1) & (k - 1)) != 0;
}
template <int IDM, int OFF, bool TAB, bool RUNS>
__global__ void __launch_bounds__(PW_NT, 1) k_pr_pull(GView g, PrArgs a) {
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  PrWarp& W = reinterpret_cast<PrWarp*>(dyn_smem)[wid];
  float* tab = reinterpret_cast<float*>(dyn_smem + PW_WARPS * sizeof(PrWarp));
  if (blockIdx.x == 0 && threadIdx.x == 0) a.sync[a.turn ^ 1u] = 0;  // the next iteration's ticket counter
  if (TAB) {
    const float4* src = reinterpret_cast<const float4*>(a.contrib_in);
    for (uint32_t i = threadIdx.x; i < a.tabn / 4; i += PW_NT) reinterpret_cast<float4*>(tab)[i] = __ldg(src + i);
    for (uint32_t i = (a.tabn & ~3u) + threadIdx.x; i < a.tabn; i += PW_NT) tab[i] = __ldg(a.contrib_in + i);
    __syncthreads();
  }
  const PrGather<TAB> G = {a.contrib_in, tab, a.tabn, a.hot, policy_stream(), policy_keep()};
  const uint32_t n1 = (uint32_t)((min(g.n, a.tile_b) - min(g.n, a.tile_a) + a.tile_nv - 1) / a.tile_nv);
  const uint32_t n2 = (uint32_t)g.n_items, k = a.items;
  const uint32_t total = n1 + n2 + (g.n > a.tile_b ? (uint32_t)((g.n - a.tile_b + PW_TV - 1) / PW_TV) : 0u);
  for (uint32_t t = first_unit(wid * gridDim.x + blockIdx.x, n1, n2, k); t < total;) {
    uint32_t next = 0;
    if (lane == 0 && !same_ticket(t, n1, n2, k)) next = atomicAdd(a.sync + a.turn, 1u);
    if (t - n1 < n2) {
      const HeavyItem h = g.items[t - n1];
      const float s = pr_item<IDM>(g, h, G, W);
      if (h.nitems == 1) {
        if (lane == 0) pr_finish(g, a, h.v, h.deg, s);
      } else {
        // the warp that brings a vertex's last sum adds them up, in the same order every time
        uint32_t last = 0;
        if (lane == 0) {
          a.part[t - n1] = s;
          __threadfence();
          last = atomicInc(a.sync + 2 + h.slot, h.nitems - 1) == h.nitems - 1;  // wraps to 0 for the next iteration
        }
        if (__shfl_sync(LG_FULL_MASK, last, 0)) {
          __threadfence();
          float sum = 0.f;
          for (uint32_t q = lane; q < h.nitems; q += 32) sum += __ldcg(a.part + h.first + q);
          sum = warp_sum<float>(sum);
          if (lane == 0) pr_finish(g, a, h.v, h.deg, sum);
        }
      }
    } else {
      const bool small = t < n1;
      const uint64_t v0 = small ? a.tile_a + (uint64_t)a.tile_nv * t : a.tile_b + (uint64_t)PW_TV * (t - n1 - n2);
      const uint64_t p0 = OFF == OFF_EF ? __ldg(a.aux + (small ? t : t - n2)) : 0;
      pr_tile<IDM, OFF, RUNS>(g, a, v0, small ? a.tile_nv : PW_TV, p0, G, W);
    }
    t = same_ticket(t, n1, n2, k) ? t + 1
                                  : first_unit(PW_WARPS * gridDim.x + __shfl_sync(LG_FULL_MASK, next, 0), n1, n2, k);
  }
}

}  // namespace lg
