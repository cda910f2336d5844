// Single-source shortest paths on the weighted compressed graph (Section
// 7.1.2: SSSP by delta-stepping; weights stored at omega bits right after each
// ID, Section 3.3).
//
// A GPU form of delta-stepping ("near / far" piles):
//   * bucket [lo, lo + delta) is processed in rounds: the arcs of the near
//     queue are spread evenly over warps, each lane decoding its arc's neighbor
//     and weight from the compressed stream and lowering dist[u] with
//     atomicMin; a vertex improved to a distance below
//     lo + delta joins the next round's near queue (a per-round stamp keeps
//     one entry per vertex), any other improved vertex joins the far list (a
//     per-bucket stamp keeps one entry per vertex, so the list never exceeds n);
//   * when a round leaves the near queue empty, the far list is reduced to its
//     smallest live distance, the next non-empty bucket starts there, and the
//     far list is split into that bucket's near queue and the rest.
// Distances are integers (sums of stored weights), so the result is the exact
// shortest-path distance whatever the order of relaxations.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <utility>

#include "lg_traverse.cuh"

namespace lg {

constexpr uint64_t DINF = ~0ull;

struct SsspArgs {
  unsigned long long* dist;  // n, stored labels
  const uint64_t* x;         // n + 1 plain arc offsets
  const uint32_t* near_in;
  uint32_t near_len;
  uint32_t* near_out;
  uint32_t* far;              // far list (append)
  uint32_t* stamp_near;       // per vertex: last round it was queued for
  uint32_t* stamp_far;        // per vertex: last bucket it was put in the far list
  uint32_t round, bucket;
  uint64_t hi;                // upper end of the current bucket
  uint32_t* near_cnt;         // near_out length
  uint32_t* far_cnt;          // far length
};

// Plain offsets x_0 .. x_n, decoded once per call: a round needs those of its
// near vertices, and a select per vertex and round (a warp each) cost 1.2 ms of
// an SSSP on R-MAT 2^22.  Tiles that hold none but heavy vertices (DM order)
// come from the schedule: their Elias-Fano blocks are thousands of words long.
template <int IDM, int OFF>
__global__ void __launch_bounds__(TNT) k_sssp_offsets(GView g, uint64_t* x, uint32_t tile0) {
  __shared__ uint64_t xs[TV + 1];
  __shared__ TileScratch ts;
  const uint32_t r = IDM == ID_CSR32 ? 32u : g.r;
  if (tile0)
    for (uint64_t i = (uint64_t)blockIdx.x * TNT + threadIdx.x; i < g.n_items; i += (uint64_t)gridDim.x * TNT)
      if (g.items[i].f0 == 0) x[g.items[i].v] = g.items[i].bit / r;
  if (blockIdx.x == 0 && threadIdx.x == 0) x[g.n] = g.arcs;  // here: every tile may come from the schedule
  const uint64_t v0 = ((uint64_t)blockIdx.x + tile0) * TV;
  if (v0 >= g.n) return;
  const int cnt = (int)min((uint64_t)TV, g.n - v0);
  tile_offsets<OFF>(g, v0, cnt, xs, ts);
  __syncthreads();
  for (int i = threadIdx.x; i < cnt; i += TNT) x[v0 + i] = xs[i];
}

// Exclusive sums of the near vertices' degrees, the round's arcs at eoff[len]:
// a block per SSC_TILE vertices.  More than one block: a first pass leaves the
// blocks' sums in part and the block that finishes it last scans them.
constexpr int SSC_IPT = 8;
constexpr uint32_t SSC_TILE = 256 * SSC_IPT;

__device__ __forceinline__ uint64_t near_degrees(const SsspArgs& a, uint64_t (&d)[SSC_IPT]) {
  uint64_t sum = 0;
#pragma unroll
  for (int e = 0; e < SSC_IPT; e++) {
    const uint32_t q = blockIdx.x * SSC_TILE + threadIdx.x * SSC_IPT + e;
    d[e] = 0;
    if (q < a.near_len) {
      const uint32_t v = a.near_in[q];
      d[e] = a.x[v + 1ull] - a.x[v];
    }
    sum += d[e];
  }
  return sum;
}

__global__ void __launch_bounds__(256) k_sssp_part(SsspArgs a, uint64_t* part, uint32_t* arrived) {
  __shared__ uint64_t tmp[8];
  __shared__ uint32_t last;
  uint64_t d[SSC_IPT], total;
  block_excl_scan<uint64_t, 256>(near_degrees(a, d), total, tmp);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = total;
    __threadfence();
    last = atomicInc(arrived, gridDim.x - 1) == gridDim.x - 1;  // wraps to 0 for the next round
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  uint64_t carry = 0;
  for (uint32_t base = 0; base < gridDim.x; base += 256) {
    const uint32_t i = base + threadIdx.x;
    const uint64_t v = i < gridDim.x ? __ldcg(part + i) : 0;
    const uint64_t pre = block_excl_scan<uint64_t, 256>(v, total, tmp) + carry;
    if (i < gridDim.x) part[i] = pre;
    carry += total;
  }
}

__global__ void __launch_bounds__(256) k_sssp_eoff(SsspArgs a, const uint64_t* part, uint64_t* eoff) {
  __shared__ uint64_t tmp[8];
  uint64_t d[SSC_IPT], total;
  uint64_t pre = block_excl_scan<uint64_t, 256>(near_degrees(a, d), total, tmp) + (part ? part[blockIdx.x] : 0);
  if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) eoff[a.near_len] = pre + total;
#pragma unroll
  for (int e = 0; e < SSC_IPT; e++) {
    const uint32_t q = blockIdx.x * SSC_TILE + threadIdx.x * SSC_IPT + e;
    if (q < a.near_len) eoff[q] = pre;
    pre += d[e];
  }
}

// Edge-balanced relaxation: a round's arcs are slots 0 .. E - 1 in the order of
// the near queue, and every warp takes a contiguous range of windows of 256
// slots, so hubs are spread over as many warps as their arcs need.  Per window
// the warp lists the near vertices that have arcs in it (distance, and the
// stream bit of slot 0 were it the vertex's), with a head bit where each
// begins; a slot then finds its vertex by counting head bits (before: a binary
// search of the queue per window and lane, then a step per vertex; the whole call 8.0 ms on R-MAT 2^22; 4.9 with this,
// the plain offsets and no transfers per round, 4.0 with wider buckets).
template <int IDM>
__global__ void __launch_bounds__(256) k_sssp_relax_lb(GView g, SsspArgs a, const uint64_t* eoff) {
  constexpr uint32_t CH = 256;  // arc slots per window
  constexpr int S = CH / 32;
  __shared__ uint64_t dist_s[8][CH + 1], bit_s[8][CH + 1];
  __shared__ uint32_t heads[8][S];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, lt = lane_lt_mask(), le = lt | (1u << lane);
  const uint32_t r = IDM == ID_CSR32 ? 32u : g.r;
  const uint64_t E = eoff[a.near_len];
  const uint64_t windows = (E + CH - 1) / CH, warps = (uint64_t)gridDim.x * 8;
  const uint64_t each = (windows + warps - 1) / warps;
  const uint64_t w0 = ((uint64_t)blockIdx.x * 8 + wid) * each, w1 = min(windows, w0 + each);
  if (w0 >= w1) return;
  uint64_t* ds = dist_s[wid];
  uint64_t* bs = bit_s[wid];
  // the last near vertex that begins at or before the first slot
  uint32_t q0 = 0;
  for (uint32_t hi = a.near_len; hi - q0 > 1;) {
    const uint32_t step = (hi - q0 + 31) / 32, at = q0 + lane * step;
    const uint32_t c = __popc(__ballot_sync(LG_FULL_MASK, at < hi && eoff[at] <= w0 * CH));
    hi = min(hi, q0 + c * step);
    q0 += (c - 1) * step;
  }
  for (uint64_t wi = w0; wi < w1; wi++) {
    const uint64_t s0 = wi * CH;
    const uint32_t ns = (uint32_t)min((uint64_t)CH, E - s0);
    if (lane < S) heads[wid][lane] = 0;
    __syncwarp();
    // entries: q0 first, then the vertices that begin inside the window and have
    // arcs; its last one is the next window's q0
    uint32_t cnt = 0, nq = q0;
    for (uint32_t base = q0;; base += 32) {
      const uint32_t q = base + lane;
      const uint64_t e0 = q < a.near_len ? eoff[q] : E, e1 = q < a.near_len ? eoff[q + 1] : E;
      const bool in = e0 < s0 + ns && e1 > s0 && e1 > e0;
      const uint32_t b = __ballot_sync(LG_FULL_MASK, in);
      if (in) {
        const uint32_t v = a.near_in[q], j = cnt + __popc(b & lt);
        ds[j] = a.dist[v];
        bs[j] = a.x[v] * r - (e0 - s0) * r;  // modulo 2^64: e0 may lie before the window
        if (e0 > s0) atomicOr(&heads[wid][(uint32_t)(e0 - s0) >> 5], 1u << ((uint32_t)(e0 - s0) & 31u));
      }
      if (b) nq = base + 31u - (uint32_t)__clz((int)b);
      cnt += __popc(b);
      if (__any_sync(LG_FULL_MASK, e0 >= s0 + ns)) break;
    }
    q0 = nq;
    __syncwarp();
    // Distances are read with ordinary (L1-cached) loads: they only decrease,
    // so a stale value is never below the true one; a stale dist[u] only costs
    // an atomicMin that changes nothing, and a stale dist[v] only weakens one
    // relaxation -- a vertex improved during a round is queued again, and the
    // next round is a new launch that sees the new value.
    // The window runs in phases so that each lane has its 8 slots' loads in
    // flight together: decode all, load all distances, then the atomics.
    uint32_t uu[S];
    uint64_t nd[S];
    uint32_t jb = 0;  // entry open before the group
#pragma unroll
    for (int t = 0; t < S; t++) {
      const uint32_t hd = heads[wid][t], slot = 32u * t + lane;
      uu[t] = 0xffffffffu;
      nd[t] = DINF;
      if (slot < ns) {
        const uint32_t j = jb + __popc(hd & le);
        const uint64_t bit = bs[j] + (uint64_t)slot * r;
        uu[t] = IDM == ID_CSR32 ? __ldg(g.A32 + (bit >> 5)) : ext32(g.A32, bit, g.s);
        const uint32_t w = IDM == ID_CSR32 ? (g.W32 ? __ldg(g.W32 + (bit >> 5)) : 1u)
                                           : (g.omega ? ext32(g.A32, bit + g.s, g.omega) : 1u);
        nd[t] = ds[j] + w;
      }
      jb += __popc(hd);
    }
    uint64_t du[S];
#pragma unroll
    for (int t = 0; t < S; t++) du[t] = uu[t] != 0xffffffffu ? a.dist[uu[t]] : 0;
    // all atomics of the window are issued before any result is used
#pragma unroll
    for (int t = 0; t < S; t++)
      du[t] = (uu[t] != 0xffffffffu && nd[t] < du[t]) ? atomicMin(a.dist + uu[t], (unsigned long long)nd[t]) : 0;
    uint32_t stamp_old[S];
#pragma unroll
    for (int t = 0; t < S; t++) {
      stamp_old[t] = 0;
      if (nd[t] < du[t]) {  // improved (du now holds the value before the atomicMin)
        stamp_old[t] = nd[t] < a.hi ? atomicExch(a.stamp_near + uu[t], a.round)
                                    : atomicExch(a.stamp_far + uu[t], a.bucket);
      }
    }
    uint32_t near_bits = 0, far_bits = 0;
#pragma unroll
    for (int t = 0; t < S; t++) {
      if (nd[t] < du[t]) {
        if (nd[t] < a.hi) {
          if (stamp_old[t] != a.round) near_bits |= 1u << t;
        } else if (stamp_old[t] != a.bucket) {
          far_bits |= 1u << t;
        }
      }
    }
    // one warp-aggregated append per list
    if (__any_sync(LG_FULL_MASK, near_bits | far_bits)) {
      const uint32_t cn = __popc(near_bits), cf = __popc(far_bits);
      const uint32_t in = warp_incl_scan<uint32_t>(cn), inf = warp_incl_scan<uint32_t>(cf);
      uint32_t bn = 0, bf = 0;
      if (lane == 31) {
        if (in) bn = atomicAdd(a.near_cnt, in);
        if (inf) bf = atomicAdd(a.far_cnt, inf);
      }
      bn = __shfl_sync(LG_FULL_MASK, bn, 31) + in - cn;
      bf = __shfl_sync(LG_FULL_MASK, bf, 31) + inf - cf;
#pragma unroll
      for (int t = 0; t < S; t++) {
        if ((near_bits >> t) & 1u) a.near_out[bn++] = uu[t];
        if ((far_bits >> t) & 1u) a.far[bf++] = uu[t];
      }
    }
  }
}

// smallest distance among far entries that are still at or above `lo`
__global__ void k_far_min(const uint32_t* far, uint32_t len, const unsigned long long* dist, uint64_t lo,
                          unsigned long long* out) {
  uint64_t m = DINF;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < len; i += gridDim.x * blockDim.x) {
    const uint64_t d = dist[far[i]];
    if (d >= lo && d < m) m = d;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t y = __shfl_xor_sync(LG_FULL_MASK, m, o);
    m = y < m ? y : m;
  }
  if ((threadIdx.x & 31) == 0 && m != DINF) atomicMin(out, (unsigned long long)m);
}

// split the far list at the new bucket [lo, hi): entries inside go to the near
// queue (once per vertex), entries above stay far (once per vertex), entries
// below lo were settled in an earlier bucket and are dropped
__global__ void k_far_split(const uint32_t* far, uint32_t len, const unsigned long long* dist, uint64_t lo,
                            uint64_t hi, uint32_t* near_out, uint32_t* far_out, uint32_t* stamp_near,
                            uint32_t* stamp_far, uint32_t round, uint32_t bucket, uint32_t* near_cnt,
                            uint32_t* far_cnt) {
  const int lane = threadIdx.x & 31;
  for (uint32_t base = blockIdx.x * blockDim.x; base < len; base += gridDim.x * blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    bool tn = false, tf = false;
    uint32_t v = 0;
    if (i < len) {
      v = far[i];
      const uint64_t d = dist[v];
      if (d >= lo && d < hi) tn = atomicExch(stamp_near + v, round) != round;
      else if (d >= hi) tf = atomicExch(stamp_far + v, bucket) != bucket;
    }
    const uint32_t bn = __ballot_sync(LG_FULL_MASK, tn), bf = __ballot_sync(LG_FULL_MASK, tf);
    uint32_t pn = 0, pf = 0;
    if (lane == 0) {
      if (bn) pn = atomicAdd(near_cnt, (uint32_t)__popc(bn));
      if (bf) pf = atomicAdd(far_cnt, (uint32_t)__popc(bf));
    }
    pn = __shfl_sync(LG_FULL_MASK, pn, 0);
    pf = __shfl_sync(LG_FULL_MASK, pf, 0);
    const uint32_t below = lane_lt_mask();
    if (tn) near_out[pn + __popc(bn & below)] = v;
    if (tf) far_out[pf + __popc(bf & below)] = v;
  }
}

__global__ void k_sssp_init(unsigned long long* dist, uint32_t* s_near, uint32_t* s_far, uint64_t n,
                            const uint32_t* perm, uint32_t src, uint32_t* near, uint32_t* src_stored) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x) {
    dist[v] = DINF;
    s_near[v] = 0xffffffffu;
    s_far[v] = 0xffffffffu;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const uint32_t s = perm ? perm[src] : src;
    *src_stored = s;
    near[0] = s;
  }
}

__global__ void k_sssp_seed(unsigned long long* dist, const uint32_t* src_stored) { dist[*src_stored] = 0; }

// distances back to original IDs: out[v] = dist[perm[v]]
__global__ void k_sssp_unpermute(const unsigned long long* dist, const uint32_t* perm, uint64_t n, uint64_t* out) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
    out[v] = dist[perm[v]];
}

template <int IDM, int OFF>
cudaError_t launch_sssp_offsets(const GView& g, uint64_t* x, cudaStream_t st) {
  const uint32_t tile0 = (uint32_t)(g.heavy_prefix / TV);
  k_sssp_offsets<IDM, OFF><<<schedule_tiles_grid(g, tile0), TNT, 0, st>>>(g, x, tile0);
  count_launch();
  return cudaGetLastError();
}

// one round: degree sums, then the relaxation (even a single near vertex can
// be a hub with 10^5 arcs, so every round is balanced by arcs)
template <int IDM>
cudaError_t launch_sssp_relax(const GView& g, const SsspArgs& a, uint64_t* eoff, uint64_t* part, uint32_t* arrived,
                              cudaStream_t st) {
  const unsigned blocks = (a.near_len + SSC_TILE - 1) / SSC_TILE;
  if (blocks > 1) {
    k_sssp_part<<<blocks, 256, 0, st>>>(a, part, arrived);
    count_launch();
  }
  k_sssp_eoff<<<blocks, 256, 0, st>>>(a, blocks > 1 ? part : nullptr, eoff);
  count_launch();
  k_sssp_relax_lb<IDM><<<152 * 4, 256, 0, st>>>(g, a, eoff);
  count_launch();
  return cudaGetLastError();
}

}  // namespace lg

using namespace lg;

namespace {

struct DevBuf {
  void* p = nullptr;
  cudaStream_t st;
  explicit DevBuf(cudaStream_t s) : st(s) {}
  ~DevBuf() {
    if (p) cudaFreeAsync(p, st);
  }
  cudaError_t alloc(size_t b) { return lg::pool_alloc(&p, b, st); }
  template <typename T>
  T* as() const {
    return reinterpret_cast<T*>(p);
  }
};

lg_status fail(const char* what, cudaError_t e) {
  char msg[256];
  snprintf(msg, sizeof msg, "%s: %s", what, cudaGetErrorString(e));
  set_error_message(msg);
  return e == cudaErrorMemoryAllocation ? LG_ENOMEM : LG_ECUDA;
}
#define STRY(call)                                 \
  do {                                             \
    cudaError_t e_ = (call);                       \
    if (e_ != cudaSuccess) return fail(#call, e_); \
  } while (0)

// Bucket width of a call that names none.  In wide buckets arcs are relaxed
// again and again, more the more short arcs a vertex has; narrow ones are a
// round and two reads each.  Measured for weights of 1 .. 255, the best width is
// inverse to the mean degree, as the method's analysis has it (width of the
// order of the largest weight over the degree); at 4096 / degree and its
// neighbors, ms at a quarter / half / taken / twice / four times: 2 M vertices of
// degree 8 3.52 2.62 2.18 2.01 2.47, 1.5 M of 40 2.89 2.79 2.77 4.18 4.64,
// 400,000 of 160 1.93 1.81 1.75 2.37 2.65, of 300 2.10 1.92 1.84 3.00 3.49.
// Where few vertices have most arcs the mean says little (R-MAT 2^18, degree 104:
// 2.14 1.50 1.12 ms in 32, 64, 128): half the largest weight there, and at least
// that below 2^24 arcs, where the rounds take longer than their arcs (3,000
// vertices of degree 2,400: 0.33 ms in 128, 0.41 in 2).
// Other weights scale it (16 bits on R-MAT 2^20: 36 ms in buckets of 128, 1.6 in
// 2^15), but below 8 bits the rounds are so few that narrower ones do not pay
// (4 bits: 0.73 ms in 128, 1.09 in 8).
uint64_t default_delta(const lg_graph* g) {
  const double w = std::max((double)g->max_weight + 1.0, 256.0);
  double width = w / 2;
  if (even_degrees(g) && g->arcs) {
    const double by_degree = 16.0 * w * (double)g->n / (double)g->arcs;
    width = g->arcs >> 24 ? by_degree : std::max(by_degree, width);
  }
  return (uint64_t)1 << (int)std::min(std::max(std::round(std::log2(width)), 0.0), 62.0);
}

}  // namespace

extern "C" lg_status lg_sssp(const lg_graph* g, uint32_t source, uint64_t delta, uint64_t* dist, void* stream) {
  set_error_message("");
  if (!g || !dist) {
    set_error_message("lg_sssp: null argument");
    return LG_EINVAL;
  }
  if (source >= g->n) {
    set_error_message("lg_sssp: source >= n");
    return LG_EINVAL;
  }
  if (!g->weighted) {
    set_error_message("lg_sssp: the graph has no weights (encode with weights, global IDs or CSR-32)");
    return LG_EUNSUPPORTED;
  }
  if (g->id_mode != ID_GLOBAL && g->id_mode != ID_CSR32) {
    set_error_message("lg_sssp: weights exist only in global-ID and CSR-32 graphs");
    return LG_EUNSUPPORTED;
  }
  if (delta == 0) delta = default_delta(g);
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != g->device) cudaSetDevice(g->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const uint64_t n = g->n;
  const GView v = make_view(g);
  lg_status status = LG_OK;
  do {
    // Counters of RING steps are zeroed together: a step takes a pair of them
    // (near queue, far list) and, between buckets, a minimum; no value goes to
    // the device per step.
    constexpr uint32_t RING = 64;
    DevBuf tdist(st), sn(st), sf(st), na(st), nb(st), fa(st), fb(st), small(st), eo(st), tx(st), tpart(st);
    unsigned long long* d = reinterpret_cast<unsigned long long*>(dist);
    if (g->perm) {
      if ((status = tdist.alloc(n * 8) == cudaSuccess ? LG_OK : LG_ENOMEM) != LG_OK) break;
      d = tdist.as<unsigned long long>();
    }
    cudaError_t e = sn.alloc(n * 4 + 16);
    if (e == cudaSuccess) e = sf.alloc(n * 4 + 16);
    if (e == cudaSuccess) e = na.alloc(n * 4 + 16);
    if (e == cudaSuccess) e = nb.alloc(n * 4 + 16);
    if (e == cudaSuccess) e = fa.alloc(n * 4 + 16);
    if (e == cudaSuccess) e = fb.alloc(n * 4 + 16);
    if (e == cudaSuccess) e = small.alloc(32 + RING * 24);
    if (e == cudaSuccess) e = eo.alloc((n + 1) * 8 + 16);
    if (e == cudaSuccess && g->id_mode != ID_CSR32) e = tx.alloc((n + 1) * 8 + 16);
    if (e == cudaSuccess) e = tpart.alloc((n / SSC_TILE + 2) * 8);
    if (e == cudaSuccess) e = cudaMemsetAsync(small.p, 0, 32, st);
    if (e != cudaSuccess) {
      status = fail("lg_sssp: scratch", e);
      break;
    }
    uint32_t* src_stored = small.as<uint32_t>();
    uint32_t* arrived = src_stored + 1;
    unsigned long long* mins = reinterpret_cast<unsigned long long*>(small.as<char>() + 32);  // RING minima
    uint32_t* counts = reinterpret_cast<uint32_t*>(mins + RING);                               // RING pairs
    uint32_t* far_cnt = src_stored + 2;  // the current far list's length
    k_sssp_init<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(d, sn.as<uint32_t>(), sf.as<uint32_t>(), n, g->perm,
                                                            source, na.as<uint32_t>(), src_stored);
    count_launch();
    k_sssp_seed<<<1, 1, 0, st>>>(d, src_stored);
    count_launch();
    e = cudaGetLastError();
    SsspArgs a;
    memset(&a, 0, sizeof(a));
    if (g->id_mode == ID_CSR32) a.x = g->O;  // the row pointer
    else a.x = tx.as<uint64_t>();
    if (e == cudaSuccess && g->id_mode != ID_CSR32)
      e = g->off_mode == OFF_EF ? launch_sssp_offsets<ID_GLOBAL, OFF_EF>(v, tx.as<uint64_t>(), st)
                                : launch_sssp_offsets<ID_GLOBAL, OFF_PACKED>(v, tx.as<uint64_t>(), st);
    if (e != cudaSuccess) {
      status = fail("lg_sssp: init", e);
      break;
    }
    uint32_t* near_in = na.as<uint32_t>();
    uint32_t* near_out = nb.as<uint32_t>();
    uint32_t* far = fa.as<uint32_t>();
    uint32_t* far_alt = fb.as<uint32_t>();
    uint32_t near_len = 1, far_len = 0, round = 0, bucket = 0;
    uint64_t lo = 0, hi = delta;
    uint64_t hmin = 0;
    a.dist = d;
    a.stamp_near = sn.as<uint32_t>();
    a.stamp_far = sf.as<uint32_t>();
    const uint64_t max_steps = 4 * n + 64;  // every step settles or moves work; this only bounds a bug
    uint64_t steps = 0;
    auto read = [&](void* to, const void* from, size_t bytes) {
      cudaError_t r = cudaMemcpyAsync(to, from, bytes, cudaMemcpyDeviceToHost, st);
      return r == cudaSuccess ? cudaStreamSynchronize(st) : r;
    };
    for (;; steps++) {
      if (steps > max_steps) {
        set_error_message("lg_sssp: no progress (internal error)");
        status = LG_ECUDA;
        break;
      }
      const uint32_t slot = (uint32_t)(steps % RING);
      if (slot == 0) {
        // the far list's length may live in the ring: carried over
        if (far_cnt != src_stored + 2) {
          if ((e = cudaMemcpyAsync(src_stored + 2, far_cnt, 4, cudaMemcpyDeviceToDevice, st)) != cudaSuccess) break;
          far_cnt = src_stored + 2;
        }
        if ((e = cudaMemsetAsync(mins, 0xff, RING * 8, st)) != cudaSuccess) break;
        if ((e = cudaMemsetAsync(counts, 0, RING * 16, st)) != cudaSuccess) break;
      }
      uint32_t* c = counts + 4 * slot;  // near queue, far list of a new bucket
      if (near_len) {
        // one round of the current bucket: next near queue into near_out, far appended
        round++;
        a.near_in = near_in;
        a.near_len = near_len;
        a.near_out = near_out;
        a.far = far;
        a.round = round;
        a.bucket = bucket;
        a.hi = hi;
        a.near_cnt = c;
        a.far_cnt = far_cnt;
        uint64_t* eoff = eo.as<uint64_t>();
        e = g->id_mode == ID_CSR32 ? launch_sssp_relax<ID_CSR32>(v, a, eoff, tpart.as<uint64_t>(), arrived, st)
                                   : launch_sssp_relax<ID_GLOBAL>(v, a, eoff, tpart.as<uint64_t>(), arrived, st);
        if (e != cudaSuccess) break;
        if ((e = read(&near_len, c, 4)) != cudaSuccess) break;
        std::swap(near_in, near_out);
        continue;
      }
      // next non-empty bucket: the smallest far distance at or above hi
      if ((e = read(&far_len, far_cnt, 4)) != cudaSuccess) break;
      if (far_len == 0) break;  // done
      k_far_min<<<grid_for(far_len, 256, 152 * 8), 256, 0, st>>>(far, far_len, d, hi, mins + slot);
      count_launch();
      if ((e = cudaGetLastError()) != cudaSuccess) break;
      if ((e = read(&hmin, mins + slot, 8)) != cudaSuccess) break;
      if (hmin == DINF) break;  // every far entry was settled: done
      lo = hmin / delta * delta;
      hi = lo + delta;
      round++;
      bucket++;
      k_far_split<<<grid_for(far_len, 256, 152 * 8), 256, 0, st>>>(far, far_len, d, lo, hi, near_in, far_alt,
                                                                   a.stamp_near, a.stamp_far, round, bucket, c,
                                                                   c + 1);
      count_launch();
      if ((e = cudaGetLastError()) != cudaSuccess) break;
      far_cnt = c + 1;
      if ((e = read(&near_len, c, 4)) != cudaSuccess) break;
      std::swap(far, far_alt);
    }
    if (status == LG_OK && e != cudaSuccess) status = fail("lg_sssp", e);
    if (status == LG_OK && g->perm) {
      k_sssp_unpermute<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(d, g->perm, n, dist);
      count_launch();
      if ((e = cudaGetLastError()) != cudaSuccess) status = fail("lg_sssp: unpermute", e);
    }
    if (status == LG_OK && (e = cudaStreamSynchronize(st)) != cudaSuccess) status = fail("lg_sssp", e);
  } while (0);
  if (prev != g->device) cudaSetDevice(prev);
  return status;
}
