// liblg.so: the C ABI declared in include/lg.h.
//
// The construction follows Listing 3 (Section 6) of the Log(Graph) paper:
// permute (DM, Section 5.6), transform A (Sections 3.2-3.6), build the offsets
// and logarithmize them (Sections 3.4 and 4.3).  getNeighbors, BFS and
// PageRank decode the structure inside their kernels.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "lg_internal.h"
#include "lg_traverse.cuh"

namespace {

thread_local char g_err[768] = "";

void set_errf(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
}

lg_status from_cuda(cudaError_t e, const char* what) {
  set_errf("%s: %s", what, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? LG_ENOMEM : LG_ECUDA;
}

#define LG_TRY(call)                                    \
  do {                                                  \
    cudaError_t e_ = (call);                            \
    if (e_ != cudaSuccess) return from_cuda(e_, #call); \
  } while (0)

// stream-ordered temporary buffer, released (stream-ordered) on scope exit
struct Tmp {
  void* p = nullptr;
  cudaStream_t st;
  explicit Tmp(cudaStream_t s) : st(s) {}
  ~Tmp() {
    if (p) cudaFreeAsync(p, st);
  }
  Tmp(const Tmp&) = delete;
  Tmp& operator=(const Tmp&) = delete;
  cudaError_t alloc(size_t bytes) { return lg::pool_alloc(&p, bytes ? bytes : 16, st); }
  template <typename T> T* as() const { return reinterpret_cast<T*>(p); }
};

struct DeviceGuard {
  int prev = -1;
  bool changed = false;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) {
      cudaSetDevice(dev);
      changed = true;
    }
  }
  ~DeviceGuard() {
    if (changed) cudaSetDevice(prev);
  }
};

lg_status describe_dev_err(int flags) {
  set_errf("invalid input:%s%s%s%s%s%s%s", (flags & lg::DERR_ROWPTR) ? " row_ptr not monotone or out of range;" : "",
           (flags & lg::DERR_COL_RANGE) ? " neighbor id >= n;" : "",
           (flags & lg::DERR_UNSORTED) ? " a row is not strictly increasing;" : "",
           (flags & lg::DERR_WEIGHT) ? " a weight does not fit weight_bits;" : "",
           (flags & lg::DERR_ASYM) ? " an arc has no reverse arc;" : "",
           (flags & lg::DERR_QUERY) ? " a vertex id is >= n;" : "",
           (flags & lg::DERR_INTERNAL) ? " internal invariant failed;" : "");
  return LG_EINVAL;
}

// graph arrays: the bit readers fetch whole 32-byte sectors of them, so a
// block that is not 32-byte aligned is refused (pool blocks are)
cudaError_t alloc_words(uint64_t** p, uint64_t words, cudaStream_t st) {
  cudaError_t e = lg::pool_alloc((void**)p, words * sizeof(uint64_t), st);
  if (e != cudaSuccess) return e;
  if (reinterpret_cast<uintptr_t>(*p) & 31u) {
    cudaFreeAsync(*p, st);
    *p = nullptr;
    return cudaErrorMisalignedAddress;
  }
  return cudaMemsetAsync(*p, 0, words * sizeof(uint64_t), st);
}

// tunables (environment overrides; include/lg.h lists them)
uint32_t env_u32(const char* name, uint32_t dflt) {
  const char* s = getenv(name);
  if (!s || !*s) return dflt;
  return (uint32_t)strtoul(s, nullptr, 10);
}
// Light/heavy degree limit and the split size of the heavy-vertex schedule,
// read at every encode (LG_HEAVY_MIN, LG_HEAVY_SEG).
uint32_t heavy_min_env() {
  const uint32_t v = env_u32("LG_HEAVY_MIN", 256);
  return v == 0 ? 256 : v > lg::PW_HEAVY_MAX ? lg::PW_HEAVY_MAX : v;
}
uint32_t heavy_seg_env() {
  const uint32_t v = env_u32("LG_HEAVY_SEG", 4096);
  return v >= 32 ? v : 4096;
}
uint32_t pull_divisor() {
  static const uint32_t v = env_u32("LG_BFS_PULL_DIV", 64);
  return v ? v : 64;
}

}  // namespace

#include <atomic>
#include <mutex>

namespace lg {

static std::atomic<unsigned long long> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

// One pool per device, created on first use, release threshold unlimited:
// repeated encodes, traversals and frees reuse mapped memory instead of
// mapping and unmapping gigabytes per call.
static std::mutex g_pool_mu;
static cudaMemPool_t g_pools[64] = {};

static cudaError_t device_pool(int dev, cudaMemPool_t* out) {
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (!g_pools[dev]) {
    cudaMemPoolProps props;
    memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    uint64_t keep = UINT64_MAX;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(pool);
      return e;
    }
    g_pools[dev] = pool;
  }
  *out = g_pools[dev];
  return cudaSuccess;
}

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  cudaMemPool_t pool = nullptr;
  if (e == cudaSuccess) e = device_pool(dev, &pool);
  if (e != cudaSuccess) return e;
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

void set_error_message(const char* msg) { snprintf(g_err, sizeof g_err, "%s", msg); }

GView make_view(const lg_graph* g) {
  GView v;
  memset(&v, 0, sizeof(v));
  v.A32 = reinterpret_cast<const uint32_t*>(g->A);
  v.A64 = g->A;
  v.O = g->O;
  v.ef_low = g->ef_low;
  v.ef_high32 = reinterpret_cast<const uint32_t*>(g->ef_high);
  v.ef_samples = g->ef_samples;
  v.perm = g->perm;
  v.inv_perm = g->inv_perm;
  v.W32 = g->W;
  v.n = g->n;
  v.arcs = g->arcs;
  v.ef_high_words32 = (g->ef_high_bits + 31) / 32;
  v.s = g->s; v.H = g->H; v.omega = g->omega; v.r = g->r; v.w_O = g->w_O; v.ef_l = g->ef_l;
  v.sample_log2 = g->sample_log2;
  v.items = g->items;
  v.multi = g->multi;
  v.n_items = g->n_items;
  v.n_multi = g->n_multi;
  v.heavy_min = g->heavy_min;
  v.heavy_seg = g->heavy_seg;
  v.max_degree = (uint32_t)g->max_degree;
  v.heavy_prefix = g->heavy_prefix;
  v.mid_prefix = g->mid_prefix;
  return v;
}

// ---------------------------------------------------------------- split vertices
// A vertex split into several heavy items: its items' partial sums are added
// in item order (deterministic), then the vertex is finished.
__global__ void k_ppr_finish_multi(GView g, PprArgs a) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < g.n_multi; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t first = g.multi[i];
    const HeavyItem h = g.items[first];
    float s[PPR_K];
    for (int k = 0; k < PPR_K; k++) s[k] = 0.f;
    for (uint32_t j = 0; j < h.nitems; j++)
      for (int k = 0; k < PPR_K; k++) s[k] += a.part[(uint64_t)(first + j) * PPR_K + k];
    ppr_finish(a, h.v, h.deg, s);
  }
}

cudaError_t ppr_finish_multi(const GView& g, const PprArgs& a, cudaStream_t st) {
  if (g.n_multi == 0) return cudaSuccess;
  k_ppr_finish_multi<<<grid_for(g.n_multi, 256, 4096), 256, 0, st>>>(g, a);
  count_launch();
  return cudaGetLastError();
}

// carries of split gap-coded vertices: exclusive sums of the item sums, in order
__global__ void k_plan_carry_scan(HeavyItem* items, const uint32_t* multi, uint64_t n_multi, const uint32_t* segsum) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_multi; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t first = multi[i];
    const uint32_t k = items[first].nitems;
    uint32_t run = 0;
    for (uint32_t j = 0; j < k; j++) {
      items[first + j].carry = run;
      run += segsum[first + j];
    }
  }
}

cudaError_t plan_carry_scan(HeavyItem* items, const uint32_t* multi, uint64_t n_multi, const uint32_t* segsum,
                            cudaStream_t st) {
  if (n_multi == 0) return cudaSuccess;
  k_plan_carry_scan<<<grid_for(n_multi, 256, 4096), 256, 0, st>>>(items, multi, n_multi, segsum);
  count_launch();
  return cudaGetLastError();
}

const TravOps* trav_ops(int id_mode, int off_mode) {
  if (id_mode == ID_CSR32) return trav_ops_csr32();
  if (id_mode == ID_GLOBAL) return off_mode == OFF_EF ? trav_ops_global_ef() : trav_ops_global_packed();
  if (id_mode == ID_LOCAL) return off_mode == OFF_EF ? trav_ops_local_ef() : trav_ops_local_packed();
  return off_mode == OFF_EF ? trav_ops_gap_ef() : trav_ops_gap_packed();
}

// ---------------------------------------------------------------- small kernels
// Start of a sweep: a thread per source (at most 64) checks and maps it, sets
// its bit in the masks and queues its vertex once.  Nothing but scratch is
// written, so a bad source leaves the caller's arrays as they were.
template <typename M>
__global__ void __launch_bounds__(64) k_bfs_start(M* vis, M* front, uint64_t n, const uint32_t* src,
                                                  const uint32_t* perm, uint32_t S, uint32_t* stored, uint32_t* queue,
                                                  uint32_t* count, int* err) {
  const uint32_t i = threadIdx.x;
  if (i >= S) return;
  if (src[i] >= n) { set_err(err, DERR_QUERY); return; }
  const uint32_t v = perm ? perm[src[i]] : src[i];
  const M bit = (M)((M)1 << i);
  stored[i] = v;
  atomic_or_mask<M>(vis + v, bit);
  if (atomic_or_mask<M>(front + v, bit) == 0) queue[atomicAdd(count, 1u)] = v;
}
__global__ void k_bfs_depth0(uint32_t* depth, uint64_t n, const uint32_t* stored, uint32_t S, uint32_t vmajor) {
  const uint32_t i = threadIdx.x;
  if (i < S) depth[vmajor ? (uint64_t)stored[i] * S + i : (uint64_t)i * n + stored[i]] = 0;
}

// zero the mask entries listed in a queue (the nonzeros of a frontier)
__global__ void k_clear_queue(uint8_t* masks, int mb, const uint32_t* queue, uint32_t len) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < len; i += gridDim.x * blockDim.x) {
    uint8_t* p = masks + (uint64_t)queue[i] * mb;
    if (mb == 2) *reinterpret_cast<uint16_t*>(p) = 0;
    else if (mb == 4) *reinterpret_cast<uint32_t*>(p) = 0;
    else *reinterpret_cast<uint64_t*>(p) = 0;
  }
}

// out[s][o] = tmp[perm[o]][s]: the relabeled depths are one record of S
// values per vertex, so a thread gathers the record of perm[o] (16-byte loads
// when S is a multiple of 4) and writes its S values, each store coalesced
// over the warp's consecutive o
template <bool VEC>
__global__ void __launch_bounds__(256) k_permute_depths(const uint32_t* __restrict__ tmp, uint32_t* __restrict__ out,
                                                        const uint32_t* __restrict__ perm, uint64_t n, uint32_t S) {
  for (uint64_t o = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t p = perm[o];
    if (VEC) {
      const uint4* rec = reinterpret_cast<const uint4*>(tmp + p * S);
      for (uint32_t q = 0; q < S / 4; q++) {
        const uint4 x = __ldg(rec + q);
        __stcs(out + (uint64_t)(4 * q) * n + o, x.x);
        __stcs(out + (uint64_t)(4 * q + 1) * n + o, x.y);
        __stcs(out + (uint64_t)(4 * q + 2) * n + o, x.z);
        __stcs(out + (uint64_t)(4 * q + 3) * n + o, x.w);
      }
    } else {
      for (uint32_t s = 0; s < S; s++) __stcs(out + (uint64_t)s * n + o, __ldg(tmp + p * S + s));
    }
  }
}

cudaError_t bfs_permute_depths(const uint32_t* tmp, uint32_t* out, const uint32_t* perm, uint64_t n, uint32_t S,
                               cudaStream_t st) {
  if (S % 4 == 0) k_permute_depths<true><<<grid_for(n, 256, 152 * 16), 256, 0, st>>>(tmp, out, perm, n, S);
  else k_permute_depths<false><<<grid_for(n, 256, 152 * 16), 256, 0, st>>>(tmp, out, perm, n, S);
  count_launch();
  return cudaGetLastError();
}

// stored labels of caller ids (perm may be null), with a range check
__global__ void k_map_ids(const uint32_t* __restrict__ in, uint32_t* __restrict__ out,
                          const uint32_t* __restrict__ perm, uint64_t k, uint64_t n, int* err) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = in[i];
    if (v >= n) { set_err(err, DERR_QUERY); out[i] = 0; continue; }
    out[i] = perm ? perm[v] : v;
  }
}

cudaError_t map_ids(const uint32_t* in, uint32_t* out, const uint32_t* perm, uint64_t k, uint64_t n, int* err,
                    cudaStream_t st) {
  if (k == 0) return cudaSuccess;
  k_map_ids<<<grid_for(k, 256, 4096), 256, 0, st>>>(in, out, perm, k, n, err);
  count_launch();
  return cudaGetLastError();
}

// r_0 written straight to the output (zero iterations)
__global__ void k_pr_fill0(float* ranks, uint64_t n, float r0, int64_t personal_orig) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
    ranks[v] = personal_orig < 0 ? r0 : ((int64_t)v == personal_orig ? 1.0f : 0.0f);
}

uint32_t hot_rows(const lg_graph* g, uint32_t elem_bytes) {
  const uint64_t all = g->n < 0xffffffffull ? g->n : 0xffffffffull;
  if (g->relabel != 1 || elem_bytes == 0) return (uint32_t)all;
  const char* e = getenv("LG_HOT_BYTES");  // read per traversal: a few ns
  const uint64_t bytes = (e && *e) ? (uint64_t)strtoull(e, nullptr, 10) : (64ull << 20);
  const uint64_t rows = bytes / elem_bytes;
  return (uint32_t)(rows < all ? rows : all);
}

// no degree far above the mean
bool even_degrees(const lg_graph* g) { return g->max_degree * g->n <= 4 * g->arcs; }

// Warp tiles hold 128 vertices, but fewer where that would make a long unit: in
// a small graph (fewer than two tiles of 128 per resident warp), and for the
// DM-ordered vertices of more than 32 arcs (a warp walks 256 fields in about
// 2 us, so 128 x 256 fields ran 250 us on one warp).  The smaller tiles trade
// the tile's own cost against the longest unit; measured per sweep at 4 / 8 /
// 16 / 32 vertices: R-MAT 2^12 in DM order 8 / 10 / 13 / 19 us, community 2^15
// 25 / 26 / 34 / 54, community 2^18 in DM order 133 / 80 / 58 / 80, R-MAT 2^18
// not relabeled 110 / 72 / 53 / 47, R-MAT 900,000 287 / 173 / 114 / 85; but
// tiles of too few fields are all cost.  Where
// no degree is above four times the mean, no unit is long for its size, and
// tiles are as large as leaves one for every second warp: 5 M vertices of
// degree 40 in DM order, local-gap IDs, 1.02 ms in tiles of 32, 0.90 in 128,
// 300,000 of degree 40 86 and 76 us.  Such a graph's heavy items, short ones,
// come after its tiles (1 M vertices of degree 250, 35 % of them heavy: 1.27 ms
// with the items first, 1.12 so), several to a ticket.  Tiles start right after
// the vertices that are all in the schedule: one that held a few hubs would have
// a warp search their Elias-Fano block alone (ten hubs of 200,000 arcs among
// 500,000 vertices: 156 us a sweep, 32 so).
//
// The shared-memory table of contributions pays when it answers some of the
// gathers of a sweep that is long enough to fill it (R-MAT 2^24 in DM order,
// 28 % of the arcs on the first 16,384 labels: 1.78 -> 1.61 ms a sweep;
// community 2^23, 9 %: 0.94 -> 0.91; 2^24, 6 %: equal; R-MAT 2^18, 76 %: 41 ->
// 43 us).  Without it the L1 answers some too, and on a small graph more, unless
// its hubs take a third of the arcs and it is not that small: degree 1,600, 40,000 vertices 147 us with
// the table, 83 without, 100,000 of 1,000 294 and 269, 200,000 of 500 348 and
// 368; R-MAT 2^17 in DM order 46 and 49, not relabeled 75 and 69.
PrPlan pr_plan(const lg_graph* g) {
  PrPlan p;
  const uint64_t warps = (uint64_t)PW_WARPS * PW_SMS;
  const bool small = g->n < 2 * warps * PW_TV;
  const bool even = even_degrees(g);
  p.tile_a = g->heavy_prefix;
  uint64_t end = small || even ? g->n : g->mid_prefix > p.tile_a ? g->mid_prefix : p.tile_a;
  if (even) {
    p.tile_nv = 2 * g->heavy_arcs > g->arcs ? 32 : 4;  // tiles of next to no light fields are not worth splitting
    while (p.tile_nv < PW_TV && g->n / (2 * p.tile_nv) >= warps / 2) p.tile_nv *= 2;
  } else {
    p.tile_nv = g->n < (1u << 14) ? 4 : g->n < (1u << 16) ? 8 : g->n < (1u << 19) && g->relabel == 1 ? 16 : 32;
    // 512 light fields a tile on the average, if there are two tiles per warp
    while (p.tile_nv < PW_TV && 2 * p.tile_nv * (g->arcs - g->heavy_arcs) <= 512 * g->n && g->n / (2 * p.tile_nv) >= 2 * warps)
      p.tile_nv *= 2;
  }
  p.tile_b = p.tile_a + ((end > p.tile_a ? end - p.tile_a : 0) + PW_TV - 1) / PW_TV * PW_TV;
  p.items = 1;  // short ones share a ticket as long as there are eight for every warp
  while (g->n_items / (2 * p.items) >= 8 * warps && (even || g->heavy_arcs <= 512 * g->n_items)) p.items *= 2;
  const uint64_t most = (PW_SMEM - PW_WARPS * sizeof(PrWarp)) / sizeof(float);
  const bool table = g->n >= 3u << 16 ? 12 * g->top_arcs >= g->arcs : g->n >= 1u << 17 && 3 * g->top_arcs >= g->arcs;
  p.tabn = g->arcs >> 24 && table ? (uint32_t)(g->n < most ? g->n : most) : 0;
  p.part_floats = g->n_multi ? g->n_items : 0;
  p.sync_words = 2 + g->n_multi;
  p.aux_words = g->off_mode == OFF_EF ? (p.tile_b - p.tile_a) / p.tile_nv + g->n / PW_TV + 1 : 0;
  return p;
}

cudaError_t pr_fill0(float* ranks, uint64_t n, int64_t personal_orig, cudaStream_t st) {
  k_pr_fill0<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(ranks, n, 1.0f / (float)n, personal_orig);
  count_launch();
  return cudaGetLastError();
}

}  // namespace lg

using namespace lg;

// =========================================================================
// C ABI
// =========================================================================
extern "C" const char* lg_last_error(void) { return g_err; }

extern "C" uint64_t lg_kernel_launches(void) { return (uint64_t)g_launches.load(std::memory_order_relaxed); }

extern "C" void lg_free(lg_graph* g) {
  if (!g) return;
  DeviceGuard dg(g->device);
  // nothing still uses g once the device is idle; the blocks go back to the
  // pool (they stay mapped for the next graph)
  cudaDeviceSynchronize();
  void* bufs[] = {g->A, g->O, g->ef_low, g->ef_high, g->ef_samples, g->perm, g->inv_perm, g->W, g->items, g->multi};
  for (void* p : bufs)
    if (p) cudaFreeAsync(p, cudaStreamLegacy);
  delete g;
}

extern "C" lg_status lg_decode(const lg_graph* g, uint64_t* row_ptr, uint32_t* col, uint32_t* weights,
                               uint64_t capacity, void* stream) {
  g_err[0] = 0;
  if (!g || !row_ptr || (g->arcs && !col)) { set_errf("lg_decode: null argument"); return LG_EINVAL; }
  if (weights && !g->weighted) { set_errf("lg_decode: weights requested from an unweighted graph"); return LG_EINVAL; }
  if (capacity < g->arcs) {
    set_errf("lg_decode: capacity %llu < %llu arcs", (unsigned long long)capacity, (unsigned long long)g->arcs);
    return LG_ERANGE;
  }
  DeviceGuard dg(g->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const uint64_t n = g->n;
  if (n == 0) {
    LG_TRY(cudaMemsetAsync(row_ptr, 0, sizeof(uint64_t), st));
    return LG_OK;
  }
  const GView v = make_view(g);
  const TravOps* ops = trav_ops((int)g->id_mode, (int)g->off_mode);
  DecArgs a;
  memset(&a, 0, sizeof(a));
  a.row_ptr = row_ptr;
  a.ids = col;
  a.weights = weights;
  if (g->id_mode == ID_GLOBAL || g->id_mode == ID_CSR32) {
    // records are in arc order: the offsets are the row offsets (one launch
    // writes both)
    a.row_out = row_ptr;
    LG_TRY(ops->dec_all(v, a, st));
    return LG_OK;
  }
  // local IDs: one launch (row offsets by a single-pass look-back over the
  // tiles, then the rows); its small state is zeroed first
  const bool even = even_degrees(g);
  dec_tiles(n, v.mid_prefix, even, a);
  a.heavy_after = 3 * g->heavy_arcs >= 2 * g->arcs;
  const uint64_t ntiles = a.tiles;
  Tmp t_state(st);
  const size_t bytes = ntiles * (sizeof(unsigned long long) + sizeof(uint32_t)) + 16;
  LG_TRY(t_state.alloc(bytes));
  LG_TRY(cudaMemsetAsync(t_state.p, 0, bytes, st));
  a.tile_status = t_state.as<unsigned long long>();
  a.tile_ready = reinterpret_cast<uint32_t*>(a.tile_status + ntiles);
  a.ticket = a.tile_ready + ntiles;
  a.err = reinterpret_cast<int*>(a.ticket + 1);
  a.row_out = row_ptr;
  a.wait_ns = 200ull * 1000 * 1000;
  LG_TRY(ops->dec_all(v, a, st));
  int err = 0;
  LG_TRY(cudaMemcpyAsync(&err, a.err, sizeof(int), cudaMemcpyDeviceToHost, st));
  LG_TRY(cudaStreamSynchronize(st));
  if (err) {
    set_errf("lg_decode: a wait between the decode's blocks ran out (row offsets incomplete)");
    return LG_ETIMEOUT;
  }
  return LG_OK;
}

extern "C" lg_status lg_free_async(lg_graph* g, void* stream) {
  g_err[0] = 0;
  if (!g) return LG_OK;
  DeviceGuard dg(g->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t first = cudaSuccess;
  void* bufs[] = {g->A, g->O, g->ef_low, g->ef_high, g->ef_samples, g->perm, g->inv_perm, g->W, g->items, g->multi};
  for (void* p : bufs) {
    if (!p) continue;
    const cudaError_t e = cudaFreeAsync(p, st);
    if (first == cudaSuccess) first = e;
  }
  delete g;
  if (first != cudaSuccess) return from_cuda(first, "lg_free_async");
  return LG_OK;
}

extern "C" lg_status lg_pool_trim(int device, uint64_t keep_bytes) {
  g_err[0] = 0;
  cudaMemPool_t pool = nullptr;
  LG_TRY(device_pool(device, &pool));
  DeviceGuard dg(device);
  LG_TRY(cudaDeviceSynchronize());
  LG_TRY(cudaMemPoolTrimTo(pool, (size_t)keep_bytes));
  return LG_OK;
}

extern "C" lg_status lg_pool_usage(int device, uint64_t* reserved, uint64_t* used) {
  g_err[0] = 0;
  if (!reserved || !used) { set_errf("lg_pool_usage: null argument"); return LG_EINVAL; }
  cudaMemPool_t pool = nullptr;
  LG_TRY(device_pool(device, &pool));
  unsigned long long r = 0, u = 0;
  LG_TRY(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &r));
  LG_TRY(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &u));
  *reserved = (uint64_t)r;
  *used = (uint64_t)u;
  return LG_OK;
}

extern "C" lg_status lg_stats_get(const lg_graph* g, lg_stats* out) {
  g_err[0] = 0;
  if (!g || !out) { set_errf("lg_stats_get: null argument"); return LG_EINVAL; }
  memset(out, 0, sizeof(*out));
  out->n = g->n; out->arcs = g->arcs;
  out->bits_A = g->bits_A; out->bits_O = g->bits_O;
  out->bytes_A = g->words_A * 8;
  out->bytes_O = (g->words_O + g->words_ef_low + g->words_ef_high + g->words_ef_samples) * 8;
  out->bytes_perm = g->perm ? 2 * g->n * sizeof(uint32_t) : 0;
  out->bytes_schedule = g->n_items * sizeof(HeavyItem) + g->n_multi * sizeof(uint32_t);
  out->bytes_total = out->bytes_A + out->bytes_O + out->bytes_perm + out->bytes_schedule + (g->W ? g->arcs * 4 : 0);
  out->max_degree = g->max_degree;
  out->id_mode = g->id_mode; out->off_mode = g->off_mode; out->relabel = g->relabel; out->weighted = g->weighted;
  out->s = g->s; out->H = g->H; out->omega = g->omega; out->w_O = g->w_O; out->ef_l = g->ef_l;
  out->select_sample = g->sample;
  out->bits_per_arc = g->arcs ? (double)(g->bits_A + g->bits_O) / (double)g->arcs : 0.0;
  return LG_OK;
}

extern "C" lg_status lg_arrays_get(const lg_graph* g, lg_arrays* out) {
  g_err[0] = 0;
  if (!g || !out) { set_errf("lg_arrays_get: null argument"); return LG_EINVAL; }
  out->A = g->A; out->words_A = g->words_A;
  out->O = g->O; out->words_O = g->words_O;
  out->ef_low = g->ef_low; out->words_ef_low = g->words_ef_low;
  out->ef_high = g->ef_high; out->words_ef_high = g->words_ef_high;
  out->ef_samples = g->ef_samples; out->words_ef_samples = g->words_ef_samples;
  out->perm = g->perm; out->inv_perm = g->inv_perm;
  return LG_OK;
}

// Heavy-vertex schedule, derived from the encoded A and the plain offsets x_0 ..
// x_n (decoding them again cost 1.5 ms at R-MAT 2^26: the hubs' Elias-Fano
// block is 200,000 words long): every vertex of degree > heavy_min becomes
// ceil(d / HEAVY_SEG) items, listed in vertex order.
static lg_status build_schedule(lg_graph* g, const uint64_t* x, cudaStream_t st) {
  g->heavy_min = heavy_min_env();
  g->heavy_seg = heavy_seg_env();
  const uint64_t ntiles = (g->n + LG_TILE_V - 1) / LG_TILE_V;
  // counts of items, then of split vertices, per tile, scanned together
  Tmp t_cnt(st), t_off(st), t_stmp(st), t_seg(st);
  struct { uint64_t end; unsigned long long top, heavy; uint32_t mid, pad; } sums;  // end: of the scan
  LG_TRY(t_cnt.alloc(2 * ntiles * sizeof(uint32_t)));
  LG_TRY(t_off.alloc(2 * ntiles * sizeof(uint64_t) + sizeof(sums)));
  LG_TRY(t_stmp.alloc(scan_tmp_words(2 * ntiles) * sizeof(uint64_t)));
  uint64_t* off = t_off.as<uint64_t>();
  LG_TRY(cudaMemsetAsync(off + 2 * ntiles, 0, sizeof(sums), st));
  PlanArgs p;
  memset(&p, 0, sizeof(p));
  p.tile_count = t_cnt.as<uint32_t>();
  p.multi_count = p.tile_count + ntiles;
  p.tile_off = off;
  p.multi_off = off + ntiles;  // behind all items
  p.top = reinterpret_cast<unsigned long long*>(off + 2 * ntiles + 1);
  p.heavy = p.top + 1;
  p.mid = g->relabel == 1 ? reinterpret_cast<uint32_t*>(p.heavy + 1) : nullptr;
  GView v = make_view(g);
  v.O = x;
  const TravOps* ops = trav_ops((int)g->id_mode, (int)g->off_mode);
  LG_TRY(ops->plan_count(v, p, st));
  LG_TRY(scan_excl_u32(p.tile_count, 2 * ntiles, off, t_stmp.as<uint64_t>(), st));
  LG_TRY(cudaMemcpyAsync(&g->n_items, off + ntiles, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
  LG_TRY(cudaMemcpyAsync(&sums, off + 2 * ntiles, sizeof(sums), cudaMemcpyDeviceToHost, st));
  LG_TRY(cudaStreamSynchronize(st));
  g->n_multi = sums.end - g->n_items;
  g->heavy_prefix = 0;
  g->mid_prefix = g->relabel == 1 ? sums.mid : 0;
  g->top_arcs = sums.top;
  g->heavy_arcs = sums.heavy;
  if (g->n_items == 0) return LG_OK;
  LG_TRY(pool_alloc((void**)&g->items, g->n_items * sizeof(HeavyItem), st));
  if (g->n_multi) LG_TRY(pool_alloc((void**)&g->multi, g->n_multi * sizeof(uint32_t), st));
  p.items = g->items;
  p.multi = g->multi;
  LG_TRY(ops->plan_fill(v, p, st));
  if (g->n_multi && g->id_mode == ID_LOCAL_GAP) {
    LG_TRY(t_seg.alloc(g->n_items * sizeof(uint32_t)));
    p.segsum = t_seg.as<uint32_t>();
    v = make_view(g);
    LG_TRY(ops->plan_carry(v, p, st));
    LG_TRY(plan_carry_scan(g->items, g->multi, g->n_multi, p.segsum, st));
  }
  HeavyItem last;
  if (g->relabel == 1)  // degrees descend: every vertex up to the last item's is heavy
    LG_TRY(cudaMemcpyAsync(&last, g->items + g->n_items - 1, sizeof(last), cudaMemcpyDeviceToHost, st));
  LG_TRY(cudaStreamSynchronize(st));
  if (g->relabel == 1) g->heavy_prefix = (uint64_t)last.v + 1;
  return LG_OK;
}

static lg_status encode_impl(lg_graph* g, const uint64_t* row_ptr, const uint32_t* col, const uint32_t* weights,
                             const lg_encode_opts& o, cudaStream_t st) {
  const uint64_t n = g->n, arcs = g->arcs;
  // ---- validation (one pass; device flag, never traps)
  Tmp small(st);
  LG_TRY(small.alloc(64));
  int* d_err = small.as<int>();
  unsigned long long* d_maxdeg = reinterpret_cast<unsigned long long*>(small.as<char>() + 8);
  uint32_t* d_maxw = reinterpret_cast<uint32_t*>(small.as<char>() + 16);
  LG_TRY(cudaMemsetAsync(small.p, 0, 64, st));
  LG_TRY(enc_validate(row_ptr, col, weights, n, arcs, o.weight_bits, d_err, d_maxdeg, d_maxw, st));
  struct { int err; int pad; unsigned long long maxdeg; uint32_t maxw; } h{};
  LG_TRY(cudaMemcpyAsync(&h, small.p, 20, cudaMemcpyDeviceToHost, st));
  LG_TRY(cudaStreamSynchronize(st));
  if (h.err) return describe_dev_err(h.err);
  if (o.flags & LG_FLAG_CHECK_SYMMETRIC) {
    LG_TRY(enc_check_symmetric(row_ptr, col, n, d_err, st));
    LG_TRY(cudaMemcpyAsync(&h.err, d_err, 4, cudaMemcpyDeviceToHost, st));
    LG_TRY(cudaStreamSynchronize(st));
    if (h.err) return describe_dev_err(h.err);
  }
  g->max_degree = h.maxdeg;

  // ---- widths (Sections 3.2.1, 3.3)
  g->s = host_bits(n - 1);
  if (g->s < 1) g->s = 1;
  g->H = host_bits(g->s);
  g->omega = 0;
  if (weights) {
    g->max_weight = h.maxw;
    g->omega = o.weight_bits ? o.weight_bits : host_bits(h.maxw);
    if (g->omega < 1) g->omega = 1;
  }
  g->r = g->s + g->omega;

  // ---- optional relabel: DM (Section 5.6) or the greedy heuristic (Listing 1)
  const uint64_t* rp = row_ptr;
  const uint32_t* cl = col;
  const uint32_t* wt = weights;
  Tmp t_nrp(st), t_ncol(st), t_nw(st);
  if (g->relabel) {
    LG_TRY(pool_alloc((void**)&g->perm, n * sizeof(uint32_t), st));
    LG_TRY(pool_alloc((void**)&g->inv_perm, n * sizeof(uint32_t), st));
    LG_TRY(t_nrp.alloc((n + 1) * sizeof(uint64_t)));
    LG_TRY(t_ncol.alloc(arcs * sizeof(uint32_t)));
    if (weights) LG_TRY(t_nw.alloc(arcs * sizeof(uint32_t)));
    LG_TRY(enc_dm_relabel(row_ptr, col, weights, n, arcs, g->max_degree, g->relabel, g->perm, g->inv_perm,
                          t_nrp.as<uint64_t>(),
                          t_ncol.as<uint32_t>(), weights ? t_nw.as<uint32_t>() : nullptr, st));
    rp = t_nrp.as<uint64_t>();
    cl = t_ncol.as<uint32_t>();
    wt = weights ? t_nw.as<uint32_t>() : nullptr;
  }

  // ---- uncompressed baseline: copy the (possibly relabeled) CSR
  if (g->id_mode == ID_CSR32) {
    g->bits_A = 32 * arcs;
    g->words_A = padded_words(g->bits_A);
    LG_TRY(alloc_words(&g->A, g->words_A, st));
    if (arcs) LG_TRY(cudaMemcpyAsync(g->A, cl, arcs * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st));
    g->bits_O = 64 * (n + 1);
    g->words_O = padded_words(g->bits_O);
    LG_TRY(alloc_words(&g->O, g->words_O, st));
    LG_TRY(cudaMemcpyAsync(g->O, rp, (n + 1) * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    if (wt) {
      LG_TRY(pool_alloc((void**)&g->W, (arcs ? arcs : 1) * sizeof(uint32_t), st));
      if (arcs) LG_TRY(cudaMemcpyAsync(g->W, wt, arcs * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st));
    }
    g->off_mode = OFF_ROWPTR;
    return build_schedule(g, rp, st);
  }

  // ---- A stream
  const uint64_t* xsrc = rp;  // offsets x_0..x_n: record index (global) or bit (local)
  uint64_t U = arcs;
  Tmp t_wid(st), t_len(st), t_x(st), t_stmp(st);
  if (g->id_mode == ID_GLOBAL) {
    g->bits_A = arcs * g->r;
    g->words_A = padded_words(g->bits_A);
    LG_TRY(alloc_words(&g->A, g->words_A, st));
    LG_TRY(enc_pack_global(cl, wt, arcs, g->s, g->omega, g->A, (g->bits_A + 63) / 64, st));
  } else {
    const int gap = g->id_mode == ID_LOCAL_GAP;
    LG_TRY(t_wid.alloc(n));
    LG_TRY(t_len.alloc(n * sizeof(uint64_t)));
    LG_TRY(t_x.alloc((n + 1) * sizeof(uint64_t)));
    LG_TRY(t_stmp.alloc(scan_tmp_words(n) * sizeof(uint64_t)));
    Tmp t_long(st);
    LongRows rows, *L = nullptr;
    const bool alike = even_degrees(g) && g->max_degree <= LONG_WINDOW && n >= 32ull * 152 * 16;
    if (g->max_degree > LONG_ROW && !alike) {
      LG_TRY(t_long.alloc(long_rows_bytes(arcs)));
      rows = long_rows(t_long.p, arcs);
      L = &rows;
      LG_TRY(enc_long_rows(rp, n, gap, rows, st));
    }
    LG_TRY(enc_local_lengths(rp, cl, n, gap, g->s, g->H, t_wid.as<uint8_t>(), t_len.as<uint64_t>(), L, st));
    LG_TRY(scan_excl_u64(t_len.as<uint64_t>(), n, t_x.as<uint64_t>(), t_stmp.as<uint64_t>(), st));
    LG_TRY(cudaMemcpyAsync(&U, t_x.as<uint64_t>() + n, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    LG_TRY(cudaStreamSynchronize(st));
    g->bits_A = U;
    g->words_A = padded_words(g->bits_A);
    LG_TRY(alloc_words(&g->A, g->words_A, st));
    LG_TRY(enc_pack_local(rp, cl, t_x.as<uint64_t>(), t_wid.as<uint8_t>(), n, gap, g->s, g->H, g->A,
                          (g->bits_A + 63) / 64, L, st));
    xsrc = t_x.as<uint64_t>();
  }

  // ---- offsets (Section 3.4 packed, Section 4.3 Elias-Fano)
  if (g->off_mode == OFF_PACKED) {
    g->w_O = host_bits(U);
    if (g->w_O < 1) g->w_O = 1;
    g->bits_O = (n + 1) * (uint64_t)g->w_O;
    g->words_O = padded_words(g->bits_O);
    LG_TRY(alloc_words(&g->O, g->words_O, st));
    LG_TRY(enc_pack_u64(xsrc, n + 1, g->w_O, g->O, (g->bits_O + 63) / 64, st));
  } else {
    const uint64_t N = n + 1, q = U / N;
    g->ef_N = N; g->ef_U = U;
    g->ef_l = q ? host_bits(q) - 1 : 0;
    g->ef_low_bits = N * (uint64_t)g->ef_l;
    g->ef_high_bits = N + (U >> g->ef_l) + 1;
    g->n_samples = (N + g->sample - 1) / g->sample;
    g->words_ef_low = padded_words(g->ef_low_bits);
    g->words_ef_high = padded_words(g->ef_high_bits);
    g->words_ef_samples = padded_words(64 * g->n_samples);
    LG_TRY(alloc_words(&g->ef_low, g->words_ef_low, st));
    LG_TRY(alloc_words(&g->ef_high, g->words_ef_high, st));
    LG_TRY(alloc_words(&g->ef_samples, g->words_ef_samples, st));
    if (g->ef_l) LG_TRY(enc_pack_u64(xsrc, N, g->ef_l, g->ef_low, (g->ef_low_bits + 63) / 64, st));
    LG_TRY(enc_ef_high(xsrc, N, g->ef_l, g->ef_high, st));
    LG_TRY(enc_ef_samples(xsrc, N, g->ef_l, g->sample, g->ef_samples, g->n_samples, st));
    g->bits_O = g->ef_low_bits + g->ef_high_bits + 64 * g->n_samples;
  }
  return build_schedule(g, xsrc, st);
}

extern "C" lg_status lg_encode(const uint64_t* row_ptr, const uint32_t* col, const uint32_t* weights, uint64_t n,
                               uint64_t arcs, const lg_encode_opts* opts, void* stream, lg_graph** out) {
  g_err[0] = 0;
  if (!out) { set_errf("lg_encode: out is NULL"); return LG_EINVAL; }
  *out = nullptr;
  if (!row_ptr || (arcs && !col)) { set_errf("lg_encode: row_ptr/col is NULL"); return LG_EINVAL; }
  if (n == 0 || n > 0xffffffffull) { set_errf("lg_encode: n must be in [1, 2^32-1], got %llu", (unsigned long long)n); return LG_EINVAL; }
  if (arcs > 0xffffffffull * 0xffffull) { set_errf("lg_encode: arcs too large"); return LG_EINVAL; }
  lg_encode_opts o = {LG_ID_GLOBAL, LG_OFF_PACKED, 0, 512, 0, 0};
  if (opts) o = *opts;
  if (o.select_sample == 0) o.select_sample = 512;
  if (o.id_mode > LG_ID_CSR32 || o.off_mode > LG_OFF_EF) { set_errf("lg_encode: unknown id_mode/off_mode"); return LG_EINVAL; }
  if (o.select_sample < 64 || o.select_sample > 65536 || (o.select_sample & (o.select_sample - 1))) {
    set_errf("lg_encode: select_sample must be a power of two in [64, 65536]");
    return LG_EINVAL;
  }
  if (o.weight_bits > 32) { set_errf("lg_encode: weight_bits must be <= 32"); return LG_EINVAL; }
  if (o.relabel > 2) { set_errf("lg_encode: relabel must be 0, 1 (DM) or 2 (greedy)"); return LG_EINVAL; }
  if (weights && (o.id_mode == LG_ID_LOCAL || o.id_mode == LG_ID_LOCAL_GAP)) {
    set_errf("lg_encode: weights are supported with LG_ID_GLOBAL and LG_ID_CSR32 only");
    return LG_EUNSUPPORTED;
  }
  lg_graph* g = new (std::nothrow) lg_graph;
  if (!g) { set_errf("lg_encode: host allocation failed"); return LG_ENOMEM; }
  memset(g, 0, sizeof(*g));
  if (cudaGetDevice(&g->device) != cudaSuccess) { delete g; set_errf("lg_encode: no CUDA device"); return LG_ECUDA; }
  g->n = n; g->arcs = arcs;
  g->id_mode = o.id_mode; g->off_mode = o.off_mode; g->relabel = o.relabel; g->weighted = weights ? 1 : 0;
  g->sample = o.select_sample;
  g->sample_log2 = host_bits(o.select_sample) - 1;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  lg_status s = encode_impl(g, row_ptr, col, weights, o, st);
  if (s != LG_OK) {
    cudaStreamSynchronize(st);
    lg_free(g);
    return s;
  }
  *out = g;
  return LG_OK;
}

extern "C" lg_status lg_neighbors(const lg_graph* g, const uint32_t* vertices, uint64_t k, uint64_t* out_offsets,
                                  uint32_t* out_ids, uint32_t* out_weights, uint64_t out_capacity, void* stream) {
  g_err[0] = 0;
  if (!g || !out_offsets || (k && !vertices)) { set_errf("lg_neighbors: null argument"); return LG_EINVAL; }
  if (out_weights && !g->weighted) { set_errf("lg_neighbors: graph has no weights"); return LG_EINVAL; }
  DeviceGuard dg(g->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  Tmp small(st), stmp(st);
  LG_TRY(small.alloc(sizeof(NbrStat)));
  LG_TRY(cudaMemsetAsync(small.p, 0, sizeof(NbrStat), st));
  const GView v = make_view(g);
  const TravOps* ops = trav_ops((int)g->id_mode, (int)g->off_mode);
  NbrArgs a;
  memset(&a, 0, sizeof(a));
  a.vertices = vertices; a.k = k; a.out_offsets = out_offsets; a.out_ids = out_ids; a.out_weights = out_weights;
  a.stat = small.as<NbrStat>();
  a.scan = k > 0 && k <= NBR_SCAN;
  a.sort = g->relabel != 0;
  LG_TRY(ops->nbr_degrees(v, a, st));
  NbrStat h{};
  LG_TRY(cudaMemcpyAsync(&h, small.p, sizeof(h), cudaMemcpyDeviceToHost, st));
  if (!a.scan) {
    LG_TRY(stmp.alloc(scan_tmp_words(k) * sizeof(uint64_t)));
    LG_TRY(scan_excl_u64(out_offsets, k, out_offsets, stmp.as<uint64_t>(), st));
    LG_TRY(cudaMemcpyAsync(&h.total, out_offsets + k, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
  }
  LG_TRY(cudaStreamSynchronize(st));
  if (h.err) return describe_dev_err(h.err);
  if (h.total > out_capacity) {
    set_errf("lg_neighbors: %llu neighbors do not fit out_capacity %llu", (unsigned long long)h.total,
             (unsigned long long)out_capacity);
    return LG_ERANGE;
  }
  if (h.total && !out_ids) { set_errf("lg_neighbors: out_ids is NULL"); return LG_EINVAL; }
  if (h.total) LG_TRY(ops->nbr_rows(v, a, st));
  if (g->relabel)
    LG_TRY(segmented_sort(out_ids, out_weights, out_offsets, k, h.total, h.max_degree, st, 32, true));
  LG_TRY(cudaStreamSynchronize(st));
  return LG_OK;
}

extern "C" lg_status lg_bfs(const lg_graph* g, const uint32_t* sources, uint32_t S, uint32_t* depths, void* stream) {
  g_err[0] = 0;
  if (!g || (S && (!sources || !depths))) { set_errf("lg_bfs: null argument"); return LG_EINVAL; }
  if (S == 0) return LG_OK;
  DeviceGuard dg(g->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const uint64_t n = g->n;
  const uint32_t maxb = S >= 64 ? 64 : S;
  const int mb = maxb <= 16 ? 2 : (maxb <= 32 ? 4 : 8);
  constexpr uint32_t RING = 64;  // levels whose counters are zeroed together
  Tmp t_vis(st), t_fa(st), t_fb(st), t_qa(st), t_qb(st), t_small(st), t_depth(st), t_hacc(st);
  LG_TRY(t_vis.alloc(n * mb + 16));
  LG_TRY(t_fa.alloc(n * mb + 16));
  LG_TRY(t_fb.alloc(n * mb + 16));
  LG_TRY(t_qa.alloc(n * sizeof(uint32_t)));
  LG_TRY(t_qb.alloc(n * sizeof(uint32_t)));
  // error and start count, stored sources, counters of RING levels
  const size_t small_bytes = 16 + 64 * sizeof(uint32_t) + RING * 8;
  LG_TRY(t_small.alloc(small_bytes));
  if (g->relabel) LG_TRY(t_depth.alloc((uint64_t)maxb * n * sizeof(uint32_t)));
  const size_t hacc_bytes = (g->n_multi * mb + 15) / 16 * 16;
  LG_TRY(t_hacc.alloc(hacc_bytes + g->n_multi * sizeof(uint32_t)));
  LG_TRY(cudaMemsetAsync(t_hacc.p, 0, hacc_bytes + g->n_multi * sizeof(uint32_t), st));
  int* d_err = t_small.as<int>();
  uint32_t* stored = t_small.as<uint32_t>() + 4;
  uint32_t* ring = stored + 64;
  if (S > 64) {  // every source is checked before the first sweep writes its depths
    Tmp t_src(st);
    LG_TRY(t_src.alloc(S * sizeof(uint32_t)));
    LG_TRY(cudaMemsetAsync(t_small.p, 0, 16, st));
    LG_TRY(map_ids(sources, t_src.as<uint32_t>(), g->perm, S, n, d_err, st));
    int herr = 0;
    LG_TRY(cudaMemcpyAsync(&herr, d_err, 4, cudaMemcpyDeviceToHost, st));
    LG_TRY(cudaStreamSynchronize(st));
    if (herr) return describe_dev_err(herr);
  }

  const GView v = make_view(g);
  const TravOps* ops = trav_ops((int)g->id_mode, (int)g->off_mode);
  const uint64_t pull_threshold = n / pull_divisor();
  for (uint32_t b0 = 0; b0 < S; b0 += 64) {
    const uint32_t Sb = (S - b0) < 64 ? (S - b0) : 64;
    uint32_t* depth_b = g->relabel ? t_depth.as<uint32_t>() : depths + (uint64_t)b0 * n;
    LG_TRY(cudaMemsetAsync(t_vis.p, 0, n * mb + 16, st));
    LG_TRY(cudaMemsetAsync(t_fa.p, 0, n * mb + 16, st));
    LG_TRY(cudaMemsetAsync(t_small.p, 0, small_bytes, st));
    uint32_t* qa = t_qa.as<uint32_t>();
    if (mb == 2) k_bfs_start<uint16_t><<<1, 64, 0, st>>>(t_vis.as<uint16_t>(), t_fa.as<uint16_t>(), n, sources + b0, g->perm, Sb, stored, qa, stored - 3, d_err);
    else if (mb == 4) k_bfs_start<uint32_t><<<1, 64, 0, st>>>(t_vis.as<uint32_t>(), t_fa.as<uint32_t>(), n, sources + b0, g->perm, Sb, stored, qa, stored - 3, d_err);
    else k_bfs_start<uint64_t><<<1, 64, 0, st>>>(t_vis.as<uint64_t>(), t_fa.as<uint64_t>(), n, sources + b0, g->perm, Sb, stored, qa, stored - 3, d_err);
    count_launch();
    LG_TRY(cudaGetLastError());
    uint32_t hc[2] = {0, 0};  // error, frontier
    LG_TRY(cudaMemcpyAsync(hc, d_err, 8, cudaMemcpyDeviceToHost, st));
    LG_TRY(cudaStreamSynchronize(st));
    if (hc[0]) return describe_dev_err((int)hc[0]);
    LG_TRY(cudaMemsetAsync(depth_b, 0xff, (uint64_t)Sb * n * sizeof(uint32_t), st));
    k_bfs_depth0<<<1, 64, 0, st>>>(depth_b, n, stored, Sb, g->relabel ? 1u : 0u);
    count_launch();
    LG_TRY(cudaGetLastError());
    uint32_t nq = hc[1], prev = 0;  // lengths of this level's frontier and of the one before
    void* cur = t_fa.p;
    void* nxt = t_fb.p;
    uint32_t* qcur = qa;
    uint32_t* qnxt = t_qb.as<uint32_t>();
    BfsArgs a;
    memset(&a, 0, sizeof(a));
    a.vis = t_vis.p;
    a.depth = depth_b;
    a.all_mask = Sb == 64 ? ~0ull : ((1ull << Sb) - 1ull);
    a.S = Sb;
    a.vmajor = g->relabel ? 1u : 0u;  // relabeled depths are permuted afterwards
    a.hacc = t_hacc.p;
    a.hcnt = reinterpret_cast<uint32_t*>(t_hacc.as<char>() + hacc_bytes);
    a.err = d_err;
    a.hot = hot_rows(g, mb);
    for (uint32_t level = 0; nq > 0; level++) {
      if (level && level % RING == 0) LG_TRY(cudaMemsetAsync(ring, 0, RING * 8, st));
      a.counters = ring + 2 * (level % RING);
      a.front_in = cur; a.front_out = nxt; a.level = level;
      a.queue_in = qcur; a.queue_in_len = nq; a.queue_out = qnxt;
      if ((uint64_t)nq > pull_threshold) {
        LG_TRY(ops->bfs_pull(v, a, mb, st));
      } else {
        // A push level adds to zeroed masks (a pull level writes them all): the
        // output masks hold the frontier of the level before, listed in qnxt.
        if (level == 0 || (uint64_t)prev * 16 >= n) {
          LG_TRY(cudaMemsetAsync(nxt, 0, n * mb, st));
        } else {
          k_clear_queue<<<grid_for(prev, 256, 4096), 256, 0, st>>>(reinterpret_cast<uint8_t*>(nxt), mb, qnxt, prev);
          count_launch();
          LG_TRY(cudaGetLastError());
        }
        LG_TRY(ops->bfs_push(v, a, mb, st));
      }
      LG_TRY(cudaMemcpyAsync(hc, a.counters, 8, cudaMemcpyDeviceToHost, st));
      LG_TRY(cudaStreamSynchronize(st));
      void* t = cur; cur = nxt; nxt = t;
      uint32_t* tq = qcur; qcur = qnxt; qnxt = tq;
      prev = nq;
      nq = hc[0];
    }
    if (g->relabel) LG_TRY(bfs_permute_depths(depth_b, depths + (uint64_t)b0 * n, g->perm, n, Sb, st));
  }
  LG_TRY(cudaStreamSynchronize(st));
  return LG_OK;
}

extern "C" lg_status lg_pagerank(const lg_graph* g, float damping, uint32_t iters, const uint32_t* personalize_source,
                                 float* ranks, void* stream) {
  g_err[0] = 0;
  if (!g || !ranks) { set_errf("lg_pagerank: null argument"); return LG_EINVAL; }
  if (!(damping >= 0.0f && damping <= 1.0f)) { set_errf("lg_pagerank: damping must be in [0, 1]"); return LG_EINVAL; }
  int64_t personal_orig = -1, personal = -1;
  if (personalize_source) {
    if (*personalize_source >= g->n) { set_errf("lg_pagerank: personalize_source >= n"); return LG_EINVAL; }
    personal_orig = *personalize_source;
  }
  DeviceGuard dg(g->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const uint64_t n = g->n;
  if (iters == 0) {
    LG_TRY(pr_fill0(ranks, n, personal_orig, st));
    return LG_OK;
  }
  if (personal_orig >= 0) {
    if (g->perm) {
      uint32_t ps = 0;
      LG_TRY(cudaMemcpyAsync(&ps, g->perm + personal_orig, 4, cudaMemcpyDeviceToHost, st));
      LG_TRY(cudaStreamSynchronize(st));
      personal = ps;
    } else {
      personal = personal_orig;
    }
  }
  const PrPlan plan = pr_plan(g);
  Tmp ca(st), cb(st), tpart(st), tsync(st), taux(st);
  LG_TRY(ca.alloc(n * sizeof(float)));
  LG_TRY(cb.alloc(n * sizeof(float)));
  if (plan.part_floats) LG_TRY(tpart.alloc(plan.part_floats * sizeof(float)));
  LG_TRY(tsync.alloc(plan.sync_words * sizeof(uint32_t)));
  if (plan.aux_words) LG_TRY(taux.alloc(plan.aux_words * sizeof(uint64_t)));
  const GView v = make_view(g);
  const TravOps* ops = trav_ops((int)g->id_mode, (int)g->off_mode);
  PrArgs a;
  memset(&a, 0, sizeof(a));
  a.damp = damping;
  a.personal = personal;
  a.base_all = personal < 0 ? (1.0f - damping) / (float)n : (1.0f - damping);
  a.r0_all = 1.0f / (float)n;
  a.part = tpart.as<float>();
  a.ranks_out = ranks;
  a.contrib_out = ca.as<float>();
  a.hot = hot_rows(g, sizeof(float));
  a.tile_a = plan.tile_a;
  a.tile_b = plan.tile_b;
  a.tile_nv = plan.tile_nv;
  a.items = plan.items;
  a.tabn = plan.tabn;
  a.sync = tsync.as<uint32_t>();
  a.nsync = plan.sync_words;
  a.aux = taux.as<uint64_t>();
  LG_TRY(ops->pr_init(v, a, st));
  float* cur = ca.as<float>();
  float* nxt = cb.as<float>();
  for (uint32_t t = 0; t < iters; t++) {
    a.contrib_in = cur;
    a.contrib_out = nxt;
    a.last = (t + 1 == iters);
    a.turn = t & 1;
    LG_TRY(ops->pr_pull(v, a, st));
    float* tt = cur; cur = nxt; nxt = tt;
  }
  return LG_OK;
}
