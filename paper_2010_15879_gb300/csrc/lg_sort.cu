// Sorting used by the encoder: a stable LSD radix sort (8-bit digits) of
// (key, value) pairs, the DM permuter of Section 5.6 (vertices ordered by
// degree descending, ties by original ID) built on it, and a segmented sort of
// CSR rows (the relabeled neighborhoods must be sorted again, Section 2.3).
#include "lg_internal.h"

#include <algorithm>

namespace lg {

// =========================================================================
// stable LSD radix sort
// =========================================================================
constexpr int RS_NT = 256;
constexpr int RS_ROUNDS = 16;
constexpr int RS_TILE = RS_NT * RS_ROUNDS;  // keys per CTA
constexpr int RS_NW = RS_NT / 32;

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename K>
__global__ void __launch_bounds__(RS_NT) k_rs_hist(const K* __restrict__ keys, uint64_t n, uint32_t shift,
                                                   uint32_t* __restrict__ hist, uint64_t ntiles) {
  __shared__ uint32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * RS_TILE;
  for (int r = 0; r < RS_ROUNDS; r++) {
    const uint64_t i = base + (uint64_t)r * RS_NT + threadIdx.x;
    if (i < n) atomicAdd(&cnt[(uint32_t)(keys[i] >> shift) & 255u], 1u);
  }
  __syncthreads();
  hist[(uint64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];  // digit-major
}

// Scatter of one tile of RS_TILE keys: the tile is first ranked stably by digit
// into shared memory (per round of RS_NT keys: a match among the warp's lanes,
// the counts of the warps before, the tile's keys of this digit in earlier
// rounds), then written out in that order, so the keys of one digit -- about
// RS_TILE / 256 of them -- go to consecutive addresses (coalesced writes).
template <typename K>
struct RsSmem {
  K keys[RS_TILE];
  uint32_t vals[RS_TILE];
  uint32_t wcnt[RS_NW][256];
  uint32_t loc[256];        // first position of each digit in the tile
  uint32_t seen[256];       // keys of each digit placed so far
  uint64_t glob[256];       // first global position of each digit for this tile
  uint32_t red[RS_NW];
};

template <typename K>
__global__ void __launch_bounds__(RS_NT) k_rs_scatter(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                      K* __restrict__ kout, uint32_t* __restrict__ vout, uint64_t n,
                                                      uint32_t shift, const uint64_t* __restrict__ off,
                                                      const uint32_t* __restrict__ hist, uint64_t ntiles) {
  extern __shared__ __align__(16) unsigned char rs_raw[];
  RsSmem<K>& sm = *reinterpret_cast<RsSmem<K>*>(rs_raw);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t cell = (uint64_t)threadIdx.x * ntiles + blockIdx.x;
  {
    uint32_t total;
    sm.loc[threadIdx.x] = block_excl_scan<uint32_t, RS_NT>(hist[cell], total, sm.red);
    sm.glob[threadIdx.x] = off[cell];
    sm.seen[threadIdx.x] = 0;
  }
  const uint64_t base = (uint64_t)blockIdx.x * RS_TILE;
  const uint32_t tn = (uint32_t)min((uint64_t)RS_TILE, n - base);
  for (int r = 0; r < RS_ROUNDS; r++) {
    for (int k = 0; k < RS_NW; k++) sm.wcnt[k][threadIdx.x] = 0;
    __syncthreads();
    const uint32_t li = (uint32_t)r * RS_NT + threadIdx.x;
    const bool ok = li < tn;
    const K key = ok ? kin[base + li] : K(0);
    const uint32_t val = (ok && vin) ? vin[base + li] : 0u;
    const uint32_t dig = ok ? ((uint32_t)(key >> shift) & 255u) : 256u;
    const uint32_t peers = __match_any_sync(LG_FULL_MASK, dig);
    const uint32_t rank = __popc(peers & lanemask_lt());
    if (ok && rank == 0) sm.wcnt[w][dig] = __popc(peers);
    __syncthreads();
    // thread t owns digit t: exclusive prefix over the warps of this round
    uint32_t acc = 0;
    for (int k = 0; k < RS_NW; k++) {
      const uint32_t c = sm.wcnt[k][threadIdx.x];
      sm.wcnt[k][threadIdx.x] = acc;
      acc += c;
    }
    __syncthreads();
    if (ok) {
      const uint32_t pos = sm.loc[dig] + sm.seen[dig] + sm.wcnt[w][dig] + rank;
      sm.keys[pos] = key;
      sm.vals[pos] = val;
    }
    __syncthreads();
    sm.seen[threadIdx.x] += acc;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < tn; i += RS_NT) {
    const K key = sm.keys[i];
    const uint32_t dig = (uint32_t)(key >> shift) & 255u;
    const uint64_t pos = sm.glob[dig] + (i - sm.loc[dig]);
    kout[pos] = key;
    if (vin) vout[pos] = sm.vals[i];
  }
  (void)lane;
}

size_t radix_tmp_bytes(uint64_t n) {
  const uint64_t ntiles = (n + RS_TILE - 1) / RS_TILE;
  const uint64_t cells = 256 * ntiles;
  return cells * sizeof(uint32_t) + (cells + 1) * sizeof(uint64_t) + scan_tmp_words(cells) * sizeof(uint64_t) + 256;
}

template <typename K>
static cudaError_t radix_impl(K* keys, uint32_t* vals, K* keys_alt, uint32_t* vals_alt, uint64_t n,
                              uint32_t key_bits, void* tmp, cudaStream_t st) {
  if (n <= 1 || key_bits == 0) return cudaSuccess;
  const uint64_t ntiles = (n + RS_TILE - 1) / RS_TILE;
  const uint64_t cells = 256 * ntiles;
  uint32_t* hist = reinterpret_cast<uint32_t*>(tmp);
  uint64_t* off = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(tmp) + ((cells * 4 + 15) & ~15ull));
  uint64_t* stmp = off + cells + 2;
  K* ka = keys; K* kb = keys_alt;
  uint32_t* va = vals; uint32_t* vb = vals_alt;
  const uint32_t passes = (key_bits + 7) / 8;
  {
    const cudaError_t e = cudaFuncSetAttribute(k_rs_scatter<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(RsSmem<K>));
    if (e != cudaSuccess) return e;
  }
  for (uint32_t p = 0; p < passes; p++) {
    const uint32_t shift = 8 * p;
    k_rs_hist<K><<<(unsigned)ntiles, RS_NT, 0, st>>>(ka, n, shift, hist, ntiles);
    count_launch();
    cudaError_t e = scan_excl_u32(hist, cells, off, stmp, st);
    if (e != cudaSuccess) return e;
    k_rs_scatter<K><<<(unsigned)ntiles, RS_NT, sizeof(RsSmem<K>), st>>>(ka, va, kb, vb, n, shift, off, hist, ntiles);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    K* t = ka; ka = kb; kb = t;
    uint32_t* tv = va; va = vb; vb = tv;
  }
  if (ka != keys) {
    cudaError_t e = cudaMemcpyAsync(keys, ka, n * sizeof(K), cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    if (vals) e = cudaMemcpyAsync(vals, va, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t radix_sort_u32(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt, uint64_t n,
                           uint32_t key_bits, void* tmp, cudaStream_t st) {
  return radix_impl<uint32_t>(keys, vals, keys_alt, vals_alt, n, key_bits, tmp, st);
}
cudaError_t radix_sort_u64(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt, uint32_t* vals_alt, uint64_t n,
                           uint32_t key_bits, void* tmp, cudaStream_t st) {
  return radix_impl<uint64_t>(keys, vals, keys_alt, vals_alt, n, key_bits, tmp, st);
}

// =========================================================================
// segmented sort of CSR rows
// =========================================================================
constexpr uint32_t SEG_SMALL = 32;    // what a row's producer sorts (a thread per row, a network in registers)
constexpr uint32_t SEG_MEDIUM = NBR_SORT;  // 4,096: what the lookups' row kernel sorts itself
constexpr uint32_t SEG_LARGE = 16384;      // what one CTA sorts
constexpr int SROW = 33;              // shared slot stride of a small row (conflict-free lanes)

// compare-exchange into ascending order, without branches
template <bool VALS>
__device__ __forceinline__ void ce_asc(uint32_t& a, uint32_t& b, uint32_t& va, uint32_t& vb) {
  if (VALS) {
    const bool sw = a > b;
    const uint32_t ta = sw ? b : a, tb = sw ? a : b;
    const uint32_t tva = sw ? vb : va, tvb = sw ? va : vb;
    a = ta; b = tb; va = tva; vb = tvb;
  } else {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo; b = hi;
  }
}

// compare-exchange into ascending (up) or descending order
template <bool VALS>
__device__ __forceinline__ void ce_dir(uint32_t& a, uint32_t& b, uint32_t& va, uint32_t& vb, bool up) {
  if (VALS) {
    const bool sw = up ? (a > b) : (a < b);
    const uint32_t ta = sw ? b : a, tb = sw ? a : b;
    const uint32_t tva = sw ? vb : va, tvb = sw ? va : vb;
    a = ta; b = tb; va = tva; vb = tvb;
  } else {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = up ? lo : hi; b = up ? hi : lo;
  }
}

// Batcher's odd-even merge sort network on N = 2^m registers (19, 63 and 191
// comparators for N = 8, 16, 32): merges of sorted runs of length p into runs
// of 2p, each merge comparing elements k apart for k = p, p/2, .., 1 within
// the same 2p-run.  One instantiation per (p, k), so that every register
// index is a compile-time constant.
template <int N, bool VALS, int P, int K>
__device__ __forceinline__ void oem_pk(uint32_t (&x)[N], uint32_t (&y)[N]) {
  if constexpr (P < N) {
    if constexpr (K == 0) {
      oem_pk<N, VALS, 2 * P, 2 * P>(x, y);
    } else {
#pragma unroll
      for (int j = K % P; j + K < N; j += 2 * K) {
#pragma unroll
        for (int i = 0; i < K; i++) {
          if (i + j + K < N && (i + j) / (2 * P) == (i + j + K) / (2 * P))
            ce_asc<VALS>(x[i + j], x[i + j + K], y[i + j], y[i + j + K]);
        }
      }
      oem_pk<N, VALS, P, K / 2>(x, y);
    }
  }
}

template <int N, bool VALS>
__device__ __forceinline__ void oem_sort(uint32_t (&x)[N], uint32_t (&y)[N]) {
  oem_pk<N, VALS, 1, 1>(x, y);
}

// one thread sorts the d <= N keys of its shared slot (padded with UINT32_MAX)
template <int N, bool VALS>
__device__ __forceinline__ void slot_sort(uint32_t* sk, uint32_t* sv, uint32_t d) {
  uint32_t x[N], y[N];
#pragma unroll
  for (int t = 0; t < N; t++) {
    x[t] = (uint32_t)t < d ? sk[t] : 0xffffffffu;
    y[t] = (VALS && (uint32_t)t < d) ? sv[t] : 0u;
  }
  oem_sort<N, VALS>(x, y);
#pragma unroll
  for (int t = 0; t < N; t++) {
    if ((uint32_t)t < d) {
      sk[t] = x[t];
      if (VALS) sv[t] = y[t];
    }
  }
}

// Each lane sorts slot `lane` (d keys, d <= 32) of its warp's 32 shared slots.
// A warp runs at most two networks: 8 keys, and 16 or 32 (32 if any of its
// rows needs it).
template <bool VALS>
__device__ __forceinline__ void warp_sort_slots(uint32_t* sk, uint32_t* sv, uint32_t d, bool small, int lane) {
  const bool any32 = __any_sync(LG_FULL_MASK, small && d > 16);
  if (small && d > 1) {
    uint32_t* k = sk + lane * SROW;
    uint32_t* v = sv + lane * SROW;
    if (d <= 8) slot_sort<8, VALS>(k, v, d);
    else if (any32) slot_sort<32, VALS>(k, v, d);
    else slot_sort<16, VALS>(k, v, d);
  }
  __syncwarp();
}

// the rows of one size class: listed, or `count` consecutive ones from `first`
struct SegRows {
  const uint32_t* list;
  uint32_t first, count;
  __device__ __forceinline__ uint64_t row(uint32_t i) const { return list ? list[i] : first + i; }
};

// ---------------------------------------------------------------------------
// Rows of 33..128 keys of a size class, and of up to 512 without values, P =
// 16 G >= d keys per row (padded with UINT32_MAX), G lanes per row.  Lane g holds keys 16 g + e, e < 16, so a
// bitonic compare-exchange at distance j is a register pair for j < 16 and a
// shuffle with lane g ^ (j / 16) beyond.  The first four levels are unrolled;
// the rest run as a loop (an unrolled network of this size would outgrow the
// instruction cache).  Values double each stage's moves, so from 129 keys on
// rows with values are quicker by radix, which moves indices (R-MAT 2^22, whole
// encode, degree order: 3.80 ms, 4.54 with the network up to 512; 3 M vertices
// of degree 200 15.2 and 20.4); rows of keys alone are not (2.99 and 2.94, 12.9
// and 7.7; in greedy order 19.7 and 10.6).
// ---------------------------------------------------------------------------
template <int J, bool VALS>
__device__ __forceinline__ void blk_pairs(uint32_t (&x)[16], uint32_t (&y)[16], uint32_t base16, uint32_t k) {
#pragma unroll
  for (int e = 0; e < 16; e++) {
    if ((e & J) == 0) ce_dir<VALS>(x[e], x[e | J], y[e], y[e | J], ((base16 | (uint32_t)e) & k) == 0);
  }
}

// the four register stages j = 8, 4, 2, 1 of a level k >= 16 (direction set
// by the lane's block only)
template <bool VALS>
__device__ __forceinline__ void blk_tail(uint32_t (&x)[16], uint32_t (&y)[16], bool up) {
#pragma unroll
  for (int j = 8; j >= 1; j >>= 1) {
#pragma unroll
    for (int e = 0; e < 16; e++) {
      if ((e & j) == 0) ce_dir<VALS>(x[e], x[e | j], y[e], y[e | j], up);
    }
  }
}

template <bool VALS>
__device__ __forceinline__ void blk_shfl(uint32_t (&x)[16], uint32_t (&y)[16], uint32_t lanemask, bool keep_min) {
#pragma unroll
  for (int e = 0; e < 16; e++) {
    const uint32_t ok = __shfl_xor_sync(LG_FULL_MASK, x[e], lanemask);
    if (VALS) {
      const uint32_t ov = __shfl_xor_sync(LG_FULL_MASK, y[e], lanemask);
      const bool take = keep_min ? (ok < x[e]) : (ok > x[e]);
      x[e] = take ? ok : x[e];
      y[e] = take ? ov : y[e];
    } else {
      x[e] = keep_min ? min(x[e], ok) : max(x[e], ok);
    }
  }
}

template <int G, bool VALS>
__global__ void __launch_bounds__(256) k_seg_blk(uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                 const uint64_t* __restrict__ off, SegRows rows) {
  constexpr uint32_t P = 16u * G;
  constexpr int RPB = 256 / G;  // rows per block pass
  const int g = threadIdx.x % G;
  const uint32_t base16 = 16u * g;
  for (uint64_t base = (uint64_t)blockIdx.x * RPB; base < rows.count; base += (uint64_t)gridDim.x * RPB) {
    const uint64_t li = base + threadIdx.x / G;
    uint64_t lo = 0;
    uint32_t d = 0;
    if (li < rows.count) {
      const uint64_t r = rows.row((uint32_t)li);
      lo = off[r];
      d = (uint32_t)(off[r + 1] - lo);
    }
    uint32_t x[16], y[16];
#pragma unroll
    for (int e = 0; e < 16; e++) {
      const uint32_t i = base16 + e;
      x[e] = i < d ? keys[lo + i] : 0xffffffffu;
      y[e] = (VALS && i < d) ? vals[lo + i] : 0u;
    }
    // levels k = 2 .. 16 inside the lane's block
    blk_pairs<1, VALS>(x, y, base16, 2);
    blk_pairs<2, VALS>(x, y, base16, 4);
    blk_pairs<1, VALS>(x, y, base16, 4);
    blk_pairs<4, VALS>(x, y, base16, 8);
    blk_pairs<2, VALS>(x, y, base16, 8);
    blk_pairs<1, VALS>(x, y, base16, 8);
    blk_tail<VALS>(x, y, (base16 & 16u) == 0);
#pragma unroll 1
    for (uint32_t k = 32; k <= P; k <<= 1) {
      const bool up = (base16 & k) == 0;
#pragma unroll 1
      for (uint32_t j = k >> 1; j >= 16; j >>= 1) {
        const uint32_t m = j >> 4;
        blk_shfl<VALS>(x, y, m, ((g & m) == 0) == up);
      }
      blk_tail<VALS>(x, y, up);
    }
#pragma unroll
    for (int e = 0; e < 16; e++) {
      const uint32_t i = base16 + e;
      if (i < d) {
        keys[lo + i] = x[e];
        if (VALS) vals[lo + i] = y[e];
      }
    }
  }
}

// size class of a row: 0 for d <= 32, k = 1..9 for 2^(4+k) < d <= 2^(5+k),
// SEG_BIG above
constexpr int SEG_BIG = 10;
constexpr int SEG_NCLASS = 11;

__device__ __forceinline__ int seg_class(uint64_t d) {
  if (d <= SEG_SMALL) return 0;
  if (d > SEG_LARGE) return SEG_BIG;
  return 27 - __clz((uint32_t)d - 1);
}

__global__ void k_seg_count(const uint64_t* __restrict__ off, uint64_t rows, uint32_t* __restrict__ cnt) {
  __shared__ uint32_t c[SEG_NCLASS];
  if (threadIdx.x < SEG_NCLASS) c[threadIdx.x] = 0;
  __syncthreads();
  for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (uint64_t)gridDim.x * blockDim.x) {
    const int k = seg_class(off[r + 1] - off[r]);
    if (k) atomicAdd(&c[k], 1u);
  }
  __syncthreads();
  if (threadIdx.x < SEG_NCLASS && c[threadIdx.x]) atomicAdd(&cnt[threadIdx.x], c[threadIdx.x]);
}

__global__ void __launch_bounds__(256) k_seg_fill(const uint64_t* __restrict__ off, uint64_t rows,
                                                  const uint32_t* __restrict__ base, uint32_t* __restrict__ cursor,
                                                  uint32_t* __restrict__ list) {
  const int lane = threadIdx.x & 31;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t r0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); r0 < rows; r0 += stride) {
    const uint64_t r = r0 + lane;
    const int k = r < rows ? seg_class(off[r + 1] - off[r]) : 0;
    // one cursor atomic per class present in the warp
    const uint32_t peers = __match_any_sync(LG_FULL_MASK, k);
    const int leader = __ffs(peers) - 1;
    uint32_t at = 0;
    if (k && lane == leader) at = base[k] + atomicAdd(&cursor[k], (uint32_t)__popc(peers));
    at = __shfl_sync(LG_FULL_MASK, at, leader);
    if (k) list[at + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)r;
  }
}

// large rows: gather (row rank, key) composite keys, radix sort, scatter back
__global__ void k_seg_big_gather(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                 const uint64_t* __restrict__ off, const uint32_t* __restrict__ big,
                                 const uint64_t* __restrict__ boff, uint32_t nbig, uint32_t* __restrict__ ck,
                                 uint32_t* __restrict__ cv) {
  for (uint32_t b = blockIdx.x; b < nbig; b += gridDim.x) {
    const uint64_t lo = off[big[b]], d = off[big[b] + 1] - lo, o = boff[b];
    for (uint64_t i = threadIdx.x; i < d; i += blockDim.x) {
      ck[o + i] = keys[lo + i];
      cv[o + i] = vals ? vals[lo + i] : 0u;
    }
  }
}
__global__ void k_seg_big_scatter(uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                  const uint64_t* __restrict__ off, const uint32_t* __restrict__ big,
                                  const uint64_t* __restrict__ boff, uint32_t nbig, const uint32_t* __restrict__ ck,
                                  const uint32_t* __restrict__ cv) {
  for (uint32_t b = blockIdx.x; b < nbig; b += gridDim.x) {
    const uint64_t lo = off[big[b]], d = off[big[b] + 1] - lo, o = boff[b];
    for (uint64_t i = threadIdx.x; i < d; i += blockDim.x) {
      keys[lo + i] = ck[o + i];
      if (vals) vals[lo + i] = cv[o + i];
    }
  }
}
__global__ void k_seg_big_sizes(const uint64_t* __restrict__ off, const uint32_t* __restrict__ big, uint32_t nbig,
                                uint64_t* __restrict__ sizes) {
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nbig; b += gridDim.x * blockDim.x)
    sizes[b] = off[big[b] + 1] - off[big[b]];
}

// -------------------------------------------------------------------------
// One stable split of up to 512 NW keys by a 9-bit digit, for the segmented
// radix sorts.  Warp w holds the consecutive chunk [c0, c0 + 32 G) with
// c0 = 32 G w, key c0 + 32 g + lane in register g: a vote per bit of the digit
// gives a key's rank among its equals, the warp's own 16-bit counts (two digits to a
// word, so the block scan adds both at once) the rank among the groups before,
// and the scan over (digit, warp) the position.  The rank is kept beside the
// digit, so the chunk goes out without another pass over the counts.  Three
// block barriers per pass, whatever the tile's length.
// -------------------------------------------------------------------------
constexpr int SPL_BITS = 9;
constexpr uint32_t SPL_NB = 1u << SPL_BITS;  // digits per pass
constexpr int SPL_G = 16;                    // groups of 32 keys per warp, at most
static_assert(SPL_G * RS_NT == RS_TILE, "a tile is one split of 8 warps");

template <int NW>
struct SplitSmem {
  uint32_t wc[NW][SPL_NB / 2];  // per warp: the counts, then the first position, of digits 2 i and 2 i + 1
  uint32_t red[NW];
  // the first position of a digit in the tile
  __device__ __forceinline__ uint32_t start(uint32_t d) const { return reinterpret_cast<const uint16_t*>(wc[0])[d]; }
};

__host__ __device__ constexpr uint32_t spl_passes(uint32_t key_bits) { return (key_bits + SPL_BITS - 1) / SPL_BITS; }

// digit(g): of the key in register g; put(g, pos): writes it.  All 32 G NW
// keys take part: the caller fills up with keys of the last digit, which stay
// behind the others.
template <int NW, typename Digit, typename Put>
__device__ __forceinline__ void split_pass(int G, SplitSmem<NW>& sp, Digit digit, Put put) {
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, lt = lanemask_lt();
  uint4* mine4 = reinterpret_cast<uint4*>(sp.wc[w]);
#pragma unroll
  for (uint32_t b = 0; b < SPL_NB / 8; b += 32) mine4[b + lane] = make_uint4(0, 0, 0, 0);
  __syncwarp();
  uint16_t* mine = reinterpret_cast<uint16_t*>(sp.wc[w]);
  uint32_t dr[SPL_G];  // digit | rank in the chunk << 16
#pragma unroll
  for (int g = 0; g < SPL_G; g++) {
    if (g >= G) continue;
    // The lanes of equal digit, by votes: a match takes longer the more digits
    // differ.  R-MAT 2^26, rows of one to 32 warps: 5.2, 4.3, 6.2 ms (4 warps),
    // 6.7 (16) and 3.3 (32) by match, 5.1, 3.8, 4.2, 4.6 and 2.1 by votes.
    const uint32_t dig = digit(g);
    uint32_t peers = LG_FULL_MASK;
#pragma unroll
    for (int b = 0; b < SPL_BITS; b++) {
      const bool bit = dig >> b & 1u;
      const uint32_t v = __ballot_sync(LG_FULL_MASK, bit);
      peers &= bit ? v : ~v;
    }
    const uint32_t rank = mine[dig] + __popc(peers & lt);
    __syncwarp();
    if (peers >> lane == 1u) mine[dig] = (uint16_t)(rank + 1);  // the last lane of the digit
    __syncwarp();
    dr[g] = dig | rank << 16;
  }
  __syncthreads();
  constexpr int WPT = NW < 8 ? 8 / NW : 1;  // count words per thread, consecutive
  const bool scans = NW <= 8 || threadIdx.x < SPL_NB / 2;
  uint32_t sum = 0;
#pragma unroll 2
  for (int q = 0; q < WPT; q++) {
    uint32_t acc = 0;
    if (scans) {
#pragma unroll 8
      for (int v = 0; v < NW; v++) acc += sp.wc[v][threadIdx.x * WPT + q];
    }
    sum += (acc & 0xffffu) + (acc >> 16);
  }
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(LG_FULL_MASK, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  if (lane == 31) sp.red[w] = incl;
  __syncthreads();
  uint32_t pre = incl - sum;
#pragma unroll
  for (int v = 0; v < (NW < 8 ? NW : 8); v++) pre += (uint32_t)v < w ? sp.red[v] : 0u;
#pragma unroll 2
  for (int q = 0; q < WPT; q++) {
    if (!scans) break;
    uint32_t acc = 0;
#pragma unroll 8
    for (int v = 0; v < NW; v++) {
      const uint32_t c = sp.wc[v][threadIdx.x * WPT + q];
      sp.wc[v][threadIdx.x * WPT + q] = acc;
      acc += c;
    }
    const uint32_t both = pre | (pre + (acc & 0xffffu)) << 16;
#pragma unroll 8
    for (int v = 0; v < NW; v++) sp.wc[v][threadIdx.x * WPT + q] += both;
    pre += (acc & 0xffffu) + (acc >> 16);
  }
  __syncthreads();
#pragma unroll
  for (int g = 0; g < SPL_G; g++)
    if (g < G) put(g, mine[dr[g] & 0xffffu] + (dr[g] >> 16));
  __syncthreads();
}

// Rows above SEG_LARGE keys: a segmented LSD radix sort of the rows gathered
// into one buffer.  Tiles of RS_TILE keys never straddle two rows; the
// histogram cells are laid out row by row, digit-major within a row, so one
// exclusive scan over all cells gives every (row, digit, tile) its output
// position inside its own row -- no row index in the keys, ceil(key_bits / 9)
// passes over 4-byte keys.
struct SrsTile {
  uint64_t start;     // first key of the tile in the gathered buffer
  uint64_t cellbase;  // first histogram cell of the tile's row
  uint32_t len;       // keys in the tile (<= RS_TILE)
  uint32_t stride;    // tiles in the row
  uint32_t tl;        // index of the tile within its row
  uint32_t row;       // the row
};

__global__ void k_srs_tile_count(const uint64_t* __restrict__ boff, uint32_t nbig, uint32_t* __restrict__ nt) {
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nbig; b += gridDim.x * blockDim.x)
    nt[b] = (uint32_t)((boff[b + 1] - boff[b] + RS_TILE - 1) / RS_TILE);
}
__global__ void k_srs_tile_fill(const uint64_t* __restrict__ boff, const uint64_t* __restrict__ tbase, uint32_t nbig,
                                SrsTile* __restrict__ tiles) {
  for (uint32_t b = blockIdx.x; b < nbig; b += gridDim.x) {
    const uint64_t size = boff[b + 1] - boff[b], t0 = tbase[b];
    const uint32_t nt = (uint32_t)(tbase[b + 1] - t0);
    for (uint32_t tl = threadIdx.x; tl < nt; tl += blockDim.x) {
      SrsTile d;
      d.start = boff[b] + (uint64_t)tl * RS_TILE;
      d.cellbase = (uint64_t)SPL_NB * t0;
      d.len = (uint32_t)min((uint64_t)RS_TILE, size - (uint64_t)tl * RS_TILE);
      d.stride = nt;
      d.tl = tl;
      d.row = b;
      tiles[t0 + tl] = d;
    }
  }
}
__global__ void __launch_bounds__(RS_NT) k_srs_hist(const uint32_t* __restrict__ keys, const SrsTile* __restrict__ tiles,
                                                    uint32_t shift, uint32_t* __restrict__ hist) {
  __shared__ uint32_t cnt[SPL_NB];
  const SrsTile d = tiles[blockIdx.x];
  for (uint32_t b = threadIdx.x; b < SPL_NB; b += RS_NT) cnt[b] = 0;
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < d.len; i += RS_NT)
    atomicAdd(&cnt[(keys[d.start + i] >> shift) & (SPL_NB - 1)], 1u);
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < SPL_NB; b += RS_NT) hist[d.cellbase + (uint64_t)b * d.stride + d.tl] = cnt[b];
}

struct SrsSmem {
  uint32_t k[RS_TILE];   // as they came
  uint32_t v[RS_TILE];
  uint16_t at[RS_TILE];  // the order by digit
  uint64_t glob[SPL_NB];  // first output position of each digit of this tile, less its first position here
  SplitSmem<RS_NW> sp;
};

// One pass: the tile is split by digit in shared memory, then each key goes to
// its digit's run for this tile (runs of one digit are consecutive in kout).
template <bool VALS>
__global__ void __launch_bounds__(RS_NT, 4) k_srs_scatter(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                       uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                       const SrsTile* __restrict__ tiles, uint32_t shift,
                                                       const uint64_t* __restrict__ off) {
  extern __shared__ __align__(16) unsigned char srs_raw[];
  SrsSmem& sm = *reinterpret_cast<SrsSmem*>(srs_raw);
  const SrsTile d = tiles[blockIdx.x];
  const int G = (int)((d.len + RS_NT - 1) / RS_NT), lane = threadIdx.x & 31;
  const uint32_t c0 = 32u * G * (threadIdx.x >> 5);
  if (VALS) {
    for (uint32_t i = threadIdx.x; i < d.len; i += RS_NT) cp_async4(&sm.v[i], vin + d.start + i);
  }
  uint32_t x[SPL_G];
#pragma unroll
  for (int g = 0; g < SPL_G; g++) {
    const uint32_t i = c0 + 32u * g + lane;
    x[g] = g < G && i < d.len ? kin[d.start + i] : 0u;
  }
#pragma unroll
  for (int g = 0; g < SPL_G; g++)
    if (g < G && c0 + 32u * g + lane < d.len) sm.k[c0 + 32u * g + lane] = x[g];
  split_pass<RS_NW>(
      G, sm.sp, [&](int g) { return c0 + 32u * g + lane < d.len ? (x[g] >> shift) & (SPL_NB - 1) : SPL_NB - 1; },
      [&](int g, uint32_t pos) { sm.at[pos] = (uint16_t)(c0 + 32u * g + lane); });
  for (uint32_t b = threadIdx.x; b < SPL_NB; b += RS_NT)
    sm.glob[b] = off[d.cellbase + (uint64_t)b * d.stride + d.tl] - sm.sp.start(b);
  if (VALS) cp_async_wait_all();
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < d.len; i += RS_NT) {
    const uint32_t at = sm.at[i], key = sm.k[at];
    const uint64_t pos = sm.glob[(key >> shift) & (SPL_NB - 1)] + i;
    kout[pos] = key;
    if (VALS) vout[pos] = sm.v[at];
  }
}

// The tiles of nbig rows held back to back, row b at [boff[b], boff[b+1]) with
// boff on the device.
struct SrsTiles {
  SrsTile* tiles = nullptr;
  uint64_t count = 0;  // tiles
  uint64_t head = 0;   // tiles of the first nhead rows
  void release(cudaStream_t st) {
    if (tiles) cudaFreeAsync(tiles, st);
    tiles = nullptr;
  }
};

static cudaError_t srs_tiles(const uint64_t* boff, uint32_t nbig, uint32_t nhead, SrsTiles* out, cudaStream_t st) {
  uint64_t *tbase = nullptr, *stmp = nullptr;
  uint32_t* nt = nullptr;
  cudaError_t e = lg::pool_alloc((void**)&tbase, (nbig + 1) * sizeof(uint64_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&nt, nbig * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&stmp, scan_tmp_words(nbig) * sizeof(uint64_t), st);
  if (e == cudaSuccess) {
    k_srs_tile_count<<<grid_for(nbig, 256, 1024), 256, 0, st>>>(boff, nbig, nt);
    count_launch();
    e = scan_excl_u32(nt, nbig, tbase, stmp, st);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&out->count, tbase + nbig, sizeof(uint64_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&out->head, tbase + nhead, sizeof(uint64_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess)
    e = lg::pool_alloc((void**)&out->tiles, (out->count ? out->count : 1) * sizeof(SrsTile), st);
  if (e == cudaSuccess) {
    k_srs_tile_fill<<<grid_for(nbig, 1, 4096), 256, 0, st>>>(boff, tbase, nbig, out->tiles);
    count_launch();
    e = cudaGetLastError();
  }
  if (tbase) cudaFreeAsync(tbase, st);
  if (nt) cudaFreeAsync(nt, st);
  if (stmp) cudaFreeAsync(stmp, st);
  return e;
}

// The segmented radix passes over the head tiles' rows in (ka, va); kb, vb hold
// as much.  On return *result_in_b says whether the sorted rows ended in (kb, vb).
static cudaError_t srs_sort(uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb, const SrsTiles& T,
                            uint32_t key_bits, bool* result_in_b, cudaStream_t st) {
  uint64_t *coff = nullptr, *ctmp = nullptr;
  uint32_t* hist = nullptr;
  *result_in_b = false;
  const uint64_t cells = (uint64_t)SPL_NB * T.head;
  cudaError_t e = lg::pool_alloc((void**)&hist, (cells ? cells : 1) * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&coff, (cells + 1) * sizeof(uint64_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&ctmp, scan_tmp_words(cells) * sizeof(uint64_t), st);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(va ? k_srs_scatter<true> : k_srs_scatter<false>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SrsSmem));
  const uint32_t passes = spl_passes(key_bits);
  for (uint32_t p = 0; p < passes && e == cudaSuccess && T.head; p++) {
    const uint32_t shift = SPL_BITS * p;
    k_srs_hist<<<(unsigned)T.head, RS_NT, 0, st>>>(ka, T.tiles, shift, hist);
    count_launch();
    e = scan_excl_u32(hist, cells, coff, ctmp, st);
    if (e != cudaSuccess) break;
    if (va)
      k_srs_scatter<true><<<(unsigned)T.head, RS_NT, sizeof(SrsSmem), st>>>(ka, va, kb, vb, T.tiles, shift, coff);
    else
      k_srs_scatter<false><<<(unsigned)T.head, RS_NT, sizeof(SrsSmem), st>>>(ka, va, kb, vb, T.tiles, shift, coff);
    count_launch();
    e = cudaGetLastError();
    uint32_t* t = ka; ka = kb; kb = t;
    t = va; va = vb; vb = t;
    *result_in_b = !*result_in_b;
  }
  if (hist) cudaFreeAsync(hist, st);
  if (coff) cudaFreeAsync(coff, st);
  if (ctmp) cudaFreeAsync(ctmp, st);
  return e;
}

// Rows above SEG_LARGE keys listed in `big`: gathered back to back, sorted,
// scattered back.
static cudaError_t seg_sort_big(uint32_t* keys, uint32_t* vals, const uint64_t* off, const uint32_t* big,
                                uint32_t nbig, uint32_t key_bits, cudaStream_t st) {
  uint64_t *sizes = nullptr, *boff = nullptr, *stmp = nullptr;
  uint32_t *ka = nullptr, *kb = nullptr, *va = nullptr, *vb = nullptr;
  uint64_t nb_total = 0;
  cudaError_t e = lg::pool_alloc((void**)&sizes, nbig * sizeof(uint64_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&boff, (nbig + 1) * sizeof(uint64_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&stmp, scan_tmp_words(nbig) * sizeof(uint64_t), st);
  if (e == cudaSuccess) {
    k_seg_big_sizes<<<grid_for(nbig, 256, 1024), 256, 0, st>>>(off, big, nbig, sizes);
    count_launch();
    e = scan_excl_u64(sizes, nbig, boff, stmp, st);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&nb_total, boff + nbig, sizeof(uint64_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&ka, nb_total * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&kb, nb_total * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&va, nb_total * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&vb, nb_total * sizeof(uint32_t), st);
  if (e == cudaSuccess) {
    k_seg_big_gather<<<grid_for(nbig, 1, 4096), 256, 0, st>>>(keys, vals, off, big, boff, nbig, ka, va);
    count_launch();
    e = cudaGetLastError();
  }
  bool in_b = false;
  SrsTiles T;
  if (e == cudaSuccess) e = srs_tiles(boff, nbig, nbig, &T, st);
  if (e == cudaSuccess) e = srs_sort(ka, vals ? va : nullptr, kb, vals ? vb : nullptr, T, key_bits, &in_b, st);
  T.release(st);
  if (e == cudaSuccess) {
    k_seg_big_scatter<<<grid_for(nbig, 1, 4096), 256, 0, st>>>(keys, vals, off, big, boff, nbig, in_b ? kb : ka,
                                                                in_b ? vb : va);
    count_launch();
    e = cudaGetLastError();
  }
  cudaFreeAsync(sizes, st); cudaFreeAsync(boff, st); cudaFreeAsync(stmp, st);
  cudaFreeAsync(ka, st); cudaFreeAsync(kb, st); cudaFreeAsync(va, st); cudaFreeAsync(vb, st);
  return e;
}

// The head tiles' rows lie back to back from 0 (the rows above SEG_LARGE keys in
// degree-descending order, `total` keys): sorted in place, with one buffer of
// the same size beside them.
static cudaError_t seg_sort_big_prefix(uint32_t* keys, uint32_t* vals, const SrsTiles& T, uint64_t total,
                                       uint32_t key_bits, cudaStream_t st) {
  uint32_t *kb = nullptr, *vb = nullptr;
  cudaError_t e = lg::pool_alloc((void**)&kb, total * sizeof(uint32_t), st);
  if (e == cudaSuccess && vals) e = lg::pool_alloc((void**)&vb, total * sizeof(uint32_t), st);
  bool in_b = false;
  if (e == cudaSuccess) e = srs_sort(keys, vals, kb, vb, T, key_bits, &in_b, st);
  if (e == cudaSuccess && in_b) {
    e = cudaMemcpyAsync(keys, kb, total * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && vals) e = cudaMemcpyAsync(vals, vb, total * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
  }
  if (kb) cudaFreeAsync(kb, st);
  if (vb) cudaFreeAsync(vb, st);
  return e;
}

// -------------------------------------------------------------------------
// Rows of 129..16384 keys (513.. without values): a CTA of NW warps per row of up to 512 NW keys, a
// stable LSD radix sort with 9-bit digits in shared memory.  The passes move
// the keys' indices only, keys and values stay where they were loaded until
// the sorted row is written.
//
// Degree-mapped rows need two passes whatever the number of vertices: a row
// arrives sorted by its old IDs, in which order the labels of one degree
// ascend, so only the degrees have to be sorted.  The sort key is a coarse
// label of 18 bits -- exact below 2^17, one of 2^13 steps per power of two
// above --, and index and key fit one word.  Labels of one step come out in
// the order they had, which is wrong only where a change of degree lies between
// them: the few such runs are sorted by insertion, and a row with a run of more
// than RUN_MAX goes through all passes of the whole label (as do rows in
// another order than the DM's).
// What bounds it is instructions and shared-memory latency.  R-MAT 2^26,
// weighted: rows of 513..4096 keys 20.3 ms with three passes of keys and values
// and a second pass over the counts, 8.0 so; rows of 129..512 9.1 ms as bitonic
// networks, 5.1; rows of 4097..16384, 490 M of the 780 M keys that went through
// the tiles' passes in global memory (20.3 ms in all), 6.7 beside 7.0 for the
// rest.
// -------------------------------------------------------------------------
constexpr uint32_t SEG_IDX_BITS = 14;
constexpr uint32_t COARSE_BITS = 2 * SPL_BITS;
constexpr uint32_t RUN_MAX = 64;
static_assert(SEG_LARGE <= 1u << SEG_IDX_BITS && SEG_IDX_BITS + COARSE_BITS <= 32, "index and key share a word");

__device__ __forceinline__ uint32_t coarse_label(uint32_t x) {
  if (x < 1u << 17) return x;
  const uint32_t e = 31u - __clz(x);
  return (1u << 17) + ((e - 17u) << 13) + ((x >> (e - 13u)) & 8191u);  // at most 2^17 + 15 2^13 - 1
}

template <int NW, bool VALS>
struct SegRadixSmem {
  uint32_t k[512 * NW];
  uint32_t v[VALS ? 512 * NW : 4];
  uint32_t at[512 * NW];  // the sorted order: the key's index in the low bits
  SplitSmem<NW> sp;
};

template <int NW, bool VALS>
__global__ void __launch_bounds__(32 * NW, NW == 1 ? 30 : 32 / NW) k_seg_radix(uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                                const uint64_t* __restrict__ off, SegRows rows,
                                                                uint32_t passes, bool coarse) {
  constexpr uint32_t NT = 32 * NW, IM = (1u << SEG_IDX_BITS) - 1;
  extern __shared__ __align__(16) unsigned char sr_raw[];
  SegRadixSmem<NW, VALS>& sm = *reinterpret_cast<SegRadixSmem<NW, VALS>*>(sr_raw);
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t li = blockIdx.x; li < rows.count; li += gridDim.x) {
    const uint64_t r = rows.row(li), lo = off[r];
    const uint32_t d = (uint32_t)(off[r + 1] - lo);
    const int G = (int)((d + NT - 1) / NT);
    const uint32_t c0 = 32u * G * (threadIdx.x >> 5);
    uint32_t x[SPL_G];
    if (VALS) {
      for (uint32_t i = threadIdx.x; i < d; i += NT) cp_async4(&sm.v[i], vals + lo + i);
    }
#pragma unroll
    for (int g = 0; g < SPL_G; g++) {
      const uint32_t i = c0 + 32u * g + lane;
      x[g] = g < G && i < d ? keys[lo + i] : 0u;
    }
#pragma unroll
    for (int g = 0; g < SPL_G; g++) {
      const uint32_t i = c0 + 32u * g + lane;
      if (g < G && i < d) sm.k[i] = x[g];
      // no coarse label reaches 2^18 - 1: the padding's word comes last
      x[g] = i < d ? i | (coarse ? coarse_label(x[g]) << SEG_IDX_BITS : 0u) : ~0u;
    }
    // a warp reads its own chunk's keys in the first pass; the passes'
    // barriers come before the others
    __syncwarp();
    for (bool part = coarse;;) {
      const uint32_t np = part ? 2u : passes;
#pragma unroll 1
      for (uint32_t p = 0; p < np; p++) {
        // the word of a key: its index, then the whole coarse label or this
        // pass's digit of the label
#pragma unroll
        for (int g = 0; g < SPL_G; g++) {
          if (g < G) {
            if (p) x[g] = sm.at[c0 + 32u * g + lane];
            if (!part && x[g] != ~0u) {
              const uint32_t at = x[g] & IM;
              x[g] = at | ((sm.k[at] >> (SPL_BITS * p)) & (SPL_NB - 1)) << SEG_IDX_BITS;
            }
          }
        }
        const uint32_t shift = SEG_IDX_BITS + (part ? SPL_BITS * p : 0u);
        split_pass<NW>(
            G, sm.sp, [&](int g) { return (x[g] >> shift) & (SPL_NB - 1); },
            [&](int g, uint32_t pos) { sm.at[pos] = x[g]; });
      }
      if (!part) break;
      // a run's first key sorts it; others read only what the run's keys share
      bool bad = false;
      for (uint32_t i = threadIdx.x; i + 1 < d; i += NT) {
        const uint32_t first = sm.at[i];
        if ((first ^ sm.at[i + 1]) > IM) continue;
        if (i && (first ^ sm.at[i - 1]) <= IM) continue;
        for (uint32_t e = i + 1; e < d; e++) {
          const uint32_t next = sm.at[e];
          if ((next ^ first) > IM) break;
          if (e - i == RUN_MAX) {
            bad = true;
            break;
          }
          const uint32_t key = sm.k[next & IM];
          uint32_t j = e;
          for (; j > i; j--) {
            const uint32_t prev = sm.at[j - 1];
            if (sm.k[prev & IM] <= key) break;
            sm.at[j] = prev;
          }
          if (j < e) sm.at[j] = next;
        }
      }
      if (!__syncthreads_or(bad)) break;
      part = false;
#pragma unroll
      for (int g = 0; g < SPL_G; g++) x[g] = c0 + 32u * g + lane < d ? c0 + 32u * g + lane : ~0u;
    }
    if (VALS) {
      cp_async_wait_all();
      __syncthreads();
    }
    for (uint32_t i = threadIdx.x; i < d; i += NT) {
      const uint32_t at = sm.at[i] & IM;
      keys[lo + i] = sm.k[at];
      if (VALS) vals[lo + i] = sm.v[at];
    }
    __syncthreads();
  }
}

template <int NW, bool VALS>
static cudaError_t seg_radix_launch(uint32_t* keys, uint32_t* vals, const uint64_t* off, SegRows rows,
                                    uint32_t key_bits, bool coarse, cudaStream_t st) {
  if (!rows.count) return cudaSuccess;
  const size_t smem = sizeof(SegRadixSmem<NW, VALS>);
  cudaError_t e = cudaFuncSetAttribute(k_seg_radix<NW, VALS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const uint32_t passes = spl_passes(key_bits);
  k_seg_radix<NW, VALS><<<grid_for(rows.count, 1, 152 * 256), 32 * NW, smem, st>>>(
      keys, vals, off, rows, passes, coarse && passes > 2);
  count_launch();
  return cudaGetLastError();
}

template <int G, bool VALS>
static cudaError_t seg_blk_launch(uint32_t* keys, uint32_t* vals, const uint64_t* off, SegRows rows, cudaStream_t st) {
  if (!rows.count) return cudaSuccess;
  k_seg_blk<G, VALS><<<grid_for(rows.count, 256 / G, 152 * 16), 256, 0, st>>>(keys, vals, off, rows);
  count_launch();
  return cudaGetLastError();
}

// classes k0..9, `rows` in each; `coarse`: rows in the order of degree-mapped labels
template <bool VALS>
static cudaError_t seg_sort_classes(uint32_t* keys, uint32_t* vals, const uint64_t* off, const SegRows (&rows)[SEG_NCLASS],
                                    int k0, uint32_t key_bits, bool coarse, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  for (int k = k0; k < SEG_BIG && e == cudaSuccess; k++) {
    switch (k) {
      case 1: e = seg_blk_launch<4, VALS>(keys, vals, off, rows[k], st); break;
      case 2: e = seg_blk_launch<8, VALS>(keys, vals, off, rows[k], st); break;
      case 3:
      case 4:
        if (VALS) e = seg_radix_launch<1, VALS>(keys, vals, off, rows[k], key_bits, coarse, st);
        else if (k == 3) e = seg_blk_launch<16, false>(keys, nullptr, off, rows[k], st);
        else e = seg_blk_launch<32, false>(keys, nullptr, off, rows[k], st);
        break;
      case 5: e = seg_radix_launch<2, VALS>(keys, vals, off, rows[k], key_bits, coarse, st); break;
      case 6: e = seg_radix_launch<4, VALS>(keys, vals, off, rows[k], key_bits, coarse, st); break;
      case 7: e = seg_radix_launch<8, VALS>(keys, vals, off, rows[k], key_bits, coarse, st); break;
      case 8: e = seg_radix_launch<16, VALS>(keys, vals, off, rows[k], key_bits, coarse, st); break;
      default: e = seg_radix_launch<32, VALS>(keys, vals, off, rows[k], key_bits, coarse, st);
    }
  }
  return e;
}

cudaError_t segmented_sort(uint32_t* keys, uint32_t* vals, const uint64_t* off, uint64_t rows, uint64_t total,
                           uint64_t max_row, cudaStream_t st, uint32_t key_bits, bool big_only) {
  if (rows == 0 || total == 0 || max_row <= (big_only ? SEG_MEDIUM : SEG_SMALL)) return cudaSuccess;
  cudaError_t e;
  // rows by power-of-two size class
  uint32_t* meta = nullptr;  // SEG_NCLASS counts, first places in the list, cursors
  if ((e = lg::pool_alloc((void**)&meta, 3 * SEG_NCLASS * sizeof(uint32_t), st)) != cudaSuccess) return e;
  cudaMemsetAsync(meta, 0, 3 * SEG_NCLASS * sizeof(uint32_t), st);
  k_seg_count<<<grid_for(rows, 256, 152 * 16), 256, 0, st>>>(off, rows, meta);
  count_launch();
  uint32_t cnt[SEG_NCLASS], base[SEG_NCLASS];
  cudaMemcpyAsync(cnt, meta, sizeof(cnt), cudaMemcpyDeviceToHost, st);
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) { cudaFreeAsync(meta, st); return e; }
  uint32_t tot = 0;
  for (int k = 0; k < SEG_NCLASS; k++) { base[k] = tot; tot += cnt[k]; }
  uint32_t* list = nullptr;
  if ((e = lg::pool_alloc((void**)&list, (tot ? tot : 1) * sizeof(uint32_t), st)) != cudaSuccess) {
    cudaFreeAsync(meta, st);
    return e;
  }
  cudaMemcpyAsync(meta + SEG_NCLASS, base, sizeof(base), cudaMemcpyHostToDevice, st);
  k_seg_fill<<<grid_for(rows, 256, 152 * 16), 256, 0, st>>>(off, rows, meta + SEG_NCLASS, meta + 2 * SEG_NCLASS, list);
  count_launch();
  SegRows rows_of[SEG_NCLASS];
  for (int k = 0; k < SEG_NCLASS; k++) rows_of[k] = {list + base[k], 0, cnt[k]};
  const int k0 = big_only ? 8 : 1;
  e = vals ? seg_sort_classes<true>(keys, vals, off, rows_of, k0, key_bits, false, st)
           : seg_sort_classes<false>(keys, vals, off, rows_of, k0, key_bits, false, st);
  if (e == cudaSuccess && cnt[SEG_BIG])
    e = seg_sort_big(keys, vals, off, list + base[SEG_BIG], cnt[SEG_BIG], key_bits, st);
  cudaFreeAsync(list, st);
  cudaFreeAsync(meta, st);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

// =========================================================================
// DM permuter (Section 5.6): label i goes to the i-th vertex in the order
// (degree descending, original ID ascending); the relabeled CSR holds row
// P(v) = sorted { P(u) : u in N_v }.
// =========================================================================
__global__ void k_dm_keys(const uint64_t* __restrict__ rp, uint64_t n, uint64_t max_deg, uint32_t* __restrict__ keys,
                          uint32_t* __restrict__ vals) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x) {
    keys[v] = (uint32_t)(max_deg - (rp[v + 1] - rp[v]));
    vals[v] = (uint32_t)v;
  }
}
__global__ void k_dm_perm(const uint32_t* __restrict__ inv, uint64_t n, uint32_t* __restrict__ perm,
                          const uint64_t* __restrict__ rp, uint32_t* __restrict__ newdeg) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = inv[i];
    perm[v] = (uint32_t)i;
    newdeg[i] = (uint32_t)(rp[v + 1] - rp[v]);
  }
}
// New rows P(v) = { P(u) : u in N_v }.  A warp takes 32 consecutive new rows.
// Rows of <= 32 arcs are gathered into the warp's shared slots (a row per
// step, coalesced reads of the old row, DM_INFLIGHT rows' perm lookups in
// flight),
// sorted one per lane in registers and written out coalesced, so they are
// final here.  Longer rows are copied unsorted (the size-class sorts follow).
// Rows stream through L2 (evict-first loads, streaming stores) so that the
// randomly gathered perm array stays resident (evict-last).
constexpr int DM_INFLIGHT = 8;  // rows whose loads and perm lookups are in flight together

// The weights of short rows: none, moved with the keys, or fetched by the old
// position that the low 5 bits of the sorted word hold (labels below 2^27: half
// the shared memory and a network on one word; R-MAT 2^26 6.4 ms moved, 4.3
// indexed).
enum { DM_PLAIN, DM_MOVED, DM_INDEXED };

template <int MODE>
__global__ void __launch_bounds__(256) k_dm_rows(const uint64_t* __restrict__ rp, const uint32_t* __restrict__ col,
                                                 const uint32_t* __restrict__ w, const uint32_t* __restrict__ inv,
                                                 const uint32_t* __restrict__ perm, const uint64_t* __restrict__ nrp,
                                                 uint32_t* __restrict__ ncol, uint32_t* __restrict__ nw, uint64_t n,
                                                 int skip_big) {
  constexpr bool VALS = MODE != DM_PLAIN, MOVED = MODE == DM_MOVED, IDX = MODE == DM_INDEXED;
  extern __shared__ uint32_t dsm[];  // 8 warps x 32 slots of keys, then of weights if they are moved
  const int lane = threadIdx.x & 31;
  uint32_t* sk = dsm + (threadIdx.x >> 5) * 32 * SROW;
  uint32_t* sv = dsm + 8 * 32 * SROW + (threadIdx.x >> 5) * 32 * SROW;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  const uint64_t pstream = policy_stream(), pkeep = policy_keep();
  for (uint64_t i0 = ((uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; i0 < n;
       i0 += warps * 32) {
    const uint64_t i = i0 + lane;
    uint64_t lo = 0, o = 0;
    uint32_t d = 0;
    if (i < n) {
      const uint32_t v = inv[i];
      lo = rp[v];
      d = (uint32_t)(rp[v + 1] - lo);
      o = nrp[i];
    }
    const bool small = d <= SEG_SMALL;
    const uint32_t todo = __ballot_sync(LG_FULL_MASK, small && d > 0);
    for (uint32_t t = todo; t;) {
      int q[DM_INFLIGHT];
      uint32_t c[DM_INFLIGHT];
      bool on[DM_INFLIGHT];
#pragma unroll
      for (int z = 0; z < DM_INFLIGHT; z++) {
        q[z] = t ? __ffs(t) - 1 : 0;
        on[z] = t != 0;
        if (t) t &= t - 1;
      }
#pragma unroll
      for (int z = 0; z < DM_INFLIGHT; z++) {
        const uint64_t lq = __shfl_sync(LG_FULL_MASK, lo, q[z]);
        const uint32_t dq = __shfl_sync(LG_FULL_MASK, d, q[z]);
        on[z] = on[z] && (uint32_t)lane < dq;
        c[z] = on[z] ? ldg_hint(col + lq + lane, pstream) : 0u;
        if (MOVED && on[z]) sv[q[z] * SROW + lane] = ldg_hint(w + lq + lane, pstream);
      }
#pragma unroll
      for (int z = 0; z < DM_INFLIGHT; z++) {
        if (on[z]) {
          const uint32_t x = ldg_hint(perm + c[z], pkeep);
          sk[q[z] * SROW + lane] = IDX ? x << 5 | (uint32_t)lane : x;
        }
      }
    }
    __syncwarp();
    warp_sort_slots<MOVED>(sk, sv, d, small, lane);
    for (uint32_t t = todo; t;) {
      int q[DM_INFLIGHT];
      uint32_t x[DM_INFLIGHT], y[DM_INFLIGHT];
#pragma unroll
      for (int z = 0; z < DM_INFLIGHT; z++) {
        q[z] = t ? __ffs(t) - 1 : -1;
        if (t) t &= t - 1;
      }
#pragma unroll
      for (int z = 0; z < DM_INFLIGHT; z++) {
        const uint64_t lq = IDX ? __shfl_sync(LG_FULL_MASK, lo, max(q[z], 0)) : 0;
        const uint32_t dq = __shfl_sync(LG_FULL_MASK, d, max(q[z], 0));
        if (q[z] < 0 || (uint32_t)lane >= dq) q[z] = -1 - max(q[z], 0);  // nothing here
        x[z] = q[z] >= 0 ? sk[q[z] * SROW + lane] : 0u;
        y[z] = MOVED && q[z] >= 0 ? sv[q[z] * SROW + lane] : 0u;
        if (IDX) {
          if (q[z] >= 0) y[z] = ldg_hint(w + lq + (x[z] & 31u), pstream);
          x[z] >>= 5;
        }
      }
#pragma unroll
      for (int z = 0; z < DM_INFLIGHT; z++) {
        const uint64_t oq = __shfl_sync(LG_FULL_MASK, o, q[z] >= 0 ? q[z] : -1 - q[z]);
        if (q[z] >= 0) {
          __stcs(ncol + oq + lane, x[z]);
          if (VALS) __stcs(nw + oq + lane, y[z]);
        }
      }
    }
    __syncwarp();
    if (skip_big) continue;  // k_dm_big copies the rows of more than SEG_SMALL arcs
    for (uint32_t t = __ballot_sync(LG_FULL_MASK, !small); t; t &= t - 1) {
      const int q = __ffs(t) - 1;
      const uint64_t lq = __shfl_sync(LG_FULL_MASK, lo, q);
      const uint64_t oq = __shfl_sync(LG_FULL_MASK, o, q);
      const uint32_t dq = __shfl_sync(LG_FULL_MASK, d, q);
      for (uint32_t k = lane; k < dq; k += 32) {
        const uint32_t cc = ldg_hint(col + lq + k, pstream);
        __stcs(ncol + oq + k, ldg_hint(perm + cc, pkeep));
        if (VALS) __stcs(nw + oq + k, ldg_hint(w + lq + k, pstream));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Rows of more than SEG_SMALL arcs in DM order, copied with their IDs mapped.
// What bounds it is the random gather of perm: once perm outgrows the L2, each
// arc fetches 51 B from DRAM for its 4 (R-MAT 2^26: 116 GB read for 15.6 GB of
// arcs).  So the rows are cut in P parts by position and all rows' part 0 goes
// first, then all part 1, ..: a row is sorted by its old IDs, so the parts of
// one phase gather from much the same n / P labels, which stay in the L2
// (gridDim.y = P: blocks start in that order).  Labels go by degree
// descending, so the rows of a size class are consecutive; a warp takes
// 2^lg of them and walks their parts as one range of slots, 4 slots a lane in
// flight (8 take more registers: 2 % slower).  Rows above SEG_MEDIUM arcs are cut in the radix sort's tiles, each
// of which belongs to one phase.
// R-MAT 2^26, weighted, 2.1 G arcs: 22.4 ms in one phase, 14.0 in 8 (the L2's
// sectors for the gathers and the arcs' 16 bytes: 7 TB/s).
// ---------------------------------------------------------------------------
constexpr uint64_t DM_PART_BYTES = 32ull << 20;  // labels a phase gathers from
constexpr uint32_t DM_MAX_PARTS = 32;
constexpr uint32_t DM_TILES = 16;                // tiles a block looks at
constexpr uint32_t DM_WARP_ARCS = 2048;          // arcs a warp takes in one phase, about
constexpr int DM_T = 4;

struct DmClass {
  uint32_t first, rows;  // the class's rows
  uint32_t lg;           // 2^lg rows per warp
  uint32_t warp0;        // first warp
};
struct DmWork {
  DmClass cls[8];
  uint32_t ncls, warps;
  const SrsTile* tiles;
  uint64_t ntiles;
  uint32_t tile_blocks;
};

template <bool VALS>
__global__ void __launch_bounds__(256) k_dm_big(const uint64_t* __restrict__ rp, const uint32_t* __restrict__ col,
                                                const uint32_t* __restrict__ w, const uint32_t* __restrict__ inv,
                                                const uint32_t* __restrict__ perm, const uint64_t* __restrict__ nrp,
                                                DmWork a, uint32_t* __restrict__ ncol, uint32_t* __restrict__ nw) {
  const uint32_t lane = threadIdx.x & 31u, part = blockIdx.y, parts = gridDim.y;
  const uint64_t pstream = policy_stream();
  if (blockIdx.x < a.tile_blocks) {
    const uint64_t t0 = (uint64_t)blockIdx.x * DM_TILES, t1 = min(t0 + DM_TILES, a.ntiles);
    for (uint64_t t = t0; t < t1; t++) {
      const SrsTile d = a.tiles[t];
      if ((uint32_t)((uint64_t)d.tl * parts / d.stride) != part) continue;
      const uint64_t old = rp[inv[d.row]] + (uint64_t)d.tl * RS_TILE;
      for (uint32_t i0 = threadIdx.x; i0 < d.len; i0 += 256 * DM_T) {
        uint32_t c[DM_T], x[DM_T];
#pragma unroll
        for (int j = 0; j < DM_T; j++) {
          const uint32_t i = i0 + 256u * j;
          c[j] = i < d.len ? ldg_hint(col + old + i, pstream) : 0u;
          x[j] = VALS && i < d.len ? ldg_hint(w + old + i, pstream) : 0u;
        }
#pragma unroll
        for (int j = 0; j < DM_T; j++) c[j] = i0 + 256u * j < d.len ? __ldg(perm + c[j]) : 0u;
#pragma unroll
        for (int j = 0; j < DM_T; j++) {
          const uint32_t i = i0 + 256u * j;
          if (i < d.len) {
            __stcs(ncol + d.start + i, c[j]);
            if (VALS) __stcs(nw + d.start + i, x[j]);
          }
        }
      }
    }
    return;
  }
  const uint32_t gw = (blockIdx.x - a.tile_blocks) * 8 + (threadIdx.x >> 5);
  if (gw >= a.warps) return;
  uint32_t k = 0;
  while (k + 1 < a.ncls && gw >= a.cls[k + 1].warp0) k++;
  const uint32_t lg = a.cls[k].lg, r = ((gw - a.cls[k].warp0) << lg) + lane;
  uint64_t src = 0, dst = 0;
  uint32_t len = 0;
  if (lane < (1u << lg) && r < a.cls[k].rows) {
    const uint32_t i = a.cls[k].first + r;
    const uint64_t lo = nrp[i], d = nrp[i + 1] - lo;
    // the cuts lie on 64-byte boundaries of the output
    const uint64_t c0 = part == 0 ? lo : max(lo, (lo + d * part / parts) & ~(uint64_t)15);
    const uint64_t c1 = part + 1 == parts ? lo + d : max(lo, (lo + d * (part + 1) / parts) & ~(uint64_t)15);
    src = rp[inv[i]] + (c0 - lo);
    dst = c0;
    len = (uint32_t)(c1 - c0);
  }
  uint32_t incl = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(LG_FULL_MASK, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  const uint32_t total = __shfl_sync(LG_FULL_MASK, incl, 31);
  src -= incl - len;  // slot s of the range lies at src + s, dst + s
  dst -= incl - len;
  for (uint32_t s0 = 0; s0 < total; s0 += 32 * DM_T) {
    uint32_t c[DM_T], x[DM_T];
    uint64_t to[DM_T];
#pragma unroll
    for (int j = 0; j < DM_T; j++) {
      const uint32_t s = s0 + 32u * j + lane;
      int o = 0;  // the slot's row: lanes with incl <= s come before it
#pragma unroll
      for (int step = 16; step; step >>= 1)
        if (__shfl_sync(LG_FULL_MASK, incl, o + step - 1) <= s) o += step;
      const uint64_t from = __shfl_sync(LG_FULL_MASK, src, o) + s;
      to[j] = __shfl_sync(LG_FULL_MASK, dst, o) + s;
      c[j] = s < total ? ldg_hint(col + from, pstream) : 0u;
      x[j] = VALS && s < total ? ldg_hint(w + from, pstream) : 0u;
    }
#pragma unroll
    for (int j = 0; j < DM_T; j++) c[j] = s0 + 32u * j + lane < total ? __ldg(perm + c[j]) : 0u;
#pragma unroll
    for (int j = 0; j < DM_T; j++) {
      if (s0 + 32u * j + lane < total) {
        __stcs(ncol + to[j], c[j]);
        if (VALS) __stcs(nw + to[j], x[j]);
      }
    }
  }
}

// Maps the rows of classes [k0, k1] (and the tiles, if any) in `parts` phases.
static cudaError_t dm_big(const uint64_t* rp, const uint32_t* col, const uint32_t* w, const uint32_t* inv,
                          const uint32_t* perm, const uint64_t* nrp, const SegRows (&rows)[SEG_NCLASS], int k0, int k1,
                          const SrsTiles& T, uint32_t parts, uint32_t* ncol, uint32_t* nw, cudaStream_t st) {
  DmWork a{};
  for (int k = k1; k >= k0; k--) {
    if (!rows[k].count) continue;
    uint32_t lg = 0;
    while (lg < 5 && (2ull << lg) << (5 + k) <= (uint64_t)DM_WARP_ARCS * parts) lg++;
    a.cls[a.ncls++] = {rows[k].first, rows[k].count, lg, a.warps};
    a.warps += (uint32_t)(((uint64_t)rows[k].count + (1u << lg) - 1) >> lg);
  }
  a.tiles = T.tiles;
  a.ntiles = T.count;
  a.tile_blocks = (uint32_t)((T.count + DM_TILES - 1) / DM_TILES);
  const uint64_t blocks = a.tile_blocks + (uint64_t)(a.warps + 7) / 8;
  if (!blocks) return cudaSuccess;
  const dim3 grid((unsigned)blocks, parts);
  if (w) k_dm_big<true><<<grid, 256, 0, st>>>(rp, col, w, inv, perm, nrp, a, ncol, nw);
  else k_dm_big<false><<<grid, 256, 0, st>>>(rp, col, w, inv, perm, nrp, a, ncol, nw);
  count_launch();
  return cudaGetLastError();
}

// =========================================================================
// Greedy permuter for local IDs (Listing 1, Section 3.2.2).  The listing walks
// the vertices by increasing degree (ties by ID) and hands the next free label
// to each neighbor that has none; so a vertex's label is the rank of its FIRST
// appearance in the neighbor lists concatenated in that order, and vertices
// that never appear follow in ID order.  That rank is computed in parallel:
// every arc offers its position in the concatenation to its target with
// atomicMin, then one sort by (first position, ID) gives the labels.
// =========================================================================
__global__ void k_gr_keys(const uint64_t* __restrict__ rp, uint64_t n, uint32_t* __restrict__ keys,
                          uint32_t* __restrict__ vals) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x) {
    keys[v] = (uint32_t)(rp[v + 1] - rp[v]);
    vals[v] = (uint32_t)v;
  }
}
__global__ void k_gr_degs(const uint64_t* __restrict__ rp, const uint32_t* __restrict__ order, uint64_t n,
                          uint32_t* __restrict__ sdeg, uint64_t* __restrict__ first, uint64_t none,
                          uint32_t* __restrict__ ids) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = order[i];
    sdeg[i] = (uint32_t)(rp[v + 1] - rp[v]);
    first[i] = none;
    ids[i] = (uint32_t)i;
  }
}
// one warp per vertex of the sorted order: its arcs offer positions pos0[i] + j
__global__ void __launch_bounds__(256) k_gr_first(const uint64_t* __restrict__ rp, const uint32_t* __restrict__ col,
                                                  const uint32_t* __restrict__ order, const uint64_t* __restrict__ pos0,
                                                  uint64_t n, unsigned long long* __restrict__ first) {
  const int lane = threadIdx.x & 31;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t i = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
    const uint32_t v = order[i];
    const uint64_t lo = rp[v], d = rp[v + 1] - lo, p = pos0[i];
    for (uint64_t k = lane; k < d; k += 32) {
      const uint32_t u = col[lo + k];
      if ((unsigned long long)(p + k) < first[u]) atomicMin(first + u, (unsigned long long)(p + k));
    }
  }
}

// The rows of more than SEG_SMALL arcs in DM order: mapped, then sorted.
static cudaError_t dm_big_rows(const uint64_t* rp, const uint32_t* col, const uint32_t* w, uint64_t n,
                               const uint32_t* perm, const uint32_t* inv_perm, const uint64_t* nrp, uint32_t* ncol,
                               uint32_t* nw, cudaStream_t st) {
  uint32_t* meta = nullptr;
  uint32_t cnt[SEG_NCLASS];
  uint64_t big_arcs = 0;
  cudaError_t e = lg::pool_alloc((void**)&meta, sizeof(cnt), st);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(meta, 0, sizeof(cnt), st);
  if (e == cudaSuccess) {
    k_seg_count<<<grid_for(n, 256, 152 * 16), 256, 0, st>>>(nrp, n, meta);
    count_launch();
    e = cudaMemcpyAsync(cnt, meta, sizeof(cnt), cudaMemcpyDeviceToHost, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(meta, st);
  if (e != cudaSuccess) return e;
  SegRows rows[SEG_NCLASS] = {};
  uint32_t at = 0;
  for (int k = SEG_BIG; k >= 1; k--) {
    rows[k] = {nullptr, at, cnt[k]};
    at += cnt[k];
  }
  SrsTiles T;
  const uint32_t tiled = rows[7].first;  // rows above SEG_MEDIUM arcs
  if (tiled) {
    e = cudaMemcpyAsync(&big_arcs, nrp + cnt[SEG_BIG], sizeof(uint64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = srs_tiles(nrp, tiled, cnt[SEG_BIG], &T, st);  // waits
  }
  const uint32_t parts = (uint32_t)std::min<uint64_t>((n * sizeof(uint32_t) + DM_PART_BYTES - 1) / DM_PART_BYTES, DM_MAX_PARTS);
  // a part below 16 arcs costs more in torn sectors than its gathers gain:
  // rows of up to 128 arcs go in one phase
  const int kp = parts > 1 ? 3 : 1;
  if (e == cudaSuccess) e = dm_big(rp, col, w, inv_perm, perm, nrp, rows, kp, 7, T, parts, ncol, nw, st);
  if (e == cudaSuccess && kp > 1) e = dm_big(rp, col, w, inv_perm, perm, nrp, rows, 1, kp - 1, SrsTiles{}, 1, ncol, nw, st);
  if (e == cudaSuccess)
    e = w ? seg_sort_classes<true>(ncol, nw, nrp, rows, 1, host_bits(n - 1), true, st)
          : seg_sort_classes<false>(ncol, nullptr, nrp, rows, 1, host_bits(n - 1), true, st);
  if (e == cudaSuccess && cnt[SEG_BIG])
    e = seg_sort_big_prefix(ncol, w ? nw : nullptr, T, big_arcs, host_bits(n - 1), st);
  T.release(st);
  return e;
}

cudaError_t enc_dm_relabel(const uint64_t* rp, const uint32_t* col, const uint32_t* w, uint64_t n, uint64_t arcs,
                           uint64_t max_deg, uint32_t mode, uint32_t* perm, uint32_t* inv_perm, uint64_t* nrp,
                           uint32_t* ncol, uint32_t* nw, cudaStream_t st) {
  cudaError_t e;
  uint32_t *keys = nullptr, *k2 = nullptr, *v2 = nullptr, *newdeg = nullptr;
  uint64_t* stmp = nullptr;
  void* rtmp = nullptr;
  e = lg::pool_alloc((void**)&keys, n * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&k2, n * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&v2, n * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&newdeg, n * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc((void**)&stmp, scan_tmp_words(n) * sizeof(uint64_t), st);
  if (e == cudaSuccess) e = lg::pool_alloc(&rtmp, radix_tmp_bytes(n), st);
  if (e == cudaSuccess && mode == 2) {
    // greedy: order by (degree asc, ID asc), first appearances, sort by them
    uint64_t *pos0 = nullptr, *first = nullptr, *first2 = nullptr;
    e = lg::pool_alloc((void**)&pos0, (n + 1) * sizeof(uint64_t), st);
    if (e == cudaSuccess) e = lg::pool_alloc((void**)&first, n * sizeof(uint64_t), st);
    if (e == cudaSuccess) e = lg::pool_alloc((void**)&first2, n * sizeof(uint64_t), st);
    if (e == cudaSuccess) {
      k_gr_keys<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(rp, n, keys, inv_perm);  // inv_perm: the order
      count_launch();
      e = radix_sort_u32(keys, inv_perm, k2, v2, n, host_bits(max_deg), rtmp, st);
    }
    if (e == cudaSuccess) {
      // first[] indexed by vertex; keys reused as the sorted degrees, v2 as vertex IDs
      k_gr_degs<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(rp, inv_perm, n, keys, first, arcs, v2);
      count_launch();
      e = scan_excl_u32(keys, n, pos0, stmp, st);
    }
    if (e == cudaSuccess) {
      k_gr_first<<<grid_for(n, 8, 152 * 64), 256, 0, st>>>(rp, col, inv_perm, pos0, n,
                                                           reinterpret_cast<unsigned long long*>(first));
      count_launch();
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
      // new label i goes to the vertex with the i-th smallest (first, ID): v2
      // holds 0..n-1, the radix sort is stable, never-seen vertices share key arcs
      e = radix_sort_u64(first, v2, first2, k2, n, host_bits(arcs), rtmp, st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(inv_perm, v2, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
    cudaFreeAsync(pos0, st);
    cudaFreeAsync(first, st);
    cudaFreeAsync(first2, st);
  } else if (e == cudaSuccess) {
    k_dm_keys<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(rp, n, max_deg, keys, inv_perm);
    count_launch();
    e = radix_sort_u32(keys, inv_perm, k2, v2, n, host_bits(max_deg), rtmp, st);
  }
  if (e == cudaSuccess) {
    k_dm_perm<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(inv_perm, n, perm, rp, newdeg);
    count_launch();
    e = scan_excl_u32(newdeg, n, nrp, stmp, st);
  }
  // DM order (degree descending): the rows of each size class are consecutive,
  // the largest first, and go to k_dm_big; the greedy order mixes sizes, so
  // k_dm_rows copies its big rows itself
  const int split_big = mode != 2;
  if (e == cudaSuccess) {
    const bool moved = w && host_bits(n - 1) > 27;
    const size_t smem = (size_t)8 * 32 * SROW * sizeof(uint32_t) * (moved ? 2 : 1);
    const auto rows = !w ? k_dm_rows<DM_PLAIN> : moved ? k_dm_rows<DM_MOVED> : k_dm_rows<DM_INDEXED>;
    if (moved) e = cudaFuncSetAttribute(rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      rows<<<grid_for(n, 256, 152 * 16), 256, smem, st>>>(rp, col, w, inv_perm, perm, nrp, ncol, nw, n, split_big);
    count_launch();
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  // rows of <= 32 arcs left k_dm_rows sorted
  if (e == cudaSuccess && split_big && max_deg > SEG_SMALL)
    e = dm_big_rows(rp, col, w, n, perm, inv_perm, nrp, ncol, nw, st);
  else if (e == cudaSuccess && !split_big)
    e = segmented_sort(ncol, w ? nw : nullptr, nrp, n, arcs, max_deg, st, host_bits(n - 1));
  cudaFreeAsync(keys, st); cudaFreeAsync(k2, st); cudaFreeAsync(v2, st); cudaFreeAsync(newdeg, st);
  cudaFreeAsync(stmp, st); cudaFreeAsync(rtmp, st);
  return e;
}

}  // namespace lg
