// Windows of a bit-packed stream, shared by the sweeps that decode them: a warp
// copies the words of up to 256 consecutive fields into shared memory and lane
// l takes the 8 consecutive fields 8 l .. 8 l + 7, whatever vertices they
// belong to (a head bit marks the first field of each vertex).
#pragma once

#include "lg_device.cuh"

namespace lg {

constexpr int PW_G = 8;                // groups of 32 fields per window
constexpr int PW_E = 8;                // consecutive fields of a window per lane
constexpr uint32_t PW_WF = 32 * PW_E;  // fields per window

__device__ __forceinline__ uint32_t lane_lt_mask() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Asynchronous copy of words [w0, w0 + nw) of a stream into shared memory by a
// warp (w0 a multiple of 4, nw <= 128 K, A on a 16-byte boundary), as one group
// of each thread's copies; the last 16 bytes may run into the stream's guard.
// Copies pass the L1 by, whose space the gathers in flight need.
template <int K>
__device__ __forceinline__ void stage_issue(uint32_t* stage, const uint32_t* A, uint64_t w0, uint32_t nw,
                                            uint64_t pol) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage) + 16u * lane;
  const uint32_t* src = A + w0 + 4u * lane;
#pragma unroll
  for (int k = 0; k < K; k++)
    if (4u * lane + 128u * k < nw)
      asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst + 512u * k),
                   "l"(src + 128 * k), "l"(pol)
                   : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// all but the newest N groups of the warp have landed and every lane sees them
template <int N>
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
  __syncwarp();
}

extern __shared__ __align__(16) unsigned char dyn_smem[];

// The 32 bits from bit p on of the CTA's dynamic shared memory: two loads and
// a funnel shift.
__device__ __forceinline__ uint32_t sh_bits(uint32_t p) {
  const uint32_t* a = reinterpret_cast<const uint32_t*>(dyn_smem + ((p >> 3) & ~3u));
  return __funnelshift_r(a[0], a[1], p);
}
__device__ __forceinline__ uint32_t sh_bit0(const void* p) {
  return (uint32_t)(reinterpret_cast<const unsigned char*>(p) - dyn_smem) * 8u;
}

// Per-vertex sums of a window: val the values of the lane's 8 fields (0 past
// the window's end), hb their head bits, je the vertex open before them, open
// the sum so far of the vertex open before the window.  Complete sums go to
// vsum[vertex]; returns the sum of the vertex open at the window's end.  A
// vertex between two heads of a lane is complete there, the part before a
// lane's first head belongs to je, and one segmented scan joins the lanes.
__device__ __forceinline__ float join_window(const float (&val)[PW_E], uint32_t hb, int je, float open,
                                             float* vsum) {
  const uint32_t lane = threadIdx.x & 31u;
  float run = 0.f, pre = 0.f;
  if (!__any_sync(LG_FULL_MASK, __popc(hb) > 1)) {
#pragma unroll
    for (int e = 0; e < PW_E; e++) {
      if (hb & ((2u << e) - 1u)) run += val[e];
      else pre += val[e];
    }
    if (!hb) run = pre;
  } else {
    int j = je;
#pragma unroll
    for (int e = 0; e < PW_E; e++) {
      const bool head = (hb >> e) & 1u, inner = head && (hb & ((1u << e) - 1u));
      if (inner) vsum[j] = run;
      pre = head && !inner ? run : pre;
      j += head;
      run = (head ? 0.f : run) + val[e];
    }
  }
  const uint32_t before = __ballot_sync(LG_FULL_MASK, hb != 0) & (lane_lt_mask() | (1u << lane));
  const int seg = 31 - __clz((int)(before | 1u));
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float z = __shfl_up_sync(LG_FULL_MASK, run, o);
    if ((int)lane - o >= seg) run += z;
  }
  if (!before) run += open;
  float in = __shfl_up_sync(LG_FULL_MASK, run, 1);
  if (lane == 0) in = open;
  if (hb && je >= 0) vsum[je] = in + pre;
  return __shfl_sync(LG_FULL_MASK, run, 31);
}

}  // namespace lg
