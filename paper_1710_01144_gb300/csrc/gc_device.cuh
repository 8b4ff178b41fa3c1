// Device helpers shared by the libgc kernels: bounded grid barrier, timers,
// warp/block reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gc_internal.cuh"

namespace gc {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// CTA barrier.  __syncthreads() is an aligned barrier: it counts a warp
// correctly only if the warp arrives converged.  A warp still split by an
// earlier single-thread branch (thread 0's bookkeeping, a poll) could be
// counted at the wrong barrier, after which its warps run one barrier apart;
// __syncwarp() first reconverges it.  Every CTA barrier of the library goes
// through here.
__device__ __forceinline__ void cta_sync() {
  __syncwarp();
  __syncthreads();
}

// The CTAs that work together on a grid-wide function: CTA b of G.  The whole
// grid, or a team of consecutive CTAs of it (the batched solver); every team
// has barriers and scratch of its own.
struct Team {
  int b, G;
};
__device__ __forceinline__ Team whole_grid() { return Team{(int)blockIdx.x, (int)gridDim.x}; }

// Grid barrier for cooperative launches (all CTAs co-resident) among the CTAs
// of one team.  One 32-bit word per barrier: in every episode CTA 0 of the team
// adds 2^31 - (G - 1) and each other CTA adds 1 (G = the team's size), so the episode adds exactly 2^31: bit 31 of the
// word flips at the last arrival and the low 31 bits come back to zero, ready
// for the next episode (of any grid size).  Arrival is a release atomic by
// thread 0, the wait an acquire poll of bit 31; the CTA barriers on both sides
// extend the ordering to every thread.  The poll is bounded twice: by
// `timeout_ns` of global time and by an iteration cap.  On expiry the CTA
// records GC_ETIMEOUT in *err and the barrier returns false; every caller then
// leaves its kernel.  Returns false as well when *err is already set.  A word
// left mid-episode by such an exit must be zeroed before its next launch.
__device__ __forceinline__ bool grid_sync(GridBar *bar, int32_t *err,
                                          unsigned long long timeout_ns, Team tm) {
  __shared__ int s_ok;
  cta_sync();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned int add = tm.b == 0 ? 0x80000000u - ((unsigned)tm.G - 1u) : 1u;
    unsigned int old;
    asm volatile("atom.add.release.gpu.u32 %0, [%1], %2;" : "=r"(old) : "l"(&bar->count), "r"(add) : "memory");
    const unsigned long long t0 = global_ns();
    unsigned int it = 0;
    for (;;) {
      unsigned int cur;
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(&bar->count) : "memory");
      if ((cur ^ old) & 0x80000000u) break;
      ++it;
      if ((it & 3u) == 0 && (global_ns() - t0 > timeout_ns || it > (1u << 30))) {
        atomicExch(err, GC_ETIMEOUT);
        ok = 0;
        break;
      }
    }
    s_ok = ok && (*(volatile int32_t *)err == 0);
  }
  cta_sync();
  return s_ok != 0;
}

__device__ __forceinline__ bool grid_sync(GridBar *bar, int32_t *err, unsigned long long timeout_ns) {
  return grid_sync(bar, err, timeout_ns, whole_grid());
}

// A load through the read-only data path when RO (the data must not change
// while the kernel can still read it), else a plain load.  For the same reason
// no pointer to data that a persistent kernel rewrites (d_S, bounds, stamps,
// selected candidates, active lists) is declared const __restrict__: the
// compiler may then load it through the non-coherent read-only path, which a
// grid barrier does not refresh.
template <bool RO>
__device__ __forceinline__ int32_t ld_ro(const int32_t *p) {
  if (RO) return __ldg(p);
  return *p;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum; every thread gets the result.  `sh` needs 32 entries.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T *sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum(v);
  cta_sync();
  if (lane == 0) sh[wid] = v;
  cta_sync();
  const int nw = (blockDim.x + 31) >> 5;
  T r = (threadIdx.x < nw) ? sh[threadIdx.x] : T(0);
  if (wid == 0) r = warp_sum(r);
  if (threadIdx.x == 0) sh[0] = r;
  cta_sync();
  r = sh[0];
  cta_sync();
  return r;
}

// Sums of the claims of one warp by batch lane: thread t won the lanes in `won`,
// each worth wt.  Thread j gets the sums of lanes j and j + 32 added to a and b, and
// with COUNT their numbers to ca and cb.  The 32 x 64 bits are transposed (10
// shuffles), so that thread j holds the threads that won lane j, and the weights are
// taken by bit planes (a gain is 1 or 2 nearly always): a fixed cost, where an
// atomic a lane and claim on 64 shared words serialises a warp whose claims hold
// many lanes, as on every level but the first few of a batch.  Lazy rounds in ms,
// before and now: BA n = 50,000, m = 1 20.2, 15.5; n = 200,000, m = 8 4.6, 3.7; R-MAT
// scale 20 6.3, 5.9; 64-lane batches of one CTA on BA n = 50,000 12.8, 8.1.
template <bool COUNT>
__device__ __forceinline__ void warp_lane_sums(unsigned long long won, unsigned wt, unsigned long long &a,
                                               unsigned long long &b, unsigned &ca, unsigned &cb) {
  const int lane = threadIdx.x & 31;
  unsigned x = (unsigned)won, y = (unsigned)(won >> 32);
  const unsigned ox = __reduce_or_sync(0xffffffffu, x), oy = __reduce_or_sync(0xffffffffu, y);
  if (!(ox | oy)) return;
  if (won == 0) wt = 0;
  if (__popc(ox) + __popc(oy) == 1) {  // one lane alone: a long row at level 0
    const unsigned n1 = COUNT ? __popc(__ballot_sync(0xffffffffu, won != 0)) : 0u;
    const unsigned long long s = (unsigned long long)__reduce_add_sync(0xffffffffu, wt & 0xffffu) +
                                 ((unsigned long long)__reduce_add_sync(0xffffffffu, wt >> 16) << 16);
    if (lane == __ffs(ox | oy) - 1) {
      if (ox) {
        a += s;
        if (COUNT) ca += n1;
      } else {
        b += s;
        if (COUNT) cb += n1;
      }
    }
    return;
  }
  unsigned low = 0x0000ffffu;  // bit positions without bit j
#pragma unroll
  for (int j = 16; j > 0; j >>= 1, low ^= low << j) {
    const unsigned p = __shfl_xor_sync(0xffffffffu, x, j), q = __shfl_xor_sync(0xffffffffu, y, j);
    if (lane & j) {
      x = (x & ~low) | ((p & ~low) >> j);
      y = (y & ~low) | ((q & ~low) >> j);
    } else {
      x = (x & low) | ((p & low) << j);
      y = (y & low) | ((q & low) << j);
    }
  }
  if (COUNT) {
    ca += __popc(x);
    cb += __popc(y);
  }
  for (unsigned m = __reduce_or_sync(0xffffffffu, wt), i = 0; m; m >>= 1, ++i) {
    const unsigned plane = __ballot_sync(0xffffffffu, (wt >> i) & 1u);
    a += (unsigned long long)__popc(x & plane) << i;
    b += (unsigned long long)__popc(y & plane) << i;
  }
}

// Block-wide exclusive scan of int32 (blockDim.x <= 1024); returns the
// exclusive prefix, *total gets the block total.  `sh` needs 33 entries.
__device__ __forceinline__ int block_excl_scan(int v, int *sh, int *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  cta_sync();
  if (lane == 31) sh[wid] = x;
  cta_sync();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    int s = (lane < nw) ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < nw) sh[lane] = s;  // inclusive prefix of warp totals
    if (lane == nw - 1) sh[32] = s;
  }
  cta_sync();
  const int warp_off = wid ? sh[wid - 1] : 0;
  *total = sh[32];
  const int r = warp_off + x - v;
  cta_sync();
  return r;
}

// Degree classes of the round-0 far counts (k_far_counts in gc_bfs.cu).
constexpr int kFarDeg = 8;

__device__ __forceinline__ unsigned long long far_class(int deg) {  // the class's unit in a packed pair of counts
  return deg < 1 || deg > kFarDeg ? 0ull : (deg <= 2 ? 1ull : 1ull << 32);
}

// (value, id) pairs ordered by larger value, then smaller id.
__device__ __forceinline__ bool better_max(long long v, int id, long long bv, int bid) {
  return v > bv || (v == bv && (unsigned)id < (unsigned)bid);
}
// (value, id) pairs ordered by smaller value, then smaller id.
__device__ __forceinline__ bool better_min(long long v, int id, long long bv, int bid) {
  return v < bv || (v == bv && (unsigned)id < (unsigned)bid);
}

}  // namespace gc
