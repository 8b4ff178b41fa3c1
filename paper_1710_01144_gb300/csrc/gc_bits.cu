// bitGreedy++ (Sec. 4.3, Theorem 1): Greedy with per-vertex bit vectors.
//
// b^i_u is the set of vertices within distance i of u (b^0_u = {u}, and b^i_u
// is b^{i-1}_u together with b^{i-1}_v of every neighbour v: the closed
// neighbourhood, see the reading of the recurrence).  Theorem 1 gives the
// marginal gain of every vertex at once: Delta(u | S) = sum_i |b^i_u AND NOT
// b^i_S|, where b^i_S holds the vertices w with d_S[w] <= i; and with S empty
// the farness f({u}) = sum_i (n - |b^i_u|) (the vertices farther than i, summed
// over i), so round 0 is the same sweep.
//
// Memory.  n-bit vectors for all n vertices need n^2 bits.  Because distances
// are symmetric, bit t of b^i_u says d(u, t) <= i, so the targets t can be
// taken in chunks of 64 W: for one chunk every vertex holds W words (bit j of
// word q: target base + 64 q + j), the sweep level by level computes those
// words for all u, and the per-vertex sums add up over the chunks.  Two
// buffers of n x W words are the whole memory (the memory limit the paper
// leaves open, with W = 32 at most: 2048 targets per chunk), plus one byte
// per vertex and buffer saying whether its row holds any bit: a level loads
// the words of a neighbour only when its row is nonzero (32 neighbours' flags
// are gathered and balloted at once).
//
// Pruning.  A target t adds to no sum at levels i >= d_S[t] (its bit is
// masked out there), so its bit is dropped from the words from that level on:
// the sweep for target t is a BFS from t cut at depth d_S[t] - 1, the pruned
// SSSP of Sec. 4.1 seen from the other end.
//
// Up to kBitsCtaN vertices (k_bits_cta): a CTA takes 32 targets, and the words
// of all vertices (two buffers of n 32-bit words) and the sums fit its shared
// memory.  The sweep of a CTA's targets needs no other CTA, so a level ends with
// a CTA barrier and its neighbour words are shared-memory reads; k_bits_pick, one
// CTA, then takes the best vertex and updates d_S, so the rounds follow one
// another on the stream without a host round trip.  Bound by the latency of a
// level (row pointers, columns, words, one barrier).  Measured in ms, k = 50
// (the last: k = 20), against the chunks below: road-like 64 x 64 33.9 -> 6.3; BA
// 2000, m = 5, 7.4 -> 2.2; R-MAT scale 12 30.7 -> 4.0, scale 14 89.6 -> 5.4.
//
// Above that (k_bits_round): chunks of 64 W targets in global memory, one
// cooperative launch per round, every level ends with a grid barrier.
#include <limits.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <string>
#include <vector>

#include "gc_device.cuh"
#include "gc_internal.cuh"

namespace gc {

typedef unsigned long long u64;

constexpr int kBitsThreads = 256;

// 32 targets per CTA: targets [32 b, 32 b + 32).  MODE and sums as in
// k_bits_round below; out starts at zero.
constexpr int kBitsCtaThreads = 1024;
// Two forms.  Sparse (ROW = 32): rows of up to 32 entries go to a thread each.  Dense
// (ROW = kBitsRow), where rows average more than kBitsDense entries: threads of a warp
// read different lines, so such rows exceed L1, and rows of 17 to 32 entries go to the
// warp, four at a time; and level 1 is taken from the targets' rows.  20 rounds in ms,
// chunks, sparse form, dense form: random n = 15,900, rows of 18 15.4, 13.7, 10.6, of 34
// 15.7, 27.9, 17.1, of 129 16.1, 30.2, 9.7; n = 4,000, rows of 482 5.9, 8.1, 5.0; ring n
// = 8,000, rows of 32 98, 207, 69, of 128 59, 38.4, 37.5; R-MAT scale 14 90, 11.6, 5.4.
constexpr int kBitsRow = 16;
constexpr int kBitsDense = 8;

template <int MODE, int ROW>
__global__ void __launch_bounds__(kBitsCtaThreads) k_bits_cta(const int32_t *__restrict__ rp,
                                                              const int32_t *__restrict__ ci, int32_t n,
                                                              const int32_t *__restrict__ dS, long long *out,
                                                              BitsCtl *ctl) {
  extern __shared__ uint32_t s_bits[];  // two word buffers and the sums, n each
  if (*(volatile int32_t *)&ctl->err) return;  // an earlier round failed (the rounds are enqueued at once)
  const int tid = threadIdx.x, lane = tid & 31, T = kBitsCtaThreads;
  uint32_t *cur = s_bits, *nxt = s_bits + n;
  int32_t *sum = reinterpret_cast<int32_t *>(s_bits + 2 * (size_t)n);
  const int base = 32 * blockIdx.x, cs = min(32, n - base);
  // every warp keeps the targets' d_S, one per lane (farness: never reached)
  const int dt = lane < cs ? (MODE == 0 ? INT_MAX : __ldg(dS + base + lane)) : 0;
  for (int u = tid; u < n; u += T) {
    const bool own = u >= base && u < base + cs;
    const bool in = own && (MODE == 0 || __ldg(dS + u) > 0);
    cur[u] = in ? 1u << (u - base) : 0u;
    sum[u] = MODE == 0 ? cs - (own ? 1 : 0) : (in ? 1 : 0);  // level 0
  }
  cta_sync();
  int i = 1;
  for (; i <= n; ++i) {
    const uint32_t mask = __ballot_sync(0xffffffffu, dt > i);  // the targets still counted at level i
    if (mask == 0u) break;  // (the same in every warp)
    bool chg = false;
    auto finish = [&](int u, uint32_t own, uint32_t x) {
      const int pc = __popc(x);
      sum[u] += MODE == 1 ? pc : cs - pc;
      chg |= x != (own & mask);
    };
    if (ROW < 32 && i == 1) {
      // level 1: the neighbours of each target, a warp a target (rows hold both
      // directions), instead of every row of the graph.  With two or three levels
      // this is half of a round: random n = 15,900, rows of 256, 43.5 -> 8.6 ms for
      // 20 rounds (17.4 by the chunks)
      for (int u = tid; u < n; u += T) nxt[u] = cur[u] & mask;
      cta_sync();
      static_assert(kBitsCtaThreads / 32 == 32, "a warp a target");
      const int t = tid >> 5;
      if ((mask >> t) & 1u) {
        const int r1 = __ldg(rp + base + t + 1);
#pragma unroll 4
        for (int e = __ldg(rp + base + t) + lane; e < r1; e += 32) atomicOr(&nxt[__ldg(ci + e)], 1u << t);
      }
      cta_sync();
      for (int u = tid; u < n; u += T) finish(u, cur[u], nxt[u]);
    } else {
      // a thread per row of at most ROW entries, the warp together for longer ones
      for (int w0 = tid & ~31; w0 < n; w0 += T) {
        const int u = w0 + lane;
        uint32_t own = 0u, x = 0u;
        int r0 = 0, r1 = 0;
        if (u < n) {
          own = x = cur[u];
          if ((own & mask) != mask) {  // (else every counted target is in already)
            r0 = __ldg(rp + u);
            r1 = __ldg(rp + u + 1);
          }
        }
        const int len = r1 - r0;
        if (len <= ROW) {
          for (int e = r0; e < r1; e += 4) {
            int v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = e + k < r1 ? __ldg(ci + e + k) : u;
#pragma unroll
            for (int k = 0; k < 4; ++k) x |= cur[v[k]];
          }
        }
        unsigned lng = __ballot_sync(0xffffffffu, len > ROW);
        if (ROW < 32 && lng) {
          const unsigned more = __ballot_sync(0xffffffffu, len > 32);
          for (unsigned m = lng & ~more; m;) {  // four rows in flight
            int q[4], w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              q[k] = m ? __ffs(m) - 1 : 32;
              m &= m - 1;
              const int a = __shfl_sync(0xffffffffu, r0, q[k] & 31), l = __shfl_sync(0xffffffffu, len, q[k] & 31);
              w[k] = q[k] < 32 && lane < l ? __ldg(ci + a + lane) : -1;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t y = __reduce_or_sync(0xffffffffu, w[k] >= 0 ? cur[w[k]] : 0u);
              if (lane == q[k]) x |= y;
            }
          }
          lng = more;
        }
        for (; lng; lng &= lng - 1) {
          const int q = __ffs(lng) - 1;
          const int a = __shfl_sync(0xffffffffu, r0, q), b = __shfl_sync(0xffffffffu, r1, q);
          uint32_t y = 0u;
          for (int e = a + lane; e < b; e += 32) y |= cur[__ldg(ci + e)];
          y = __reduce_or_sync(0xffffffffu, y);
          if (lane == q) x |= y;
        }
        if (u < n) {
          x &= mask;
          nxt[u] = x;
          finish(u, own, x);
        }
      }
    }
    uint32_t *t = cur;
    cur = nxt;
    nxt = t;
    // farness: once no word changed, every later level adds nothing
    __syncwarp();
    const int any = __syncthreads_or(chg ? 1 : 0);
    if (MODE == 0 && !any) break;
  }
  for (int u = tid; u < n; u += T)
    if (sum[u]) atomicAdd(reinterpret_cast<u64 *>(&out[u]), (u64)(long long)sum[u]);
  if (tid == 0) atomicAdd(&ctl->levels, (u64)i);
}

// One CTA: the round's pick from the sums (MODE 0 the smallest farness, MODE 1
// the largest gain among u with d_S[u] > 0; ties: smaller id) to picks[r] and
// pgain[r], the sums back to zero, and d_S updated by the pruned relabel BFS from
// the pick (Sec. 4.1; MODE 0: a fresh BFS), its decrease (MODE 0: the farness) to
// pdec[r].  A vertex that round 0 does not reach: *err.
template <int MODE>
__global__ void __launch_bounds__(kBitsCtaThreads) k_bits_pick(const int32_t *__restrict__ rp,
                                                               const int32_t *__restrict__ ci, int32_t n, int32_t *dS,
                                                               long long *out, int32_t r, int32_t *picks,
                                                               long long *pgain, long long *pdec, int32_t *err) {
  extern __shared__ uint32_t s_bits[];  // the BFS queue: every relabelled vertex in BFS order
  if (*(volatile int32_t *)err) return;
  __shared__ long long s_v[32];
  __shared__ int s_id[32];
  __shared__ int s_n;
  int32_t *q = reinterpret_cast<int32_t *>(s_bits);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, T = kBitsCtaThreads;
  long long bv = LLONG_MIN;
  int bid = -1;
  for (int u = tid; u < n; u += T) {
    const long long v = MODE == 0 ? -out[u] : (dS[u] > 0 ? out[u] : LLONG_MIN);
    out[u] = 0;
    if (v != LLONG_MIN && better_max(v, u, bv, bid)) {
      bv = v;
      bid = u;
    }
    if (MODE == 0) dS[u] = kInf;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oid = __shfl_xor_sync(0xffffffffu, bid, o);
    if (better_max(ov, oid, bv, bid)) {
      bv = ov;
      bid = oid;
    }
  }
  if (lane == 0) {
    s_v[wid] = bv;
    s_id[wid] = bid;
  }
  cta_sync();
  bv = s_v[0];
  bid = s_id[0];
  for (int w = 1; w < T / 32; ++w)
    if (better_max(s_v[w], s_id[w], bv, bid)) {
      bv = s_v[w];
      bid = s_id[w];
    }
  cta_sync();  // (s_v is the reduction scratch below)
  if (bid < 0) {  // no vertex left: k <= n rules it out
    if (tid == 0) atomicExch(err, GC_EINTERNAL);
    return;
  }
  long long dec = 0;
  if (tid == 0) {
    picks[r] = bid;
    pgain[r] = MODE == 0 ? -bv : bv;
    if (MODE == 1) dec = dS[bid];
    dS[bid] = 0;
    q[0] = bid;
    s_n = 1;
  }
  cta_sync();
  int a = 0, b = 1;
  for (int nd = 1; a < b; ++nd) {  // the vertices at distance nd - 1 are q[a..b)
    auto claim = [&](int w) {
      if (nd >= *(volatile int32_t *)&dS[w]) return;
      const int old = atomicMin(&dS[w], nd);
      if (old <= nd) return;
      dec += MODE == 0 ? (long long)nd : (long long)(old - nd);
      q[atomicAdd(&s_n, 1)] = w;
    };
    for (int i0 = a + (tid & ~31); i0 < b; i0 += T) {
      const int i = i0 + lane;
      int r0 = 0, r1 = 0;
      if (i < b) {
        r0 = __ldg(rp + q[i]);
        r1 = __ldg(rp + q[i] + 1);
      }
      const bool lng = r1 - r0 > 32;
      if (!lng)
        for (int e = r0; e < r1; ++e) claim(__ldg(ci + e));
      for (unsigned m = __ballot_sync(0xffffffffu, lng); m; m &= m - 1) {
        const int t = __ffs(m) - 1;
        const int x = __shfl_sync(0xffffffffu, r0, t), y = __shfl_sync(0xffffffffu, r1, t);
        for (int e = x + lane; e < y; e += 32) claim(__ldg(ci + e));
      }
    }
    cta_sync();
    a = b;
    b = s_n;
    cta_sync();
  }
  dec = block_sum(dec, s_v);
  if (tid == 0) {
    pdec[r] = dec;
    if (MODE == 0 && b != n) atomicExch(err, GC_EDISCONNECTED);
  }
}

// k rounds of bitGreedy++ on a graph of at most kBitsCtaN vertices, enqueued on
// the handle's stream: picks, gains (round 0: the farness) and d_S decreases to
// g->picks, g->pgain, g->pdec; out (n sums) and ctl are zeroed here.  After a round
// that failed the others return at once: on a disconnected graph each would sweep n
// levels for targets that are never reached (4,096 vertices in 64 components, k = 200:
// 1,107 ms without the look, 1.4 with it).
int launch_bits_small(gc_graph *g, int32_t k, long long *out, BitsCtl *ctl) {
  const int n = g->n, grid = (n + 31) / 32;
  const size_t smem = (size_t)n * 12, smem_q = (size_t)n * 4;
  GC_CUDA(cudaMemsetAsync(ctl, 0, sizeof(BitsCtl), g->stream));
  GC_CUDA(cudaMemsetAsync(out, 0, (size_t)n * sizeof(long long), g->stream));
  const bool dense = g->nnz > (int64_t)kBitsDense * n;
  const auto far = dense ? k_bits_cta<0, kBitsRow> : k_bits_cta<0, 32>;
  const auto gain = dense ? k_bits_cta<1, kBitsRow> : k_bits_cta<1, 32>;
  for (const void *f : {(const void *)far, (const void *)gain})
    GC_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kBitsCtaN * 12));
  for (const void *f : {(const void *)k_bits_pick<0>, (const void *)k_bits_pick<1>})
    GC_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kBitsCtaN * 4));
  g->launches += 2 * k;
  for (int32_t r = 0; r < k; ++r) {
    if (r == 0) {
      far<<<grid, kBitsCtaThreads, smem, g->stream>>>(g->rp, g->ci, n, g->dS, out, ctl);
      k_bits_pick<0><<<1, kBitsCtaThreads, smem_q, g->stream>>>(g->rp, g->ci, n, g->dS, out, r, g->picks, g->pgain,
                                                                g->pdec, &ctl->err);
    } else {
      gain<<<grid, kBitsCtaThreads, smem, g->stream>>>(g->rp, g->ci, n, g->dS, out, ctl);
      k_bits_pick<1><<<1, kBitsCtaThreads, smem_q, g->stream>>>(g->rp, g->ci, n, g->dS, out, r, g->picks, g->pgain,
                                                                g->pdec, &ctl->err);
    }
  }
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// MODE 0: out[u] += sum_i (cs - |b^i_u|) over the chunk (farness, S empty).
// MODE 1: out[u] += sum_i |b^i_u AND NOT b^i_S| over the chunk (gains).
template <int MODE>
__global__ void __launch_bounds__(kBitsThreads) k_bits_round(const int32_t *__restrict__ rp,
                                                             const int32_t *__restrict__ ci, int32_t n,
                                                             const int32_t *dS, int W, u64 *B0, u64 *B1,
                                                             unsigned char *A0, unsigned char *A1,
                                                             long long *out, BitsCtl *ctl,
                                                             unsigned long long tns) {
  __shared__ u64 s_mask[32];
  __shared__ int s_live;
  const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.x, G = gridDim.x, T = blockDim.x;
  const int gw = (b * T + tid) >> 5, nw = (G * T) >> 5;
  const int chunk = 64 * W;
  int32_t *err = &ctl->err;
  u64 lev_total = 0;
  for (int base = 0; base < n; base += chunk) {
    const int cs = min(chunk, n - base);
    // level 0: every target's own bit (gains: only targets outside S)
    for (size_t x = (size_t)b * T + tid; x < (size_t)n * W; x += (size_t)G * T) B0[x] = 0ull;
    for (int u = b * T + tid; u < n; u += G * T) A0[u] = 0;
    if (!grid_sync(&ctl->bar, err, tns)) return;
    for (int j = b * T + tid; j < cs; j += G * T) {
      const int t = base + j;
      if (MODE == 0 || dS[t] > 0) {
        B0[(size_t)t * W + (j >> 6)] = 1ull << (j & 63);
        A0[t] = 1;
        if (MODE == 1) out[t] += 1;  // |b^0_t AND NOT b^0_S| = [d_S[t] > 0]
      }
    }
    if (MODE == 0)  // level 0: every target but u itself is farther than 0
      for (int u = b * T + tid; u < n; u += G * T) out[u] += cs - ((u >= base && u < base + cs) ? 1 : 0);
    if (b == 0 && tid == 0) ctl->changed[0] = ctl->changed[1] = ctl->changed[2] = 0u;
    if (!grid_sync(&ctl->bar, err, tns)) return;
    u64 *cur = B0, *nxt = B1;
    unsigned char *acur = A0, *anxt = A1;  // row nonzero, per vertex
    for (int i = 1;; ++i) {
      // the targets still counted at level i
      if (tid < W) {
        u64 m = 0ull;
        for (int q = 0; q < 64; ++q) {
          const int j = tid * 64 + q;
          if (j < cs && (MODE == 0 || dS[base + j] > i)) m |= 1ull << q;
        }
        s_mask[tid] = m;
      }
      if (tid == 0) s_live = 0;
      cta_sync();
      if (tid < W && s_mask[tid]) atomicOr(&s_live, 1);
      cta_sync();
      if (!s_live || i > n) break;  // no target left (the same decision in every CTA); i > n: never on a connected graph
      if (b == 0 && tid == 0) ctl->changed[(i + 1) % 3] = 0u;  // read two levels from now
      unsigned int chg = 0u;
      for (int u = gw; u < n; u += nw) {
        const u64 own = (lane < W && acur[u]) ? cur[(size_t)u * W + lane] : 0ull;
        u64 x = own;
        for (int e0 = rp[u]; e0 < rp[u + 1]; e0 += 32) {
          // 32 neighbours at once: their row flags, then only the nonzero rows
          const int cnt = min(32, rp[u + 1] - e0);
          const int mine = lane < cnt ? ci[e0 + lane] : 0;
          unsigned live = __ballot_sync(0xffffffffu, lane < cnt && acur[mine] != 0);
          while (live) {
            const int q = __ffs(live) - 1;
            live &= live - 1;
            const int v = __shfl_sync(0xffffffffu, mine, q);
            if (lane < W) x |= cur[(size_t)v * W + lane];
          }
        }
        int pc = 0;
        if (lane < W) {
          x &= s_mask[lane];
          nxt[(size_t)u * W + lane] = x;
          pc = __popcll(x);
          chg |= x != (own & s_mask[lane]);
        }
        const bool nz = __ballot_sync(0xffffffffu, lane < W && x != 0ull) != 0u;
        pc = warp_sum(pc);
        if (lane == 0) {
          anxt[u] = nz ? 1 : 0;
          out[u] += MODE == 1 ? (long long)pc : (long long)(cs - pc);
        }
      }
      if (MODE == 0 && __any_sync(0xffffffffu, chg) && lane == 0) atomicOr(&ctl->changed[i % 3], 1u);
      if (!grid_sync(&ctl->bar, err, tns)) return;
      ++lev_total;
      u64 *t = cur;
      cur = nxt;
      nxt = t;
      unsigned char *ta = acur;
      acur = anxt;
      anxt = ta;
      // farness: once no word changed, every later level adds cs - |b_u| = 0
      // (connected graph: all of the chunk is reached)
      if (MODE == 0 && *(volatile unsigned int *)&ctl->changed[i % 3] == 0u) break;
    }
    if (!grid_sync(&ctl->bar, err, tns)) return;  // the chunk's buffers are reused
  }
  if (b == 0 && tid == 0) ctl->levels = lev_total;
}

// Packed arg-best over the sums: MODE 0 the smallest farness (ties: smaller
// id), MODE 1 the largest gain among u with d_S[u] > 0 (ties: smaller id).
// Values below 2^31 (checked by the host: n <= kBitsMaxN).
template <int MODE>
__global__ void __launch_bounds__(kBitsThreads) k_bits_argbest(const long long *out, const int32_t *dS, int32_t n,
                                                               BitsCtl *ctl) {
  u64 best = 0ull;
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
    if (MODE == 1 && dS[u] <= 0) continue;
    const long long v = out[u];
    const u64 val = MODE == 0 ? (u64)(v >= 0x7fffffffll ? 0ll : 0x7fffffffll - v) : (u64)v;
    const u64 key = (val << 32) | (u64)(0xffffffffu - (unsigned)u);
    best = best > key ? best : key;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const u64 x = __shfl_xor_sync(0xffffffffu, best, o);
    best = best > x ? best : x;
  }
  if ((threadIdx.x & 31) == 0 && best) atomicMax(&ctl->best, best);
}

static int bits_occupancy(int *blocks_per_sm) {
  int a = 0, b = 0;
  GC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_bits_round<0>, kBitsThreads, 0));
  GC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_bits_round<1>, kBitsThreads, 0));
  *blocks_per_sm = std::min(a, b);
  return GC_OK;
}

int launch_bits_round(gc_graph *g, int mode, unsigned long long *B, long long *out, BitsCtl *ctl, int W,
                      int64_t tns) {
  int occ = 0;
  const int rc = bits_occupancy(&occ);
  if (rc != GC_OK) return rc;
  const int grid = std::min(kMaxGridCtas, std::max(1, occ) * g->num_sms);
  const int32_t *rp = g->rp, *ci = g->ci, *dS = g->dS;
  int32_t n = g->n;
  u64 *B0 = B, *B1 = B + (size_t)n * W;
  unsigned char *A0 = (unsigned char *)(B + 2 * (size_t)n * W), *A1 = A0 + n;
  unsigned long long t = (unsigned long long)tns;
  void *args[] = {(void *)&rp, (void *)&ci, (void *)&n, (void *)&dS, (void *)&W, (void *)&B0, (void *)&B1,
                  (void *)&A0, (void *)&A1, (void *)&out, (void *)&ctl, (void *)&t};
  GC_CUDA(cudaMemsetAsync(ctl, 0, sizeof(BitsCtl), g->stream));
  GC_CUDA(cudaMemsetAsync(out, 0, (size_t)n * sizeof(long long), g->stream));
  g->launches += 2;
  GC_CUDA(cudaLaunchCooperativeKernel(mode == 0 ? (const void *)k_bits_round<0> : (const void *)k_bits_round<1>,
                                      dim3(grid), dim3(kBitsThreads), args, 0, g->stream));
  const int rb = std::min(g->num_sms * 4, std::max(1, (n + kBitsThreads - 1) / kBitsThreads));
  if (mode == 0) k_bits_argbest<0><<<rb, kBitsThreads, 0, g->stream>>>(out, g->dS, n, ctl);
  else k_bits_argbest<1><<<rb, kBitsThreads, 0, g->stream>>>(out, g->dS, n, ctl);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

}  // namespace gc
