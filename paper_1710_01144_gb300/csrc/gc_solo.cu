// Deep graphs (roads, paths, grids): one source per small CTA.
//
// Why a kernel of its own.  The 64-lane batches (gc_gain.cu) share a row scan
// among the lanes that reach a vertex at the same level.  On deep graphs
// distinct candidates, even neighbours, reach most vertices at different
// levels, so a scan serves 1.4 lanes on average, while every claim pays for
// 32-byte lane-word records in a working set that does not fit L2 (44 bytes
// per vertex and CTA) and a whole 512-thread CTA waits at every one of several
// hundred levels.  A single search needs one visited bit per vertex: 8 KB of
// shared memory for 65,536 vertices, so a claim is a shared-memory atomic, the
// sums stay in registers, and up to sixteen 128-thread CTAs share an SM and
// cover each other's level barriers.
//
// The search.  Level-synchronous BFS from one source; the queue (one int32 per
// vertex in global memory, written and read by this CTA alone) keeps every
// visited vertex in BFS order, so level L is a slice of it.  The queues lie in the
// memory of the 64-lane batches' workspaces, which are zero at rest: a CTA puts
// zeros back where it wrote once it has no more sources (kernels of the same stream
// run before or after, never beside).  Queues of their own were 640 MB at 65,536 vertices, for every sparse
// handle; greedy on road-like 256 x 256, k = 20, takes 37.8 ms, 37.5 with those.  A thread takes a
// frontier vertex and its row, four entries in flight; rows longer than
// kSoloRow are taken by the warp together.  One CTA barrier per level: the
// level's claims are counted in one of three counters in rotation.
//
// kModeGain: Delta(v | S) with the pruning of Sec. 4.1, relaxed by `slack`:
// vertices with d_S + slack > d(v, .) are visited, those with d_S > d(v, .)
// contribute.  region[i] is the number visited.  For any candidate x at
// distance t <= slack from v,
//   Delta(x | S) <= Delta(v | S) + t * region(v):
// d(x, u) >= d(v, u) - t for every u, and only the u with d(v, u) - t < d_S(u)
// can gain from it (a shortest path to such a u stays inside the region).
// kModeFarness: f({v}), cut like BFScut (Sec. 3.1) once the distances counted
// so far exceed the best farness even if every unvisited vertex is in the next
// level.  For every x at distance t from v, f({x}) >= f({v}) - t (n - 2).
// k_relax passes both kinds of bounds from the searched vertices to their
// neighbourhoods, so that most candidates are never searched.
//
// Bound by the latency of a level (dependent loads of the queue, the row, d_S and
// one barrier, about 1 us) that many small CTAs overlap.  Measured, against the
// 64-lane batches: road-like 256 x 256, k = 20: 589 -> 45.9 ms (round 0 154 -> 10
// ms: 40,273 searches -> 5,400; rounds 1 to 19: 357,000 evaluations -> 71,000);
// 300 x 300, k = 20: 1058 -> 62 ms; 1001 gains on 512 x 512 against a group of 50:
// 9.03 -> 1.91 ms; top-60 closeness on 220 x 220: 226 -> 38 ms.
#include <limits.h>

#include <algorithm>

#include "gc_device.cuh"
#include "gc_internal.cuh"

namespace gc {

typedef unsigned long long u64;

constexpr int kSoloThreads = 128;
constexpr int kSoloRow = 32;  // longer rows are shared by the warp

// With `deep_only`, the kernel runs only if the BFS that filled d_S went deeper
// than kWideLevels (bctl->levels); otherwise the 64-lane kernel launched beside
// it does the work.  With MANY, the first `head` searches count what they scan, and the
// first CTA to come for a later one decides whether the 64-lane batches take the rest.
template <int MODE, bool MANY = false>
__global__ void __launch_bounds__(kSoloThreads, 16)
    k_solo(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n, const int32_t *__restrict__ dS,
           const int32_t *__restrict__ mx, const int32_t *__restrict__ cand, int32_t n_cand_arg,
           const int32_t *__restrict__ n_cand_dev, long long *__restrict__ out, int32_t *__restrict__ region,
           int32_t *queues, long long q_stride, GainCtl *ctl, const BfsCtl *deep_only, int32_t slack, int32_t no_cut,
           int32_t head, const SelCtl *sctl) {
  extern __shared__ __align__(16) uint32_t s_seen[];  // one bit per vertex
  __shared__ int s_task;
  __shared__ int s_new[3];
  __shared__ long long s_best;
  __shared__ long long s_red[32];
  if (deep_only && *(volatile const int32_t *)&deep_only->levels <= kWideLevels) return;
  const int tid = threadIdx.x, lane = tid & 31, T = kSoloThreads;
  const int nw4 = ((n + 31) / 32 + 3) / 4;  // bitmap in 16-byte units
  uint4 *seen4 = reinterpret_cast<uint4 *>(s_seen);
  int32_t *q = queues + (size_t)blockIdx.x * q_stride;
  const int n_cand = n_cand_dev ? *n_cand_dev : n_cand_arg;
  u64 w_edges = 0, w_levels = 0, w_front = 0, w_tasks = 0;
  unsigned w_head = 0;  // searches whose counts are in *ctl already
  bool stop = false;    // thread 0
  int high = 0;  // entries of the queue that were written
  for (int i = tid; i < nw4; i += T) seen4[i] = make_uint4(0, 0, 0, 0);
  for (;;) {
    if (tid == 0) {
      const int rest = MANY ? *(volatile int32_t *)&ctl->lanes_rest : 0;
      s_task = MANY && stop ? n_cand : (int)atomicAdd(&ctl->batch_next, 1u);
      stop = rest == 2;  // (after the one just taken)
      if (MANY && rest == 0 && s_task >= head)  // the first searches are through, or nearly
        atomicCAS(&ctl->lanes_rest, 0,
                  lanes_take_rest(*(volatile u64 *)&ctl->edges_scalar, *(volatile u64 *)&ctl->lanes, __ldg(rp + n),
                                  (int64_t) * (volatile unsigned long long *)&sctl->sum, n)
                      ? 2
                      : 1);
      s_new[0] = s_new[1] = s_new[2] = 0;
      if (MODE == kModeFarness) s_best = no_cut ? LLONG_MAX : *(volatile long long *)&ctl->best_f;
    }
    cta_sync();
    const int task = s_task;
    if (task >= n_cand) break;
    const int c = cand[task];
    const int dc = (MODE == kModeGain && c >= 0 && c < n) ? __ldg(dS + c) : 1;
    if (c < 0 || c >= n || dc <= 0) {  // invalid id, or a member of S
      cta_sync();
      if (tid == 0) {
        out[task] = c < 0 || c >= n ? -1 : 0;
        if (c < 0 || c >= n) atomicExch(&ctl->err, GC_EINVAL);
        if (region) region[task] = 0;
      }
      continue;
    }
    const long long best = MODE == kModeFarness ? s_best : 0;
    if (tid == 0) {
      s_seen[c >> 5] = 1u << (c & 31);
      q[0] = c;
    }
    cta_sync();
    long long acc = 0;             // gain: this thread's contributions
    long long sum = 0;             // farness: the distances counted (same in every thread)
    int a = 0, b = 1;              // the level's slice of the queue
    bool cut = false;
    int L = 0;
    for (; a < b; ++L) {
      const int nlev = L + 1;
      int *cnt = &s_new[L % 3];
      if (tid == 0) s_new[(L + 1) % 3] = 0;  // the next level's; every thread read it last before the barrier of level L - 1
      for (int base = a; base < b; base += T) {
        const int i = base + tid;
        int r0 = 0, r1 = 0;
        if (i < b) {
          const int u = q[i];
          r0 = __ldg(rp + u);
          r1 = __ldg(rp + u + 1);
          // no neighbour of u can be visited: skip its row
          if (MODE == kModeGain && mx && __ldg(mx + u) + slack <= nlev) r1 = r0;
          w_edges += (u64)(r1 - r0);
        }
        // entries e0, e0 + step, ... (four per round) of this thread's row
        auto scan = [&](int e0, int end, int step) {
          int w[4], d[4];
          unsigned won = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) w[k] = e0 + k * step < end ? __ldg(ci + e0 + k * step) : -1;
          if (MODE == kModeGain) {
#pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = w[k] >= 0 ? __ldg(dS + w[k]) : 0;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (w[k] < 0 || (MODE == kModeGain && d[k] + slack <= nlev)) continue;
            const uint32_t bit = 1u << (w[k] & 31);
            if (s_seen[w[k] >> 5] & bit) continue;
            if (atomicOr(&s_seen[w[k] >> 5], bit) & bit) continue;
            won |= 1u << k;
            if (MODE == kModeGain && d[k] > nlev) acc += d[k] - nlev;
          }
          const int mine = __popc(won);
          int incl = mine;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          const int all = __shfl_sync(0xffffffffu, incl, 31);
          if (!all) return;
          int at = 0;
          if (lane == 0) at = atomicAdd(cnt, all);
          at = b + __shfl_sync(0xffffffffu, at, 0) + incl - mine;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if ((won >> k) & 1u) q[at++] = w[k];
        };
        const bool lng = r1 - r0 > kSoloRow;
        int most = __reduce_max_sync(0xffffffffu, lng ? 0u : (unsigned)(r1 - r0));
        for (int e = 0; e < most; e += 4) scan(r0 + e, lng ? r0 : r1, 1);  // (warp-uniform trip count)
        for (unsigned m = __ballot_sync(0xffffffffu, lng); m; m &= m - 1) {
          const int t = __ffs(m) - 1;
          const int x0 = __shfl_sync(0xffffffffu, r0, t), x1 = __shfl_sync(0xffffffffu, r1, t);
          for (int e = x0; e < x1; e += 128) scan(e + lane, x1, 32);
        }
      }
      if (MODE == kModeGain && tid == 0) w_front += (u64)(b - a);
      cta_sync();
      const int fresh = *cnt;
      a = b;
      b += fresh;
      if (MODE == kModeFarness) {
        sum += (long long)nlev * fresh;
        // b vertices within distance L + 1, the rest at L + 2 or more
        if (fresh > 0 && sum + (long long)(L + 2) * (long long)(n - b) > best) {
          cut = true;
          ++L;
          break;
        }
      }
    }
    w_levels += (u64)L;
    ++w_tasks;
    if (MODE == kModeGain) acc = block_sum(acc, s_red);
    if (MANY && task < head) {
      w_edges = block_sum(w_edges, (u64 *)s_red);
      if (tid == 0) {
        atomicAdd(&ctl->edges_scalar, w_edges);
        atomicAdd(&ctl->edges_union, w_edges);
        atomicAdd(&ctl->lanes, 1ull);
      }
      w_edges = 0;
      ++w_head;
    }
    if (tid == 0) {
      if (MODE == kModeGain) {
        out[task] = (long long)dc + acc;
        if (region) region[task] = b;
      } else if (cut) {
        out[task] = -1;
      } else if (b != n) {
        out[task] = -1;
        ctl->short_vertex = c;
        ctl->short_count = b;
        atomicExch(&ctl->err, GC_EDISCONNECTED);
      } else {
        out[task] = sum;
        if (!ctl->fixed_best) atomicMin(&ctl->best_f, sum);
      }
    }
    // the bitmap back to zero: by the queue while that is the shorter list
    high = max(high, b);
    cta_sync();
    if (b < 2 * nw4) {
      for (int i = tid; i < b; i += T) s_seen[q[i] >> 5] = 0u;
    } else {
      for (int i = tid; i < nw4; i += T) seen4[i] = make_uint4(0, 0, 0, 0);
    }
    cta_sync();
  }
  uint4 *q4 = reinterpret_cast<uint4 *>(q);  // (a queue's length is a multiple of 4)
  for (int i = tid; i < (high + 3) / 4; i += T) q4[i] = make_uint4(0, 0, 0, 0);
  w_edges = block_sum(w_edges, (u64 *)s_red);
  if (tid == 0 && w_tasks) {
    atomicAdd(&ctl->edges_scalar, w_edges);
    atomicAdd(&ctl->edges_union, w_edges);
    atomicAdd(&ctl->levels, w_levels);
    atomicAdd(&ctl->batches, w_tasks);
    atomicAdd(&ctl->frontier, w_front);
    atomicAdd(&ctl->pushes, w_front);
    atomicAdd(&ctl->lanes, w_tasks - w_head);
  }
}

static size_t solo_smem(int32_t n) { return (size_t)((n + 31) / 32 + 3) / 4 * 16; }

static size_t solo_queue_bytes(int32_t n) { return ws_align((size_t)n * sizeof(int32_t)); }

// CTAs of the solo kernel for a graph of n vertices (0: its bitmap does not fit
// shared memory), with queues in ws_bytes of workspaces.
int solo_plan(int32_t n, int num_sms, size_t ws_bytes, int *ctas) {
  *ctas = 0;
  const size_t smem = solo_smem(n);
  if (smem > 200 * 1024) return GC_OK;
  int x = 0, y = 0;
  GC_CUDA(cudaFuncSetAttribute(k_solo<kModeGain>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  GC_CUDA(cudaFuncSetAttribute(k_solo<kModeGain, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  GC_CUDA(cudaFuncSetAttribute(k_solo<kModeFarness>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  GC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x, k_solo<kModeGain>, kSoloThreads, smem));
  GC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&y, k_solo<kModeFarness>, kSoloThreads, smem));
  const size_t fit = ws_bytes / solo_queue_bytes(n);
  *ctas = (int)std::min<size_t>((size_t)std::min(x, y) * num_sms, fit);
  return GC_OK;
}

int launch_solo(gc_graph *g, int mode, const int32_t *cand, int32_t n_cand, const int32_t *n_cand_dev, long long *out,
                int32_t *region, int32_t slack, bool no_cut, bool deep_only, int32_t head) {
  if (!n_cand_dev && n_cand <= 0) return GC_OK;
  // (with deep_only the caller has just zeroed *gctl)
  if (!deep_only) GC_CUDA(cudaMemsetAsync(&g->gctl->batch_next, 0, sizeof(unsigned int), g->stream));
  int ctas = g->solo_ctas;
  if (!n_cand_dev) ctas = std::min(ctas, n_cand);
  ++g->launches;
  const BfsCtl *deep = deep_only ? g->bctl : nullptr;
  const size_t smem = solo_smem(g->n);
  int32_t *queues = (int32_t *)g->ws;
  const long long q_stride = (long long)(solo_queue_bytes(g->n) / sizeof(int32_t));
  if (mode == kModeGain && head > 0)
    k_solo<kModeGain, true><<<ctas, kSoloThreads, smem, g->stream>>>(g->rp, g->ci, g->n, g->dS, g->mx, cand, n_cand,
                                                                     n_cand_dev, out, region, queues, q_stride,
                                                                     g->gctl, deep, slack, 0, head, g->sctl);
  else if (mode == kModeGain)
    k_solo<kModeGain><<<ctas, kSoloThreads, smem, g->stream>>>(g->rp, g->ci, g->n, g->dS, g->mx, cand, n_cand,
                                                               n_cand_dev, out, region, queues, q_stride, g->gctl,
                                                               deep, slack, 0, 0, nullptr);
  else
    k_solo<kModeFarness><<<ctas, kSoloThreads, smem, g->stream>>>(g->rp, g->ci, g->n, g->dS, nullptr, cand, n_cand,
                                                                  n_cand_dev, out, nullptr, queues, q_stride, g->gctl,
                                                                  deep, 0, no_cut ? 1 : 0, 0, nullptr);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// What the one-source searches left to the 64-lane batches (all in stream order, so that
// the call needs no host read and can be captured).
__global__ void k_lanes_rest(GainCtl *ctl, int32_t n_cand) {
  ctl->rest_first = ctl->lanes_rest == 2 ? (int32_t)min(ctl->batch_next, (unsigned)n_cand) : n_cand;
  ctl->batch_next = 0;
}

int launch_deep_gains(gc_graph *g, const int32_t *cand, int32_t n_cand, long long *out, bool deep_only) {
  const bool many = n_cand > kLanesFrom && g->n >= kLanesMinN;
  const int rc = launch_solo(g, kModeGain, cand, n_cand, nullptr, out, nullptr, 0, false, deep_only,
                             many ? kLanesHead : 0);
  if (rc != GC_OK || !many) return rc;
  ++g->launches;
  k_lanes_rest<<<1, 1, 0, g->stream>>>(g->gctl, n_cand);
  GC_CUDA(cudaGetLastError());
  return launch_gains(g, kModeGain, cand, n_cand, nullptr, out, 0, kLanes, false, true, false, true);
}

// ---- bounds for the neighbourhoods of searched vertices ----

// val[v] <- +infinity, then val[list[i]] <- (MODE gain: the gain; farness:
// -f) and slope[list[i]] <- region[i] for the searched vertices.  Cut searches
// (out < 0) start nothing.
__global__ void k_relax_init(int32_t n, long long *val) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) val[v] = LLONG_MAX;
}

__global__ void k_relax_seed(const int32_t *__restrict__ list, const int32_t *m_dev, const long long *__restrict__ out,
                             const int32_t *__restrict__ region, int32_t farness, long long *val, int32_t *slope) {
  const int m = *m_dev;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const long long o = out[i];
    if (o < 0) continue;
    val[list[i]] = farness ? -o : o;
    if (region) slope[list[i]] = region[i];
  }
}

// One hop: val1[v] <- min(val0[v], min over neighbours w of val0[w] + slope[w]),
// the slope following the value taken.  slope0 == nullptr: the constant `step`.  A
// thread per row of at most kSoloRow entries, the warp together for longer ones, the
// CTA for those of the list of long rows: deep graphs may have hubs (a broom of
// 100,000 leaves, k = 5, on this path: 1,240 ms with a thread per row, 68 so; road-like
// 120 x 120 with a vertex of 50,000 leaves, k = 10: 816, 88).
constexpr int kRelaxThreads = 256;

__global__ void __launch_bounds__(kRelaxThreads)
    k_relax(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n,
            const long long *__restrict__ val0, const int32_t *__restrict__ slope0, long long *__restrict__ val1,
            int32_t *__restrict__ slope1, long long step, const int32_t *__restrict__ heavy,
            const int32_t *__restrict__ nh) {
  __shared__ long long s_v[kRelaxThreads / 32];
  __shared__ int s_sl[kRelaxThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  long long best;
  int sl;
  auto start = [&](int v) {
    best = val0[v];
    sl = slope0 ? slope0[v] : 0;
  };
  auto take = [&](long long y, int s) {
    if (y < best) {
      best = y;
      sl = s;
    }
  };
  auto scan = [&](int e0, int e1, int by) {
    for (int e = e0; e < e1; e += by) {
      const int w = ci[e];
      const long long x = val0[w];
      if (x == LLONG_MAX) continue;
      const int s = slope0 ? slope0[w] : 0;
      take(x + (slope0 ? (long long)s : step), s);
    }
  };
  auto fold_warp = [&]() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long y = __shfl_xor_sync(0xffffffffu, best, o);
      const int s = __shfl_xor_sync(0xffffffffu, sl, o);
      if (y < best || (y == best && s < sl)) {
        best = y;
        sl = s;
      }
    }
  };
  auto put = [&](int v) {
    val1[v] = best;
    if (slope1) slope1[v] = sl;
  };
  for (int base = (blockIdx.x * kRelaxThreads + tid) & ~31; base < n; base += gridDim.x * kRelaxThreads) {
    const int v = base + lane;
    const int r0 = v < n ? rp[v] : 0, r1 = v < n ? rp[v + 1] : 0, len = r1 - r0;
    if (v < n && len <= kSoloRow) {
      start(v);
      scan(r0, r1, 1);
      put(v);
    }
    for (unsigned m = __ballot_sync(0xffffffffu, len > kSoloRow && len <= kHeavyRow); m; m &= m - 1) {
      const int t = __ffs(m) - 1;
      const int x0 = __shfl_sync(0xffffffffu, r0, t), x1 = __shfl_sync(0xffffffffu, r1, t);
      start(base + t);
      scan(x0 + lane, x1, 32);
      fold_warp();
      if (lane == 0) put(base + t);
    }
  }
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int v = heavy[i];
    start(v);
    scan(rp[v] + tid, rp[v + 1], kRelaxThreads);
    fold_warp();
    cta_sync();  // the last row's readers
    if (lane == 0) {
      s_v[tid >> 5] = best;
      s_sl[tid >> 5] = sl;
    }
    cta_sync();
    if (tid == 0) {
      for (int w = 1; w < kRelaxThreads / 32; ++w) take(s_v[w], s_sl[w]);
      put(v);
    }
  }
}

// ub[v] lowered to val[v] for candidates not evaluated in `round`; or (farness)
// key[v] for undecided vertices.
__global__ void k_relax_apply(int32_t n, const long long *__restrict__ val, long long *key, const int32_t *stamp,
                              int32_t round) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const long long k = key[v];
    if (stamp ? (k < 0 || stamp[v] == round) : k == LLONG_MIN) continue;
    if (val[v] < k) key[v] = val[v];
  }
}

int launch_relax(gc_graph *g, bool farness, const int32_t *region, int32_t hops, int32_t round) {
  // round 0 keeps key and f0, later rounds keep ub: the other arrays are free
  long long *v0 = g->akey, *v1 = farness ? g->ub : g->key;
  int32_t *s0 = farness ? nullptr : g->gx, *s1 = farness ? nullptr : g->gx + g->n;
  const int blocks = std::min((g->n + 255) / 256, g->num_sms * 8);
  g->launches += 3 + hops;
  k_relax_init<<<blocks, 256, 0, g->stream>>>(g->n, v0);
  k_relax_seed<<<g->red_blocks, 256, 0, g->stream>>>(g->list, &g->sctl->n_sel, g->lgain, region, farness ? 1 : 0, v0,
                                                     s0);
  for (int h = 0; h < hops; ++h) {
    k_relax<<<blocks, kRelaxThreads, 0, g->stream>>>(g->rp, g->ci, g->n, v0, s0, v1, s1, (long long)g->n - 2, g->heavy,
                                                     g->n_heavy);
    std::swap(v0, v1);
    std::swap(s0, s1);
  }
  k_relax_apply<<<blocks, 256, 0, g->stream>>>(g->n, v0, farness ? g->key : g->ub, farness ? nullptr : g->stamp,
                                               round);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// About `want` of the m listed vertices (sample_takes) into `sample`; *count (zeroed
// by the caller) gets how many, 1 to m.
__global__ void k_sample(const int32_t *__restrict__ list, const int32_t *m_dev, int32_t want, uint32_t salt,
                         int32_t *sample, int32_t *count) {
  const int m = *m_dev;
  const int lane = threadIdx.x & 31;
  for (int base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; base < m; base += gridDim.x * blockDim.x) {
    const int i = base + lane;
    const int v = i < m ? list[i] : 0;
    const bool take = i < m && sample_takes(i, v, m, want, salt);
    const unsigned tm = __ballot_sync(0xffffffffu, take);
    int at = 0;
    if (lane == 0 && tm) at = atomicAdd(count, __popc(tm));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (take) sample[at + __popc(tm & ((1u << lane) - 1u))] = v;
  }
}

int launch_sample(gc_graph *g, int32_t want, uint32_t salt) {
  // io_b <- the sample of list, then the two change places
  int32_t *count = g->blk + g->red_blocks + 4;
  GC_CUDA(cudaMemsetAsync(count, 0, sizeof(int32_t), g->stream));
  ++g->launches;
  k_sample<<<g->red_blocks, 256, 0, g->stream>>>(g->list, &g->sctl->n_sel, want, salt, g->io_b, count);
  GC_CUDA(cudaGetLastError());
  GC_CUDA(cudaMemcpyAsync(&g->sctl->n_sel, count, sizeof(int32_t), cudaMemcpyDeviceToDevice, g->stream));
  std::swap(g->list, g->io_b);
  return GC_OK;
}

}  // namespace gc
