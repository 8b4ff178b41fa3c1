// Weighted graphs (positive integer edge weights): the paper's Greedy with
// every SSSP a shortest-path search instead of a BFS (Sec. 3.2: Dijkstra,
// O(kn(m + n log n))), and the pruning of Sec. 4.1, which carries over: if
// d(v, w) < d_S[w] then every vertex x on a shortest v-w path has d(v, x) <
// d_S[x] (d(v, x) = d(v, w) - d(x, w) < d_S[w] - d(x, w) <= d_S[x]), so
// relaxing only into vertices the candidate would bring strictly closer finds
// the exact distance of every vertex that contributes to the gain.
//
// One search per CTA (k_wsearch), in distance order.  Modes:
//   kWFarness  f({v}) of each source, cut by the best farness (round 0);
//   kWGain     Delta(v | S) of each listed candidate against d_S;
//   kWRelabel  d_S <- min(d_S, d(s, .)) in place from one source (the d_S
//              update), the decrease summed for the gain check.
#include <limits.h>

#include <algorithm>

#include "gc_device.cuh"
#include "gc_internal.cuh"

namespace gc {

// Rows ordered by weight (built once per gc_set_weights): stable counting passes over 8
// bits of the weights each, least significant first.  A middle pass moves entry numbers
// alone, the last one the ids and weights.  A warp takes a segment of a row, 32 entries
// at a time, and ranks the equal digits of a tile by match-any: a row is one segment,
// rows of more than kHeavyRow entries are kWSortWarps, by a CTA.  The whole call, ms, a
// warp a row and scratch weights allocated, now: star of 16,000, weights up to 1000,
// 0.54, 0.21; of 1,000,000 33, 12; R-MAT scale 18 1.50, 0.64; complete n = 600 0.21, 0.10.
constexpr int kWSortWarps = 32;

struct WSort {
  const int32_t *ci, *wt;   // the rows as they are
  const int32_t *from;      // the order so far (entry numbers; null: as they are)
  int32_t *to;              // the order after this pass (null: the last pass)
  int32_t *ci_w, *wt_w;
  int shift;
};

// at[0 .. 256): the digits' counts of entries [e0, e1), by one warp
__device__ __forceinline__ void wsort_count(const WSort &w, int e0, int e1, int *at) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < 256; i += 32) at[i] = 0;
  __syncwarp();
  for (int e = e0 + lane; e < e1; e += 32) atomicAdd(&at[(w.wt[w.from ? w.from[e] : e] >> w.shift) & 255], 1);
  __syncwarp();
}

// the entries to their slots; at: the digits' next slots
__device__ __forceinline__ void wsort_move(const WSort &w, int e0, int e1, int *at) {
  const int lane = threadIdx.x & 31;
  for (int base = e0; base < e1; base += 32) {
    const int e = base + lane;
    const int x = e < e1 ? (w.from ? w.from[e] : e) : 0;
    const int v = e < e1 ? w.wt[x] : 0;
    const int g = e < e1 ? (v >> w.shift) & 255 : 256 + lane;  // (idle lanes match nobody)
    const unsigned same = __match_any_sync(0xffffffffu, g);
    if (e < e1) {
      const int slot = at[g] + __popc(same & ((1u << lane) - 1u));
      if (w.to) {
        w.to[slot] = x;
      } else {
        w.ci_w[slot] = w.ci[x];
        w.wt_w[slot] = v;
      }
    }
    __syncwarp();
    if (e < e1 && lane == __ffs(same) - 1) at[g] += __popc(same);
    __syncwarp();
  }
}

// Long rows first, a CTA each, then the others, a warp each.
__global__ void __launch_bounds__(32 * kWSortWarps) k_wsort(const int32_t *__restrict__ rp, int32_t n,
                                                            const int32_t *__restrict__ heavy,
                                                            const int32_t *__restrict__ nh, const WSort w) {
  __shared__ int s_at[kWSortWarps][256];
  __shared__ int s_scan[33];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int *at = s_at[wid];
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int e0 = rp[heavy[i]], len = rp[heavy[i] + 1] - e0;
    // warp k: entries [len k / 32, len (k + 1) / 32)
    const int a = e0 + (int)((long long)len * wid / kWSortWarps);
    const int b = e0 + (int)((long long)len * (wid + 1) / kWSortWarps);
    wsort_count(w, a, b, at);
    cta_sync();
    // counts -> first slots: digits in order, a digit's segments in order
    int sum = 0;
    if (tid < 256)
      for (int k = 0; k < kWSortWarps; ++k) sum += s_at[k][tid];
    int total;
    int first = e0 + block_excl_scan(sum, s_scan, &total);
    if (tid < 256)
      for (int k = 0; k < kWSortWarps; ++k) {
        const int c = s_at[k][tid];
        s_at[k][tid] = first;
        first += c;
      }
    cta_sync();
    wsort_move(w, a, b, at);
    cta_sync();  // s_at is reused
  }
  for (int v = blockIdx.x * kWSortWarps + wid; v < n; v += gridDim.x * kWSortWarps) {
    const int e0 = rp[v], e1 = rp[v + 1];
    if (e1 - e0 > kHeavyRow) continue;
    wsort_count(w, e0, e1, at);
    int carry = e0;  // counts -> first slots
    for (int base = 0; base < 256; base += 32) {
      const int c = at[base + lane];
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      at[base + lane] = carry + incl - c;
      carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    wsort_move(w, e0, e1, at);
  }
}

// A search settles the vertices in buckets [., T): within a bucket it is a
// label-correcting search that relaxes only the entries with dist[u] + weight <
// T, a prefix of u's row, since rows are ordered by weight; ptr[u] keeps where
// the prefix ended, and u stays in the pending list until T has passed its last
// entry.  At the end of a bucket everything below T is final.  Gains and the d_S
// update relax only into vertices they bring strictly closer than d_S.
//
// Farness, BFScut (Sec. 3.1) on weighted distances: at the end of a bucket every
// unsettled vertex is at least as far as the nearest pending entry reaches, so
// with `cnt` settled vertices of distance sum `sum`,
//   f({v}) >= sum + (nearest pending) (n - cnt),
// and a search whose bound exceeds the best farness is cut: on R-MAT scale 14
// with weights in [1, 16] after 11% of the entries on average, where a full
// search of every vertex reads the whole graph n times over.  Measured, round 0
// at scale 14 in ms, weights up to 1, 16, 1000: 25, 47, 99 -> 1.7, 11.8, 37; the
// whole call (k = 50) 34, 60, 119 -> 7.6, 19.5, 47.
//
// A search's random accesses are its distances and two flags per vertex.  For
// 300 to 1,200 searches at a time they do not fit L2 (round 0 at scale 14: 26 ms
// with them in the workspace, bound by DRAM sectors), so up to kWFarSmemN
// vertices they live in shared memory (SM: 13 ms; four CTAs of 512 threads per SM up
// to about 11,000 vertices, three at scale 14, one of 1024 beyond 24,000); the queues and lists in
// global memory are written and read in order.  Larger graphs keep them in the
// workspace.
constexpr int kWFarSmemN = 48000;  // 199 KB, and 13 KB of static arrays at 1024 threads
// Steps of at most 32 queued vertices belong to warp 0: their rows by a scan over its
// lanes, and up to this many entries relaxed without a CTA barrier; more go to the CTA
// (five barriers a step instead of nine).  Paths and strips have little but such steps.
// k = 6, ms, with one warp a row and no buckets, with every step by the CTA, now: path
// n = 2,000, weights up to 1000, 17.0, 27.7, 16.4; grid strip 5 x 1,000, unit weights
// 21.8, 27.2, 20.0; road-like 100 x 100, up to 16, 78.8, 23.8, 20.6.
constexpr int kWWarpEntries = 128;
constexpr unsigned kWNear = 1u, kWBucket = 2u;  // queued; listed in a bucket (settled at its end)

// per CTA: near queues, pending and bucket lists, ptr, and without SM the
// distances, the flags and the touched list
size_t wws_stride(int32_t n) { return 8 * ws_align((size_t)n * 4); }
static size_t wfar_smem(int32_t n) { return (size_t)n * 4 + 2 * (((size_t)n + 31) / 32) * 4; }

// How a graph is searched: 0 shared memory, 512 threads (two CTAs per SM or
// more); 1 shared memory, one CTA of 1024 threads per SM; 2 workspace, 512
// threads.  Between 24,000 and kWFarSmemN vertices, 1 gives up the many CTAs
// that hide a sparse search's latency and pays off on dense rows only: R-MAT
// scale 16 (46,693 vertices, 39 entries each) round 0 279 ms by 1, 624 by 2; BA
// n = 47,000, m = 3, 38 by 1, and n = 49,000 28 by 2.
static int wform(const gc_graph *g) {
  if (g->n <= kWFarSmemN / 2) return 0;
  return g->n <= kWFarSmemN && g->nnz >= 16ll * g->n ? 1 : 2;
}
static int wthreads(int mode, int form) { return form == 1 || (form == 0 && mode == kWRelabel) ? 1024 : 512; }

// The workspaces' dist words to kInf and flags to 0.
__global__ void k_wfar_init(unsigned char *base, size_t stride, int32_t n) {
  unsigned char *p = base + stride * (size_t)blockIdx.x;
  const size_t a4 = ws_align((size_t)n * 4);
  int32_t *d = (int32_t *)(p + 5 * a4);
  unsigned int *fl = (unsigned int *)(p + 6 * a4);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    d[i] = kInf;
    fl[i] = 0u;
  }
}

// Sources list[i] (list == nullptr: every vertex i), i < m.  ci, wt: the rows
// ordered by weight.  delta > 0: the bucket width; 0: from the best farness.
// kWFarness  out[v]: the farness of source v, -1 if cut; sources whose out[v] is
//            already >= 0 are skipped.  *best: the smallest farness found so far,
//            lowered as searches complete.
// kWGain     out[i]: the gain (0 for a member of S).
// kWRelabel  out[0]: the decrease of d_S over labels with a finite old value.
template <int MODE, int TH, bool SM>
__global__ void __launch_bounds__(TH, TH == 512 ? 4 : 1)
    k_wsearch(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const int32_t *__restrict__ wt,
              int32_t n, int32_t *dS, const int32_t *list, const int32_t *m_dev, int32_t m_arg, long long *out,
              unsigned char *ws_base, size_t ws_stride, unsigned int *task, long long *best, int32_t w_max,
              int32_t delta_arg, int32_t *err) {
  extern __shared__ __align__(16) int32_t s_dist[];  // SM: distances, then the two flag bitmaps
  __shared__ int s_i, s_F, s_nt, s_np, s_nb, s_min, s_state, s_rows, s_total;
  __shared__ int s_off[TH], s_e0[TH], s_du[TH];
  __shared__ int s_scan[33];
  __shared__ long long s_bst;
  __shared__ long long s_red[32];
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t a4 = ws_align((size_t)n * 4);
  unsigned char *base_p = ws_base + ws_stride * (size_t)blockIdx.x;
  auto arr = [&](int k) { return (int32_t *)(base_p + k * a4); };
  int32_t *q0 = arr(0), *q1 = arr(1), *pend = arr(2), *bucket = arr(3), *ptr = arr(4), *gd = arr(5),
          *touched = arr(7);
  unsigned int *fl = (unsigned int *)arr(6);
  const int nw = (n + 31) / 32;
  unsigned int *s_near = (unsigned int *)(s_dist + n), *s_buck = s_near + nw;
  auto dist = [&](int v) -> int { return SM ? *(volatile int32_t *)&s_dist[v] : __ldcg(&gd[v]); };
  auto lower = [&](int v, int x) -> int { return atomicMin(SM ? &s_dist[v] : &gd[v], x); };
  // set a flag; true if it was clear
  auto flag = [&](int v, unsigned f) -> bool {
    if (SM) return !(atomicOr((f == kWNear ? s_near : s_buck) + (v >> 5), 1u << (v & 31)) & (1u << (v & 31)));
    return !(atomicOr(&fl[v], f) & f);
  };
  auto unqueue = [&](int v) {
    if (SM) atomicAnd(&s_near[v >> 5], ~(1u << (v & 31)));
    else atomicAnd(&fl[v], ~kWNear);
  };
  int T = 0;
  // the part of a queued vertex's row up to T, entries [e0, lo): from the start,
  // or, for a settled vertex taken up again (queued as ~u), from where the last
  // bucket stopped; its distance is one value for the whole row (if it is lowered
  // meanwhile the vertex is queued again)
  auto row_part = [&](int x, int &du, int &e0, int &lo) -> int {
    const int u = x < 0 ? ~x : x;
    du = dist(u);
    const int e1 = rp[u + 1];
    e0 = x < 0 ? ptr[u] : rp[u];
    // (the last bucket: the whole row)
    lo = T == kInf - 1 ? e1 : e0;
    int step = 4;  // galloping: the prefixes are short
    while (lo + step <= e1 && du + wt[lo + step - 1] < T) {
      lo += step;
      step *= 2;
    }
    int hi = min(e1, lo + step);
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (du + wt[mid] < T) lo = mid + 1;
      else hi = mid;
    }
    return u;
  };
  auto take = [&](int x, int u, int lo) {
    if (x >= 0) {
      unqueue(u);
      if (flag(u, kWBucket)) bucket[atomicAdd(&s_nb, 1)] = u;
    }
    ptr[u] = lo;
  };
  // entry e of `total` in the parts of `rows` rows: row j is the largest with
  // s_off[j] <= e.  A thread's entries ascend, so j starts at the last one's: with
  // long parts the next row is a step or two away (galloping), with short ones it
  // is searched for.  A search over all TH rows for every entry was half of the time
  // on dense graphs (random n = 4,000, rows of 400, weights up to 16: 10.9 -> 7.9 ms
  // a call).
  auto relax = [&](int e, int rows, int total, int &j, int32_t *nxt) {
    int hi = rows - 1;
    if (total >= 32 * rows) {
      int step = 1;
      while (j + step <= hi && s_off[j + step] <= e) {
        j += step;
        step *= 2;
      }
      hi = min(hi, j + step - 1);
    }
    while (j < hi) {
      const int mid = (j + hi + 1) >> 1;
      if (s_off[mid] <= e) j = mid;
      else hi = mid - 1;
    }
    const int x = s_e0[j] + (e - s_off[j]);
    const int w = ci[x], nd = s_du[j] + wt[x];
    if (MODE != kWFarness && nd >= dS[w]) return;  // pruned (Sec. 4.1)
    if (nd >= dist(w)) return;
    const int old = lower(w, nd);
    if (nd >= old) return;
    if (!SM && old == kInf) touched[atomicAdd(&s_nt, 1)] = w;
    if (flag(w, kWNear)) nxt[atomicAdd(&s_F, 1)] = w;
  };
  const int m = m_dev ? *m_dev : m_arg;
  for (;;) {
    if (SM) {
      for (int i = tid; i < n; i += TH) s_dist[i] = kInf;
      for (int i = tid; i < 2 * nw; i += TH) s_near[i] = 0u;
    }
    if (tid == 0) {
      s_i = (int)atomicAdd(task, 1u);
      s_bst = MODE == kWFarness ? *(volatile long long *)best : LLONG_MAX;
    }
    cta_sync();
    const int i = s_i;
    const long long bst = s_bst;
    cta_sync();
    if (i >= m) break;
    const int s = list ? list[i] : i;
    if (MODE == kWFarness && out[s] >= 0) continue;  // searched before (uniform)
    if (s < 0 || s >= n) {
      if (tid == 0) {
        out[i] = -1;
        atomicExch(err, GC_EINVAL);
      }
      continue;
    }
    if (MODE == kWGain && dS[s] == 0) {  // a member: no gain
      if (tid == 0) out[i] = 0;
      continue;
    }
    // bucket width: given, or an eighth of the best mean distance
    const int delta = delta_arg > 0 ? delta_arg
                      : bst < LLONG_MAX ? (int)max(1ll, bst / (8ll * n)) : max(1, w_max / 4);
    if (tid == 0) {
      lower(s, 0);
      if (!SM) touched[0] = s;
      flag(s, kWNear);
      q0[0] = s;
      s_nt = 1;
      s_F = 1;
      s_np = 0;
    }
    T = min(delta, kInf - 1);
    long long sum = 0, cnt = 0;  // settled: farness, gain or decrease, and vertices (the same in every thread)
    bool cut = false;
    int32_t *cur = q0, *nxt = q1;
    cta_sync();
    for (;;) {
      if (tid == 0) s_nb = 0;
      // ---- one bucket: label-correcting below T ----
      for (;;) {
        cta_sync();
        int F = s_F;
        cta_sync();
        if (F == 0) break;
        if (F <= 32) {
          // few queued vertices: warp 0 alone, step after step, while they stay few;
          // the entries of a step by the whole CTA if they are many, and back here
          if (tid < 32) {
            int32_t *c = cur, *x = nxt;
            int state = 0, total = 0;  // bit 0: the queues have changed places, bit 1: entries for the CTA
            for (int f = F; f > 0 && f <= 32; state ^= 1) {
              int q = 0, u = 0, du = 0, e0 = 0, lo = 0;
              if (lane < f) {
                q = c[lane];
                u = row_part(q, du, e0, lo);
                take(q, u, lo);
              }
              int incl = lo - e0;
#pragma unroll
              for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
              }
              total = __shfl_sync(0xffffffffu, incl, 31);
              s_off[lane] = incl - (lo - e0);
              s_e0[lane] = e0;
              s_du[lane] = du;
              if (lane == 0) s_F = 0;
              if (total > kWWarpEntries) {
                state |= 2;
                if (lane == 0) s_rows = f;
                break;
              }
              __syncwarp();
              int j = 0;
              for (int e = lane; e < total; e += 32) relax(e, f, total, j, x);
              __syncwarp();
              int32_t *t = c;
              c = x;
              x = t;
              f = *(volatile int *)&s_F;
              __syncwarp();
            }
            if (lane == 0) {
              s_state = state;
              s_total = total;
            }
          }
          cta_sync();
          const int state = s_state;
          F = s_F;
          if (state & 1) {
            int32_t *t = cur;
            cur = nxt;
            nxt = t;
          }
          cta_sync();
          if (state & 2) {
            const int rows = s_rows, total = s_total;
            int j = 0;
            for (int e = tid; e < total; e += TH) relax(e, rows, total, j, nxt);
            int32_t *t = cur;
            cur = nxt;
            nxt = t;
            continue;
          }
          if (F == 0) break;
        }
        if (tid == 0) s_F = 0;
        for (int base = 0; base < F; base += TH) {  // a thread per queued vertex
          const int q = base + tid;
          int u = -1, du = 0, e0 = 0, lo = 0;
          if (q < F) {
            u = row_part(cur[q], du, e0, lo);
            take(cur[q], u, lo);
          }
          const int len = lo - e0;
          int total;
          const int off = block_excl_scan(len, s_scan, &total);
          s_off[tid] = off;
          s_e0[tid] = e0;
          s_du[tid] = du;
          cta_sync();
          // the chunk's entries, spread over the threads
          const int rows = min(TH, F - base);
          int j = 0;
          for (int e = tid; e < total; e += TH) relax(e, rows, total, j, nxt);
          cta_sync();
        }
        int32_t *t = cur;
        cur = nxt;
        nxt = t;
      }
      // ---- everything below T is settled; the pending entries ----
      const int nb = s_nb, np = s_np;
      long long x = 0;
      for (int q = tid; q < nb; q += TH) {
        const int v = bucket[q], dv = dist(v);
        if (MODE == kWFarness) {
          x += dv;
        } else {
          const int old = dS[v];
          if (old < kInf) x += old - dv;
          if (MODE == kWRelabel) dS[v] = dv;
        }
      }
      x = block_sum(x, s_red);
      sum += x;
      cnt += nb;
      if (MODE == kWFarness && cnt == n) break;  // complete
      if (tid == 0) {
        s_np = 0;
        s_min = kInf;
      }
      int mn = kInf;
      const int all = np + nb;
      for (int base = 0; base < all; base += TH) {  // in place: reads stay ahead of writes
        const int q = base + tid;
        const int u = q < np ? pend[q] : q < all ? bucket[q - np] : -1;
        bool keep = false;
        if (u >= 0) {
          const int e = ptr[u];
          keep = e < rp[u + 1];
          if (keep) mn = min(mn, dist(u) + wt[e]);
        }
        cta_sync();
        if (keep) pend[atomicAdd(&s_np, 1)] = u;
        cta_sync();
      }
      mn = __reduce_min_sync(0xffffffffu, mn);
      if (lane == 0) atomicMin(&s_min, mn);
      cta_sync();
      mn = s_min;
      const int left = s_np;
      if (left == 0) break;  // nothing more to reach (farness short of n: disconnected)
      if (MODE == kWFarness && sum + (long long)mn * ((long long)n - cnt) > bst) {
        cut = true;
        break;
      }
      // ---- the next bucket: rows with an entry below the new T go on ----
      T = w_bucket_end(mn, delta);
      for (int q = tid; q < left; q += TH) {
        const int u = pend[q];
        if (w_in_bucket(dist(u) + wt[ptr[u]], T)) cur[atomicAdd(&s_F, 1)] = ~u;
      }
    }
    cta_sync();
    if (tid == 0) {
      if (MODE != kWFarness) {
        out[i] = sum;
      } else if (cut) {
        out[s] = -1;
      } else if (cnt != n) {
        out[s] = -1;
        atomicExch(err, GC_EDISCONNECTED);
      } else {
        out[s] = sum;
        atomicMin(best, sum);
      }
    }
    if (!SM) {  // the workspace back to rest
      const int nt = s_nt;
      for (int q = tid; q < nt; q += TH) {
        const int w = touched[q];
        gd[w] = kInf;
        fl[w] = 0u;
      }
    }
    cta_sync();
  }
}

// weights: w >= 1 everywhere, the same in both rows of an edge (binary search
// of the mirror entry in its sorted row), and the largest below max_w_out
__global__ void k_wcheck(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                         const int32_t *__restrict__ wt, int32_t n, int check_mirror, int32_t *bad,
                         int32_t *max_w) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
  int mx = 0;
  for (int u = gw; u < n; u += nw) {
    for (int e = rp[u] + lane; e < rp[u + 1]; e += 32) {
      const int w = wt[e];
      mx = max(mx, w);
      bool ok = w >= 1;
      if (ok && check_mirror) {
        const int x = ci[e];
        int lo = rp[x], hi = rp[x + 1];
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (ci[mid] < u) lo = mid + 1;
          else hi = mid;
        }
        ok = lo < rp[x + 1] && ci[lo] == u && wt[lo] == w;
      }
      if (!ok) atomicExch(bad, 1);
    }
  }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  if (lane == 0 && mx) atomicMax(max_w, mx);
}

template <int MODE>
static const void *wsearch_fn(int form) {
  return form == 2 ? (const void *)k_wsearch<MODE, 512, false>
         : wthreads(MODE, form) == 512 ? (const void *)k_wsearch<MODE, 512, true>
                                       : (const void *)k_wsearch<MODE, 1024, true>;
}

static const void *wsearch_fn(int mode, int form) {
  return mode == kWFarness ? wsearch_fn<kWFarness>(form)
         : mode == kWGain  ? wsearch_fn<kWGain>(form)
                           : wsearch_fn<kWRelabel>(form);
}

int launch_wfar_init(gc_graph *g) {
  ++g->launches;
  k_wfar_init<<<g->w_ctas, 512, 0, g->stream>>>(g->w_ws, g->w_stride, g->n);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_wsearch(gc_graph *g, int mode, const int32_t *list, const int32_t *m_dev, int32_t m, long long *out,
                   long long *best, int32_t delta) {
  GC_CUDA(cudaMemsetAsync(g->w_task, 0, sizeof(unsigned int), g->stream));
  ++g->launches;
  const int32_t *rp = g->rp, *ci = g->ci_w, *wt = g->wt_w;
  int32_t n = g->n, w_max = g->w_max, *err = &g->sctl->err, *dS = g->dS;
  unsigned char *ws = g->w_ws;
  size_t stride = g->w_stride;
  unsigned int *task = g->w_task;
  void *args[] = {(void *)&rp, (void *)&ci,  (void *)&wt,     (void *)&n,    (void *)&dS,   (void *)&list,
                  (void *)&m_dev, (void *)&m, (void *)&out, (void *)&ws, (void *)&stride, (void *)&task, (void *)&best,
                  (void *)&w_max, (void *)&delta, (void *)&err};
  const int form = wform(g);
  GC_CUDA(cudaLaunchKernel(wsearch_fn(mode, form), dim3(mode == kWRelabel ? 1 : g->w_ctas), dim3(wthreads(mode, form)),
                           args, form == 2 ? 0 : wfar_smem(n), g->stream));
  return GC_OK;
}

// ci_w, wt_w <- the rows ordered by weight, a pass per 8 bits of w_max; tmp (nnz
// entries) holds the order between two passes, ci_w before that one
int launch_wsort(gc_graph *g, int32_t *tmp) {
  int passes = 1;
  while (passes < 4 && (g->w_max >> (8 * passes)) > 0) ++passes;
  const int grid = std::min(g->num_sms * 2, (g->n + kWSortWarps - 1) / kWSortWarps);
  WSort w{g->ci, g->wt, nullptr, nullptr, g->ci_w, g->wt_w, 0};
  for (int p = 0; p < passes; ++p) {
    const int left = passes - 1 - p;
    w.to = left == 0 ? nullptr : (left & 1) ? tmp : g->ci_w;
    w.shift = 8 * p;
    ++g->launches;
    k_wsort<<<grid, 32 * kWSortWarps, 0, g->stream>>>(g->rp, g->n, g->heavy, g->n_heavy, w);
    w.from = w.to;
  }
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int wsearch_occupancy(const gc_graph *g, int *blocks_per_sm) {
  const int form = wform(g);
  const size_t smem = form == 2 ? 0 : wfar_smem(g->n);
  for (int mode : {kWRelabel, kWGain, kWFarness}) {  // the result is the farness searches'
    if (smem)  // (the limit is the process's, not the graph's: the largest any graph needs)
      GC_CUDA(cudaFuncSetAttribute(wsearch_fn(mode, form), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)wfar_smem(kWFarSmemN)));
    GC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, wsearch_fn(mode, form), wthreads(mode, form),
                                                          smem));
  }
  return GC_OK;
}

int launch_wcheck(gc_graph *g, bool mirror, int32_t *bad, int32_t *max_w) {
  ++g->launches;
  k_wcheck<<<g->num_sms * 8, 256, 0, g->stream>>>(g->rp, g->ci, g->wt, g->n, mirror ? 1 : 0, bad, max_w);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

}  // namespace gc
