// Batched Greedy++ over many graphs: three persistent cooperative launches, no
// host round trip between them.
//
// The batch is stored as one block-diagonal union CSR (global vertex ids;
// graph g owns ids [off[g], off[g+1])).  Distances never cross components, so
// the multi-source relabel BFS computes every graph's BFS at once (one seed
// per graph), and 64-lane gain batches stay inside one graph.  What is per
// graph -- round-0 cut thresholds, argmin/argmax, the lazy round state and its
// acceptance test (Sec. 4.2), the group -- lives in per-graph arrays.
//
// Phases (bounded grid barriers between them); P0 to P5 are k_batch_solve, P6
// k_batch_lazy, P7 k_batch_check:
//   P0  lower bounds LB(v) and, per graph, the vertex v_a of smallest bound
//   P1  BFS from all v_a; per-graph farness f_a
//   P2  every v with LB(v) <= f_a evaluated by the 64-lane BFS in farness
//       mode with per-graph cuts (graph-aligned batches, by teams of CTAs on
//       graphs with few survivors), after the far counts have raised the
//       bounds; per graph s0 = argmin (f, id).  With round 1's batches by
//       teams too, rounds 0 and 1 of 24 mixed graphs went from 45 + 32 to 17 + 12
//       ms, of 256 graphs from 623 + 190 to 493 + 167 (other kernels as they were
//       then)
//   P3  BFS from all s0 (d_S), per-graph farness, neighbour bound mx
//   P4  round 1: every candidate of every graph, graph-aligned 64-lane batches
//       from a dynamic task counter; per-graph argmax; picks; BFS from picks
//   P5  per graph (one CTA): active list of the largest bounds
//   P6  lazy rounds: teams of CTAs, each running the rounds of one graph after
//       another (longest first) to completion -- fold, decide, select 64,
//       evaluate them by the whole team, update d_S from the pick's claim log --
//       so no graph waits for another.  A team's steps are those of the
//       single-graph persistent kernel.  One CTA per graph, as before, left
//       most of the GPU idle behind the slowest graph: 24 mixed graphs 717 ms
//       (lazy rounds 634), 256 graphs 1468; by teams, with the sweeps and all later
//       steps, 34 to 37 and 377.
//   P7  check: one BFS from every graph's whole group; each graph's farness
//       must equal f(s0) minus the sum of its accepted gains.
#include <limits.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <functional>
#include <queue>
#include <string>
#include <vector>

#include "gc_cta.cuh"
#include "gc_lazy.cuh"

namespace gc {

struct BatchCtl {
  GridBar bar;
  int32_t err;
  int32_t remaining;  // graphs that still need lazy rounds
  int32_t nseeds;     // seeds of the next relabel BFS
  int32_t task, task2;  // dynamic task counters (P2, P4): the teams', the single CTAs'
  int32_t pad0;
  unsigned long long pk[3];  // relabel BFS frontiers (see BfsCtl)
  int32_t pad;
  unsigned long long decrease;
  long long iterations;
  long long dbg[4];  // first failed check: phase, graph, expected, found
  unsigned long long ns_ph[6];  // end of round 0 (P2), round 1 (P5), lazy rounds (P6), check (P7),
                                // start and end of the round-1 gains (P4)
  unsigned long long ns_lazy[3];  // lazy rounds, summed over graphs: selection (with list
                                  // rebuilds), gain batches, d_S updates
  int32_t blk_tot[kMaxGridCtas];
  unsigned long long t_start;  // the solve's start (CTA 0's clock)
  int32_t stage;               // kernels of the solve that have completed without an error
  int32_t lazy_next;           // next entry of the lazy rounds' graph order
};

// One team of the lazy rounds: its barrier, the graph it works on and its
// grid-batch control block.
struct TeamCtl {
  GridBar bar;
  int32_t g;
  int32_t sweep_n, sweep_next;  // sweep: candidates listed, next one to take
  int32_t pad;
  long long best;                 // round 0: the cut threshold of the current task
  unsigned long long sweep_best;  // its best exact gain: gain << 32 | ~(id in the graph)
  GridGainCtl gg;
};

static __device__ void check_fail(BatchCtl *c, int phase, int g, long long want, long long got) {
  if (atomicCAS((unsigned long long *)&c->dbg[0], 0ull, (unsigned long long)phase) == 0ull) {
    c->dbg[1] = g;
    c->dbg[2] = want;
    c->dbg[3] = got;
  }
  atomicExch(&c->err, GC_EINTERNAL);
}

struct BatchArgs {
  const int32_t *rp, *ci;
  int32_t N;
  int32_t count;
  const int32_t *gid, *off, *ng, *kk, *iota;
  const int32_t *bstart;  // round-1 task prefix per graph ([count+1])
  int32_t lanes1;         // candidates per round-1 batch
  int32_t max_n;          // vertices of the largest graph (workspace layout)
  int32_t *dS, *mx, *stamp, *q0, *q1, *goff, *st1;
  int32_t *rpf, *cif, *c3;  // pruned adjacency for rounds >= 1 (built in P3)
  int32_t *dS1;             // d(s0, .) as of P3, never written after: round 1 reads it read-only
  long long *ub, *key, *f0;
  unsigned char *ws;
  size_t ws_stride;
  unsigned long long *packed;
  long long *fa, *farness, *bestf;
  LazyCtl *lc;
  int32_t *act, *act_n;
  int32_t A;
  int32_t kmax;
  int32_t *picks;
  long long *pgain;
  int32_t *seeds;  // [max(count, sum k)]
  int32_t *slist;  // round-0 survivors, graph-aligned [N]
  int32_t *scount, *tstart;  // per-graph survivor counts, task prefixes [2 (count+1)]
  BatchCtl *ctl;
  GainCtl *gctl;
  // lazy rounds (k_batch_lazy): teams of team_size CTAs, each with its control
  // block and selection scratch; 3 n_g entries of gx and 2 n_g of the claim log
  // per graph, at 3 off[g] and 2 off[g]; wide steps: 64 candidates per CTA
  TeamCtl *teams;
  GridSelScratch *gsel;
  int32_t *gx;
  ClaimRec *clog;
  int32_t *wsel;
  long long *wgain;
  int32_t *depth;     // BFS levels of the deepest round-1 batch, per graph
  unsigned long long *cls;  // [2 count]: members of the two degree classes of each graph (far counts)
  const int32_t *order;  // graphs of the team phase, longest first; order_n of them
  int32_t order_n;
  int32_t team_size;
  int32_t list_cap;   // entries of a shared-memory list (a power of two, at most kCta0SelectMax)
  int32_t grid_min_n; // graphs with at least this many vertices run their lazy rounds grid-wide
  int32_t team_entries, far;  // entries from which a graph's short lists go to teams; 1: round 0 takes the far counts
  int32_t simple;     // no row holds an entry twice or its own vertex
  int32_t bounded;    // round 1 with two-hop bounds (batch_round1_bounded) and the refresh after it
  long long *g3;      // [2 * count]: sum of (d - 3)^+ per graph for round 1, then for the refresh
  unsigned long long tns;
};

constexpr int kBatchThreads = kGainThreads;
// lazy rounds grid-wide from this many vertices: graphs of 10^4 to 5 x 10^5
// vertices finish sooner by teams side by side than by taking the grid in turn
constexpr int32_t kBatchGridMinN = 1 << 21;

// lazy rounds: a list that cannot certify a pick starts a sweep when more than
// this many bounds reach the best gain (16 steps of 64): when they came, 24 mixed
// graphs 207 -> 102 ms, 256 graphs 1109 -> 976 (34 to 37 and 377 with all later steps)
constexpr int kBatchSweepMin = 1024;

static __device__ __forceinline__ bool bsync(const BatchArgs &a) { return grid_sync(&a.ctl->bar, &a.ctl->err, a.tns); }

// The pruned adjacency of the single-graph path (k_row_stats in gc_rows.cu)
// over the union CSR, built inside the solve once d_S = d(s0, .) is known:
// rows keep the neighbours with d_S >= 2, those with d_S >= 3 first (c3 of
// them).  Count per vertex into a.q0 (free here), scan across CTAs (each
// CTA owns a contiguous vertex range), fill.  Three grid barriers.
static __device__ bool batch_prune(const BatchArgs &a) {
  __shared__ int s_scan[33];
  __shared__ long long s_off[kMaxGridCtas + 1];
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x, G = gridDim.x, b = blockIdx.x;
  const int gw = (b * T + tid) >> 5, nw = (G * T) >> 5;
  for (int u = gw; u < a.N; u += nw) {
    int a2 = 0, a3 = 0;
    for (int e = a.rp[u] + lane; e < a.rp[u + 1]; e += 32) {
      const int d = a.dS[a.ci[e]];
      a2 += d >= 2;
      a3 += d >= 3;
    }
    a2 = warp_sum(a2);
    a3 = warp_sum(a3);
    if (lane == 0) {
      a.q0[u] = a2;
      a.c3[u] = a3;
    }
  }
  if (!bsync(a)) return false;
  const int P = (a.N + G - 1) / G;
  const int lo = min(a.N, b * P), hi = min(a.N, lo + P);
  long long mine = 0;
  for (int v = lo + tid; v < hi; v += T) mine += a.q0[v];
  mine = block_sum(mine, (long long *)s_off);
  if (tid == 0) a.ctl->blk_tot[b] = (int32_t)mine;  // < 2^31: the CSR has fewer entries
  if (!bsync(a)) return false;
  long long run = 0;
  for (int base = 0; base < G; base += T) {
    const int j = base + tid;
    const int v = j < G ? ((volatile int32_t *)a.ctl->blk_tot)[j] : 0;
    int total;
    const int off = block_excl_scan(v, s_scan, &total);
    if (j < G) s_off[j] = run + off;
    run += total;
    cta_sync();
  }
  long long carry = s_off[b];
  cta_sync();
  for (int base = lo; base < hi; base += T) {
    const int v = base + tid;
    const int x = v < hi ? a.q0[v] : 0;
    int total;
    const int off = block_excl_scan(x, s_scan, &total);
    if (v < hi) a.rpf[v] = (int32_t)(carry + off);
    carry += total;
  }
  if (b == G - 1 && tid == 0) a.rpf[a.N] = (int32_t)run;
  if (!bsync(a)) return false;
  for (int u = gw; u < a.N; u += nw) {
    int pos = a.rpf[u];
    for (int pass = 0; pass < 2; ++pass) {  // d_S >= 3 first, then d_S == 2
      for (int e0 = a.rp[u]; e0 < a.rp[u + 1]; e0 += 32) {
        const int e = e0 + lane;
        int w = 0;
        bool keep = false;
        if (e < a.rp[u + 1]) {
          w = a.ci[e];
          const int d = a.dS[w];
          keep = pass == 0 ? d >= 3 : d == 2;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) a.cif[pos + __popc(m & ((1u << lane) - 1u))] = w;
        pos += __popc(m);
      }
    }
  }
  return bsync(a);
}


// per-graph sum of d over all vertices (warp-aggregated when a warp's vertices
// share a graph); unreached vertices raise GC_EDISCONNECTED
static __device__ void seg_sum_dist(const BatchArgs &a, long long *out) {
  const int lane = threadIdx.x & 31;
  for (int base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; base < a.N; base += gridDim.x * blockDim.x) {
    const int v = base + lane;
    long long d = 0;
    int g = -1;
    if (v < a.N) {
      const int x = a.dS[v];
      if (x >= kInf) atomicExch(&a.ctl->err, GC_EDISCONNECTED);
      else d = x;
      g = a.gid[v];
    }
    const int g0 = __shfl_sync(0xffffffffu, g, 0);
    const bool uniform = __all_sync(0xffffffffu, g == g0 || g < 0);
    if (uniform) {
      const long long s = warp_sum(d);
      if (lane == 0 && g0 >= 0 && s) atomicAdd((unsigned long long *)&out[g0], (unsigned long long)s);
    } else if (g >= 0 && d) {
      atomicAdd((unsigned long long *)&out[g], (unsigned long long)d);
    }
  }
}

// one CTA: argmin (f0, local id) over graph g's vertices with f0 >= 0
static __device__ int cta_argmin_f0(const BatchArgs &a, int g) {
  __shared__ long long s_v[32];
  __shared__ int s_id[32];
  const int o = a.off[g], n = a.ng[g];
  long long bv = LLONG_MAX;
  int bid = -1;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const long long f = a.f0[o + i];
    if (f >= 0 && better_min(f, i, bv, bid)) {
      bv = f;
      bid = i;
    }
  }
  // block arg-min through the arg-max helper on negated values
  long long nv = bv == LLONG_MAX ? LLONG_MIN : -bv;
  block_argmax_all(nv, bid, s_v, s_id);
  return bid;
}

// One CTA: the want-th largest of graph g's bounds ub >= 0, by a radix select
// over their bytes (256-bin shared histograms, most significant byte first).
// *c gets how many bounds are >= 0; when *c <= want the result is -1.  *need
// gets how many of the bounds equal to the result belong to the top `want`
// (the others above it: want - *need of them).
static __device__ long long cta_kth_bound(const long long *ub, int o, int n, int want, long long *c,
                                          int *need) {
  __shared__ int s_hist[256];
  __shared__ int s_pick[2];
  __shared__ long long s_ll[32];
  const int tid = threadIdx.x, T = blockDim.x;
  long long umax = -1, cnt = 0;
  for (int i = tid; i < n; i += T) {
    const long long u = ub[o + i];
    if (u >= 0) {
      umax = max(umax, u);
      ++cnt;
    }
  }
  umax = block_max_ll(umax, s_ll);
  cnt = block_sum(cnt, s_ll);
  *c = cnt;
  *need = 0;
  if (cnt <= want) return -1;
  unsigned long long prefix = 0, mask = 0;
  int nd = want;
  const int top = umax > 0 ? 63 - __clzll((unsigned long long)umax) : 0;
  for (int shift = (top / 8) * 8; shift >= 0; shift -= 8) {
    for (int j = tid; j < 256; j += T) s_hist[j] = 0;
    cta_sync();
    for (int i = tid; i < n; i += T) {
      const long long u = ub[o + i];
      if (u >= 0 && ((unsigned long long)u & mask) == prefix)
        atomicAdd(&s_hist[((unsigned long long)u >> shift) & 255], 1);
    }
    cta_sync();
    if (tid == 0) {  // the bin holding the nd-th largest of the matching values
      int acc = 0, bin = 255;
      for (; bin > 0; --bin) {
        if (acc + s_hist[bin] >= nd) break;
        acc += s_hist[bin];
      }
      s_pick[0] = bin;
      s_pick[1] = acc;
    }
    cta_sync();
    prefix |= (unsigned long long)s_pick[0] << shift;
    mask |= 255ull << shift;
    nd -= s_pick[1];
    cta_sync();
  }
  *need = nd;
  return (long long)prefix;
}

// One CTA: the `want` candidates of graph g with the largest bounds, ordered by
// (ub desc, id asc) with ub >= 0, written to out[] in id order; returns their
// count.  Every candidate above the want-th largest bound T is taken, then the
// smallest ids of those equal to T.
static __device__ int cta_top_bounds(const long long *ub, int o, int n, int want, int32_t *out) {
  __shared__ int s_scan[33];
  const int tid = threadIdx.x, T = blockDim.x;
  long long c;
  int need;
  const long long thr = cta_kth_bound(ub, o, n, want, &c, &need);  // -1: take every ub >= 0
  int carry = 0, eq_seen = 0;
  for (int base = 0; base < n; base += T) {
    const int i = base + tid;
    const long long u = i < n ? ub[o + i] : -1;
    const int eq = u >= 0 && u == thr;
    int eq_total;
    const int eq_pos = block_excl_scan(eq, s_scan, &eq_total);
    const int take = (u >= 0 && u > thr) || (eq && eq_seen + eq_pos < need);
    int total;
    const int pos = block_excl_scan(take, s_scan, &total);
    if (take) out[carry + pos] = o + i;
    carry += total;
    eq_seen += eq_total;
  }
  return carry;
}

// One CTA: graph g's active list = {ub >= L} (ids in increasing order, at most
// A of them) with L the smallest value whose list fits, and theta = the
// largest bound left out, plus one (LLONG_MIN when nothing is left out): every
// candidate outside the list has ub < theta.
static __device__ void cta_build_list(const BatchArgs &a, int g) {
  __shared__ long long s_ll[32];
  __shared__ int s_scan[33];
  const int tid = threadIdx.x, T = blockDim.x;
  const int o = a.off[g], n = a.ng[g];
  long long c;
  int need;
  const long long kth = cta_kth_bound(a.ub, o, n, a.A, &c, &need);
  long long L = 0, theta = LLONG_MIN;
  if (c > a.A) {
    // the bounds equal to kth that the top A leaves out decide whether kth fits
    long long eq = 0, below = -1;
    for (int i = tid; i < n; i += T) {
      const long long u = a.ub[o + i];
      eq += u == kth;
      if (u >= 0 && u < kth) below = max(below, u);
    }
    eq = block_sum(eq, s_ll);
    below = block_max_ll(below, s_ll);
    if (eq > need) {
      L = kth + 1;
      theta = kth + 1;
    } else {
      L = kth;
      theta = below + 1;  // c > A leaves some bound below kth
    }
  }
  int32_t *act = a.act + (size_t)g * a.A;
  int carry = 0;
  for (int base = 0; base < n; base += T) {
    const int i = base + tid;
    const int f = i < n && a.ub[o + i] >= 0 && a.ub[o + i] >= L;
    int total;
    const int pos = block_excl_scan(f, s_scan, &total);
    if (f && carry + pos < a.A) act[carry + pos] = o + i;
    carry += total;
  }
  if (carry > a.A) {  // cannot happen (count(ub >= L) <= A); never write past the list
    if (tid == 0) check_fail(a.ctl, 5, g, a.A, carry);
    carry = a.A;
  }
  if (tid == 0) {
    a.act_n[g] = carry;
    a.lc[g].theta = theta;
  }
  cta_sync();
}

// Two-hop upper bound of Delta(v|S) for the group whose distances are d (the
// inequality and its derivation are those of the round-1 bounds in gc_rows.cu):
// d[v] + sum over the pruned row of v of ((d[w] - 1)^+ + c3[w]), plus the
// graph's G3 = sum_u (d[u] - 3)^+ added by the caller.  One warp per v.
static __device__ __forceinline__ long long warp_two_hop(const BatchArgs &a, const int32_t *d, const int32_t *c3,
                                                         int v) {
  const int lane = threadIdx.x & 31;
  long long s = 0;
  for (int e = a.rpf[v] + lane; e < a.rpf[v + 1]; e += 32) {
    const int w = a.cif[e];
    s += (long long)max(d[w] - 1, 0) + (long long)c3[w];
  }
  return warp_sum(s) + (long long)d[v];
}

// per-graph sum of (d - 3)^+ into out[g] (warp-aggregated like seg_sum_dist)
static __device__ void seg_sum_excess3(const BatchArgs &a, const int32_t *d, long long *out) {
  const int lane = threadIdx.x & 31;
  for (int base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; base < a.N; base += gridDim.x * blockDim.x) {
    const int v = base + lane;
    long long x = 0;
    int g = -1;
    if (v < a.N) {
      x = max(d[v] - 3, 0);
      g = a.gid[v];
    }
    const int g0 = __shfl_sync(0xffffffffu, g, 0);
    if (__all_sync(0xffffffffu, g == g0 || g < 0)) {
      const long long s = warp_sum(x);
      if (lane == 0 && g0 >= 0 && s) atomicAdd((unsigned long long *)&out[g0], (unsigned long long)s);
    } else if (g >= 0 && x) {
      atomicAdd((unsigned long long *)&out[g], (unsigned long long)x);
    }
  }
}

// Graphs with at most this many listed vertices and at least kTeamEntries adjacency
// entries run their tasks by teams: a CTA alone finishes a small graph's batch before
// a team has met at its barriers.  Rounds 0 and 1 in ms by teams and by CTAs: 180
// graphs of 63 to 300 vertices 1.23, 0.46; 8 R-MAT graphs of 59,000 entries 0.48, 0.36;
// one attachment graph of 80,000 entries 0.43, 0.57, of 480,000 0.67, 1.22.
constexpr int kTeamListMax = 4 * kLanes;
constexpr int32_t kTeamEntries = 1 << 16;
// Batches whose largest graph is smaller go without the far counts: their searches
// cost less than the pass and its two barriers (60 vertices: round 0 0.12, 0.10 ms).
constexpr int32_t kFarMinN = 4096;

// tstart[g] = tasks (64 listed vertices each) of the graphs before g that go to
// teams, tstart[count + 1 + g] = of those that go to single CTAs; both task counters
// start again.  One CTA.
static __device__ void task_prefix(const BatchArgs &a) {
  __shared__ int s_scan[33];
  const int tid = threadIdx.x, T = blockDim.x;
  int32_t *const solo = a.tstart + a.count + 1;
  int teams = 0, ctas = 0;
  for (int base = 0; base < a.count; base += T) {
    const int g = base + tid;
    int t = 0, c = 0;
    if (g < a.count) {
      const int m = a.scount[g], o = a.off[g];
      (m <= kTeamListMax && a.rp[o + a.ng[g]] - a.rp[o] >= a.team_entries ? t : c) = (m + kLanes - 1) / kLanes;
    }
    int all_t, all_c;
    const int x = block_excl_scan(t, s_scan, &all_t), y = block_excl_scan(c, s_scan, &all_c);
    if (g < a.count) {
      a.tstart[g] = teams + x;
      solo[g] = ctas + y;
    }
    teams += all_t;
    ctas += all_c;
  }
  if (tid == 0) {
    a.tstart[a.count] = teams;
    solo[a.count] = ctas;
    a.ctl->task = a.ctl->task2 = 0;
  }
}

// the graph with start[g] <= task < start[g + 1]
static __device__ int task_graph(const BatchArgs &a, const int32_t *start, int task) {
  int lo = 0, hi = a.count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= task) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// CTAs of a team for n_tasks tasks of short lists on G CTAs.  Such lists are
// the vertices whose searches reach everything (round-0 survivors of a graph
// with few, the 64 largest bounds of round 1): one CTA takes 38 ms for a 64-lane
// batch on the largest graph of a mix (10.7M entries), the grid 1 ms, so few
// tasks leave most of the GPU idle behind the longest one.  Up to four tasks
// per CTA go to teams.  Long lists (graphs whose every vertex survives the
// bounds; searches that are cut early) keep one CTA per batch.
static __device__ __forceinline__ int task_team(int n_tasks, int G) {
  return max(1, min(G, 4 * G / max(1, n_tasks)));
}

// One 64-lane batch of graph g by a team (its own control block, its first
// CTA's workspace, the queues of its second CTA's workspace as scratch).
// Results in s_out of the team's CTA 0.  Not inlined: the CTA-local phases keep
// their registers.
template <int MODE>
static __device__ __noinline__ bool team_batch(const BatchArgs &a, int g, const int32_t *cand, int nl, TeamCtl *tc,
                                               Team tm, long long *s_out) {
  const int first = blockIdx.x - tm.b, o = a.off[g];
  unsigned char *ws0 = a.ws + a.ws_stride * (size_t)first;
  int32_t *gx = gain_ws(a.ws, a.ws_stride, a.max_n, first + 1).qv0;
  const int gx_n = (int)(ws_align((size_t)a.max_n * sizeof(int32_t)) / sizeof(int32_t));
  const bool gain = MODE == kModeGain;
  return grid_gain_batch<MODE>(gain ? a.rpf : a.rp, gain ? a.cif : a.ci, a.N, gain ? a.dS1 : a.dS, cand, nl, nullptr,
                               s_out, ws0, gx, a.goff, &tc->gg, a.gctl, &tc->bar, &a.ctl->err, a.tns,
                               gain ? a.mx : nullptr, gain ? a.c3 : nullptr, o, a.max_n, kBatchAll, nullptr, nullptr,
                               0, nullptr, tm, gx_n, gain ? nullptr : &tc->best, a.ng[g], a.simple != 0);
}

// The tasks of the lists in slist (scount entries per graph) that start counts, from
// the counter *task_next, by teams of S CTAs:
// kModeFarness  f0[v] <- f({v}) or -1, cut by the graph's best (round 0);
// kModeGain     ub[v] <- Delta(v | {s0}), stamp[v] <- 1, bestf[g] <- the best gain.
// Ends without a grid barrier.
template <int MODE>
static __device__ bool run_tasks(const BatchArgs &a, const GainWs &myws, GainCounters &cnt, long long *s_out,
                                 const int32_t *start, int32_t *task_next, const int S) {
  __shared__ int s_task;
  __shared__ long long s_ll[32];
  const int tid = threadIdx.x;
  const int n_tasks = start[a.count];
  const int t = blockIdx.x / S;
  const Team tm{(int)blockIdx.x - t * S, S};
  if ((t + 1) * S > (int)gridDim.x) return true;  // a remainder of fewer than S CTAs
  TeamCtl *tc = &a.teams[1 + t];
  const LaneGraphs lg = MODE == kModeFarness ? LaneGraphs{a.gid, a.ng, a.bestf} : LaneGraphs();
  for (;;) {
    if (S == 1) {
      if (tid == 0) s_task = atomicAdd(task_next, 1);
      cta_sync();
    } else {
      if (tm.b == 0) {  // the next task and a fresh control block for its batch
        unsigned int *w = reinterpret_cast<unsigned int *>(&tc->gg);
        for (int i = tid; i < (int)(sizeof(GridGainCtl) / 4); i += blockDim.x) w[i] = 0;
        if (tid == 0) {
          const int next = atomicAdd(task_next, 1);
          tc->g = next;
          // one threshold for the whole team: other teams may lower the graph's
          // best while this batch runs, and every CTA must cut the same lanes
          if (MODE == kModeFarness && next < n_tasks)
            tc->best = *(volatile long long *)&a.bestf[task_graph(a, start, next)];
        }
      }
      if (!grid_sync(&tc->bar, &a.ctl->err, a.tns, tm)) return false;
      if (tid == 0) s_task = *(volatile int32_t *)&tc->g;
      cta_sync();
    }
    const int task = s_task;
    cta_sync();
    if (task >= n_tasks) return true;
    const int g = task_graph(a, start, task), o = a.off[g], first = (task - start[g]) * kLanes;
    const int nl = min(kLanes, a.scount[g] - first);
    const int32_t *cand = a.slist + o + first;
    int levels = 0;
    if (S > 1) {
      if (!team_batch<MODE>(a, g, cand, nl, tc, tm, s_out)) return false;
      if (tm.b != 0) continue;
      cta_sync();  // s_out
      if (tid == 0) levels = tc->gg.levels;
    } else if (MODE == kModeFarness) {
      cta_gain_batch<MODE, true, false>(a.rp, a.ci, a.N, a.dS, cand, nl, s_out, myws, a.gctl, nullptr, lg, cnt, o);
    } else {
      const unsigned long long lev0 = cnt.levels;
      cta_gain_batch<MODE, true, true>(a.rpf, a.cif, a.N, a.dS1, cand, nl, s_out, myws, a.gctl, a.mx, lg, cnt, o,
                                       a.c3);
      levels = (int)(cnt.levels - lev0);
    }
    if (MODE == kModeFarness) {
      if (tid < nl) {
        a.f0[cand[tid]] = s_out[tid];
        if (S > 1 && s_out[tid] >= 0) atomicMin(&a.bestf[g], s_out[tid]);
      }
    } else {
      if (tid < nl) {
        a.ub[cand[tid]] = s_out[tid];
        a.stamp[cand[tid]] = 1;
      }
      const long long best = block_max_ll(tid < nl ? s_out[tid] : -1ll, s_ll);
      if (tid == 0) {
        atomicMax(&a.bestf[g], best);
        atomicMax(&a.depth[g], levels);
      }
    }
    cta_sync();
  }
}

// Every task of the lists: the teams' first, then the single CTAs'; who is done with
// one kind goes on to the other.  Called after a grid barrier (the lists are
// complete), ends with one.
template <int MODE>
static __device__ bool batch_tasks(const BatchArgs &a, const GainWs &myws, GainCounters &cnt, long long *s_out) {
  if (blockIdx.x == 0) task_prefix(a);
  if (!bsync(a)) return false;
  const int32_t *solo = a.tstart + a.count + 1;
  const int n_team = a.tstart[a.count], n_solo = solo[a.count];
  if (n_team && !run_tasks<MODE>(a, myws, cnt, s_out, a.tstart, &a.ctl->task, task_team(n_team, gridDim.x)))
    return false;
  if (n_solo && !run_tasks<MODE>(a, myws, cnt, s_out, solo, &a.ctl->task2, 1)) return false;
  return bsync(a);
}

// Round 0: the far counts of the single-graph path (k_far_counts, k_far_bound in
// gc_bfs.cu) over the union: per vertex the neighbours of degree 1 to kFarDeg in
// two classes (packed in ub, zero so far), per graph the members of each class,
// then a tighter key for every survivor.  One thread per counted row, a warp
// per survivor's row.
static __device__ bool batch_far_bounds(const BatchArgs &a) {
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x, G = gridDim.x;
  unsigned long long *cnt = reinterpret_cast<unsigned long long *>(a.ub);
  for (int base = (blockIdx.x * T + tid) & ~31; base < a.N; base += G * T) {
    const int u = base + lane;
    int g = -1, beg = 0, end = 0;
    if (u < a.N) {
      g = a.gid[u];
      beg = a.rp[u];
      end = a.rp[u + 1];
    }
    const unsigned long long c = far_class(end - beg);
    if (c)
      for (int e = beg; e < end; ++e) atomicAdd(&cnt[a.ci[e]], c);
    const int g0 = __shfl_sync(0xffffffffu, g, 0);
    if (__all_sync(0xffffffffu, g == g0 || g < 0)) {
      const unsigned lo = __ballot_sync(0xffffffffu, c == 1ull), hi = __ballot_sync(0xffffffffu, c > 1ull);
      if (lane == 0 && lo) atomicAdd(&a.cls[2 * g0], (unsigned long long)__popc(lo));
      if (lane == 0 && hi) atomicAdd(&a.cls[2 * g0 + 1], (unsigned long long)__popc(hi));
    } else if (c) {
      atomicAdd(&a.cls[2 * g + (c == 1ull ? 0 : 1)], 1ull);
    }
  }
  if (!bsync(a)) return false;
  for (int base = (blockIdx.x * T + tid) & ~31; base < a.N; base += G * T) {
    const int v = base + lane;
    int g = -1, deg = 0, beg = 0;
    long long k = LLONG_MIN, fa = 0;
    if (v < a.N) {
      g = a.gid[v];
      fa = a.fa[g];
      k = a.key[v];
      beg = a.rp[v];
      deg = a.rp[v + 1] - beg;
    }
    unsigned todo = __ballot_sync(0xffffffffu, v < a.N && -k <= fa);
    long long near0 = 0, near1 = 0;
    for (unsigned m = todo; m; m &= m - 1) {
      const int q = __ffs(m) - 1;
      const int rb = __shfl_sync(0xffffffffu, beg, q), rd = __shfl_sync(0xffffffffu, deg, q);
      long long x0 = 0, x1 = 0;
#pragma unroll 4
      for (int e = rb + lane; e < rb + rd; e += 32) {
        const unsigned long long x = cnt[a.ci[e]];
        x0 += (long long)(x & 0xffffffffull);
        x1 += (long long)(x >> 32);
      }
      x0 = warp_sum(x0);
      x1 = warp_sum(x1);
      if (lane == q) {
        near0 = x0;
        near1 = x1;
      }
    }
    if ((todo >> lane) & 1u) {
      const unsigned long long c = far_class(deg), own = cnt[v];
      const long long rest = max(0ll, (long long)a.ng[g] - 1 - deg);
      const long long f0 = (long long)a.cls[2 * g] - (c == 1ull) - near0 - (long long)(own & 0xffffffffull);
      const long long f1 = (long long)a.cls[2 * g + 1] - (c > 1ull) - near1 - (long long)(own >> 32);
      const long long far = min(rest, max(0ll, f0) + max(0ll, f1));
      const long long c2 = min((long long)deg + 3 * rest + k, rest - far);  // the degree bound's c2 from its key
      a.key[v] = -((long long)deg + 2 * c2 + 3 * (rest - c2));
    }
  }
  return bsync(a);
}

// Round 1 with two-hop bounds (the single-graph path's round 1, per graph):
// every candidate gets the bound for S = {s0}; the 64 largest bounds of each
// graph are evaluated as one CTA batch, then every candidate whose bound
// reaches that batch's best exact gain.  After that no unevaluated candidate
// can beat the best exact gain (its bound is below it), so the lazy rule of
// Sec. 4.2 accepts the best one.  Evaluated candidates get stamp 1 and their
// exact gain in ub; the rest keep stamp 0 and their bound.
static __device__ bool batch_round1_bounded(const BatchArgs &a, const GainWs &myws, GainCounters &cnt,
                                            long long *s_out) {
  __shared__ int s_task;
  __shared__ long long s_ll[32];
  __shared__ int s_scan[33];
  const int tid = threadIdx.x, b = blockIdx.x, G = gridDim.x, T = blockDim.x;
  seg_sum_excess3(a, a.dS1, a.g3);
  if (!bsync(a)) return false;
  {
    const int lane = tid & 31, gw = (b * T + tid) >> 5, nw = (G * T) >> 5;
    for (int v = gw; v < a.N; v += nw) {
      const long long s = warp_two_hop(a, a.dS1, a.c3, v);
      if (lane == 0) {
        a.ub[v] = a.dS1[v] == 0 ? -1ll : s + a.g3[a.gid[v]];
        a.stamp[v] = 0;
      }
    }
  }
  if (!bsync(a)) return false;
  // the first batch of each graph: its 64 largest bounds
  for (int g = b; g < a.count; g += G) {
    const int m = a.kk[g] >= 2 ? cta_top_bounds(a.ub, a.off[g], a.ng[g], kLanes, a.slist + a.off[g]) : 0;
    if (tid == 0) {
      a.scount[g] = m;
      a.bestf[g] = -1;  // the best exact gain of round 1 so far
    }
    cta_sync();
  }
  if (!bsync(a)) return false;
  if (!batch_tasks<kModeGain>(a, myws, cnt, s_out)) return false;
  // every other candidate whose bound reaches the first batch's best
  for (int g = b; g < a.count; g += G) {
    const int o = a.off[g], n = a.ng[g];
    const long long b1 = a.bestf[g];
    int carry = 0;
    if (a.kk[g] >= 2) {
      for (int base = 0; base < n; base += T) {
        const int i = base + tid;
        int flag = 0;
        if (i < n) {
          const long long u = a.ub[o + i];
          flag = u >= 0 && u >= b1 && a.stamp[o + i] == 0;
        }
        int total;
        const int pos = block_excl_scan(flag, s_scan, &total);
        if (flag) a.slist[o + carry + pos] = o + i;
        carry += total;
      }
    }
    if (tid == 0) a.scount[g] = carry;
    cta_sync();
  }
  if (!bsync(a)) return false;
  return batch_tasks<kModeGain>(a, myws, cnt, s_out);
}

// Bound refresh before the lazy rounds: the two-hop bound for the group after
// round 1 (d = the current d_S, c3 recounted into q0, G3 into g3[count + g])
// lowers every candidate's bound, as before each persistent launch of the
// single-graph path.
static __device__ bool batch_bound_refresh(const BatchArgs &a) {
  const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.x, G = gridDim.x, T = blockDim.x;
  const int gw = (b * T + tid) >> 5, nw = (G * T) >> 5;
  for (int u = gw; u < a.N; u += nw) {
    int c = 0;
    for (int e = a.rpf[u] + lane; e < a.rpf[u + 1]; e += 32) c += a.dS[a.cif[e]] >= 3;
    c = warp_sum(c);
    if (lane == 0) a.q0[u] = c;
  }
  seg_sum_excess3(a, a.dS, a.g3 + a.count);
  if (!bsync(a)) return false;
  for (int v = gw; v < a.N; v += nw) {
    const int g = a.gid[v];
    if (a.kk[g] <= 2 || a.ub[v] < 0) continue;  // warp-uniform: one v per warp
    const long long s = warp_two_hop(a, a.dS, a.q0, v) + a.g3[a.count + g];
    if (lane == 0 && s < a.ub[v]) a.ub[v] = s;
  }
  return bsync(a);
}

// Refresh of one graph's bounds in the lazy rounds, when its active list can no
// longer certify a pick (the single-graph path refreshes before each rebuild
// of its list the same way): c3 for the current d_S into q0, G3 of the graph,
// then every candidate's bound lowered to the two-hop bound for the current
// group.  By the CTAs of one team, with three team barriers.
static __device__ bool team_refresh_graph(const BatchArgs &a, int g, TeamCtl *tc, Team tm) {
  __shared__ long long s_ll[32];
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
  const int gw = (tm.b * T + tid) >> 5, nw = (tm.G * T) >> 5;
  const int o = a.off[g], n = a.ng[g];
  long long *g3 = a.g3 + a.count + g;
  if (tm.b == 0 && tid == 0) *g3 = 0;
  if (!grid_sync(&tc->bar, &a.ctl->err, a.tns, tm)) return false;
  long long x3 = 0;
  for (int i = tm.b * T + tid; i < n; i += tm.G * T) x3 += max(a.dS[o + i] - 3, 0);
  x3 = block_sum(x3, s_ll);
  if (tid == 0 && x3) atomicAdd((unsigned long long *)g3, (unsigned long long)x3);
  for (int u = o + gw; u < o + n; u += nw) {
    int c = 0;
    for (int e = a.rpf[u] + lane; e < a.rpf[u + 1]; e += 32) c += a.dS[a.cif[e]] >= 3;
    c = warp_sum(c);
    if (lane == 0) a.q0[u] = c;
  }
  if (!grid_sync(&tc->bar, &a.ctl->err, a.tns, tm)) return false;
  const long long G3 = *(volatile long long *)g3;
  for (int v = o + gw; v < o + n; v += nw) {
    if (a.ub[v] < 0) continue;  // a member (warp-uniform)
    const long long s = warp_two_hop(a, a.dS, a.q0, v) + G3;
    if (lane == 0 && s < a.ub[v]) a.ub[v] = s;
  }
  return grid_sync(&tc->bar, &a.ctl->err, a.tns, tm);
}

// Sweep of graph g in round r by one team: every candidate not evaluated in
// this round whose bound reaches the round's best exact gain is evaluated, one
// 64-lane batch per CTA at a time (listed in slist, free after round 1).  After
// that no unevaluated bound reaches the best.
static __device__ bool team_sweep(const BatchArgs &a, int g, int r, TeamCtl *tc, Team tm, const GainWs &myws,
                                  GainCounters &cnt) {
  __shared__ int s_at;
  __shared__ long long s_out[kLanes];
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
  LazyCtl *lc = &a.lc[g];
  const int o = a.off[g], n = a.ng[g];
  const bool lead = tm.b == 0 && tid == 0;
  if (lead) {
    tc->sweep_n = tc->sweep_next = 0;
    tc->sweep_best = 0;
  }
  if (!grid_sync(&tc->bar, &a.ctl->err, a.tns, tm)) return false;
  const long long gb = *(volatile long long *)&lc->best_gain;
  for (int base = tm.b * T + (tid & ~31); base < n; base += tm.G * T) {
    const int i = base + lane;
    const bool want = i < n && a.ub[o + i] >= max(gb, 0ll) && a.stamp[o + i] != r;
    const unsigned wm = __ballot_sync(0xffffffffu, want);
    int at = 0;
    if (lane == 0 && wm) at = atomicAdd(&tc->sweep_n, __popc(wm));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (want) a.slist[o + at + __popc(wm & ((1u << lane) - 1u))] = o + i;
  }
  if (!grid_sync(&tc->bar, &a.ctl->err, a.tns, tm)) return false;
  const int m = *(volatile int32_t *)&tc->sweep_n;
  if (m > kBatchSweepMin) {
    for (;;) {
      if (tid == 0) s_at = atomicAdd(&tc->sweep_next, kLanes);
      cta_sync();
      const int at = s_at;
      cta_sync();
      if (at >= m) break;
      const int nl = min(kLanes, m - at);
      cta_gain_batch<kModeGain, true, false>(a.rpf, a.cif, a.N, a.dS, a.slist + o + at, nl, s_out, myws, a.gctl, a.mx,
                                             LaneGraphs(), cnt, o, a.c3);
      if (tid < nl) {
        const int v = a.slist[o + at + tid];
        a.ub[v] = s_out[tid];
        a.stamp[v] = r;
        // gains are below 2^31 (checked in round 1, and they only decrease)
        atomicMax(&tc->sweep_best, ((u64)s_out[tid] << 32) | (u64)(0xffffffffu - (unsigned)(v - o)));
      }
      cta_sync();
    }
    if (!grid_sync(&tc->bar, &a.ctl->err, a.tns, tm)) return false;
    if (lead && tc->sweep_best) {
      const long long sg = (long long)(tc->sweep_best >> 32);
      const int sv = o + (int)(0xffffffffu - (unsigned)(tc->sweep_best & 0xffffffffull));
      if (better_max(sg, sv, lc->best_gain, lc->best_id)) {
        lc->best_gain = sg;
        lc->best_id = sv;
        lc->best_lane = -1;  // its search is not in the claim log
      }
    }
  }
  return true;
}

// Lazy rounds (Sec. 4.2) of graph g by one team of CTAs, from its list built in
// P5 to its last pick: the loop of the single-graph persistent kernel
// (gc_lazy.cu) on a part of the grid.  Three forms of a step:
//   lean  (list of at most list_cap entries): the team's CTA 0 keeps the list in
//         shared memory with its sorted view, folds, decides, selects and runs
//         level 0; the team runs the rest of the 64-lane batch, and a pick
//         updates d_S from the claim log (or the relabel BFS past its capacity);
//   wide  (deep graphs: more than kWideLevels levels per round-1 batch): one
//         64-lane batch per CTA of the team, no team barrier inside;
//   grid  (longer lists): the whole team selects (grid_lazy_step).
// When the list cannot certify a pick, the graph's bounds are refreshed, the
// candidates that still reach the best gain are swept if they are many, and the
// list is rebuilt; a second failure in the same round lists every candidate
// from then on.  Every CTA of the team runs the same loop.
static __device__ bool team_lazy(const BatchArgs &a, int g, TeamCtl *tc, Team tm, GridSelScratch *gsel,
                                 GainCounters &cnt, GridCounts &gcnt, unsigned char *s_list) {
  __shared__ Cta0State s_st;
  __shared__ int s_nord;
  __shared__ u64 s_red[32];
  const int tid = threadIdx.x, b = tm.b;
  const bool lead = b == 0 && tid == 0;
  LazyCtl *lc = &a.lc[g];
  const int o = a.off[g], ng = a.ng[g], k = a.kk[g];
  const int first = blockIdx.x - b;  // the team's first CTA: its workspace serves the team's batches
  unsigned char *ws0 = a.ws + a.ws_stride * (size_t)first;
  const GainWs myws = gain_ws(a.ws, a.ws_stride, a.max_n, blockIdx.x);
  int32_t *gx = a.gx + 3 * (size_t)o;
  ClaimRec *clog = a.clog + 2 * (size_t)o;
  const u64 clog_cap = 2 * (u64)ng;
  int32_t *wsel = a.wsel + (size_t)first * kLanes;
  long long *wgain = a.wgain + (size_t)first * kLanes;
  const bool wide = a.depth[g] > kWideLevels;
  auto sync = [&]() { return grid_sync(&tc->bar, &a.ctl->err, a.tns, tm); };

  // CTA 0's list: bounds, ids, stamps, and the sorted view of them
  const int cap = a.list_cap;
  long long *sk = reinterpret_cast<long long *>(s_list);
  int32_t *sa = reinterpret_cast<int32_t *>(sk + cap), *ss = sa + cap;
  SortedView view;
  view.ord = reinterpret_cast<uint16_t *>(ss + cap);
  view.tmp = view.ord + cap;
  view.mark = reinterpret_cast<unsigned char *>(view.tmp + cap);
  view.nord = &s_nord;
  bool every = false, fold = false;
  int rebuilt = -1;  // round of the last rebuild
  const int32_t *list = nullptr;
  int m = 0;
  bool lean = false;
  // the list of the coming steps (every CTA), and CTA 0's copy of it
  auto load = [&]() {
    list = every ? a.iota + o : a.act + (size_t)g * a.A;
    m = every ? ng : *(volatile int32_t *)&a.act_n[g];
    lean = !wide && m <= cap;
    if (!lean || b != 0) return;
    if (tid == 0) {
      s_st.bpos = -1;
      s_st.bid = lc->best_id;
      s_st.bgain = lc->best_gain;
      s_st.theta = lc->theta;
      s_st.log_mark = lc->log_mark;
      s_st.nsel = 0;
      s_st.dec = 0;
    }
    cta_sync();
    for (int i = tid; i < m; i += blockDim.x) {
      const int v = list[i];
      sa[i] = v;
      sk[i] = a.ub[v];
      ss[i] = a.stamp[v];
      if (v == s_st.bid) {
        s_st.bpos = i;
        lc->best_pos = i;
      }
    }
    cta_sync();
    sv_build(sk, m, view);
  };
  unsigned long long t_ph[3] = {0, 0, 0}, t_mark = lead ? global_ns() : 0;  // phase clocks
  auto lap = [&](int q) {
    if (lead) {
      const unsigned long long now = global_ns();
      t_ph[q] += now - t_mark;
      t_mark = now;
    }
    __syncwarp();  // reconverge warp 0 before the warp-synchronous code that follows
  };
  load();
  int r = *(volatile int32_t *)&lc->round;
  if (!sync()) return false;
  while (r < k) {
    if (lean) {
      if (b == 0) {
        lean_step(sa, a.ub, a.stamp, lc, &tc->gg, fold, r, sk, ss, view, s_st);
        cta_sync();  // s_st.dec, the batch and the reset batch control block
        const int d = s_st.dec;
        if (d == 0)
          grid_gain_batch<kModeGain>(a.rpf, a.cif, a.N, a.dS, s_st.sel, 0, &s_st.nsel, s_st.gout, ws0, gx, a.goff,
                                     &tc->gg, a.gctl, &tc->bar, &a.ctl->err, a.tns, a.mx, a.c3, o, a.max_n,
                                     kBatchLevel0, clog, &lc->log_n, clog_cap, nullptr, tm, ng);  // (the candidates alone)
      }
    } else if (wide) {
      if (b == 0)
        lazy_cta0_step(list, m, a.ub, a.stamp, lc, nullptr, fold, nullptr, 0, nullptr, nullptr, wsel, wgain, nullptr,
                       tm.G * kLanes);
    } else {
      int dec_local;
      if (!grid_lazy_step(list, m, a.ub, a.stamp, nullptr, nullptr, lc, &tc->gg, fold, lc->sel, lc->selpos, lc->gsel,
                          kLanes, gsel, &tc->bar, &a.ctl->err, a.tns, &dec_local, tm))
        return false;
    }
    if (lead) {  // an accepted pick's update starts from zero
      lc->pk[0] = lc->pk[1] = lc->pk[2] = 0;
      lc->decrease = 0;
    }
    if (!sync()) return false;
    const int dec = *(volatile int32_t *)&lc->dec;
    lap(0);
    if (dec == 2) {
      if (every) {  // cannot happen with every candidate listed
        if (lead) check_fail(a.ctl, 6, g, 1, 2);
        return false;
      }
      if (rebuilt == r) {
        every = true;
        if (lead) lc->theta = LLONG_MIN;
      } else {
        rebuilt = r;
        if (!team_refresh_graph(a, g, tc, tm)) return false;
        if (!team_sweep(a, g, r, tc, tm, myws, cnt)) return false;
        if (b == 0) cta_build_list(a, g);
      }
      if (!sync()) return false;
      load();
      fold = false;
      lap(0);
      continue;
    }
    if (dec == 0) {
      if (wide) {
        const int ns = *(volatile int32_t *)&lc->n_sel, nb = (ns + kLanes - 1) / kLanes;
        for (int bi = b; bi < nb; bi += tm.G)
          cta_gain_batch<kModeGain, true, false>(a.rpf, a.cif, a.N, a.dS, wsel + bi * kLanes,
                                                 min(kLanes, ns - bi * kLanes), wgain + bi * kLanes, myws, a.gctl,
                                                 a.mx, LaneGraphs(), cnt, o, a.c3);
        if (!sync()) return false;  // gains visible to CTA 0
      } else {
        // CTA 0 keeps a lean batch in shared memory, the others read its copy
        const bool st0 = lean && b == 0;
        if (!grid_gain_batch<kModeGain>(a.rpf, a.cif, a.N, a.dS, st0 ? s_st.sel : lc->sel, 0,
                                        st0 ? &s_st.nsel : &lc->n_sel, st0 ? s_st.gout : lc->gsel, ws0, gx, a.goff,
                                        &tc->gg, a.gctl, &tc->bar, &a.ctl->err, a.tns, a.mx, a.c3, o, a.max_n,
                                        lean ? kBatchRest : kBatchAll, clog, &lc->log_n, clog_cap, &gcnt, tm, ng,
                                        nullptr, 0, a.simple != 0))
          return false;
        if (!lean && !sync()) return false;  // a team-wide fold reads the gains CTA 0 wrote
        if (lead && *(volatile int32_t *)&tc->gg.err) atomicExch(&a.ctl->err, *(volatile int32_t *)&tc->gg.err);
      }
      lap(1);
      fold = true;
      continue;
    }
    // accept the round's best and update d_S from it
    fold = false;
    const int blane = *(volatile int32_t *)&lc->best_lane, pick = *(volatile int32_t *)&lc->best_id;
    const u64 l0 = *(volatile u64 *)&lc->best_seg0, l1 = *(volatile u64 *)&lc->best_seg1;
    if (!wide && blane >= 0 && blane < kLanes && l0 <= l1 && l1 <= clog_cap) {
      const u64 bit = 1ull << blane;
      u64 dec_sum = 0, rel = 0;
      log_update_row(a.rpf, a.cif, a.dS, pick, dec_sum, rel, tm);
      for (u64 i = l0 + (u64)b * blockDim.x + tid; i < l1; i += (u64)tm.G * blockDim.x) {
        const int4 e = *reinterpret_cast<const int4 *>(clog + i);
        if (!(((u64)(unsigned)e.z | ((u64)(unsigned)e.w << 32)) & bit)) continue;
        const int old = atomicMin(&a.dS[e.x], e.y);
        if (old > e.y) dec_sum += (u64)(old - e.y);
      }
      if (lead) {  // the pick itself (level 0)
        const int old = atomicMin(&a.dS[pick], 0);
        if (old > 0) dec_sum += (u64)old;
      }
      dec_sum = block_sum(dec_sum, s_red);
      if (tid == 0 && dec_sum) atomicAdd(&lc->decrease, dec_sum);
    } else if (!grid_relabel_bfs(a.rpf, a.cif, a.N, a.dS, &lc->best_id, 1, a.q0 + o, a.q1 + o, lc->pk, nullptr,
                                 &lc->decrease, nullptr, a.goff + o, a.st1 + o, &tc->bar, &a.ctl->err, a.tns, nullptr,
                                 a.c3, tm)) {
      return false;
    }
    if (!sync()) return false;
    if (lead) {
      const long long gain = lean ? s_st.bgain : lc->best_gain;
      const u64 d = *(volatile u64 *)&lc->decrease;
      if ((long long)d != gain) check_fail(a.ctl, 6, g, gain, (long long)d);
      a.picks[(size_t)g * a.kmax + r] = pick;
      a.pgain[(size_t)g * a.kmax + r] = gain;
      a.ub[pick] = -1;  // a member: never a candidate again
      if (lean && s_st.bpos >= 0 && s_st.bpos < m && sa[s_st.bpos] == pick) sk[s_st.bpos] = -1;
      lc->last_gain = gain;
      lc->best_id = -1;
      lc->best_gain = -1;
      lc->best_lane = -1;
      lc->log_n = 0;  // the next round's log (its first batch starts after a barrier)
      lc->log_mark = 0;
      if (lean) {
        s_st.bid = -1;
        s_st.bgain = -1;
        s_st.bpos = -1;
        s_st.log_mark = 0;
      }
      lc->round = r + 1;
    }
    ++r;
    if (lean) cta_sync();  // only CTA 0 reads the bookkeeping before the next step's barrier
    else if (!sync()) return false;
    lap(2);
  }
  if (lead) {
    atomicAdd((unsigned long long *)&a.ctl->iterations, (unsigned long long)lc->steps);
    for (int q = 0; q < 3; ++q) atomicAdd(&a.ctl->ns_lazy[q], t_ph[q]);
  }
  return true;
}

// Two CTAs per SM (64 registers, no spills): the CTA-local phases are latency
// bound and gain from the second resident CTA.
__global__ void __launch_bounds__(kBatchThreads, 2) k_batch_solve(const BatchArgs a) {
  __shared__ long long s_out[kLanes];
  __shared__ int s_task;
  __shared__ int s_scan[33];
  __shared__ unsigned long long s_red[32];
  const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.x, G = gridDim.x, T = blockDim.x;
  GainCounters cnt;
  const unsigned long long t_start = global_ns();
  if (b == 0 && tid == 0) a.ctl->t_start = t_start;
  const GainWs myws = gain_ws(a.ws, a.ws_stride, a.max_n, b);  // this CTA's workspace, sized for the largest graph
  // ---- P0: lower bounds, per-graph argmin ----
  {
    const int gw = (b * T + tid) >> 5, nw = (G * T) >> 5;
    for (int v = gw; v < a.N; v += nw) {
      const int beg = a.rp[v], end = a.rp[v + 1];
      long long x = 0;
      for (int e = beg + lane; e < end; e += 32) {
        const int w = a.ci[e];
        x += (long long)(a.rp[w + 1] - a.rp[w] - 1);
      }
      x = warp_sum(x);
      if (lane == 0) {
        const int g = a.gid[v];
        const long long deg = end - beg;
        long long rest = (long long)a.ng[g] - 1 - deg;
        if (rest < 0) rest = 0;
        const long long c2 = x < rest ? x : rest;
        const long long lb = deg + 2 * c2 + 3 * (rest - c2);
        a.key[v] = -lb;
        a.f0[v] = -1;
        a.dS[v] = kInf;
        a.stamp[v] = 0;
        a.ub[v] = 0;  // the far counts of P2 (bounds and gains come in round 1)
        atomicMin(&a.packed[g], ((unsigned long long)lb << 32) | (unsigned long long)(v - a.off[g]));
      }
    }
  }
  for (int g = b * T + tid; g < 2 * a.count; g += G * T) a.g3[g] = 0;
  if (!bsync(a)) return;
  // ---- P1: BFS from all v_a ----
  for (int g = b * T + tid; g < a.count; g += G * T) a.seeds[g] = a.off[g] + (int)(a.packed[g] & 0xffffffffull);
  if (!bsync(a)) return;
  if (!grid_relabel_bfs(a.rp, a.ci, a.N, a.dS, a.seeds, a.count, a.q0, a.q1, a.ctl->pk, nullptr,
                        &a.ctl->decrease, nullptr, a.goff, a.st1, &a.ctl->bar, &a.ctl->err, a.tns))
    return;
  if (!bsync(a)) return;
  seg_sum_dist(a, a.fa);
  if (b == 0 && tid == 0) a.ctl->pk[0] = a.ctl->pk[1] = a.ctl->pk[2] = 0;
  if (!bsync(a)) return;
  // ---- P2: round-0 survivors (every v with LB(v) <= f_a) ----
  if (a.far && !batch_far_bounds(a)) return;
  // P2a, one CTA per graph: compact the graph's survivors into its own region
  // of slist (graph-aligned, so batches never mix graphs)
  for (int g = b; g < a.count; g += G) {
    const int o = a.off[g], n = a.ng[g];
    const long long fa = a.fa[g];
    const int va = a.seeds[g];
    if (tid == 0) {
      a.bestf[g] = fa;
      a.f0[va] = fa;
      a.key[va] = LLONG_MIN;
    }
    cta_sync();
    int carry = 0;
    for (int base = 0; base < n; base += T) {
      const int i = base + tid;
      int flag = 0;
      if (i < n) {
        const long long k = a.key[o + i];
        flag = k != LLONG_MIN && -k <= fa;
      }
      int total;
      const int pos = block_excl_scan(flag, s_scan, &total);
      if (flag) a.slist[o + carry + pos] = o + i;
      carry += total;
    }
    if (tid == 0) a.scount[g] = carry;
    cta_sync();
  }
  if (!bsync(a)) return;
  // P2b: 64 survivors per task, by teams or CTAs
  if (!batch_tasks<kModeFarness>(a, myws, cnt, s_out)) return;
  // P2d, one CTA per graph: s0 = argmin (f, id) over the exact farness values
  for (int g = b; g < a.count; g += G) {
    const int s0 = cta_argmin_f0(a, g);
    if (tid == 0) a.seeds[g] = a.off[g] + (s0 >= 0 ? s0 : 0);
    cta_sync();
  }
  if (!bsync(a)) return;
  if (b == 0 && tid == 0) a.ctl->ns_ph[0] = global_ns() - t_start;
  // ---- P3: d_S = BFS from all s0; farness; neighbour bound ----
  for (int v = b * T + tid; v < a.N; v += G * T) a.dS[v] = kInf;
  if (!bsync(a)) return;
  if (!grid_relabel_bfs(a.rp, a.ci, a.N, a.dS, a.seeds, a.count, a.q0, a.q1, a.ctl->pk, nullptr,
                        &a.ctl->decrease, nullptr, a.goff, a.st1, &a.ctl->bar, &a.ctl->err, a.tns))
    return;
  if (!bsync(a)) return;
  seg_sum_dist(a, a.farness);
  for (int v = b * T + tid; v < a.N; v += G * T) a.dS1[v] = a.dS[v];  // round 1's read-only d_S
  {
    const int gw = (b * T + tid) >> 5, nw = (G * T) >> 5;
    for (int v = gw; v < a.N; v += nw) {
      int m = 0;
      for (int e = a.rp[v] + lane; e < a.rp[v + 1]; e += 32) m = max(m, a.dS[a.ci[e]]);
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 4));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      if (lane == 0) a.mx[v] = m;
    }
  }
  if (b == 0 && tid == 0) {
    a.ctl->pk[0] = a.ctl->pk[1] = a.ctl->pk[2] = 0;
    a.ctl->task = 0;
  }
  if (!bsync(a)) return;
  if (!batch_prune(a)) return;
  for (int g = b * T + tid; g < a.count; g += G * T) {
    const int s0 = a.seeds[g];
    if (a.f0[s0] != a.farness[g]) check_fail(a.ctl, 3, g, a.f0[s0], a.farness[g]);
    a.picks[(size_t)g * a.kmax] = s0;
    a.pgain[(size_t)g * a.kmax] = a.farness[g];
    a.packed[g] = 0;  // reused as the round-1 arg-max key
  }
  // ---- P4: round 1 (graph-aligned batches from a dynamic counter) ----
  if (b == 0 && tid == 0) a.ctl->ns_ph[4] = global_ns() - t_start;
  if (a.bounded) {
    if (!bsync(a)) return;  // the pruned adjacency's c3 and the picks above are in place
    if (!batch_round1_bounded(a, myws, cnt, s_out)) return;
  }
  const int n_tasks = a.bounded ? 0 : a.bstart[a.count];
  for (;;) {
    if (tid == 0) s_task = atomicAdd(&a.ctl->task, 1);
    cta_sync();
    const int t = s_task;
    cta_sync();
    if (t >= n_tasks) break;
    int lo = 0, hi = a.count - 1;  // graph with bstart[g] <= t < bstart[g+1]
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.bstart[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    const int g = lo;
    if (a.kk[g] < 2) continue;
    const int o = a.off[g], first = (t - a.bstart[g]) * a.lanes1;
    const int nl = min(a.lanes1, a.ng[g] - first);
    const unsigned long long lev0 = cnt.levels;
    cta_gain_batch<kModeGain, true, true>(a.rpf, a.cif, a.N, a.dS1, a.iota + o + first, nl, a.ub + o + first, myws,
                                          a.gctl, a.mx, LaneGraphs(), cnt, o, a.c3);
    if (tid == 0) atomicMax(&a.depth[g], (int)(cnt.levels - lev0));
  }
  if (!bsync(a)) return;
  if (b == 0 && tid == 0) a.ctl->ns_ph[5] = global_ns() - t_start;
  if (!a.bounded)  // every candidate was evaluated in round 1
    for (int v = b * T + tid; v < a.N; v += G * T) a.stamp[v] = 1;
  for (int g = b * T + tid; g < a.count; g += G * T) a.ub[a.seeds[g]] = -1;  // s0 is a member
  if (!bsync(a)) return;
  // per-graph argmax (gain desc, id asc) of round 1
  for (int base = (b * T + tid) & ~31; base < a.N; base += G * T) {
    const int v = base + lane;
    unsigned long long key = 0;
    int g = -1;
    if (v < a.N) {
      g = a.gid[v];
      const long long u = a.ub[v];
      if (u >= 0 && a.kk[g] >= 2 && a.stamp[v] == 1) {  // exact round-1 gains only
        if (u >= (1ll << 31)) atomicExch(&a.ctl->err, GC_ERANGE);
        key = ((unsigned long long)u << 32) | (0xffffffffull - (unsigned long long)(v - a.off[g]));
      }
    }
    const int g0 = __shfl_sync(0xffffffffu, g, 0);
    if (__all_sync(0xffffffffu, g == g0 || g < 0)) {
      unsigned long long m = key;
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, s));
      if (lane == 0 && g0 >= 0 && m) atomicMax(&a.packed[g0], m);
    } else if (g >= 0 && key) {
      atomicMax(&a.packed[g], key);
    }
  }
  if (!bsync(a)) return;
  if (b == 0) {
    if (tid == 0) {
      a.ctl->nseeds = 0;
      a.ctl->remaining = 0;
    }
    cta_sync();
    for (int g = tid; g < a.count; g += T) {
      if (a.kk[g] < 2) {
        a.lc[g].round = a.kk[g];  // nothing after round 0
        continue;
      }
      const unsigned long long key = a.packed[g];
      const int v = a.off[g] + (int)(0xffffffffull - (key & 0xffffffffull));
      const long long gain = (long long)(key >> 32);
      a.picks[(size_t)g * a.kmax + 1] = v;
      a.pgain[(size_t)g * a.kmax + 1] = gain;
      a.ub[v] = -1;
      a.seeds[atomicAdd(&a.ctl->nseeds, 1)] = v;
      LazyCtl *lc = &a.lc[g];
      lc->round = 2;
      lc->best_id = -1;
      lc->best_gain = -1;
      lc->last_gain = gain;
      lc->pad = 0;  // fold flag
      if (a.kk[g] > 2) atomicAdd(&a.ctl->remaining, 1);
    }
  }
  if (!bsync(a)) return;
  if (!grid_relabel_bfs(a.rpf, a.cif, a.N, a.dS, a.seeds, *(volatile int32_t *)&a.ctl->nseeds, a.q0, a.q1,
                        a.ctl->pk, nullptr, &a.ctl->decrease, nullptr, a.goff, a.st1, &a.ctl->bar,
                        &a.ctl->err, a.tns, nullptr, a.c3))
    return;
  if (!bsync(a)) return;
  if (b == 0 && tid == 0) {
    a.ctl->pk[0] = a.ctl->pk[1] = a.ctl->pk[2] = 0;
    a.ctl->nseeds = 0;
  }
  if (a.bounded && !batch_bound_refresh(a)) return;
  // ---- P5: active lists (one CTA per graph) ----
  for (int g = b; g < a.count; g += G) {
    if (a.kk[g] <= 2) continue;
    cta_build_list(a, g);
  }
  if (!bsync(a)) return;
  if (b == 0 && tid == 0) {
    a.ctl->ns_ph[1] = global_ns() - t_start;
    a.ctl->stage = 1;
  }
  // work counters
  u64 c_scalar = block_sum(cnt.scalar, s_red);
  u64 c_union = block_sum(cnt.uni, s_red);
  u64 c_front = block_sum(cnt.front, s_red);
  u64 c_push = block_sum(cnt.push, s_red);
  if (tid == 0) {
    atomicAdd(&a.gctl->edges_scalar, c_scalar);
    atomicAdd(&a.gctl->edges_union, c_union);
    atomicAdd(&a.gctl->frontier, c_front);
    atomicAdd(&a.gctl->pushes, c_push);
    atomicAdd(&a.gctl->levels, cnt.levels);
    atomicAdd(&a.gctl->batches, cnt.batches);
    atomicAdd(&a.gctl->lanes, cnt.lanes);
  }
}

// P6: the lazy rounds.  Graphs of at least grid_min_n vertices take the whole
// grid in turn; the others go to teams of team_size consecutive CTAs, each team
// taking the next graph of `order` (longest first) and running it to
// completion, so that no graph waits for another graph's step.  One CTA per SM
// (128 registers), as in the single-graph kernel; two (64 registers) where more small
// graphs than SMs go to single CTAs (200 attachment graphs of 1,000 vertices, k = 40,
// lazy rounds: 1.77 ms against 2.58; of 300, 1.46 against 2.11).
template <int PER_SM>
__global__ void __launch_bounds__(kBatchThreads, PER_SM) k_batch_lazy(const BatchArgs a) {
  extern __shared__ __align__(16) unsigned char s_list[];  // list_cap * 21 bytes
  __shared__ u64 s_red[32];
  if (*(volatile int32_t *)&a.ctl->stage != 1) return;  // an earlier phase failed
  const int tid = threadIdx.x, b = blockIdx.x;
  GainCounters cnt;
  GridCounts gcnt;
  bool ok = true;
  for (int g = 0; g < a.count && ok; ++g)
    if (a.ng[g] >= a.grid_min_n && a.kk[g] > 2)
      ok = team_lazy(a, g, &a.teams[0], whole_grid(), a.gsel, cnt, gcnt, s_list);
  const int S = a.team_size, t = b / S;
  const Team tm{b - t * S, S};
  if ((t + 1) * S <= (int)gridDim.x) {  // (a remainder of fewer than S CTAs stays idle)
    TeamCtl *tc = &a.teams[1 + t];
    while (ok) {
      if (tm.b == 0 && tid == 0) {
        const int i = atomicAdd(&a.ctl->lazy_next, 1);
        tc->g = i < a.order_n ? a.order[i] : -1;
      }
      ok = grid_sync(&tc->bar, &a.ctl->err, a.tns, tm);
      if (!ok) break;
      const int g = *(volatile int32_t *)&tc->g;
      if (g < 0) break;
      ok = team_lazy(a, g, tc, tm, a.gsel + 1 + t, cnt, gcnt, s_list) &&
           grid_sync(&tc->bar, &a.ctl->err, a.tns, tm);  // everyone has read tc->g
    }
  }
  u64 c_scalar = block_sum(cnt.scalar + gcnt.scalar, s_red);
  u64 c_union = block_sum(cnt.uni + gcnt.uni, s_red);
  u64 c_front = block_sum(cnt.front + gcnt.front, s_red);
  u64 c_push = block_sum(cnt.push + gcnt.push, s_red);
  if (tid == 0) {
    atomicAdd(&a.gctl->edges_scalar, c_scalar);
    atomicAdd(&a.gctl->edges_union, c_union);
    atomicAdd(&a.gctl->frontier, c_front);
    atomicAdd(&a.gctl->pushes, c_push);
    atomicAdd(&a.gctl->levels, cnt.levels);
    atomicAdd(&a.gctl->batches, cnt.batches);
    atomicAdd(&a.gctl->lanes, cnt.lanes);
    atomicMax(&a.ctl->ns_ph[2], global_ns() - a.ctl->t_start);
  }
}

// P7: every group's farness by one BFS from all picks of all graphs.
__global__ void __launch_bounds__(kBatchThreads, 2) k_batch_check(const BatchArgs a) {
  if (*(volatile int32_t *)&a.ctl->stage != 1 || *(volatile int32_t *)&a.ctl->err != 0) return;  // set before the launch
  const int tid = threadIdx.x, b = blockIdx.x, G = gridDim.x, T = blockDim.x;
  // ---- P7: check every group's farness with one BFS ----
  for (int v = b * T + tid; v < a.N; v += G * T) a.dS[v] = kInf;
  if (b == 0) {
    if (tid == 0) {
      a.ctl->nseeds = 0;
      a.ctl->pk[0] = a.ctl->pk[1] = a.ctl->pk[2] = 0;  // the grid lazy rounds leave them set
    }
    cta_sync();
    for (int g = tid; g < a.count; g += T) {
      long long f = a.pgain[(size_t)g * a.kmax];
      for (int r = 1; r < a.kk[g]; ++r) f -= a.pgain[(size_t)g * a.kmax + r];
      a.fa[g] = f;  // farness implied by the accepted gains
      a.farness[g] = 0;
    }
  }
  if (!bsync(a)) return;
  if (b == 0) {
    for (int g = 0; g < a.count; ++g) {
      for (int r = tid; r < a.kk[g]; r += T) a.seeds[atomicAdd(&a.ctl->nseeds, 1)] = a.picks[(size_t)g * a.kmax + r];
    }
  }
  if (!bsync(a)) return;
  if (!grid_relabel_bfs(a.rp, a.ci, a.N, a.dS, a.seeds, *(volatile int32_t *)&a.ctl->nseeds, a.q0, a.q1,
                        a.ctl->pk, nullptr, &a.ctl->decrease, nullptr, a.goff, a.st1, &a.ctl->bar,
                        &a.ctl->err, a.tns))
    return;
  if (!bsync(a)) return;
  seg_sum_dist(a, a.farness);
  if (!bsync(a)) return;
  for (int g = b * T + tid; g < a.count; g += G * T)
    if (a.farness[g] != a.fa[g]) check_fail(a.ctl, 7, g, a.fa[g], a.farness[g]);
  if (b == 0 && tid == 0) a.ctl->ns_ph[3] = global_ns() - a.ctl->t_start;
}

__global__ void k_iota(int32_t *p, int32_t n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = i;
}

// union CSR: shift graph g's row pointers by its first edge and its neighbour
// ids by its first vertex; gid[v] = graph of v
__global__ void k_union_fix(int32_t *rp, int32_t *ci, int32_t *gid, const int32_t *off, const int64_t *eoff,
                            int32_t count, int32_t N, int64_t nnz) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < N; v += stride) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (off[mid] <= v) lo = mid;
      else hi = mid - 1;
    }
    gid[v] = lo;
    rp[v] += (int32_t)eoff[lo];
  }
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += stride) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (eoff[mid] <= e) lo = mid;
      else hi = mid - 1;
    }
    ci[e] += off[lo];
  }
}

}  // namespace gc

using namespace gc;

struct gc_batch {
  int32_t count = 0;
  int32_t N = 0;
  int64_t nnz = 0;
  int32_t max_n = 0;
  cudaStream_t stream = nullptr;
  int num_sms = 0, ctas = 0;
  std::vector<int32_t> h_off, h_n;
  int32_t *rp = nullptr, *ci = nullptr, *gid = nullptr, *off = nullptr, *ng = nullptr, *iota = nullptr;
  int32_t *dS = nullptr, *mx = nullptr, *stamp = nullptr, *q0 = nullptr, *q1 = nullptr, *goff = nullptr,
          *st1 = nullptr;
  int32_t *rpf = nullptr, *cif = nullptr, *c3 = nullptr, *gx = nullptr, *dS1 = nullptr;
  GridSelScratch *gsel = nullptr;
  TeamCtl *teams = nullptr;     // [1 + ctas]: the whole grid's, then the teams'
  ClaimRec *clog = nullptr;
  int32_t *wsel = nullptr, *depth = nullptr, *order = nullptr;
  long long *wgain = nullptr;
  int lazy_ctas = 0;            // CTAs of the lazy rounds (one per SM)
  std::vector<int64_t> h_nnz;   // adjacency entries per graph
  long long *ub = nullptr, *key = nullptr, *f0 = nullptr;
  unsigned char *ws = nullptr;
  size_t ws_stride = 0;
  unsigned long long *packed = nullptr;
  unsigned long long *cls = nullptr;
  int32_t simple = 0;
  long long *fa = nullptr, *farness = nullptr, *bestf = nullptr, *g3 = nullptr;
  LazyCtl *lc = nullptr;
  int32_t *act = nullptr, *act_n = nullptr, *kk = nullptr, *bstart = nullptr;
  int32_t A = 0, act_cap = 0;
  int32_t kcap = 0, h_kcap = 0;  // picks a graph that the device buffers, the pinned copy hold
  int32_t *picks = nullptr;
  long long *pgain = nullptr;
  int32_t *seeds = nullptr;
  int64_t seeds_cap = 0;
  int32_t *slist = nullptr, *scount = nullptr, *tstart = nullptr;
  BatchCtl *ctl = nullptr, *h_ctl = nullptr;
  GainCtl *gctl = nullptr, *h_gctl = nullptr;
  // captured launch sequence
  cudaGraphExec_t exec = nullptr;
  cudaGraph_t graph = nullptr;
  cudaStream_t cap_stream = nullptr;  // private stream the sequence is captured on
  std::vector<int32_t> cap_k;
  int32_t cap_A = 0, cap_lanes = 0, cap_grid_min_n = 0, cap_lazy_ctas = 0;
  uint32_t cap_flags = 0;
  std::vector<int32_t> h_picks;
  std::vector<long long> h_pgain, h_far;
  int32_t *h_picks_pinned = nullptr;
  long long *h_far_pinned = nullptr;
  int32_t *h_k_pinned = nullptr, *h_bstart_pinned = nullptr, *h_order_pinned = nullptr;  // sources of the captured copies
};

static void batch_release(gc_batch *b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
  void *dev[] = {b->rp, b->ci, b->gid, b->off, b->ng, b->iota, b->dS, b->mx, b->stamp, b->q0, b->q1, b->goff, b->st1,
                 b->ub, b->key, b->f0, b->ws, b->packed, b->fa, b->farness, b->bestf, b->lc, b->act, b->act_n,
                 b->kk, b->bstart, b->picks, b->pgain, b->seeds, b->ctl, b->gctl, b->slist,
                 b->scount, b->tstart, b->rpf, b->cif, b->c3, b->gx, b->teams, b->gsel, b->dS1, b->g3, b->clog, b->wsel, b->wgain, b->depth,
                 b->order, b->cls};
  for (void *p : dev)
    if (p) cudaFree(p);
  if (b->h_ctl) cudaFreeHost(b->h_ctl);
  if (b->h_gctl) cudaFreeHost(b->h_gctl);
  if (b->h_picks_pinned) cudaFreeHost(b->h_picks_pinned);
  if (b->h_far_pinned) cudaFreeHost(b->h_far_pinned);
  if (b->h_k_pinned) cudaFreeHost(b->h_k_pinned);
  if (b->h_bstart_pinned) cudaFreeHost(b->h_bstart_pinned);
  if (b->h_order_pinned) cudaFreeHost(b->h_order_pinned);
  delete b;
}

template <typename T>
static bool balloc(T **p, size_t count) {
  if (count == 0) count = 1;
  if (cudaMalloc((void **)p, count * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return false;
  }
  return true;
}

// The lazy rounds' plan: sorts the graphs by estimated time (longest first)
// and returns the CTAs of a team: the power of two with about the shortest list
// schedule.  `ctas` > 0 asks for that size.  The estimate of a round in
// microseconds is fitted to team sizes 1 to 76: a step's barriers, selection and
// dependent loads do not shrink with the team, its edges and the bound refreshes
// do.  Lazy rounds in ms at 1, 4, 8, 16, 38 CTAs: 24 graphs of 10^4 to 5 x 10^5
// vertices 173, 48, 26, 14, 18; 24 of 10^4 to 3 x 10^4: 13.8, 4.8, 3.3, 4.8,
// 7.6; 256 of 10^4 to 5 x 10^5 (1, 4, 8, 16): 408, 150, 121, 125.
static int plan_teams(const gc_batch *b, const int32_t *ks, std::vector<int32_t> &order, int32_t ctas) {
  auto est = [&](int32_t g, int s) {
    const double e = (double)b->h_nnz[g];
    return (double)(ks[g] - 2) * (60.0 + (0.1 * std::sqrt(e) + 6e-4 * e) / s);
  };
  std::sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
    const double a = est(x, 1), c = est(y, 1);
    return a > c || (a == c && x < y);
  });
  const int G = b->lazy_ctas;
  if (ctas > 0) return std::min<int>(ctas, G);
  std::vector<double> end;  // of the whole schedule, for teams of 1, 2, 4, ...
  for (int s = 1; s <= G; s *= 2) {
    // list scheduling in that order: the next graph goes to the team that is free first
    std::priority_queue<double, std::vector<double>, std::greater<double>> load(
        std::greater<double>(), std::vector<double>((size_t)(G / s), 0.0));
    double t = 0;
    for (int32_t g : order) {
      const double e = load.top() + est(g, s);
      load.pop();
      load.push(e);
      t = std::max(t, e);
    }
    end.push_back(t);
  }
  // the smallest team within 5% of the best: a larger one's barriers cost more than the
  // estimate knows (one graph of 60 vertices, k = 20: 0.46 ms on one CTA, 0.55 on 128)
  const double limit = 1.05 * *std::min_element(end.begin(), end.end());
  int s = 0;
  while (end[s] > limit) ++s;
  return 1 << s;
}

// The union CSR of `count` graphs.  Host arrays (nnzs == nullptr: the entry
// counts are read from row_ptrs[g][ns[g]]), or device arrays of existing
// handles (nnzs given; the handles were checked when they were loaded).  The
// copies use cudaMemcpyDefault, which takes either kind of pointer.
static int batch_load_impl(int32_t count, const int32_t *const *row_ptrs, const int32_t *const *col_idxs,
                           const int32_t *ns, const int64_t *nnzs, void *stream, gc_batch **out) {
  if (!out || count < 1 || !row_ptrs || !col_idxs || !ns) {
    set_error("bad argument to gc_batch_load");
    return GC_EINVAL;
  }
  *out = nullptr;
  gc_batch *b = new gc_batch();
  b->count = count;
  b->stream = (cudaStream_t)stream;
  b->h_off.resize(count + 1);
  b->h_n.assign(ns, ns + count);
  std::vector<int64_t> eoff(count + 1);
  int64_t N = 0, E = 0;
  b->h_nnz.resize(count);
  for (int32_t g = 0; g < count; ++g) {
    const int64_t e = nnzs ? nnzs[g] : (ns[g] >= 1 && row_ptrs[g] ? row_ptrs[g][ns[g]] : -1);
    if (ns[g] < 1 || !row_ptrs[g] || e < 0 || (!nnzs && row_ptrs[g][0] != 0) || (e > 0 && !col_idxs[g])) {
      batch_release(b);
      set_error("gc_batch_load: graph " + std::to_string(g) + " is malformed");
      return GC_EINVAL;
    }
    b->h_off[g] = (int32_t)N;
    eoff[g] = E;
    b->h_nnz[g] = e;
    N += ns[g];
    E += e;
    b->max_n = std::max(b->max_n, ns[g]);
    if (N >= INT32_MAX || E >= INT32_MAX) {
      batch_release(b);
      set_error("gc_batch_load: the union exceeds int32 CSR limits");
      return GC_ERANGE;
    }
  }
  b->h_off[count] = (int32_t)N;
  eoff[count] = E;
  b->N = (int32_t)N;
  b->nnz = E;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&b->num_sms, cudaDevAttrMultiProcessorCount, dev);
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_solve, kBatchThreads, 0) != cudaSuccess || occ < 1) {
    batch_release(b);
    set_error("gc_batch_load: the batch kernel cannot be resident");
    return GC_ECUDA;
  }
  b->ctas = std::min(kMaxGridCtas, occ * b->num_sms);
  if (cudaFuncSetAttribute(k_batch_lazy<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLazyListSmem) !=
          cudaSuccess ||
      cudaFuncSetAttribute(k_batch_lazy<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLazyListSmem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_lazy<1>, kBatchThreads, kLazyListSmem) !=
          cudaSuccess ||
      occ < 1 ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_check, kBatchThreads, 0) != cudaSuccess || occ < 1) {
    batch_release(b);
    set_error("gc_batch_load: the batch kernels cannot be resident");
    return GC_ECUDA;
  }
  b->lazy_ctas = std::min(b->ctas, b->num_sms);
  const size_t Nn = (size_t)N;
  bool ok = balloc(&b->rp, Nn + 1) && balloc(&b->ci, (size_t)E) && balloc(&b->gid, Nn) &&
            balloc(&b->off, (size_t)count + 1) && balloc(&b->ng, (size_t)count) && balloc(&b->iota, Nn) &&
            balloc(&b->dS, Nn) && balloc(&b->mx, Nn) && balloc(&b->stamp, Nn) && balloc(&b->q0, Nn) &&
            balloc(&b->q1, Nn) && balloc(&b->goff, Nn + 1) && balloc(&b->st1, Nn) && balloc(&b->ub, Nn) && balloc(&b->key, Nn) &&
            balloc(&b->f0, Nn) && balloc(&b->packed, (size_t)count) && balloc(&b->fa, (size_t)count) &&
            balloc(&b->farness, (size_t)count) && balloc(&b->bestf, (size_t)count) &&
            balloc(&b->lc, (size_t)count) && balloc(&b->act_n, (size_t)count) &&
            balloc(&b->kk, (size_t)count) && balloc(&b->bstart, (size_t)count + 1) && balloc(&b->ctl, 1) &&
            balloc(&b->slist, Nn) && balloc(&b->scount, (size_t)count) && balloc(&b->tstart, 2 * ((size_t)count + 1)) &&
            balloc(&b->rpf, Nn + 1) && balloc(&b->cif, std::max<size_t>(1, (size_t)E)) && balloc(&b->c3, Nn) &&
            balloc(&b->dS1, Nn) && balloc(&b->g3, 2 * (size_t)count) &&
            balloc(&b->gx, 3 * Nn) && balloc(&b->clog, 2 * Nn) && balloc(&b->teams, (size_t)b->ctas + 1) &&
            balloc(&b->gsel, (size_t)b->ctas + 1) && balloc(&b->wsel, (size_t)b->ctas * kLanes) &&
            balloc(&b->wgain, (size_t)b->ctas * kLanes) && balloc(&b->depth, (size_t)count) &&
            balloc(&b->order, (size_t)count) && balloc(&b->cls, 2 * (size_t)count) &&
            balloc(&b->gctl, 1) && cudaMallocHost((void **)&b->h_ctl, sizeof(BatchCtl)) == cudaSuccess &&
            cudaMallocHost((void **)&b->h_gctl, sizeof(GainCtl)) == cudaSuccess;
  int64_t *d_eoff = nullptr;
  ok = ok && balloc(&d_eoff, (size_t)count + 1);
  // one workspace per CTA, sized for the largest graph
  b->ws_stride = gain_ws_stride(b->max_n);
  ok = ok && balloc(&b->ws, b->ws_stride * (size_t)b->ctas);
  if (!ok) {
    cudaFree(d_eoff);
    batch_release(b);
    set_error("gc_batch_load: device allocation failed");
    return GC_ENOMEM;
  }
  cudaStream_t st = b->stream;
  bool cp = true;
  for (int32_t g = 0; g < count; ++g) {
    cp = cp && cudaMemcpyAsync(b->rp + b->h_off[g], row_ptrs[g], (size_t)ns[g] * sizeof(int32_t),
                               cudaMemcpyDefault, st) == cudaSuccess;
    const int64_t e = eoff[g + 1] - eoff[g];
    if (e) cp = cp && cudaMemcpyAsync(b->ci + eoff[g], col_idxs[g], (size_t)e * sizeof(int32_t),
                                      cudaMemcpyDefault, st) == cudaSuccess;
  }
  const int32_t last = (int32_t)E;
  cp = cp && cudaMemcpyAsync(b->rp + N, &last, sizeof(int32_t), cudaMemcpyHostToDevice, st) == cudaSuccess &&
       cudaMemcpyAsync(b->off, b->h_off.data(), ((size_t)count + 1) * sizeof(int32_t), cudaMemcpyHostToDevice,
                       st) == cudaSuccess &&
       cudaMemcpyAsync(b->ng, ns, (size_t)count * sizeof(int32_t), cudaMemcpyHostToDevice, st) == cudaSuccess &&
       cudaMemcpyAsync(d_eoff, eoff.data(), ((size_t)count + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, st) ==
           cudaSuccess &&
       cudaMemsetAsync(b->ws, 0, b->ws_stride * (size_t)b->ctas, st) == cudaSuccess;
  if (cp) {
    k_union_fix<<<b->num_sms * 8, 256, 0, st>>>(b->rp, b->ci, b->gid, b->off, d_eoff, count, (int32_t)N, E);
    k_iota<<<b->num_sms * 8, 256, 0, st>>>(b->iota, (int32_t)N);
    cp = cudaGetLastError() == cudaSuccess && simple_rows(b->rp, b->ci, (int32_t)N, E, b->num_sms, st,
                                                          reinterpret_cast<unsigned long long *>(b->g3), &b->simple) == GC_OK;
  }
  cudaFree(d_eoff);
  if (!cp) {
    batch_release(b);
    set_error("gc_batch_load: copy to the device failed");
    return GC_ECUDA;
  }
  *out = b;
  return GC_OK;
}

extern "C" {

int gc_batch_load(int32_t count, const int32_t *const *row_ptrs, const int32_t *const *col_idxs, const int32_t *ns,
                  uint32_t flags, void *stream, gc_batch **out) {
  (void)flags;
  return batch_load_impl(count, row_ptrs, col_idxs, ns, nullptr, stream, out);
}

int gc_batch_free(gc_batch *b) {
  if (b) {
    cudaStreamSynchronize(b->stream);
    batch_release(b);
  }
  return GC_OK;
}

int64_t gc_batch_vertices(const gc_batch *b) { return b ? b->N : -1; }

int gc_batch_greedy(gc_batch *b, const int32_t *ks, const gc_opts *opts_in, int32_t *groups, int64_t *farness,
                    gc_stats *stats) {
  if (!b || !ks || !groups || !farness) {
    set_error("bad argument to gc_batch_greedy");
    return GC_EINVAL;
  }
  gc_opts opts;
  if (opts_in) opts = *opts_in;
  else gc_opts_default(&opts);
  int32_t kmax = 1;
  int64_t ksum = 0;
  for (int32_t g = 0; g < b->count; ++g) {
    if (ks[g] < 1 || ks[g] > b->h_n[g]) {
      set_error("gc_batch_greedy: k of graph " + std::to_string(g) + " outside [1, n]");
      return GC_EINVAL;
    }
    kmax = std::max(kmax, ks[g]);
    ksum += ks[g];
  }
  const int32_t A = opts.active_target > 0 ? opts.active_target : 1024;
  const int32_t lanes1 = (opts.step_lanes > 0 && opts.step_lanes <= kLanes) ? opts.step_lanes : kLanes;
  const bool capture = (opts.flags & GC_OPT_CAPTURE) != 0;
  auto t0 = std::chrono::steady_clock::now();
  cudaStream_t st = b->stream;
  // (re)size per-call buffers; a resize, or a failed one, invalidates a captured sequence
  const int64_t need_seeds = std::max<int64_t>(b->count, ksum);
  if (kmax > b->kcap || need_seeds > b->seeds_cap || A > b->act_cap) b->cap_k.clear();
  const auto dev = [](size_t count) { return [count](auto *&p) { return balloc(&p, count); }; };
  const auto dev_free = [](void *p) { cudaFree(p); };
  const auto pin = [](size_t count) {
    return [count](auto *&p) { return cudaMallocHost((void **)&p, count * sizeof(*p)) == cudaSuccess; };
  };
  const auto pin_free = [](void *p) { cudaFreeHost(p); };
  const size_t graphs = (size_t)b->count;
  if (!grow_buffers(b->kcap, kmax, dev(graphs * kmax), dev_free, b->picks, b->pgain) ||
      !grow_buffers(b->seeds_cap, need_seeds, dev((size_t)need_seeds), dev_free, b->seeds) ||
      !grow_buffers(b->act_cap, A, dev(graphs * A), dev_free, b->act)) {
    set_error("gc_batch_greedy: allocation failed");
    return GC_ENOMEM;
  }
  if (!grow_buffers(b->h_kcap, kmax, pin(graphs * kmax), pin_free, b->h_picks_pinned) ||
      !alloc_missing(pin(graphs + 1), pin_free, b->h_far_pinned, b->h_k_pinned, b->h_bstart_pinned, b->h_order_pinned)) {
    cudaGetLastError();
    set_error("gc_batch_greedy: pinned allocation failed");
    return GC_ENOMEM;
  }
  std::vector<int32_t> bstart(b->count + 1, 0);
  for (int32_t g = 0; g < b->count; ++g) bstart[g + 1] = bstart[g] + (b->h_n[g] + lanes1 - 1) / lanes1;
  const bool same = b->exec && b->cap_k == std::vector<int32_t>(ks, ks + b->count) && b->cap_A == A && b->cap_grid_min_n == opts.batch_grid_min_n && b->cap_flags == opts.flags &&
                    b->cap_lanes == lanes1 && b->cap_lazy_ctas == opts.lazy_ctas;
  BatchArgs a;
  a.rp = b->rp;
  a.ci = b->ci;
  a.N = b->N;
  a.count = b->count;
  a.gid = b->gid;
  a.off = b->off;
  a.ng = b->ng;
  a.kk = b->kk;
  a.iota = b->iota;
  a.bstart = b->bstart;
  a.lanes1 = lanes1;
  a.max_n = b->max_n;
  a.dS = b->dS;
  a.mx = b->mx;
  a.stamp = b->stamp;
  a.q0 = b->q0;
  a.q1 = b->q1;
  a.goff = b->goff;
  a.st1 = b->st1;
  a.rpf = b->rpf;
  a.cif = b->cif;
  a.c3 = b->c3;
  a.dS1 = b->dS1;
  a.teams = b->teams;
  a.gsel = b->gsel;
  a.gx = b->gx;
  a.clog = b->clog;
  a.wsel = b->wsel;
  a.wgain = b->wgain;
  a.depth = b->depth;
  a.order = b->order;
  a.cls = b->cls;
  a.bounded = (opts.flags & GC_OPT_NO_ROUND1_BOUND) ? 0 : 1;
  a.g3 = b->g3;
  a.simple = b->simple;
  a.team_entries = kTeamEntries;
  a.far = b->max_n >= kFarMinN;
  a.grid_min_n = opts.batch_grid_min_n == 0 ? kBatchGridMinN
                 : (opts.batch_grid_min_n < 0 ? INT32_MAX : opts.batch_grid_min_n);
  // the lazy rounds' plan: the graphs left to teams, longest first, and the
  // size of a team
  std::vector<int32_t> order;
  for (int32_t g = 0; g < b->count; ++g)
    if (ks[g] > 2 && b->h_n[g] < a.grid_min_n) order.push_back(g);
  a.order_n = (int32_t)order.size();
  a.team_size = plan_teams(b, ks, order, opts.lazy_ctas);
  a.list_cap = kLanes;
  while (a.list_cap < A && a.list_cap < kCta0SelectMax) a.list_cap *= 2;
  const size_t list_smem = (size_t)a.list_cap * 21;
  // two CTAs per SM for many small graphs (all of them: big ones need the registers)
  int lazy_ctas = b->lazy_ctas;
  const void *lazy_fn = (const void *)k_batch_lazy<1>;
  if (a.team_size == 1 && a.order_n > lazy_ctas && a.order_n == b->count &&
      *std::max_element(b->h_nnz.begin(), b->h_nnz.end()) < kTeamEntries) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_lazy<2>, kBatchThreads, list_smem) ==
            cudaSuccess && occ >= 2) {
      lazy_ctas = std::min(b->ctas, 2 * b->num_sms);
      lazy_fn = (const void *)k_batch_lazy<2>;
    }
  }
  a.ub = b->ub;
  a.key = b->key;
  a.f0 = b->f0;
  a.ws = b->ws;
  a.ws_stride = b->ws_stride;
  a.packed = b->packed;
  a.fa = b->fa;
  a.farness = b->farness;
  a.bestf = b->bestf;
  a.lc = b->lc;
  a.act = b->act;
  a.act_n = b->act_n;
  a.A = A;
  a.kmax = kmax;
  a.picks = b->picks;
  a.pgain = b->pgain;
  a.seeds = b->seeds;
  a.slist = b->slist;
  a.scount = b->scount;
  a.tstart = b->tstart;
  a.ctl = b->ctl;
  a.gctl = b->gctl;
  a.tns = opts.timeout_us > 0 ? (unsigned long long)opts.timeout_us * 1000ull
                              : (unsigned long long)((opts.timeout_ms > 0 ? opts.timeout_ms : 10000) * 1000000LL);
  auto enqueue = [&](cudaStream_t st) -> cudaError_t {
    cudaError_t e;
    if ((e = cudaMemcpyAsync(b->kk, b->h_k_pinned, (size_t)b->count * sizeof(int32_t), cudaMemcpyHostToDevice, st)))
      return e;
    if ((e = cudaMemcpyAsync(b->bstart, b->h_bstart_pinned, bstart.size() * sizeof(int32_t), cudaMemcpyHostToDevice,
                             st)))
      return e;
    if ((e = cudaMemsetAsync(b->packed, 0xff, (size_t)b->count * sizeof(unsigned long long), st))) return e;
    if ((e = cudaMemsetAsync(b->fa, 0, (size_t)b->count * sizeof(long long), st))) return e;
    if ((e = cudaMemsetAsync(b->farness, 0, (size_t)b->count * sizeof(long long), st))) return e;
    if ((e = cudaMemsetAsync(b->lc, 0, (size_t)b->count * sizeof(LazyCtl), st))) return e;
    if ((e = cudaMemsetAsync(b->ctl, 0, sizeof(BatchCtl), st))) return e;
    if ((e = cudaMemsetAsync(b->gctl, 0, sizeof(GainCtl), st))) return e;
    if ((e = cudaMemcpyAsync(b->order, b->h_order_pinned, (size_t)b->count * sizeof(int32_t), cudaMemcpyHostToDevice,
                             st)))
      return e;
    if ((e = cudaMemsetAsync(b->teams, 0, (1 + (size_t)b->ctas) * sizeof(TeamCtl), st))) return e;
    if ((e = cudaMemsetAsync(b->gsel, 0, (1 + (size_t)(lazy_ctas / a.team_size)) * sizeof(GridSelScratch), st)))
      return e;
    if ((e = cudaMemsetAsync(b->cls, 0, 2 * (size_t)b->count * sizeof(unsigned long long), st))) return e;
    if ((e = cudaMemsetAsync(b->depth, 0, (size_t)b->count * sizeof(int32_t), st))) return e;
    void *args[] = {(void *)&a};
    if ((e = cudaLaunchCooperativeKernel((const void *)k_batch_solve, dim3(b->ctas), dim3(kBatchThreads), args, 0,
                                         st)))
      return e;
    if (kmax > 2 &&
        (e = cudaLaunchCooperativeKernel(lazy_fn, dim3(lazy_ctas), dim3(kBatchThreads), args, list_smem, st)))
      return e;
    if ((e = cudaLaunchCooperativeKernel((const void *)k_batch_check, dim3(b->ctas), dim3(kBatchThreads), args, 0,
                                         st)))
      return e;
    if ((e = cudaMemcpyAsync(b->h_picks_pinned, b->picks, (size_t)b->count * kmax * sizeof(int32_t),
                             cudaMemcpyDeviceToHost, st)))
      return e;
    if ((e = cudaMemcpyAsync(b->h_far_pinned, b->farness, (size_t)b->count * sizeof(long long),
                             cudaMemcpyDeviceToHost, st)))
      return e;
    if ((e = cudaMemcpyAsync(b->h_ctl, b->ctl, sizeof(BatchCtl), cudaMemcpyDeviceToHost, st))) return e;
    return cudaMemcpyAsync(b->h_gctl, b->gctl, sizeof(GainCtl), cudaMemcpyDeviceToHost, st);
  };
  bool used_graph = false;
  if (!(capture && same)) {  // a replay reads the pinned buffers it was captured from (same contents)
    cudaStreamSynchronize(st);  // no earlier copy may still read them
    b->cap_k.clear();           // an earlier captured sequence reads the same buffers: record it again
    memcpy(b->h_k_pinned, ks, (size_t)b->count * sizeof(int32_t));
    memcpy(b->h_bstart_pinned, bstart.data(), bstart.size() * sizeof(int32_t));
    std::copy(order.begin(), order.end(), b->h_order_pinned);
  }
  if (capture && same) {
    if (cudaGraphLaunch(b->exec, st) != cudaSuccess) return cuda_fail(cudaGetLastError(), "cudaGraphLaunch");
    used_graph = true;
  } else if (capture) {
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      cudaGraphDestroy(b->graph);
      b->exec = nullptr;
      b->graph = nullptr;
    }
    b->cap_k.assign(ks, ks + b->count);
    b->cap_A = A;
    b->cap_lanes = lanes1;
    b->cap_grid_min_n = opts.batch_grid_min_n;
    b->cap_lazy_ctas = opts.lazy_ctas;
    b->cap_flags = opts.flags;
    // capture on a private non-blocking stream (the legacy default stream
    // cannot be captured); the graph is then launched on the caller's stream
    cudaError_t e = cudaSuccess;
    if (!b->cap_stream) e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      e = enqueue(b->cap_stream);
      cudaGraph_t graph = nullptr;
      const cudaError_t e2 = cudaStreamEndCapture(b->cap_stream, &graph);
      if (e == cudaSuccess) e = e2;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, graph, 0);
      b->graph = graph;
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      if (b->exec) cudaGraphExecDestroy(b->exec);
      if (b->graph) cudaGraphDestroy(b->graph);
      b->exec = nullptr;
      b->graph = nullptr;
      return cuda_fail(e, "capture of the batched solve");
    }
    if (cudaGraphLaunch(b->exec, st) != cudaSuccess) return cuda_fail(cudaGetLastError(), "cudaGraphLaunch");
    used_graph = true;
  } else {
    const cudaError_t e = enqueue(st);
    if (e != cudaSuccess) return cuda_fail(e, "batched solve launch");
  }
  GC_CUDA(cudaStreamSynchronize(st));
  if (b->h_ctl->err) {
    cudaMemsetAsync(b->ws, 0, b->ws_stride * (size_t)b->ctas, st);
    cudaStreamSynchronize(st);
    const int e = b->h_ctl->err;
    set_error(e == GC_ETIMEOUT ? "device-side wait timed out" : e == GC_EDISCONNECTED ? "a graph is disconnected"
              : e == GC_ERANGE ? "a gain exceeds the batched solver's 31-bit key"
                               : "device-side check failed (phase " + std::to_string(b->h_ctl->dbg[0]) + ", graph " +
                                     std::to_string(b->h_ctl->dbg[1]) + ": expected " +
                                     std::to_string(b->h_ctl->dbg[2]) + ", found " +
                                     std::to_string(b->h_ctl->dbg[3]) + ")");
    return e;
  }
  int64_t pos = 0;
  for (int32_t g = 0; g < b->count; ++g) {
    for (int32_t r = 0; r < ks[g]; ++r) groups[pos + r] = b->h_picks_pinned[(size_t)g * kmax + r];
    for (int32_t r = 0; r < ks[g]; ++r) groups[pos + r] -= b->h_off[g];  // local ids
    pos += ks[g];
    farness[g] = b->h_far_pinned[g];
  }
  if (stats) {
    memset(stats, 0, sizeof(*stats));
    stats->rounds = ksum;
    stats->steps = b->h_ctl->iterations;
    stats->batches = (int64_t)b->h_gctl->batches;
    stats->edges_scalar = (int64_t)b->h_gctl->edges_scalar;
    stats->edges_union = (int64_t)b->h_gctl->edges_union;
    stats->levels = (int64_t)b->h_gctl->levels;
    stats->frontier = (int64_t)b->h_gctl->frontier;
    stats->pushes = (int64_t)b->h_gctl->pushes;
    stats->lanes = (int64_t)b->h_gctl->lanes;
    stats->kernel_launches = kmax > 2 ? 3 : 2;
    stats->graph_replay = used_graph ? 1 : 0;
    // phases of the solve (CTA 0's clock): rounds 0, 1, the lazy rounds, the check
    const unsigned long long *ph = b->h_ctl->ns_ph;
    stats->ms_round0 = ph[0] * 1e-6;
    stats->ms_round1 = (ph[1] - ph[0]) * 1e-6;
    stats->ms_lazy_kernel = ph[2] > ph[1] ? (ph[2] - ph[1]) * 1e-6 : 0.0;  // the lazy rounds of every graph (P6)
    stats->ms_lazy_select = b->h_ctl->ns_lazy[0] * 1e-6;  // their phases, summed over graphs
    stats->ms_lazy_gain = b->h_ctl->ns_lazy[1] * 1e-6;
    stats->ms_lazy_update = b->h_ctl->ns_lazy[2] * 1e-6;
    stats->ms_gain_kernel = (ph[5] - ph[4]) * 1e-6;  // round-1 gains of every graph (P4)
    stats->ms_total = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  }
  return GC_OK;
}

// gc_greedy_batch: the batched solve over graphs already loaded as handles.
// Their device CSRs are gathered into one union (device-to-device copies), the
// union is solved by gc_batch_greedy, and each group is handed back through its
// own output pointer.
int gc_greedy_batch(gc_graph *const *gs, const int32_t *ks, int32_t count, const gc_opts *opts,
                    int32_t *const *out_groups, int64_t *out_farness, gc_stats *stats) {
  if (!gs || !ks || count < 1 || !out_groups || !out_farness) {
    set_error("bad argument to gc_greedy_batch");
    return GC_EINVAL;
  }
  std::vector<const int32_t *> rps(count), cis(count);
  std::vector<int32_t> ns(count);
  std::vector<int64_t> nnz(count);
  int64_t ksum = 0;
  for (int32_t g = 0; g < count; ++g) {
    if (!gs[g] || !out_groups[g] || gs[g]->device != gs[0]->device) {
      set_error("gc_greedy_batch: graph " + std::to_string(g) +
                " is NULL, has no output array, or lives on another device");
      return GC_EINVAL;
    }
    rps[g] = gs[g]->rp;
    cis[g] = gs[g]->ci;
    ns[g] = gs[g]->n;
    nnz[g] = gs[g]->nnz;
    ksum += ks[g] > 0 ? ks[g] : 0;
  }
  // the handles' own streams may still be writing their CSRs (adopted arrays)
  for (int32_t g = 0; g < count; ++g)
    if (cudaStreamSynchronize(gs[g]->stream) != cudaSuccess) {
      set_error("gc_greedy_batch: a handle's stream failed");
      return GC_ECUDA;
    }
  gc_batch *b = nullptr;
  int rc = batch_load_impl(count, rps.data(), cis.data(), ns.data(), nnz.data(), gs[0]->stream, &b);
  if (rc != GC_OK) return rc;
  std::vector<int32_t> flat((size_t)std::max<int64_t>(1, ksum));
  rc = gc_batch_greedy(b, ks, opts, flat.data(), out_farness, stats);
  gc_batch_free(b);
  if (rc != GC_OK) return rc;
  size_t pos = 0;
  for (int32_t g = 0; g < count; ++g) {
    memcpy(out_groups[g], flat.data() + pos, (size_t)ks[g] * sizeof(int32_t));
    pos += (size_t)ks[g];
  }
  return GC_OK;
}

}  // extern "C"
