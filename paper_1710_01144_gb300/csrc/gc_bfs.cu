// Grid-wide BFS kernels of libgc: the distance-to-group array d_S
// (Algorithm 2: SSSP from s0, then d_S <- min(d_S, d(s, .)) after each pick,
// done as a pruned SSSP per Sec. 4.1), group farness (Sec. 2), the round-0
// lower bound, and CSR validation.
#include <cooperative_groups.h>
#include <limits.h>

#include <algorithm>

#include "gc_device.cuh"
#include "gc_grid.cuh"
#include "gc_internal.cuh"

namespace gc {

__global__ void k_fill_i32(int32_t *p, int32_t v, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}
__global__ void k_fill_i64(long long *p, long long v, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

// BFS over the whole grid (cooperative, one launch for all levels).
//
// fresh: dist <- the distances from the seeds, with their sum and the number of
// unreached vertices.  Not fresh: dist <- min(dist, distance from the seeds),
// expanding only where a label drops (the pruned SSSP of Sec. 4.1 that turns d_S
// into min(d_S, d(s, .))); ctl->decrease collects sum(old - new) over the
// relabelled vertices with a finite old label, the farness decrease Delta(s | S).
// With c3 (pruned adjacency) levels >= 1 scan only the first c3[u] entries.
//
// Three ways to take a level, chosen by every CTA alike from the frontier's size:
// - spread (top-down): every CTA takes an equal slice of the frontier's adjacency
//   entries; a claimed vertex takes its slot in the next list and its range there
//   with one packed atomicAdd (entries << 32 | adjacency entries), so no pass runs
//   between levels.
// - local: a frontier of at most kBfsLocal entries is expanded by CTA 0 alone,
//   level after level until it grows past that, while the others wait at one grid
//   barrier.  A level then costs a CTA's dependent loads (2 us) without the grid
//   barrier and the list's trip through L2: deep graphs have nothing but such levels.
//   After kBfsLocalLevels of them all CTAs meet, so that no wait grows with the depth
//   of the graph (the time limit is each wait's, and a path of millions of vertices
//   takes seconds).
// - bottom-up (fresh only): when the frontier holds more entries than an eighth of
//   those left, every unreached vertex looks in its own row for a neighbour at the
//   frontier's distance and stops at the first: on R-MAT graphs the frontier at
//   distance 1 holds most of the edges, and nearly every vertex finds one in its
//   first few entries.  No list is kept; going back to top-down (a small frontier
//   with vertices still unreached) collects it in one pass over dist.
//
// Measured (farness of a group of 100, R-MAT scale 20, 31.4M entries): 630 -> 154
// us; the BFS of R-MAT scale 24 9.7 -> about 4 ms; gains with 3 to 100 seeds on road-
// like graphs of 574 to 48,301 vertices 1.2 to 2.6 times faster, among them those
// with short distances, where a larger kBfsLocal (4096) lost (64 x 64, 100 seeds:
// 243 against 171 us, 216 before).
constexpr int kBfsLocal = 768;   // adjacency entries (three per thread)
constexpr int kBfsLocalLevels = 256;  // half a millisecond
constexpr int kBfsStage = 256;    // frontier entries staged at a time (= threads)

__global__ void __launch_bounds__(kBfsThreads) k_bfs(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                                     int32_t n, int32_t *dist, const int32_t *seeds, int32_t n_seeds,
                                                     int32_t *q0, int32_t *q1, int32_t *st0, int32_t *st1, BfsCtl *ctl,
                                                     SelCtl *sctl, unsigned long long tns,
                                                     const int32_t *__restrict__ c3, int32_t fresh) {
  __shared__ unsigned long long s_red[32];
  __shared__ int s_go[kBfsStage + 1];
  __shared__ int s_rs[kBfsStage];
  __shared__ int s_x0;
  __shared__ unsigned long long s_pk;
  const int tid = threadIdx.x, lane = tid & 31, T = kBfsThreads, G = gridDim.x, b = blockIdx.x;
  unsigned long long dec = 0, rel = 0;
  const long long nnz = __ldg(rp + n);
  if (fresh) {
    for (int i = b * T + tid; i < n; i += G * T) dist[i] = kInf;
    if (!grid_sync(&ctl->bar, &ctl->err, tns)) return;
  }
  // queue w for level lev through the counter *cnt (whole warp)
  auto enqueue = [&](bool q, int w, int lev, int deg, unsigned long long *cnt) {
    const unsigned qm = __ballot_sync(0xffffffffu, q);
    if (!qm) return;
    if (!q) deg = 0;
    int incl = deg;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int sum = __shfl_sync(0xffffffffu, incl, 31);
    const int leader = __ffs(qm) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(cnt, ((unsigned long long)__popc(qm) << 32) | (unsigned long long)sum);
    base = __shfl_sync(0xffffffffu, base, leader);
    if (q) {
      const int slot = (int)(base >> 32) + __popc(qm & ((1u << lane) - 1u));
      ((lev & 1) ? q1 : q0)[slot] = w;
      ((lev & 1) ? st1 : st0)[slot] = (int)(base & 0xffffffffull) + incl - deg;
    }
  };
  // entries [es, ee) of the level-L frontier (F vertices, E entries)
  auto expand = [&](int L, int F, long long E, long long es, long long ee, unsigned long long *cnt) {
    const int32_t *qc = (L & 1) ? q1 : q0;
    const int32_t *qs = (L & 1) ? st1 : st0;
    const int nl = L + 1;
    if (es >= ee) return;
    if (tid < 32) {
      const int x = warp_find_start(qs, F, es);
      if (tid == 0) s_x0 = x;
    }
    cta_sync();
    int x = s_x0;
    while (x < F) {
      const int xi = x + tid, cntx = min(T, F - x);
      if (xi < F) {
        s_go[tid] = qs[xi];
        s_rs[tid] = __ldg(rp + qc[xi]);
      }
      if (tid == 0) s_go[cntx] = (x + cntx < F) ? qs[x + cntx] : (int)E;
      cta_sync();
      const long long a0 = max((long long)s_go[0], es), a1 = min((long long)s_go[cntx], ee);
      for (long long e0 = a0 + (tid & ~31); e0 < a1; e0 += T) {  // warp-uniform trip count
        const long long e = e0 + lane;
        bool q = false;
        int w = 0, lw = 0;
        if (e < a1) {
          int l = 0, h = cntx - 1;  // staged entry holding e (every entry's range is non-empty)
          while (l < h) {
            const int mid = (l + h + 1) >> 1;
            if (s_go[mid] <= e) l = mid;
            else h = mid - 1;
          }
          w = __ldg(ci + s_rs[l] + (int)(e - s_go[l]));
          const int dcur = __ldcg(dist + w);
          lw = row_len(rp, c3, w, nl);  // with the label: no load waits in enqueue
          if (nl < dcur) {
            const int old = atomicMin(&dist[w], nl);
            if (old > nl) {
              q = true;
              if (old < kInf) dec += (unsigned long long)(old - nl);
              ++rel;
            }
          }
        }
        enqueue(q, w, nl, lw, cnt);
      }
      const int done_end = s_go[cntx];
      cta_sync();  // the staged arrays are reused
      if ((long long)done_end >= ee) break;
      x += cntx;
    }
  };

  for (int base = b * T; base < n_seeds; base += G * T) {  // warp-uniform trip count
    const int i = base + tid;
    bool q = false;
    int s = 0;
    if (i < n_seeds) {
      s = ((volatile const int32_t *)seeds)[i];
      if (s < 0 || s >= n) {
        atomicExch(&ctl->err, GC_EINVAL);
      } else {
        const int old = atomicMin(&dist[s], 0);
        if (old > 0) {
          q = true;
          if (old < kInf) dec += (unsigned long long)old;
          ++rel;
        }
      }
    }
    enqueue(q, s, 0, q ? row_len(rp, c3, s, 0) : 0, &ctl->pk[0]);
  }
  bool ok = grid_sync(&ctl->bar, &ctl->err, tns);
  int L = 0;
  long long seen = 0, esum = 0, sum = 0;  // vertices and entries of the levels so far, their distances (every CTA alike)
  bool up = false, after_local = false;
  for (; ok;) {
    unsigned long long pk = *(volatile unsigned long long *)(after_local ? &ctl->local_pk : &ctl->pk[L % 3]);
    after_local = false;
    int F = (int)(pk >> 32);
    long long E = (long long)(pk & 0xffffffffull);
    if (F == 0) break;
    if (b == 0 && tid == 0) ctl->pk[(L + 2) % 3] = 0;  // the frontier after next (read two levels ago)
    const bool was_up = up;
    if (fresh) up = up ? F >= n / 64 : E > (nnz - esum) / 8 && E > nnz / 32;
    if (was_up && !up) {  // collect the frontier's list
      if (seen + F == n) {
        seen += F;
        sum += (long long)L * F;
        ++L;
        break;
      }
      for (int base = b * T; base < n; base += G * T) {
        const int v = base + tid;
        const bool q = v < n && __ldcg(dist + v) == L;
        enqueue(q, v, L, q ? row_len(rp, c3, v, L) : 0, &ctl->list);
      }
      ok = grid_sync(&ctl->bar, &ctl->err, tns);
      if (!ok) break;
      if (b == 0 && tid == 0) ctl->list = 0;
    }
    if (!up && E <= kBfsLocal) {
      // ---- local: CTA 0 alone, while the frontier stays small ----
      ok = grid_sync(&ctl->bar, &ctl->err, tns);  // every CTA has read this level's counters
      if (!ok) break;
      if (b == 0) {
        int l = L;
        for (;;) {
          if (tid == 0) s_pk = 0;
          cta_sync();
          seen += F;
          esum += E;
          sum += (long long)l * F;
          expand(l, F, E, 0, E, &s_pk);
          cta_sync();
          pk = s_pk;
          cta_sync();
          ++l;
          F = (int)(pk >> 32);
          E = (long long)(pk & 0xffffffffull);
          if (F == 0 || E > kBfsLocal || l - L >= kBfsLocalLevels) break;
        }
        if (tid == 0) {
          ctl->local_pk = pk;
          ctl->pk[0] = ctl->pk[1] = ctl->pk[2] = 0;
          ctl->lev = l;
          ctl->seen = seen;
          ctl->esum = esum;
          ctl->sum = sum;
        }
      }
      ok = grid_sync(&ctl->bar, &ctl->err, tns);
      L = *(volatile int32_t *)&ctl->lev;
      seen = *(volatile long long *)&ctl->seen;
      esum = *(volatile long long *)&ctl->esum;
      sum = *(volatile long long *)&ctl->sum;
      after_local = true;
      continue;
    }
    seen += F;
    esum += E;
    sum += (long long)L * F;
    if (fresh && seen == n) {  // every vertex has its distance: the last frontier claims nothing
      ++L;
      break;
    }
    if (!up) {
      expand(L, F, E, E * b / G, E * (b + 1) / G, &ctl->pk[(L + 1) % 3]);
    } else {
      // ---- bottom-up: unreached vertices look for a neighbour at distance L ----
      unsigned long long found = 0;  // vertices << 32 | their entries
      for (int base = (b * T + tid) & ~31; base < n; base += G * T) {
        const int v = base + lane;
        int r0 = 0, r1 = 0;
        if (v < n && __ldcg(dist + v) == kInf) {
          r0 = __ldg(rp + v);
          r1 = __ldg(rp + v + 1);
        }
        bool hit = false;
        const int e1 = min(r1, r0 + 32);
        for (int e = r0; e < e1 && !hit; e += 4) {
          int w[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) w[k] = e + k < e1 ? __ldg(ci + e + k) : -1;
#pragma unroll
          for (int k = 0; k < 4; ++k) hit |= w[k] >= 0 && dist[w[k]] == L;
        }
        // the rest of a long row by the whole warp
        for (unsigned m = __ballot_sync(0xffffffffu, !hit && r1 - r0 > 32); m; m &= m - 1) {
          const int t = __ffs(m) - 1;
          const int x0 = __shfl_sync(0xffffffffu, r0, t) + 32, x1 = __shfl_sync(0xffffffffu, r1, t);
          bool any = false;
          for (int e = x0; e < x1 && !any; e += 32)
            any = __any_sync(0xffffffffu, e + lane < x1 && dist[__ldg(ci + e + lane)] == L);
          if (lane == t) hit = any;
        }
        if (hit) {
          dist[v] = L + 1;
          found += (1ull << 32) | (unsigned long long)(r1 - r0);
          ++rel;
        }
      }
      found = block_sum(found, s_red);
      if (tid == 0 && found) atomicAdd(&ctl->pk[(L + 1) % 3], found);
    }
    ok = grid_sync(&ctl->bar, &ctl->err, tns);
    ++L;
  }
  dec = block_sum(dec, s_red);
  rel = block_sum(rel, s_red);
  if (tid == 0) {
    if (dec) atomicAdd(&ctl->decrease, dec);
    if (rel) atomicAdd(&ctl->relabelled, rel);
    if (b == 0 && ok) {
      ctl->levels = L;
      if (fresh && sctl) {
        sctl->sum = sum;
        sctl->count = (long long)n - seen;
      }
    }
  }
}

// sum(dist) and the count of unreached vertices; the last CTA to finish folds
// the per-CTA partials (ticket pattern, no waiting) into ctl->sum / ctl->count.
__global__ void __launch_bounds__(kRedThreads) k_sum_dist(const int32_t *__restrict__ dist, int32_t n,
                                                         long long *partial, SelCtl *ctl) {
  __shared__ long long sh[32];
  __shared__ bool last;
  long long s = 0, c = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int d = dist[i];
    if (d >= kInf) ++c;
    else s += d;
  }
  s = block_sum(s, sh);
  c = block_sum(c, sh);
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = s;
    partial[2 * blockIdx.x + 1] = c;
    __threadfence();
    last = atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1;
  }
  cta_sync();
  if (!last) return;
  __threadfence();
  s = 0;
  c = 0;
  for (int b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    s += ((volatile long long *)partial)[2 * b];
    c += ((volatile long long *)partial)[2 * b + 1];
  }
  s = block_sum(s, sh);
  c = block_sum(c, sh);
  if (threadIdx.x == 0) {
    ctl->sum = s;
    ctl->count = c;
    ctl->ticket = 0;
  }
}

// Row-wise kernels leave rows of more than kHeavyRow entries (hubs) to a CTA in a
// companion kernel, so that no warp walks a hub's row alone while the rest of the
// grid has finished.  The companions walk the list of long rows built once per
// graph (k_heavy_rows).

// heavy[0..*nh) = the rows with more than kHeavyRow entries (any order)
__global__ void __launch_bounds__(kRedThreads) k_heavy_rows(const int32_t *__restrict__ rp, int32_t n,
                                                            int32_t *heavy, int32_t *nh) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (rp[v + 1] - rp[v] > kHeavyRow) heavy[atomicAdd(nh, 1)] = v;
}

// Round 0, a tighter second level: how many vertices of small degree can be
// within distance 2 of v at most.  For a degree class C, every u in C at
// distance 1 or 2 from v is a neighbour of v or of some w in N(v), so
//   #{u in C : 1 <= d(v, u) <= 2} <= near_C(v) = cnt_C(v) + sum_{w in N(v)} cnt_C(w),
// cnt_C(w) = neighbours of w in C, and at least
//   far_C(v) = |C| - [v in C] - near_C(v)
// members of C are at distance >= 3.  The sum over C of max(0, far_C) then caps
// c2 of the degree bound: c2 <= n - 1 - deg(v) - far.  Two classes, degrees
// {1, 2} and {3 .. kFarDeg}: near_C counts a vertex once per common neighbour,
// so it is exact for degree 1 and loose only by the degree beyond.
//
// Why.  The plain degree bound gives up (c2 = everything) on vertices next to
// hubs, and each of those then needs a search: 55,455 on R-MAT scale 24, whose
// bit-parallel searches took 154 ms.  Half of such a graph has degree <= 4 and
// over 90% of that half is three or more hops from any one vertex, which the
// counts show without a search: all 55,454 other survivors fall.  Only the rows
// of degree <= kFarDeg and the survivors' own rows are read (R-MAT scale 24:
// about 3% and 45% of the entries).  Bound by the random 8-byte gathers and
// atomics on the count array (71 MB at scale 24, it stays in L2).  Measured:
// R-MAT scale 24, k = 50: round 0 166.5 -> 14.7 ms, the call 215.6 -> 64.2 ms;
// top-100 closeness at scale 18: 17.4 -> 3.60 ms (12,848 survivors -> 57); one
// survivor batch at scale 20: 9.88 -> 9.84 ms.  They run on shallow graphs with more
// than 64 survivors: up to 64 are one batch, which costs no more than the counts.

// cnt[w] += the classes of w's neighbours of degree 1 .. kFarDeg (low half
// {1, 2}, high half the rest), one thread per such neighbour's row;
// total[0..1] = members per class.  cnt and total start at zero.
__global__ void __launch_bounds__(kRedThreads) k_far_counts(const int32_t *__restrict__ rp,
                                                            const int32_t *__restrict__ ci, int32_t n,
                                                            unsigned long long *cnt, unsigned long long *total) {
  __shared__ long long sh[32];
  long long t0 = 0, t1 = 0;
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
    const int beg = rp[u], end = rp[u + 1];
    const unsigned long long c = far_class(end - beg);
    if (!c) continue;
    t0 += c == 1ull;
    t1 += c != 1ull;
    for (int e = beg; e < end; ++e) atomicAdd(&cnt[ci[e]], c);
  }
  t0 = block_sum(t0, sh);
  t1 = block_sum(t1, sh);
  if (threadIdx.x == 0) {
    if (t0) atomicAdd(&total[0], (unsigned long long)t0);
    if (t1) atomicAdd(&total[1], (unsigned long long)t1);
  }
}

// key[v] from the bound with c2 <= rest - far (never raised: the old bound holds too)
__device__ __forceinline__ void far_key(int v, int deg_i, int32_t n, long long near0, long long near1,
                                        const unsigned long long *total, unsigned long long own,
                                        const long long *two_hop, long long *key) {
  const unsigned long long c = far_class(deg_i);
  const long long deg = deg_i, rest = max(0ll, (long long)n - 1 - deg);
  const long long f0 = (long long)total[0] - (c == 1ull) - near0 - (long long)(own & 0xffffffffull);
  const long long f1 = (long long)total[1] - (c > 1ull) - near1 - (long long)(own >> 32);
  const long long far = min(rest, max(0ll, f0) + max(0ll, f1));
  const long long c2 = min(two_hop[v], rest - far);
  const long long k = -(deg + 2 * c2 + 3 * (rest - c2));
  if (k < key[v]) key[v] = k;
}

// A warp per survivor list[i]; rows longer than kHeavyRow are left to k_far_bound_heavy.
__global__ void __launch_bounds__(kRedThreads) k_far_bound(const int32_t *__restrict__ rp,
                                                           const int32_t *__restrict__ ci, int32_t n,
                                                           const int32_t *__restrict__ list, const int32_t *m_dev,
                                                           const unsigned long long *__restrict__ cnt,
                                                           const unsigned long long *__restrict__ total,
                                                           const long long *__restrict__ two_hop, long long *key) {
  const int lane = threadIdx.x & 31;
  const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  const int m = *m_dev;
  for (int i = gwarp; i < m; i += nwarps) {
    const int v = list[i];
    const int beg = rp[v], end = rp[v + 1];
    if (end - beg > kHeavyRow) continue;
    long long a0 = 0, a1 = 0;
#pragma unroll 4
    for (int e = beg + lane; e < end; e += 32) {
      const unsigned long long x = cnt[ci[e]];
      a0 += (long long)(x & 0xffffffffull);
      a1 += (long long)(x >> 32);
    }
    a0 = warp_sum(a0);
    a1 = warp_sum(a1);
    if (lane == 0) far_key(v, end - beg, n, a0, a1, total, cnt[v], two_hop, key);
  }
}

// The long rows of k_far_bound among the undecided vertices with bound <= the
// selection threshold (key >= tau), a CTA per row.
__global__ void __launch_bounds__(1024) k_far_bound_heavy(const int32_t *__restrict__ rp,
                                                         const int32_t *__restrict__ ci, int32_t n,
                                                         const unsigned long long *__restrict__ cnt,
                                                         const unsigned long long *__restrict__ total,
                                                         const long long *__restrict__ two_hop, long long *key,
                                                         const int32_t *__restrict__ heavy,
                                                         const int32_t *__restrict__ nh, const SelCtl *ctl) {
  __shared__ long long s_red[32];
  __shared__ bool s_go;
  const long long tau = ctl->tau;
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int v = heavy[i];
    cta_sync();
    if (threadIdx.x == 0) s_go = key[v] != LLONG_MIN && key[v] >= tau;
    cta_sync();
    if (!s_go) continue;
    const int beg = rp[v], end = rp[v + 1];
    long long a0 = 0, a1 = 0;
#pragma unroll 4
    for (int e = beg + threadIdx.x; e < end; e += 1024) {
      const unsigned long long x = cnt[ci[e]];
      a0 += (long long)(x & 0xffffffffull);
      a1 += (long long)(x >> 32);
    }
    a0 = block_sum(a0, s_red);
    a1 = block_sum(a1, s_red);
    if (threadIdx.x == 0) far_key(v, end - beg, n, a0, a1, total, cnt[v], two_hop, key);
  }
}

// Pivot lower bound for round 0.  For any vertex p and every w,
// d(v, w) >= |d(p, w) - d(p, v)| (triangle inequality), so with n_l vertices
// at distance l from p,
//   f({v}) >= LB_p(v) = sum_l n_l * |l - d(p, v)|,
// which prefix counts C[x] = sum_{l<x} n_l and prefix sums M[x] = sum_{l<x} l n_l
// give in O(1) per vertex:  x C[x] - M[x] + (M[D+1] - M[x+1]) - x (n - C[x+1]).
// The bound only decides which vertices still need an exact search.
__global__ void __launch_bounds__(kRedThreads) k_level_hist(const int32_t *__restrict__ dist, int32_t n,
                                                            unsigned long long *cnt, int32_t *maxlev) {
  int mloc = 0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const int x = dist[v];
    if (x >= 0 && x < n) {
      atomicAdd(&cnt[x], 1ull);
      mloc = max(mloc, x);
    }
  }
  for (int o = 16; o > 0; o >>= 1) mloc = max(mloc, __shfl_xor_sync(0xffffffffu, mloc, o));
  if ((threadIdx.x & 31) == 0) atomicMax(maxlev, mloc);
}

// One CTA: cnt[0..D] -> C[0..D+1] (exclusive prefix counts, in place of cnt
// shifted by one) and M[0..D+1]; D = *maxlev.  cnt is cleared for the next use.
__global__ void __launch_bounds__(1024) k_level_prefix(unsigned long long *cnt, const int32_t *maxlev,
                                                       unsigned long long *C, unsigned long long *M) {
  __shared__ unsigned long long s_c[1024], s_m[1024];
  __shared__ unsigned long long carry_c, carry_m;
  const int D = *maxlev;
  if (threadIdx.x == 0) {
    carry_c = 0;
    carry_m = 0;
  }
  cta_sync();
  for (int base = 0; base <= D; base += 1024) {
    const int l = base + threadIdx.x;
    const unsigned long long c = l <= D ? cnt[l] : 0ull;
    s_c[threadIdx.x] = c;
    s_m[threadIdx.x] = c * (unsigned long long)(l <= D ? l : 0);
    cta_sync();
    for (int o = 1; o < 1024; o <<= 1) {  // inclusive Hillis-Steele scan
      unsigned long long a = 0, b = 0;
      if (threadIdx.x >= o) {
        a = s_c[threadIdx.x - o];
        b = s_m[threadIdx.x - o];
      }
      cta_sync();
      s_c[threadIdx.x] += a;
      s_m[threadIdx.x] += b;
      cta_sync();
    }
    if (l <= D) {
      C[l + 1] = carry_c + s_c[threadIdx.x];
      M[l + 1] = carry_m + s_m[threadIdx.x];
      cnt[l] = 0;
    }
    cta_sync();
    if (threadIdx.x == 1023) {
      carry_c += s_c[1023];
      carry_m += s_m[1023];
    }
    cta_sync();
  }
  if (threadIdx.x == 0) {
    C[0] = 0;
    M[0] = 0;
  }
}

// key[v] = -max(LB(v), LB_p(v)) for vertices still undecided (key != INT64_MIN).
__global__ void __launch_bounds__(kRedThreads) k_pivot_bound(const int32_t *__restrict__ dist, int32_t n,
                                                             const unsigned long long *__restrict__ C,
                                                             const unsigned long long *__restrict__ M,
                                                             const int32_t *maxlev, long long *key) {
  const int D = *maxlev;
  const long long Mt = (long long)M[D + 1];
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const long long k0 = key[v];
    const int x = dist[v];
    if (k0 == LLONG_MIN || x < 0 || x > D) continue;
    const long long cx = (long long)C[x], cx1 = (long long)C[x + 1];
    const long long lb = (long long)x * cx - (long long)M[x] + (Mt - (long long)M[x + 1]) - (long long)x * ((long long)n - cx1);
    if (-lb < k0) key[v] = -lb;
  }
}

// CSR validation, part 1: row_ptr monotone within [0, nnz].
__global__ void k_validate_rowptr(const int32_t *__restrict__ rp, int32_t n, int64_t nnz,
                                  SelCtl *ctl) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int a = rp[i], b = rp[i + 1];
    if (a < 0 || b < a || (int64_t)b > nnz) atomicExch(&ctl->err, GC_EINVAL);
  }
}

// CSR validation, part 2 (only after part 1 passed): ids in range, no
// self-loop, strictly increasing rows, and every edge (u, w) mirrored by
// (w, u) (binary search in the sorted row of w).
__global__ void k_validate_rows(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                int32_t n, SelCtl *ctl) {
  const int lane = threadIdx.x & 31;
  const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int u = gwarp; u < n; u += nwarps) {
    const int beg = rp[u], end = rp[u + 1];
    for (int e = beg + lane; e < end; e += 32) {
      const int w = ci[e];
      bool bad = (w < 0 || w >= n || w == u || (e > beg && ci[e - 1] >= w));
      if (!bad) {
        int lo = rp[w], hi = rp[w + 1];
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (ci[mid] < u) lo = mid + 1;
          else hi = mid;
        }
        bad = !(lo < rp[w + 1] && ci[lo] == u);
      }
      if (bad) atomicExch(&ctl->err, GC_EINVAL);
    }
  }
}

// ------------------------------------------------------------- launchers ----
static int grid_for(int64_t count, int threads, int cap) {
  int64_t b = (count + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (int)b;
}

int launch_fill_i32(gc_graph *g, int32_t *p, int32_t v, int64_t count) {
  if (count <= 0) return GC_OK;
  ++g->launches;
  k_fill_i32<<<grid_for(count, 256, g->num_sms * 8), 256, 0, g->stream>>>(p, v, count);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}
int launch_fill_i64(gc_graph *g, long long *p, long long v, int64_t count) {
  if (count <= 0) return GC_OK;
  ++g->launches;
  k_fill_i64<<<grid_for(count, 256, g->num_sms * 8), 256, 0, g->stream>>>(p, v, count);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_bfs(gc_graph *g, int32_t *dist, const int32_t *seeds, int32_t n_seeds, int64_t timeout_ns, bool fresh,
               bool pruned) {
  GC_CUDA(cudaMemsetAsync(g->bctl, 0, sizeof(BfsCtl), g->stream));
  const int32_t *rp = pruned ? g->rpf : g->rp, *ci = pruned ? g->cif : g->ci;
  const int32_t *c3 = pruned ? g->c3 : nullptr;
  int32_t n = g->n, fr = fresh ? 1 : 0;
  int32_t *q0 = g->bq0, *q1 = g->bq1, *st0 = g->goff, *st1 = g->gx;
  BfsCtl *ctl = g->bctl;
  SelCtl *sctl = g->sctl;
  unsigned long long tns = (unsigned long long)timeout_ns;
  void *args[] = {(void *)&rp, (void *)&ci,  (void *)&n,   (void *)&dist, (void *)&seeds, (void *)&n_seeds, (void *)&q0,
                  (void *)&q1, (void *)&st0, (void *)&st1, (void *)&ctl,  (void *)&sctl,  (void *)&tns,     (void *)&c3,
                  (void *)&fr};
  static_assert(kBfsThreads == 256, "bfs_grid counts CTAs of 256 threads");
  const int grid = (int)std::min<int64_t>(std::min(g->bfs_ctas, kMaxGridCtas), bfs_grid(n, g->nnz));
  ++g->launches;
  GC_CUDA(cudaLaunchCooperativeKernel((const void *)k_bfs, dim3(grid), dim3(kBfsThreads), args, 0, g->stream));
  return GC_OK;
}

int bfs_kernel_occupancy(int *blocks_per_sm) {
  GC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_bfs, kBfsThreads, 0));
  return GC_OK;
}

int launch_sum_dist(gc_graph *g, const int32_t *dist) {
  ++g->launches;
  k_sum_dist<<<g->red_blocks, kRedThreads, 0, g->stream>>>(dist, g->n, g->partial, g->sctl);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_far_bound(gc_graph *g) {
  // counts in lgain (8 bytes per vertex, free until the survivors are searched)
  unsigned long long *cnt = (unsigned long long *)g->lgain, *total = (unsigned long long *)g->partial;
  GC_CUDA(cudaMemsetAsync(cnt, 0, (size_t)g->n * sizeof(unsigned long long), g->stream));
  GC_CUDA(cudaMemsetAsync(total, 0, 2 * sizeof(unsigned long long), g->stream));
  g->launches += 3;
  k_far_counts<<<grid_for(g->n, kRedThreads, g->num_sms * 8), kRedThreads, 0, g->stream>>>(g->rp, g->ci, g->n, cnt,
                                                                                           total);
  k_far_bound<<<g->num_sms * 8, kRedThreads, 0, g->stream>>>(g->rp, g->ci, g->n, g->list, &g->sctl->n_sel, cnt,
                                                             total, g->two_hop, g->key);
  k_far_bound_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rp, g->ci, g->n, cnt, total, g->two_hop, g->key,
                                                            g->heavy, g->n_heavy, g->sctl);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_pivot_bound(gc_graph *g) {
  g->launches += 3;
  GC_CUDA(cudaMemsetAsync(g->lev_max, 0, sizeof(int32_t), g->stream));
  k_level_hist<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->dS, g->n, g->lev_cnt, g->lev_max);
  k_level_prefix<<<1, 1024, 0, g->stream>>>(g->lev_cnt, g->lev_max, g->lev_C, g->lev_M);
  k_pivot_bound<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->dS, g->n, g->lev_C, g->lev_M, g->lev_max,
                                                              g->key);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// Round-0 work estimate: the sum over list[0..m) of two_hop[v] (sum over the
// neighbours of v of deg - 1), the adjacency entries a search from v scans to
// reach distance 2.  Accumulated into *out (zeroed by the caller).
__global__ void k_sum_two_hop(const int32_t *__restrict__ list, const int32_t *m_dev,
                              const long long *__restrict__ two_hop, unsigned long long *out) {
  __shared__ long long sh[32];
  const int m = *m_dev;
  long long s = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) s += two_hop[list[i]];
  s = block_sum(s, sh);
  if (threadIdx.x == 0 && s) atomicAdd(out, (unsigned long long)s);
}

int launch_sum_two_hop(gc_graph *g, unsigned long long *out) {
  ++g->launches;
  GC_CUDA(cudaMemsetAsync(out, 0, sizeof(unsigned long long), g->stream));
  k_sum_two_hop<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->list, &g->sctl->n_sel, g->two_hop, out);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// ub[v] = -1 for members (d_S[v] = 0), +infinity for every other vertex: the
// starting point of k_bound_refresh when no earlier bound exists.
__global__ void k_init_ub(const int32_t *__restrict__ dS, int32_t n, long long *ub) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    ub[v] = dS[v] == 0 ? -1ll : LLONG_MAX;
}

int launch_init_ub(gc_graph *g) {
  ++g->launches;
  k_init_ub<<<grid_for(g->n, 256, g->num_sms * 8), 256, 0, g->stream>>>(g->dS, g->n, g->ub);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_heavy_rows(gc_graph *g) {
  ++g->launches;
  GC_CUDA(cudaMemsetAsync(g->n_heavy, 0, sizeof(int32_t), g->stream));
  k_heavy_rows<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->rp, g->n, g->heavy, g->n_heavy);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_validate(gc_graph *g) {
  GC_CUDA(cudaMemsetAsync(&g->sctl->err, 0, sizeof(int32_t), g->stream));
  ++g->launches;
  k_validate_rowptr<<<grid_for(g->n, 256, g->num_sms * 8), 256, 0, g->stream>>>(g->rp, g->n, g->nnz,
                                                                                 g->sctl);
  GC_CUDA(cudaGetLastError());
  GC_CUDA(cudaMemcpyAsync(&g->h_sctl->err, &g->sctl->err, sizeof(int32_t), cudaMemcpyDeviceToHost,
                          g->stream));
  GC_CUDA(cudaStreamSynchronize(g->stream));
  if (g->h_sctl->err) return GC_EINVAL;
  ++g->launches;
  k_validate_rows<<<grid_for((int64_t)g->n * 32, 256, g->num_sms * 8), 256, 0, g->stream>>>(
      g->rp, g->ci, g->n, g->sctl);
  GC_CUDA(cudaGetLastError());
  GC_CUDA(cudaMemcpyAsync(&g->h_sctl->err, &g->sctl->err, sizeof(int32_t), cudaMemcpyDeviceToHost,
                          g->stream));
  GC_CUDA(cudaStreamSynchronize(g->stream));
  return g->h_sctl->err ? GC_EINVAL : GC_OK;
}

}  // namespace gc
