// Passes of the single-graph path over whole adjacencies: round-0 bounds, the
// neighbour maxima and the pruned adjacency after round 0, the two-hop bounds of
// round 1 and their refresh.  Each reads every entry of a CSR once and gathers one
// value a neighbour.
//
// What bounds them: a warp a row spends three dependent loads (row pointers, entry,
// value) on rows that mostly fill a few lanes, so the latency of those chains, not
// the 4 bytes an entry, was the time (R-MAT scale 24, 520M entries in 8.9M rows: 1.5
// to 2.4 ms a pass where the entries alone take 0.3); beyond that, the gathers' 32-
// byte sectors out of L2.  So
// - a warp takes a window of up to 32 consecutive rows, whose entries are one
//   contiguous range: 128 entries and their values are in flight at a time, and the
//   lane that owns a row picks its part of each 32 by the row's bounds (counts and
//   maxima from ballots, sums from a scan);
// - what is gathered is small: distances as 4-bit classes (packed first, one pass
//   over n), the distance-3 test as one bit, degrees and the two terms of the
//   two-hop bounds as one word;
// - rows of more than kHeavyRow entries are left to a CTA each, as elsewhere.
// Windows shrink with n so that every warp of the grid has at least two: one row a
// warp below about 40,000 rows, 32 above 600,000.
// R-MAT scale 24, k 50, long rows included, before and now in ms: keys 3.2, 2.6;
// maxima, sizes and fill 10.4, 4.9; round-1 bounds 3.1, 1.5; a refresh 5.2, 2.2; the
// whole call 53.1, 35.2.  BA n = 2,000 is unchanged (1.05 ms, one row a warp).
#include <limits.h>

#include <algorithm>

#include "gc_device.cuh"
#include "gc_internal.cuh"

namespace gc {

constexpr int kRowsCtasPerSm = 8;
constexpr int kScanTile = 4096;

// Bits [lo, hi) of a 32-entry chunk.
__device__ __forceinline__ unsigned chunk_mask(int lo, int hi) {
  return lo < hi ? (0xffffffffu >> (32 - (hi - lo))) << lo : 0u;
}

// Windows of wn rows over the whole grid.  begin(v, own): a window's start (lane v
// - v0 owns row v); gather(w): the value of neighbour w; fold(w, x, lo, hi): 32
// entries, one a lane (w < 0 past the range), of which [lo, hi) are the owned row's;
// done(v, own): own rows that are not long.  All lanes call all of them together.
template <class Begin, class Gather, class Fold, class Done>
__device__ __forceinline__ void row_windows(const int32_t *__restrict__ rp, const int32_t *__restrict__ rows,
                                            const int32_t *__restrict__ ci, int32_t n, int wn, Begin begin,
                                            Gather gather, Fold fold, Done done) {
  const int lane = threadIdx.x & 31;
  const long long gwarp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long v0 = gwarp * wn; v0 < n; v0 += nwarps * wn) {
    const bool own = lane < wn && v0 + lane < n;
    const int v = own ? (int)v0 + lane : 0;
    int a = INT_MAX, b = INT_MAX;
    bool heavy = false;
    if (own) {
      a = rows[v];
      b = rows[v + 1];
      heavy = rp[v + 1] - rp[v] > kHeavyRow;
    }
    begin(v, own, a, b);
    const unsigned hm = __ballot_sync(0xffffffffu, heavy);
    const int cnt = __popc(__ballot_sync(0xffffffffu, own));
    for (int s = 0; s < cnt;) {  // runs of rows between long ones
      const unsigned rest = hm >> s;
      const int t = rest ? min(cnt, s + __ffs(rest) - 1) : cnt;
      if (t > s) {
        const unsigned E1 = (unsigned)__shfl_sync(0xffffffffu, b, t - 1);
        for (unsigned c0 = (unsigned)__shfl_sync(0xffffffffu, a, s); c0 < E1; c0 += 128) {
          int w[4], x[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const unsigned e = c0 + 32 * k + lane;
            w[k] = e < E1 ? __ldg(ci + e) : -1;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) x[k] = w[k] >= 0 ? gather(w[k]) : 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int c = (int)(c0 + 32 * k);
            if ((unsigned)c >= E1) break;
            fold(w[k], x[k], min(max(a - c, 0), 32), min(max(b - c, 0), 32));
          }
        }
      }
      s = t + 1;
    }
    done(v, own && !heavy);
  }
}

// Sum of the values x of the entries [lo, hi) of a 32-entry chunk, 0 <= x.
__device__ __forceinline__ long long chunk_sum(int x, int lo, int hi) {
  const int lane = threadIdx.x & 31;
  if (!__any_sync(0xffffffffu, x >= 1 << 26)) {
    int p = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p += y;
    }
    const int h = __shfl_sync(0xffffffffu, p, (hi - 1) & 31), l = __shfl_sync(0xffffffffu, p, (lo - 1) & 31);
    return lo < hi ? (long long)(h - (lo > 0 ? l : 0)) : 0;
  }
  long long p = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, p, o);
    if (lane >= o) p += y;
  }
  const long long h = __shfl_sync(0xffffffffu, p, (hi - 1) & 31), l = __shfl_sync(0xffffffffu, p, (lo - 1) & 31);
  return lo < hi ? h - (lo > 0 ? l : 0) : 0;
}

// Rows a window.
static int window_rows(int32_t n, int num_sms) {
  const int64_t warps = (int64_t)num_sms * kRowsCtasPerSm * (kRedThreads / 32);
  int wn = 1;
  while (wn < 32 && n >= 4 * warps * wn) wn *= 2;
  return wn;
}

static int rows_grid(const gc_graph *g, int wn) {
  const int64_t warps = ((int64_t)g->n + wn - 1) / wn;
  return (int)std::max<int64_t>(
      1, std::min<int64_t>((warps + kRedThreads / 32 - 1) / (kRedThreads / 32), (int64_t)g->num_sms * kRowsCtasPerSm));
}

// Distances as classes min(d, 15), 8 a word, in vertex order.
__device__ __forceinline__ int dist_class(const uint32_t *__restrict__ cls, int w) {
  return (int)(__ldg(cls + (w >> 3)) >> (4 * (w & 7))) & 15;
}

__global__ void __launch_bounds__(kRedThreads) k_classes(const int32_t *__restrict__ dS, int32_t n, uint32_t *cls) {
  const int words = (int)(((long long)n + 7) >> 3);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
    const long long v0 = (long long)i * 8;
    uint32_t c = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (v0 + j < n) c |= (uint32_t)min(dS[v0 + j], 15) << (4 * j);
    cls[i] = c;
  }
}

// Bit v of far: d_S[v] >= 3.
__global__ void __launch_bounds__(kRedThreads) k_far_bits(const int32_t *__restrict__ dS, int32_t n, uint32_t *far) {
  const long long lanes = ((long long)n + 31) & ~31ll;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < lanes;
       i += (long long)gridDim.x * blockDim.x) {
    const unsigned m = __ballot_sync(0xffffffffu, i < n && dS[i] >= 3);
    if ((threadIdx.x & 31) == 0) far[i >> 5] = m;
  }
}

__global__ void __launch_bounds__(kRedThreads) k_degrees(const int32_t *__restrict__ rp, int32_t n, int32_t *deg1) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    deg1[v] = rp[v + 1] - rp[v] - 1;
}

// ---------------------------------------------------------------- load --
// Whether the grid-wide gain batches may count a candidate's neighbours at d_S = 2
// without marking them visited (gc_grid.cuh): only if no row holds an entry twice
// or its own vertex.  Rows that are not increasing are taken for such rows: their
// results are the same, by the claims that every other neighbour takes.
// Two passes in one kernel: the entries that are not above the one before them, but
// for the first of each row, and each row's search for its own vertex.  Bound by one
// read of the adjacency: R-MAT scale 24 (520M entries), device arrays, loads in 5.1 ms,
// 4.5 without.
__global__ void __launch_bounds__(kRedThreads)
    k_simple_rows(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n, long long nnz,
                  unsigned long long *bad) {
  __shared__ long long sh[32];
  const long long at = blockIdx.x * (long long)blockDim.x + threadIdx.x, all = (long long)gridDim.x * blockDim.x;
  long long c = 0;
#pragma unroll 4
  for (long long e = at + 1; e < nnz; e += all) c += __ldg(ci + e) <= __ldg(ci + e - 1);
  for (long long v = at; v < n; v += all) {
    const long long beg = rp[v], end = rp[v + 1];
    if (beg < 0 || beg >= end || end > nnz) continue;  // (an empty row, or row pointers that nobody checked)
    if (beg > 0) c -= __ldg(ci + beg) <= __ldg(ci + beg - 1);
    long long lo = beg, hi = end;
    while (lo < hi) {
      const long long mid = (lo + hi) >> 1;
      if (__ldg(ci + mid) < (int)v) lo = mid + 1;
      else hi = mid;
    }
    if (lo < end && __ldg(ci + lo) == (int)v) c += 1ll << 32;
  }
  c = block_sum(c, sh);
  if (threadIdx.x == 0 && c) atomicAdd(bad, (unsigned long long)c);
}

int simple_rows(const int32_t *rp, const int32_t *ci, int32_t n, int64_t nnz, int num_sms, cudaStream_t stream,
                unsigned long long *bad, int32_t *simple) {
  unsigned long long h = 0;
  GC_CUDA(cudaMemsetAsync(bad, 0, sizeof(*bad), stream));
  k_simple_rows<<<num_sms * kRowsCtasPerSm, kRedThreads, 0, stream>>>(rp, ci, n, (long long)nnz, bad);
  GC_CUDA(cudaGetLastError());
  GC_CUDA(cudaMemcpyAsync(&h, bad, sizeof(h), cudaMemcpyDeviceToHost, stream));
  GC_CUDA(cudaStreamSynchronize(stream));
  *simple = h == 0;
  return GC_OK;
}

// ------------------------------------------------------------- round 0 --
// Lower bound on f({v}) (the BFScut idea of Sec. 3.1 with a degree bound for
// the second level): the deg(v) neighbours sit at distance 1; at most c2 =
// min(sum_{w in N(v)} (deg(w) - 1), n - 1 - deg(v)) vertices sit at distance 2
// (every neighbour has v among its own neighbours); everything else is at
// least 3 away.  key[v] = -(deg + 2 c2 + 3 (n - 1 - deg - c2)); deg1[w] =
// deg(w) - 1.
__device__ __forceinline__ void write_key(int v, long long deg, long long x, int32_t n, long long *key,
                                          long long *two_hop) {
  const long long rest = max((long long)n - 1 - deg, 0ll);
  const long long c2 = min(x, rest);
  key[v] = -(deg + 2 * c2 + 3 * (rest - c2));
  two_hop[v] = x;
}

__global__ void __launch_bounds__(kRedThreads)
    k_round0_keys(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n, int wn,
                  const int32_t *__restrict__ deg1, long long *key, long long *two_hop) {
  long long x, deg;
  row_windows(
      rp, rp, ci, n, wn, [&](int, bool, int a, int b) { x = 0; deg = b - a; }, [&](int w) { return __ldg(deg1 + w); },
      [&](int, int d, int lo, int hi) { x += chunk_sum(d, lo, hi); },
      [&](int v, bool own) {
        if (own) write_key(v, deg, x, n, key, two_hop);
      });
}

__global__ void __launch_bounds__(1024)
    k_round0_keys_heavy(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n,
                        const int32_t *__restrict__ deg1, long long *key, long long *two_hop,
                        const int32_t *__restrict__ heavy, const int32_t *__restrict__ nh) {
  __shared__ long long s_red[32];
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int v = heavy[i], beg = rp[v], end = rp[v + 1];
    long long x = 0;
#pragma unroll 4
    for (int e = beg + threadIdx.x; e < end; e += 1024) x += (long long)__ldg(deg1 + ci[e]);
    x = block_sum(x, s_red);
    if (threadIdx.x == 0) write_key(v, end - beg, x, n, key, two_hop);
  }
}

int launch_round0_keys(gc_graph *g) {
  const int wn = window_rows(g->n, g->num_sms);
  g->launches += 3;
  k_degrees<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->rp, g->n, g->bq0);
  k_round0_keys<<<rows_grid(g, wn), kRedThreads, 0, g->stream>>>(g->rp, g->ci, g->n, wn, g->bq0, g->key, g->two_hop);
  k_round0_keys_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rp, g->ci, g->n, g->bq0, g->key, g->two_hop,
                                                              g->heavy, g->n_heavy);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// ------------------------------------------- after round 0: d_S = d(s0, .) --
// One pass for all that the later rounds take from the full adjacency:
// - mx[u] = max over neighbours w of d_S[w].  d_S only decreases as the group
//   grows, so the value stays an upper bound; a frontier vertex u at level L can
//   claim a neighbour only if that neighbour's d_S exceeds L+1, so mx[u] <= L+1
//   means expanding u is useless (the pruning test of Sec. 4.1 applied one level
//   ahead);
// - the pruned adjacency's sizes.  A neighbour w of u can be claimed (or
//   relabelled) at level L+1 only if d_S[w] > L+1 >= 1, and d_S only decreases,
//   so entries with d_S[w] <= 1 at the time of the build are useless in every
//   later round.  The pruned row of u keeps the cnt2[u] entries with d_S[w] >= 2,
//   the c3[u] with d_S[w] >= 3 first: level 0 scans the whole pruned row, levels
//   >= 1 (where d_S[w] > 2 is needed) only its first c3[u];
// - reach[u] = (d_S[u] - 1)^+ + c3[u], u's part in its neighbours' round-1 bounds.
// Separate passes for mx and the sizes took 5.3 ms on R-MAT scale 24, this one 2.2.
__global__ void __launch_bounds__(kRedThreads)
    k_row_stats(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n, int wn,
                const int32_t *__restrict__ dS, const uint32_t *__restrict__ cls, int32_t *mx, int32_t *cnt2,
                int32_t *c3, int32_t *reach) {
  int a2, a3, m;
  row_windows(
      rp, rp, ci, n, wn, [&](int, bool, int, int) { a2 = a3 = m = 0; }, [&](int w) { return dist_class(cls, w); },
      [&](int w, int c, int lo, int hi) {
        const unsigned row = chunk_mask(lo, hi);
        const unsigned p0 = __ballot_sync(0xffffffffu, c & 1), p1 = __ballot_sync(0xffffffffu, c & 2),
                       p2 = __ballot_sync(0xffffffffu, c & 4), p3 = __ballot_sync(0xffffffffu, c & 8);
        const unsigned ge2 = p1 | p2 | p3, ge3 = (p0 & p1) | p2 | p3;
        a2 += __popc(ge2 & row);
        a3 += __popc(ge3 & row);
        // the largest class of the row's entries, from the top bit down
        unsigned cand = row;
        int q = 0;
        if (cand & p3) cand &= p3, q |= 8;
        if (cand & p2) cand &= p2, q |= 4;
        if (cand & p1) cand &= p1, q |= 2;
        if (cand & p0) q |= 1;
        m = max(m, q);
        unsigned top = p0 & p1 & p2 & p3;  // class 15: the distance itself
        if (top) {
          const int d = c == 15 ? dS[w] : 0;
          for (; top; top &= top - 1) {
            const int k = __ffs(top) - 1, dk = __shfl_sync(0xffffffffu, d, k);
            if ((row >> k) & 1u) m = max(m, dk);
          }
        }
      },
      [&](int v, bool own) {
        if (!own) return;
        mx[v] = m;
        cnt2[v] = a2;
        c3[v] = a3;
        reach[v] = max(dS[v] - 1, 0) + a3;
      });
}

__global__ void __launch_bounds__(1024)
    k_row_stats_heavy(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                      const int32_t *__restrict__ dS, const uint32_t *__restrict__ cls, int32_t *mx, int32_t *cnt2,
                      int32_t *c3, int32_t *reach, const int32_t *__restrict__ heavy,
                      const int32_t *__restrict__ nh) {
  __shared__ long long s_red[32];
  __shared__ int s_m;
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int u = heavy[i], r0 = rp[u], r1 = rp[u + 1];
    if (threadIdx.x == 0) s_m = 0;
    long long a = 0;  // both counts: each below 2^31
    int m = 0;
#pragma unroll 4
    for (int e = r0 + threadIdx.x; e < r1; e += 1024) {
      const int w = ci[e];
      int c = dist_class(cls, w);
      a += (long long)(c >= 2) << 32 | (long long)(c >= 3);
      if (c == 15) c = dS[w];
      m = max(m, c);
    }
    a = block_sum(a, s_red);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_m, m);
    cta_sync();
    if (threadIdx.x == 0) {
      const int a3 = (int)(a & 0xffffffffll);
      mx[u] = s_m;
      cnt2[u] = (int)(a >> 32);
      c3[u] = a3;
      reach[u] = max(dS[u] - 1, 0) + a3;
    }
    cta_sync();
  }
}

int launch_row_stats(gc_graph *g) {
  const int wn = window_rows(g->n, g->num_sms);
  uint32_t *cls = (uint32_t *)g->bq0;
  g->launches += 3;
  k_classes<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->dS, g->n, cls);
  k_row_stats<<<rows_grid(g, wn), kRedThreads, 0, g->stream>>>(g->rp, g->ci, g->n, wn, g->dS, cls, g->mx_buf, g->io_a,
                                                              g->c3, g->c3s);
  k_row_stats_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rp, g->ci, g->dS, cls, g->mx_buf, g->io_a, g->c3,
                                                            g->c3s, g->heavy, g->n_heavy);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// Pruned rows, two cursors each: entries with d_S >= 3 go to the front of the
// row, entries with d_S == 2 after the c3[u] of them, both in CSR order.
__global__ void __launch_bounds__(kRedThreads)
    k_prune_fill(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int32_t n, int wn,
                 const uint32_t *__restrict__ cls, const int32_t *__restrict__ rpf, const int32_t *__restrict__ c3,
                 int32_t *cif) {
  const int lane = threadIdx.x & 31;
  int q3, q2;  // the owned row's cursors
  row_windows(
      rp, rp, ci, n, wn,
      [&](int v, bool own, int, int) {
        q3 = own ? rpf[v] : 0;
        q2 = own ? q3 + c3[v] : 0;
      },
      [&](int w) { return dist_class(cls, w); },
      [&](int w, int c, int lo, int hi) {
        const unsigned m3 = __ballot_sync(0xffffffffu, c >= 3), m2 = __ballot_sync(0xffffffffu, c == 2);
        if (!(m3 | m2)) return;
        // the row of this lane's entry: as many rows end at or before it
        int o = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
          if (__shfl_sync(0xffffffffu, hi, o + step - 1) <= lane) o += step;
        const int st = __shfl_sync(0xffffffffu, lo, o), b3 = __shfl_sync(0xffffffffu, q3, o),
                  b2 = __shfl_sync(0xffffffffu, q2, o);
        const unsigned before = chunk_mask(st, lane);
        if (c >= 3) cif[b3 + __popc(m3 & before)] = w;
        else if (c == 2) cif[b2 + __popc(m2 & before)] = w;
        const unsigned row = chunk_mask(lo, hi);
        q3 += __popc(m3 & row);
        q2 += __popc(m2 & row);
      },
      [](int, bool) {});
}

// The long rows, a CTA each: 4096 entries at a time with one scan for both cursors.
__global__ void __launch_bounds__(1024)
    k_prune_fill_heavy(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                       const uint32_t *__restrict__ cls, const int32_t *__restrict__ rpf,
                       const int32_t *__restrict__ c3, int32_t *cif, const int32_t *__restrict__ heavy,
                       const int32_t *__restrict__ nh) {
  __shared__ int s_scan[33];
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int u = heavy[i];
    const unsigned r1 = (unsigned)rp[u + 1];
    int p3 = rpf[u], p2 = p3 + c3[u];
    for (unsigned e0 = (unsigned)rp[u]; e0 < r1; e0 += 4096) {
      int w[4], c[4], f = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const unsigned e = e0 + 1024 * k + threadIdx.x;
        w[k] = e < r1 ? __ldg(ci + e) : -1;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        c[k] = w[k] >= 0 ? dist_class(cls, w[k]) : 0;
        f += c[k] >= 3 ? 1 : c[k] == 2 ? 1 << 16 : 0;
      }
      int tot;
      const int x = block_excl_scan(f, s_scan, &tot);
      int x3 = p3 + (x & 0xffff), x2 = p2 + (x >> 16);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (c[k] >= 3) cif[x3++] = w[k];
        else if (c[k] == 2) cif[x2++] = w[k];
      }
      p3 += tot & 0xffff;
      p2 += tot >> 16;
    }
  }
}

// Exclusive prefix sum of cnt[0..n) into out[0..n] (out[n] = total), three
// launches: per-tile sums, a one-CTA scan of the tile sums, per-tile scans.
__global__ void __launch_bounds__(1024) k_scan_tiles(const int32_t *__restrict__ cnt, int32_t n,
                                                    long long *tile_sum) {
  __shared__ long long s[32];
  long long a = 0;
  const int base = blockIdx.x * kScanTile;
  for (int i = threadIdx.x; i < kScanTile; i += 1024)
    if (base + i < n) a += cnt[base + i];
  a = block_sum(a, s);
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = a;
}

__global__ void __launch_bounds__(1024) k_scan_tops(long long *tile_sum, int32_t tiles) {
  __shared__ int s_scan[33];
  long long carry = 0;
  for (int base = 0; base < tiles; base += 1024) {
    const int i = base + threadIdx.x;
    const long long v = i < tiles ? tile_sum[i] : 0;
    int tot;
    // tile sums fit int32 here: the CSR has fewer than 2^31 entries
    const int ex = block_excl_scan((int)v, s_scan, &tot);
    if (i < tiles) tile_sum[i] = carry + ex;
    carry += tot;
    cta_sync();
  }
}

__global__ void __launch_bounds__(1024) k_scan_apply(const int32_t *__restrict__ cnt, int32_t n,
                                                    const long long *__restrict__ tile_sum, int32_t *out) {
  __shared__ int s_scan[33];
  const int base = blockIdx.x * kScanTile;
  long long carry = tile_sum[blockIdx.x];
  for (int off = 0; off < kScanTile; off += 1024) {
    const int i = base + off + threadIdx.x;
    const int v = i < n ? cnt[i] : 0;
    int tot;
    const int ex = block_excl_scan(v, s_scan, &tot);
    if (i < n) out[i] = (int32_t)(carry + ex);
    if (i == n - 1) out[n] = (int32_t)(carry + ex + v);
    carry += tot;
    cta_sync();
  }
}

int launch_prune_csr(gc_graph *g) {
  const int n = g->n, wn = window_rows(n, g->num_sms);
  const int tiles = (n + kScanTile - 1) / kScanTile;
  const uint32_t *cls = (const uint32_t *)g->bq0;
  g->launches += 5;
  k_scan_tiles<<<tiles, 1024, 0, g->stream>>>(g->io_a, n, g->lgain);
  k_scan_tops<<<1, 1024, 0, g->stream>>>(g->lgain, tiles);
  k_scan_apply<<<tiles, 1024, 0, g->stream>>>(g->io_a, n, g->lgain, g->rpf);
  k_prune_fill<<<rows_grid(g, wn), kRedThreads, 0, g->stream>>>(g->rp, g->ci, n, wn, cls, g->rpf, g->c3, g->cif);
  k_prune_fill_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rp, g->ci, cls, g->rpf, g->c3, g->cif, g->heavy,
                                                             g->n_heavy);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// -------------------------------------------------------- two-hop bounds --
// Round-1 upper bounds.  With S = {s0} and d_S = d(s0, .), every candidate v
// satisfies
//   Delta(v|S) <= d_S[v] + sum_{w in N(v)} ((d_S[w] - 1)^+ + c3[w]) + G3,
//   G3 = sum_u (d_S[u] - 3)^+,
// because a vertex u at distance 1 from v gains at most d_S[u] - 1; one at
// distance 2 gains at most (d_S[u] - 2)^+ = [d_S[u] >= 3] + (d_S[u] - 3)^+,
// and each such u with d_S[u] >= 3 is a neighbour of some w in N(v), counted
// by c3[w] (neighbours of w with d_S >= 3); farther vertices gain at most
// (d_S[u] - 3)^+; and the (d_S - 3)^+ terms of all of them sum to at most G3.
// A neighbour w with d_S[w] <= 1 adds nothing (its own term is 0 and its
// neighbours have d_S <= 2), so the pruned rows (d_S[w] >= 2) suffice.  The
// bounds replace the +infinity of round 1 (Sec. 4.2 gives none), so the lazy
// rule of round 1 evaluates only the candidates whose bound reaches the best
// exact gain.  ub[v] <- the bound (members of S: -1), stamp[v] <- 0.
__global__ void __launch_bounds__(kRedThreads) k_excess3(const int32_t *__restrict__ dS, int32_t n,
                                                         unsigned long long *g3) {
  __shared__ long long sh[32];
  long long s = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int d = dS[i];
    if (d > 3) s += d - 3;
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0 && s) atomicAdd(g3, (unsigned long long)s);
}

__device__ __forceinline__ void write_bound1(int v, long long s, int dv, long long G3, long long *ub,
                                             int32_t *stamp) {
  ub[v] = dv == 0 ? -1ll : (long long)dv + s + G3;
  stamp[v] = 0;
}

__global__ void __launch_bounds__(kRedThreads)
    k_round1_bound(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif, const int32_t *__restrict__ rp,
                   int32_t n, int wn, const int32_t *__restrict__ dS, const int32_t *__restrict__ reach,
                   const unsigned long long *__restrict__ g3, long long *ub, int32_t *stamp) {
  const long long G3 = (long long)*g3;
  long long s;
  row_windows(
      rp, rpf, cif, n, wn, [&](int, bool, int, int) { s = 0; }, [&](int w) { return __ldg(reach + w); },
      [&](int, int x, int lo, int hi) { s += chunk_sum(x, lo, hi); },
      [&](int v, bool own) {
        if (own) write_bound1(v, s, dS[v], G3, ub, stamp);
      });
}

__device__ __forceinline__ long long heavy_sum(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif,
                                               const int32_t *__restrict__ reach, int v, long long *s_red) {
  long long s = 0;
  const int end = rpf[v + 1];
#pragma unroll 4
  for (int e = rpf[v] + threadIdx.x; e < end; e += 1024) s += (long long)__ldg(reach + cif[e]);
  return block_sum(s, s_red);
}

__global__ void __launch_bounds__(1024)
    k_round1_bound_heavy(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif,
                         const int32_t *__restrict__ dS, const int32_t *__restrict__ reach,
                         const unsigned long long *__restrict__ g3, long long *ub, int32_t *stamp,
                         const int32_t *__restrict__ heavy, const int32_t *__restrict__ nh) {
  __shared__ long long s_red[32];
  const long long G3 = (long long)*g3;
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int v = heavy[i];
    const long long s = heavy_sum(rpf, cif, reach, v, s_red);
    if (threadIdx.x == 0) write_bound1(v, s, dS[v], G3, ub, stamp);
  }
}

int launch_round1_bound(gc_graph *g) {
  const int wn = window_rows(g->n, g->num_sms);
  g->launches += 3;
  GC_CUDA(cudaMemsetAsync(g->g3, 0, sizeof(unsigned long long), g->stream));
  k_excess3<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->dS, g->n, g->g3);
  k_round1_bound<<<rows_grid(g, wn), kRedThreads, 0, g->stream>>>(g->rpf, g->cif, g->rp, g->n, wn, g->dS, g->c3s,
                                                                 g->g3, g->ub, g->stamp);
  k_round1_bound_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rpf, g->cif, g->dS, g->c3s, g->g3, g->ub,
                                                               g->stamp, g->heavy, g->n_heavy);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// Bound refresh for later rounds.  The inequality of the round-1 bounds holds
// for any group S with d_S, c3 and G3 taken for that S, and it tightens as S
// grows.  k_count3 recounts, for the current d_S, the neighbours with d_S >= 3 of
// every vertex (they are all in the pruned rows: d_S only decreases) into
// reach[u]; k_bound_refresh lowers every candidate's bound to the recomputed
// value.  A candidate already evaluated in the current round keeps its exact gain
// (the bound is above it).
__device__ __forceinline__ int far_bit(const uint32_t *__restrict__ far, int w) {
  return (int)(__ldg(far + (w >> 5)) >> (w & 31)) & 1;
}

__global__ void __launch_bounds__(kRedThreads)
    k_count3(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif, const int32_t *__restrict__ rp,
             int32_t n, int wn, const int32_t *__restrict__ dS, const uint32_t *__restrict__ far, int32_t *reach) {
  int a;
  row_windows(
      rp, rpf, cif, n, wn, [&](int, bool, int, int) { a = 0; }, [&](int w) { return far_bit(far, w); },
      [&](int, int x, int lo, int hi) { a += __popc(__ballot_sync(0xffffffffu, x) & chunk_mask(lo, hi)); },
      [&](int v, bool own) {
        if (own) reach[v] = max(dS[v] - 1, 0) + a;
      });
}

__global__ void __launch_bounds__(1024)
    k_count3_heavy(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif, const int32_t *__restrict__ dS,
                   const uint32_t *__restrict__ far, int32_t *reach, const int32_t *__restrict__ heavy,
                   const int32_t *__restrict__ nh) {
  __shared__ int s_red[32];
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int u = heavy[i], end = rpf[u + 1];
    int a = 0;
#pragma unroll 4
    for (int e = rpf[u] + threadIdx.x; e < end; e += 1024) a += far_bit(far, cif[e]);
    a = block_sum(a, s_red);
    if (threadIdx.x == 0) reach[u] = max(dS[u] - 1, 0) + a;
  }
}

// ub[v] < 0 marks members; a bound is never raised.
__device__ __forceinline__ void lower_bound1(int v, long long s, const int32_t *__restrict__ dS, long long G3,
                                             long long *ub) {
  const long long b = (long long)dS[v] + s + G3;
  if (b < ub[v]) ub[v] = b;
}

__global__ void __launch_bounds__(kRedThreads)
    k_bound_refresh(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif, const int32_t *__restrict__ rp,
                    int32_t n, int wn, const int32_t *__restrict__ dS, const int32_t *__restrict__ reach,
                    const unsigned long long *__restrict__ g3, long long *ub) {
  const long long G3 = (long long)*g3;
  long long s;
  row_windows(
      rp, rpf, cif, n, wn, [&](int, bool, int, int) { s = 0; }, [&](int w) { return __ldg(reach + w); },
      [&](int, int x, int lo, int hi) { s += chunk_sum(x, lo, hi); },
      [&](int v, bool own) {
        if (own) lower_bound1(v, s, dS, G3, ub);
      });
}

__global__ void __launch_bounds__(1024)
    k_bound_refresh_heavy(const int32_t *__restrict__ rpf, const int32_t *__restrict__ cif,
                          const int32_t *__restrict__ dS, const int32_t *__restrict__ reach,
                          const unsigned long long *__restrict__ g3, long long *ub, const int32_t *__restrict__ heavy,
                          const int32_t *__restrict__ nh) {
  __shared__ long long s_red[32];
  const long long G3 = (long long)*g3;
  for (int i = blockIdx.x; i < *nh; i += gridDim.x) {
    const int v = heavy[i];
    if (ub[v] < 0) continue;  // block-uniform
    const long long s = heavy_sum(rpf, cif, reach, v, s_red);
    if (threadIdx.x == 0) lower_bound1(v, s, dS, G3, ub);
  }
}

int launch_bound_refresh(gc_graph *g) {
  const int wn = window_rows(g->n, g->num_sms), grid = rows_grid(g, wn);
  uint32_t *far = (uint32_t *)g->bq0;
  g->launches += 6;
  GC_CUDA(cudaMemsetAsync(g->g3, 0, sizeof(unsigned long long), g->stream));
  k_excess3<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->dS, g->n, g->g3);
  k_far_bits<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->dS, g->n, far);
  k_count3<<<grid, kRedThreads, 0, g->stream>>>(g->rpf, g->cif, g->rp, g->n, wn, g->dS, far, g->c3s);
  k_count3_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rpf, g->cif, g->dS, far, g->c3s, g->heavy, g->n_heavy);
  k_bound_refresh<<<grid, kRedThreads, 0, g->stream>>>(g->rpf, g->cif, g->rp, g->n, wn, g->dS, g->c3s, g->g3, g->ub);
  k_bound_refresh_heavy<<<g->num_sms * 2, 1024, 0, g->stream>>>(g->rpf, g->cif, g->dS, g->c3s, g->g3, g->ub,
                                                                g->heavy, g->n_heavy);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

}  // namespace gc
