// Rules that need neither a device nor the CUDA runtime: plain functions, the same
// in kernels, host code and host-only programs.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GC_HD __host__ __device__ __forceinline__
#else
#define GC_HD inline
#endif

namespace gc {

constexpr int32_t kInf = 0x3fffffff;  // "unreached" distance (d + 1 cannot overflow)

// Buckets of the weighted searches (gc_weighted.cu).  A bucket takes the entries
// that lead to less than its end T; T = kInf - 1 is the last one and takes every
// entry.  The end of the bucket after the nearest pending entry mn, `delta` wide:
GC_HD int32_t w_bucket_end(int32_t mn, int32_t delta) { return mn > kInf - 1 - delta ? kInf - 1 : mn + delta; }
// An entry that leads to distance x is in the bucket that ends at T.  The nearest
// pending entry always is in the next bucket, so every bucket makes progress: an
// entry may lead to exactly kInf - 1 (n vertices, weights of (2^30 - 2) / (n - 1)),
// which x < T alone would leave pending for ever.
GC_HD bool w_in_bucket(int32_t x, int32_t T) { return T == kInf - 1 || x < T; }

// Whether round 0 of the weighted greedy searches every vertex in full, in one bucket
// and one wave of CTAs, instead of in buckets with a cut.  Dense rows hold mostly
// entries that no shortest path takes, which buckets never read.  Measured, k = 6, ms
// (in full, in buckets), weights up to 1 and 1000: complete n = 1,000 3.4 and 12.1, 1.3
// and 5.4; n = 300 0.85 and 1.70, 0.78 and 1.42; n = 150 0.69 and 0.99, 0.75 and 0.96;
// random n = 1,000, rows of 182 1.78 and 3.93, 1.35 and 2.22, of 22 1.06 and 1.37, 1.08
// and 1.34; ring n = 1,000, rows of 32 1.47 and 4.0, 1.90 and 2.9; random n = 500, rows
// of 21 0.72 and 0.99, 0.80 and 1.10.
GC_HD bool w_whole_search(int64_t n, int64_t nnz) { return n <= 1024 && (n < 256 || nnz <= 64 * n); }

// Whether the mean distance `sum` / n of a search is long for n vertices: on roads,
// grids and lattices its square is a share of n (a quarter on a square grid), on
// graphs that a search fills in a few levels it is not, whatever tail of a few
// vertices makes them deep.  On the latter one-source searches lose to the 64-lane
// batches, which share rows among sources that reach them at one level, and to the
// degree and two-hop bounds.  Measured, greedy k = 5 (one-source, 64-lane, ms; mean^2
// / n): attachment graph of 100,000 vertices with a path of 40 at one of them 285, 8
// (0.0001); broom of 30,000 leaves 40, 12 (0.0002); recursive tree n = 5,000 5.8, 2.2
// (0.003); 6 attachment graphs of 5,000 in a row 14.0, 13.9 (0.003); tree of 5,000 with
// such a path 2.0, 3.9 (0.006); ring of 30,000 with 2,500 chords 9.5, 18.8 (0.009);
// road-like 40 x 40 1.6, 4.4 (0.25), 200 x 200 14, 138.
GC_HD bool far_apart(int64_t sum, int64_t n) {
  const double mean = (double)sum / (double)n;
  return mean * mean * 200.0 >= (double)n;
}

// CTAs of 256 threads for a BFS over a whole graph: few on small graphs, for cheaper
// barriers, but enough for the entries of the level that holds nearly all of them.  By
// the vertices alone, two a thread, a random graph of 4,000 vertices and 1.6M entries
// had 8 CTAs: farness from one vertex 115 us, 87 with every CTA, 53 with 97 (64
// entries a thread); top-1 closeness there 488, 423, 412 us.
GC_HD int64_t bfs_grid(int64_t n, int64_t nnz) {
  const int64_t v = (n + 511) / 512, e = nnz / 16384;
  return v > e ? (v > 1 ? v : 1) : e;
}

// Gains of many candidates on a large deep graph, after the first of them by one-source
// searches, `lanes` searches of `edges` adjacency entries: whether the 64-lane batches
// take the rest.  Searches that reach much of a graph whose distances are short share
// their rows; with many of them the batches win.  Measured on graphs of short distances
// with a path of 20 or 40, all vertices as candidates (share of the entries a search
// scans; all by one-source searches, by this rule, ms): attachment graph n = 100,000, m
// = 3, groups of 1, 2, 4, 8 (0.32; 195, 86), (0.22; 133, 70), (0.15; 89, 56), (0.03; 21,
// 21); n = 300,000 (0.14; 777, 412), (0.20; 1142, 489), (0.12; 663, 387), (0.03, but
// more for the first ids; 149, 170); random n = 100,000 (0.34; 232, 102), (0.17; 113,
// 67), (0.11; 76, 54), (0.05; 36, 35).  40,000 candidates on the first 79, 44.  50,000
// vertices, all of them: 42 by the 64-lane batches as they were before the one-source
// searches, 35 by these (130 and 195 at 100,000).
constexpr int32_t kLanesHead = 8192, kLanesFrom = 32768, kLanesMinN = 65536;
GC_HD bool lanes_take_rest(uint64_t edges, uint64_t lanes, int64_t nnz, int64_t sum, int64_t n) {
  return !far_apart(sum, n) && (double)edges * 9.0 >= (double)lanes * (double)nnz;
}

// Whether vertex v, entry i of a list of m, is in the list's sample of about `want`:
// spread by a hash of its id and `salt`.  The first entry always is, so that no
// sample is empty (one of few CTAs' worth often would be: want = 1 in 37 of 100
// lists) and a lazy step always has a candidate to search.
GC_HD bool sample_takes(int32_t i, int32_t v, int32_t m, int32_t want, uint32_t salt) {
  const uint64_t lim = m > want ? ((uint64_t)want << 32) / (uint64_t)m : ~0ull;
  uint32_t h = ((uint32_t)v + 1u + salt * 0x10001u) * 0x9E3779B1u;  // multiplicative hashing (2^32 over the golden ratio)
  h ^= h >> 16;
  h *= 0x9E3779B1u;
  h ^= h >> 13;
  h *= 0x9E3779B1u;
  h ^= h >> 16;
  return i == 0 || (uint64_t)h < lim;
}

// Buffers that are only of use together: alloc(p) for each that is null, which sets
// p and returns true, or returns false.  After a failure those that this call made
// are given back by release(p) and null again, so that a later call starts over and
// none is used while another is missing.
template <class Alloc, class Release, class... T>
bool alloc_missing(Alloc alloc, Release release, T *&...p) {
  const bool had[] = {p != nullptr...};
  bool ok = true;
  ((ok = ok && (p || alloc(p))), ...);
  if (ok) return true;
  int i = 0;
  auto back = [&](auto *&q, bool keep) {
    if (keep) return;
    if (q) release(q);
    q = nullptr;
  };
  (back(p, had[i++]), ...);
  return false;
}

// Buffers that grow together: cap follows what is there, also when a growth fails
// (0 then, with every pointer null).  False on a failure.
template <class Cap, class Alloc, class Release, class... T>
bool grow_buffers(Cap &cap, Cap want, Alloc alloc, Release release, T *&...p) {
  if (want <= cap) return true;
  auto drop = [&](auto *&q) {
    if (q) release(q);
    q = nullptr;
  };
  (drop(p), ...);
  cap = 0;
  if (!alloc_missing(alloc, release, p...)) return false;
  cap = want;
  return true;
}

}  // namespace gc
