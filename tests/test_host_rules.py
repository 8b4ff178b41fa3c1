"""The library's host-device rules (csrc/gc_rules.h), compiled by the host's
C++ compiler alone."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_01144_gb300", "csrc")
INF = 0x3FFFFFFF

SOURCE = r"""
#include "gc_rules.h"
using namespace gc;
extern "C" {
int32_t bucket_end(int32_t mn, int32_t delta) { return w_bucket_end(mn, delta); }
int in_bucket(int32_t x, int32_t T) { return w_in_bucket(x, T); }
int far(int64_t sum, int64_t n) { return far_apart(sum, n); }
int lanes_rest(uint64_t edges, uint64_t lanes, int64_t nnz, int64_t sum, int64_t n) {
  return lanes_take_rest(edges, lanes, nnz, sum, n);
}
int whole_search(int64_t n, int64_t nnz) { return w_whole_search(n, nnz); }
int64_t grid_of_bfs(int64_t n, int64_t nnz) { return bfs_grid(n, nnz); }

int sample(const int32_t *list, int m, int want, uint32_t salt) {
  int c = 0;
  for (int i = 0; i < m; ++i) c += sample_takes(i, list[i], m, want, salt);
  return c;
}

// a stand-in for a device allocator: the allocation of index `fail` fails
static int g_live, g_made, g_fail;
static int g_cells[64];
static bool fake_alloc(int *&p) {
  if (g_made++ == g_fail) return false;
  ++g_live;
  p = &g_cells[g_made];
  return true;
}
// three buffers, of which the bits of `had` are there already; returns the bits of
// those that are there after the call, with bit 8 set if it succeeded
static int *g_p[3];
int buffers(int had, int fail) {
  g_live = g_made = 0;
  g_fail = fail;
  for (int i = 0; i < 3; ++i) g_p[i] = (had >> i) & 1 ? &g_cells[40 + i] : nullptr;
  const bool ok = alloc_missing(fake_alloc, [](int *) { --g_live; }, g_p[0], g_p[1], g_p[2]);
  int there = 0;
  for (int i = 0; i < 3; ++i) there |= (g_p[i] != nullptr) << i;
  return there | (ok ? 256 : 0);
}
int live() { return g_live; }

// two buffers of one capacity: bit 0 and 1 for those that are there, bit 8 for
// success, and the capacity from bit 9 on
static int *g_q[2];
static int g_cap;
void grow_start() { g_q[0] = g_q[1] = nullptr; g_cap = g_live = 0; }
int grow(int want, int fail) {
  g_made = 0;
  g_fail = fail;
  const bool ok = grow_buffers(g_cap, want, fake_alloc, [](int *) { --g_live; }, g_q[0], g_q[1]);
  return (g_q[0] != nullptr) | (g_q[1] != nullptr) << 1 | (ok ? 256 : 0) | g_cap << 9;
}
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "rules.cpp", d / "librules.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(src),
                           "-o", str(lib)])
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("delta", [1, 2, 8, 243368, INF // 2, INF])
@pytest.mark.parametrize("mn", [1, 2, 1000, INF // 2, INF - 3, INF - 2, INF - 1, INF])
def test_next_bucket_takes_the_nearest_entry(rules, mn, delta):
    T = rules.bucket_end(mn, delta)
    assert rules.in_bucket(mn, T)
    assert T <= INF - 1 and (T == INF - 1 or T == mn + delta)
    if T < INF - 1:  # and nothing past its end
        assert not rules.in_bucket(T, T) and rules.in_bucket(T - 1, T)


@pytest.mark.parametrize("had", range(8))
def test_buffers_of_a_group_come_and_go_together(rules, had):
    missing = 3 - bin(had).count("1")
    for fail in range(missing):  # none stays behind without the others, none is lost
        assert rules.buffers(had, fail) == had
        assert rules.live() == 0
    assert rules.buffers(had, missing) == 256 | 7
    assert rules.live() == missing


def test_capacity_follows_the_buffers(rules):
    rules.grow_start()
    assert rules.grow(5, 9) == 3 | 256 | 5 << 9
    assert rules.grow(4, 0) == 3 | 256 | 5 << 9  # large enough: nothing is allocated
    for fail in (0, 1):
        assert rules.grow(8, fail) == 0 and rules.live() == 0  # no buffer, and no capacity either
        assert rules.grow(4, fail) == 0  # so a smaller want is not taken for granted
        assert rules.grow(4, 9) == 3 | 256 | 4 << 9 and rules.live() == 2


@pytest.mark.parametrize("want", [1, 2, 5, 64, 2432])
def test_samples_are_never_empty(rules, want):
    rng = np.random.default_rng(want)
    sizes = []
    for salt in range(60):
        for m in (1, want, 2 * want + 1, 40 * want):
            v = np.sort(rng.choice(100 * want + 50, m, replace=False)).astype(np.int32)
            c = rules.sample(v.ctypes.data_as(ctypes.c_void_p), m, want, salt)
            assert 1 <= c <= m
            if m <= want:
                assert c == m
            elif m == 40 * want:
                sizes.append(c)
    assert abs(np.mean(sizes) - want) <= 1 + 4 * np.sqrt(want / len(sizes))  # the mean of binomial counts, and the first entry


def test_far_apart(rules):
    far = lambda s, n: bool(rules.far(ctypes.c_int64(s), ctypes.c_int64(n)))
    for n in (1, 2, 100, 10**6, 2**31 - 1):
        assert far(n * n // 4 + 1, n)                       # a path
        assert far(int(n * 0.5 * n**0.5) + 1, n)            # a square grid
        assert far(2**62, n)                                # (no overflow)
    for n in (10**3, 10**5, 2**31 - 1):
        assert not far(2 * n, n) and not far(0, n)          # a star
    assert far(10000 * 1000, 10000) and not far(10000 * 7, 10000)
    assert far(10**6 * 71, 10**6) and not far(10**6 * 70, 10**6)  # mean^2 = n / 200 between the two


@pytest.mark.parametrize("n,nnz,ctas", [(1, 0, 1), (512, 511, 1), (513, 2000, 2), (2000, 20000, 4), (4000, 1600000, 97),
                                        (600, 359400, 21), (10**6, 4 * 10**6, 1954), (2**31 - 1, 2**31 - 1, 2**22)])
def test_bfs_grid_has_ctas_for_the_entries(rules, n, nnz, ctas):
    rules.grid_of_bfs.restype = ctypes.c_int64
    assert rules.grid_of_bfs(ctypes.c_int64(n), ctypes.c_int64(nnz)) == ctas


@pytest.mark.parametrize("n,nnz,whole", [(1, 0, 1), (255, 255 * 254, 1), (256, 256 * 64, 1), (256, 256 * 64 + 1, 0),
                                         (1024, 65536, 1), (1024, 65538, 0), (1025, 2050, 0), (2**30, 2**31 - 1, 0)])
def test_whole_weighted_searches(rules, n, nnz, whole):
    assert rules.whole_search(ctypes.c_int64(n), ctypes.c_int64(nnz)) == whole


def test_lanes_take_the_rest(rules):
    def rest(share, mean, n=100000, nnz=600000, lanes=8192):
        return bool(rules.lanes_rest(ctypes.c_uint64(int(share * lanes * nnz)), ctypes.c_uint64(lanes), ctypes.c_int64(nnz),
                                     ctypes.c_int64(int(mean * n)), ctypes.c_int64(n)))

    assert rest(0.3, 5.2) and rest(0.112, 5.2) and not rest(0.110, 5.2)
    assert not rest(0.5, 200.0)                      # a road network
    assert rest(1.0, 5.0, 2**31 - 1, 2**31 - 1, 2**31 - 1)  # (no overflow)
