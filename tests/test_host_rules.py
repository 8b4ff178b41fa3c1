"""The library's host-device rules (csrc/gc_rules.h), compiled by the host's
C++ compiler alone."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_01144_gb300", "csrc")
INF = 0x3FFFFFFF

SOURCE = r"""
#include "gc_rules.h"
using namespace gc;
extern "C" {
int32_t bucket_end(int32_t mn, int32_t delta) { return w_bucket_end(mn, delta); }
int in_bucket(int32_t x, int32_t T) { return w_in_bucket(x, T); }
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
