"""Capacity of the ACA term pool (csrc/rt_pool.h), on the host: however often it grows, terms stay on
16-byte boundaries and the growth makes room for the blocks that wait."""
from __future__ import annotations

import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2306_05789_gb300", "csrc")


@pytest.fixture(scope="module")
def pool(tmp_path_factory):
    d = tmp_path_factory.mktemp("pool")
    src = d / "pool.cpp"
    src.write_text('#include "rt_pool.h"\n'
                   'extern "C" int64_t first(int64_t need) { return rt::pool_first(need); }\n'
                   'extern "C" int64_t grown(int64_t cap, int64_t need) { return rt::pool_grown(cap, need); }\n')
    so = str(d / "pool.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for f in (lib.first, lib.grown):
        f.restype = ctypes.c_int64
    lib.first.argtypes = [ctypes.c_int64]
    lib.grown.argtypes = [ctypes.c_int64, ctypes.c_int64]
    return lib


def _round4(x):
    return (x + 3) // 4 * 4


# one block of odd size and of an odd number of float4s, several groups, a whole wave, large blocks
@pytest.mark.parametrize("G,blocks", [(1, [(1, 1)]), (1, [(333, 332)]), (3, [(665, 666)]), (5, [(64, 61), (33, 31)]),
                                      (17, [(665, 666)] * 2 + [(166, 167)] * 8), (64, [(1 << 17, (1 << 17) - 3)])])
def test_every_capacity_holds_whole_float4s(pool, G, blocks):
    terms = [G * (_round4(m) + _round4(n)) for m, n in blocks]
    need = sum(terms)
    cap = pool.first(need)
    assert cap >= 24 * need and cap % 4 == 0
    limit = max(m * n // (m + n) for m, n in blocks) * need
    for k in range(60):
        some = max(terms) if k % 2 else need   # fewer blocks are active later on
        new = pool.grown(cap, some)
        assert new % 4 == 0, (k, cap, new)
        assert new >= cap + 8 * some and new >= cap + cap // 2
        assert new <= max(cap + cap // 2, cap + 8 * some) + 64   # and no more than it has to
        cap = new
        if cap > 64 * limit:
            break
