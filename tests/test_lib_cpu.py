"""CPU tests of the native library: it loads, exports every entry point that
include/hqr.h declares, and its host-side elimination-list generator and
validator agree with the oracle. No device work here."""
import itertools
import os
import re

import numpy as np
import pytest

from oracle.elim_list import BINARY, FIBONACCI, FLAT, GREEDY, TS, TT, hqr_elim_list, validate

hqr = pytest.importorskip("paper_1110_1553_gb300.hqr")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_1110_1553_gb300 import _build
    _build.build()
    return hqr.load()


def header_functions():
    src = open(os.path.join(ROOT, "include", "hqr.h")).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(hqr_[a-z_0-9]+)\s*\(", src)))


def test_exports_every_declared_symbol(lib):
    names = header_functions()
    assert len(names) >= 15
    for name in names:
        assert hasattr(lib, name), name
    assert sorted(hqr.EXPORTS) == names


def test_strerror(lib):
    for code in range(8):
        assert lib.hqr_strerror(code)
    assert b"invalid" in lib.hqr_strerror(-3)


def test_lists_bit_exact_small(lib):
    trees = (FLAT, BINARY, GREEDY, FIBONACCI)
    for m in range(1, 8):
        for n in range(1, m + 1):
            for a in range(1, m + 1):
                for p in range(1, m + 1):
                    for lo, hi in itertools.product(trees, trees):
                        got = hqr.as_records(hqr.elim_list(m, n, a, p, lo, hi))
                        assert got == [tuple(r) for r in hqr_elim_list(m, n, a, p, lo, hi)]


@pytest.mark.parametrize("m,n,a,p", [(512, 8, 4, 16), (64, 64, 4, 1), (8, 8, 8, 1), (24, 10, 2, 3),
                                     (100, 37, 3, 7), (128, 16, 1, 1)])
def test_lists_bit_exact_workload_shapes(lib, m, n, a, p):
    for lo in (FLAT, BINARY, GREEDY, FIBONACCI):
        for hi in (FIBONACCI, GREEDY):
            got = hqr.elim_list(m, n, a, p, lo, hi)
            ref = hqr_elim_list(m, n, a, p, lo, hi)
            assert hqr.as_records(got) == [tuple(r) for r in ref]
            assert hqr.validate_list(m, n, got) == 0


def test_domino_lists_bit_exact(lib):
    trees = (FLAT, BINARY, GREEDY, FIBONACCI)
    for m in range(1, 8):
        for n in range(1, m + 1):
            for a in range(1, m + 1):
                for p in range(1, m + 1):
                    for lo, hi in itertools.product(trees, trees):
                        got = hqr.as_records(hqr.elim_list(m, n, a, p, lo, hi, domino=True))
                        assert got == [tuple(r) for r in hqr_elim_list(m, n, a, p, lo, hi, domino=True)]
    for (m, n, a, p) in [(24, 10, 2, 3), (512, 8, 4, 16), (100, 37, 3, 7)]:
        got = hqr.elim_list(m, n, a, p, GREEDY, FIBONACCI, domino=True)
        assert hqr.as_records(got) == [tuple(r) for r in hqr_elim_list(m, n, a, p, GREEDY, FIBONACCI, domino=True)]
        assert hqr.validate_list(m, n, got) == 0


def test_capacity_and_argument_errors(lib):
    import ctypes
    cnt = ctypes.c_size_t(0)
    assert lib.hqr_elim_list(8, 4, 2, 2, 0, 0, None, 0, ctypes.byref(cnt)) == hqr.ERR_CAPACITY
    assert cnt.value == 7 + 6 + 5 + 4
    assert lib.hqr_elim_list(0, 1, 1, 1, 0, 0, None, 0, ctypes.byref(cnt)) == -1
    assert lib.hqr_elim_list(4, 5, 1, 1, 0, 0, None, 0, ctypes.byref(cnt)) == -2
    assert lib.hqr_elim_list(4, 2, 0, 1, 0, 0, None, 0, ctypes.byref(cnt)) == -3
    assert lib.hqr_elim_list(4, 2, 1, 0, 0, 0, None, 0, ctypes.byref(cnt)) == -4
    assert lib.hqr_elim_list(4, 2, 1, 1, 7, 0, None, 0, ctypes.byref(cnt)) == -5
    assert lib.hqr_geqrf(None, 4, 4, 4, 0, 8, 4, None, 0, None, None) == -1
    # the widening entry point checks its arguments before any device work
    assert lib.hqr_widen_f32(None, None, -1, None) == -3
    assert lib.hqr_widen_f32(None, None, 0, None) == 0
    assert lib.hqr_widen_f32(None, ctypes.c_void_p(16), 4, None) == -1
    assert lib.hqr_widen_f32(ctypes.c_void_p(16), None, 4, None) == -2


def test_validator_agrees_with_oracle_on_mutations(lib):
    from tests.test_oracle_lists import _mutations
    L = hqr_elim_list(16, 4, 2, 2, BINARY, BINARY)
    assert hqr.validate_list(16, 4, L) == 0
    for name, M in _mutations(L):
        assert validate(M, 16, 4) is not None
        assert hqr.validate_list(16, 4, M) == hqr.ERR_INVALID_LIST, name


SMEM_LIMITS = r"""
#include "smem_limits.h"
#include <cstdio>
#include <thread>
#include <vector>
using namespace hqr;
static size_t attr[3][2];  // what a device's kernel was set to: 2 devices in the record, one beyond
static int calls;
int main() {
  SmemLimits<2, 2> rec;
  auto raise = [&](int dev, int k, size_t b) { return rec.raise(dev, k, b, [&] { ++calls; attr[dev][k] = b; return true; }); };
  // every launch on every device finds at least its bytes, and no limit is lowered
  const size_t seq[][3] = {{0, 0, 90}, {1, 0, 60}, {0, 0, 70}, {0, 1, 50}, {1, 1, 50}, {1, 0, 95}, {0, 0, 90}, {2, 0, 40}, {2, 0, 30}};
  for (auto &q : seq) {
    const size_t before = attr[q[0]][q[1]];
    if (!raise((int)q[0], (int)q[1], q[2]) || attr[q[0]][q[1]] < q[2]) return 1;
    if (q[0] < 2 && attr[q[0]][q[1]] < before) return 2;
  }
  if (calls != 7) return 3;
  // a failed set is reported and tried again
  if (rec.raise(0, 1, 80, [] { return false; }) || !raise(0, 1, 80) || attr[0][1] != 80) return 4;
  // two threads: the largest value stays
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i) t.emplace_back([&, i] { for (int b = 100 + i; b < 4000; b += 8) raise(0, 0, (size_t)b); });
  for (auto &x : t) x.join();
  return attr[0][0] == 3999 ? 0 : 5;
}
"""


def test_shared_memory_limits_per_device(tmp_path):
    """The record behind the scheduler launches, on a fake of the attribute: a
    limit that one device was granted says nothing about another device."""
    import shutil
    import subprocess
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(SMEM_LIMITS)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_1110_1553_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
