"""The launch rule of the solves' levels (csrc/solve_shape.h), compiled here for the host (CPU
only): the backward launches cover every right-hand side once, and the arrival counters they use
lie inside the smallest array a factor with such a level has (3 per level, 8, and one per
supernode).  And flat elimination trees of the GPU tests do reach the rule's limit."""
import ctypes
import os
import subprocess

import pytest

import paper_2202_09288_gb300 as P
from conftest import ROOT
from flat_trees import FLAT, flat, level_tasks

SOURCE = """
#include "solve_shape.h"
// one group of right-hand sides counts on its supernode's counter (< nsup <= counters), several
// groups of a launch on groups * ntasks from the array's start
extern "C" int check(int ntasks, int nsup, int nrhs, long long counters) {
  const chol::SolveShape s = chol::solve_shape(nrhs, ntasks, nsup, counters);
  if (s.nr < 1 || s.nr > 16 || (long long)s.groups * s.nr < nrhs || (s.groups - 1) * s.nr >= nrhs) return 1;
  if (s.bwd_groups < 1 || s.groups % s.bwd_groups != 0) return 2;
  if (s.mode == chol::kNarrow && ntasks > chol::kWave) return 3;
  if (s.mode == chol::kLeaf && s.bwd_groups != 1) return 4;
  if (s.mode != chol::kSplit && s.bwd_groups > 1 && (long long)s.bwd_groups * ntasks > counters) return 5;
  return 0;
}
extern "C" int sweep(int ntasks, int* nsup, int* nrhs) {
  for (*nsup = 1; *nsup <= ntasks; ++*nsup)
    for (*nrhs = 1; *nrhs <= 32; ++*nrhs)
      if (int rc = check(ntasks, *nsup, *nrhs, 3 + 8 + *nsup)) return rc;
  return 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    src, so = d / "shape.cpp", d / "shape.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2202_09288_gb300", "csrc"), str(src), "-o", str(so)])
    return ctypes.CDLL(str(so))


def test_counters_stay_inside(rule):
    nsup, nrhs = ctypes.c_int(), ctypes.c_int()
    for ntasks in list(range(1, 160)) + [304, 305, 1000]:
        rc = rule.sweep(ntasks, ctypes.byref(nsup), ctypes.byref(nrhs))
        assert rc == 0, (rc, ntasks, nsup.value, nrhs.value)


@pytest.mark.parametrize("name", FLAT)
def test_flat_trees(rule, name):
    A, perm = flat(name)
    sym = P.Symbolic(P.make_opts(), A, perm)
    tasks, counters = level_tasks(sym)
    rule.check.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_longlong]
    for ntasks, nsup in tasks:
        for k in range(1, 33):
            assert rule.check(ntasks, nsup, k, counters) == 0, (ntasks, nsup, k)
    # two groups of right-hand sides in a level of one wave, and too few counters for both
    assert any(n <= 152 and n < 2 * s and 2 * n > counters for n, s in tasks)
