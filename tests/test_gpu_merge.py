"""GPU tests of the merged Schur updates of a separator's chunks (groups of two in FP64, of up
to four in FP32): chains whose last chunk is narrow, odd or not a multiple of 8 wide, updates of
one strip and of several, groups inside a tree, batches of different patterns, and a tile
policy changed after the analysis is on the device."""
import numpy as np
import pytest

import oracle
import paper_2202_09288_gb300 as P
from conftest import column_error
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu

ALL128 = {"min_rows_tile64": 1, "min_rows_tile32": 1, "min_level_tiles64": 0, "min_rows_tile128": 1,
          "min_level_tiles128": 0}


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def problem(name):
    if name.startswith("dense"):
        A = inputs.random_spd_dense(int(name[5:]), 3)
        return A, np.arange(A.n, dtype=np.int32)
    return inputs.workload(name)




@pytest.mark.parametrize("name,width", [("dense129", 64), ("dense200", 64), ("dense325", 64),
                                        ("dense392", 64), ("dense600", 64), ("dense300", 40),
                                        ("dense310", 24), ("dense300", 20), ("st27x3_11", 64),
                                        ("st27x3_14", 64), ("diff3d7_14", 32)])
def test_chains(torch, name, width):
    A, perm = problem(name)
    ref = oracle.cholesky(A, perm)
    ctx = P.Context(width_cap=width)
    sym = P.Symbolic(ctx, A, perm)
    P.chol_sym_set_tile_policy(sym.handle, ALL128)
    num = P.Factor(ctx, sym, A.vals)
    assert num.status()[0] == P.CHOL_OK
    lp, li, lx = num.export()
    assert column_error(lp, lx, ref.lx) <= 1e-12
    num.refactor(A.vals)  # the scratch in use again
    assert column_error(lp, num.export()[2], ref.lx) <= 1e-12
    mixed = P.Factor(ctx, sym, A.vals, P.CHOL_MIXED)
    lp, li, lx = mixed.export()
    lx = lx * np.sqrt(A.vals[A.colptr[:-1]])[perm][li]
    # sums of up to n products of FP32 panels: n 2^-24 covers every workload here
    assert column_error(lp, lx, ref.lx) <= A.n * 2.0 ** -24
    b = A.to_scipy_full() @ inputs.rhs_block(1, A.n, 1)[:, 0]
    x, info = mixed.refine(b)
    assert info["residual"] <= 1e-12 and not info["fell_back"]


@pytest.mark.parametrize("precision", [P.CHOL_FP64, P.CHOL_MIXED])
def test_batch_of_different_patterns(torch, precision):
    ctx = P.Context()
    names = ["dense325", "st27x3_9", "dense200", "diff3d7_12"]
    mats = [problem(n) for n in names]
    syms = [P.Symbolic(ctx, A, perm) for A, perm in mats]
    for s in syms:
        P.chol_sym_set_tile_policy(s.handle, ALL128)
    alone = [P.Factor(ctx, s, A.vals, precision) for s, (A, _) in zip(syms, mats)]
    nums = [P.Factor(ctx, s, A.vals, precision) for s, (A, _) in zip(syms, mats)]
    batch = P.Batch(ctx, nums)
    for graph in (False, True, True):
        batch.factorize([A.vals for A, _ in mats], use_graph=graph)
        for a, b in zip(alone, nums):
            assert b.status()[0] == P.CHOL_OK
            lp, li, lx = a.export()
            tol = 1e-13 if precision == P.CHOL_FP64 else 1e-4
            assert column_error(lp, b.export()[2], lx) <= tol


def test_policy_changed_on_the_device(torch):
    A, perm = problem("st27x3_14")
    ref = oracle.cholesky(A, perm)
    ctx = P.Context()
    sym = P.Symbolic(ctx, A, perm)
    num = P.Factor(ctx, sym, A.vals)
    default = P.chol_sym_get_tile_policy(sym.handle)
    for policy in (ALL128, dict(ALL128, min_rows_tile128=300), default):
        P.chol_sym_set_tile_policy(sym.handle, policy)
        num.refactor(A.vals)
        assert num.status()[0] == P.CHOL_OK
        lp, li, lx = num.export()
        assert column_error(lp, lx, ref.lx) <= 1e-12
