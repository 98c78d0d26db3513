"""GPU tests of the solve kernels' forms (narrow, split and leaf levels; right-hand sides split
over CTAs, padded and in several passes) and of the small FP64 Schur tiles' virtual tasks."""
import numpy as np
import pytest

import oracle
import paper_2202_09288_gb300 as P
from conftest import column_error
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def workload(name):
    if name.startswith("dense"):
        A = inputs.random_spd_dense(int(name[5:]), 3)
        return A, np.arange(A.n, dtype=np.int32)
    if name.startswith("diag"):  # supernodes of one column, one level
        A = inputs.from_dense(np.diag(1.0 + np.arange(float(name[4:]))))
        return A, np.arange(A.n, dtype=np.int32)
    return inputs.workload(name)


# narrow levels with every number of right-hand sides per CTA and its remainders, split levels
# (st27x3_20 from 8 right-hand sides on: 40 tasks of 4 supernodes), leaf levels in one and
# two passes (lap2d_150, diag600), supernodes of one column and without rows below
@pytest.mark.parametrize("name", ["diag1", "diag600", "dense65", "dense700", "lap2d_33", "lap2d_150",
                                  "st27x3_20"])
@pytest.mark.parametrize("owner", [False, True])
def test_right_hand_sides(torch, name, owner):
    A, perm = workload(name)
    ctx = P.Context(assembly=P.CHOL_ASSEMBLY_OWNER if owner else P.CHOL_ASSEMBLY_ATOMIC)
    sym = P.Symbolic(ctx, A, perm)
    num = P.Factor(ctx, sym, A.vals)
    mixed = P.Factor(ctx, sym, A.vals, P.CHOL_MIXED)
    full = A.to_scipy_full()
    for k in (1, 2, 3, 4, 5, 8, 9, 12, 13, 16, 17, 25, 32, 33):
        B = np.asfortranarray(full @ inputs.rhs_block(k, A.n, k))
        X = num.solve(B)
        assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, B, X) <= 1e-13, k
        X, info = mixed.refine(B)
        assert info["fell_back"] is False and info["residual"] <= 1e-12, k
        assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, B, X) <= 1e-12, k
        if owner:  # a fixed order of every sum: the same bits again
            assert np.array_equal(num.solve(B), num.solve(B)), k


# levels of a few 32-tiles (done as 16 x 16 virtual tasks) and of many
@pytest.mark.parametrize("name", ["lap2d_20", "lap2d_100", "lap3d_12"])
def test_small_tiles(torch, name):
    A, perm = workload(name)
    ref = oracle.cholesky(A, perm)
    ctx = P.Context()
    num = P.Factor(ctx, P.Symbolic(ctx, A, perm), A.vals)
    lp, li, lx = num.export()
    assert np.array_equal(li, ref.li)
    assert column_error(lp, lx, ref.lx) <= 1e-12
