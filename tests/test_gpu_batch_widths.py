"""GPU test of batches whose members differ in supernode width: up to 64 columns (kept inverses, slices on
the tensor cores) beside wider ones, in every order."""
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


@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0), (1, 0, 2)])
@pytest.mark.parametrize("precision", [P.CHOL_FP64, P.CHOL_MIXED])
@pytest.mark.parametrize("owner", [False, True])
def test_widths(torch, order, precision, owner):
    ctx = P.Context(width_cap=128,
                    assembly=P.CHOL_ASSEMBLY_OWNER if owner else P.CHOL_ASSEMBLY_ATOMIC)
    specs = [("st27x3_10", 64), ("st27x3_10", 128), ("lap3d_12", 100)]
    mats, nums = [], []
    for name, width in (specs[i] for i in order):
        A, perm = inputs.workload(name)
        sym = P.Symbolic(P.make_opts(width_cap=width), A, perm)
        P.chol_sym_set_tile_policy(sym.handle, {"min_level_tiles128": 0, "min_rows_tile128": 65,
                                                "min_rows_trsm_tc": 1})
        mats.append((A, perm))
        nums.append(P.Factor(ctx, sym, A.vals, precision))
    assert max(f.sym.info["max_width"] for f in nums) > 64 >= min(f.sym.info["max_width"] for f in nums)
    batch = P.Batch(ctx, nums)
    for use_graph in (False, True):
        batch.factorize([A.vals for A, _ in mats], use_graph=use_graph)
        for f, (A, perm) in zip(nums, mats):
            assert f.status()[0] == P.CHOL_OK
            b = A.to_scipy_full() @ inputs.rhs_block(9, A.n, 1)[:, 0]
            if precision == P.CHOL_FP64:
                lp, _, lx = f.export()
                assert column_error(lp, lx, oracle.cholesky(A, perm).lx) <= 1e-12
                assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, b, f.solve(b)) <= 1e-13
            else:
                assert f.refine(b)[1]["residual"] <= 1e-12
