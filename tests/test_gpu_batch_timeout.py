"""A wait of the tensor-core Schur kernels that gives up in a batch's launch (the test hook of
test_gpu_wait_timeout.py) is reported by every member with work in that launch, not by the first
one alone; the batch and its members work again afterwards."""
import numpy as np
import pytest

import oracle
import paper_2202_09288_gb300 as P
from conftest import column_error
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu

ALL128 = {"min_rows_tile64": 1, "min_rows_tile32": 1, "min_level_tiles64": 0,
          "min_rows_tile128": 1, "min_level_tiles128": 0, "min_rows_trsm_tc": 1}


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("precision", [P.CHOL_FP64, P.CHOL_MIXED])
def test_every_member_reports(torch, precision):
    ctx = P.Context()
    mats = [inputs.workload(w) for w in ("st27x3_6", "st27x3_7", "lap3d_9")]
    syms = [P.Symbolic(ctx, A, perm) for A, perm in mats]
    for s in syms:
        P.chol_sym_set_tile_policy(s.handle, ALL128)
    nums = [P.Factor(ctx, s, A.vals, precision) for s, (A, _) in zip(syms, mats)]
    assert all(f.status()[0] == P.CHOL_OK for f in nums)
    batch = P.Batch(ctx, nums)
    P.chol_set_device_wait(ctx.handle, 1000)
    batch.factorize([A.vals for A, _ in mats], use_graph=False)
    got = [P.lib().chol_factor_status(ctx.handle, f.handle, None) for f in nums]
    P.chol_set_device_wait(ctx.handle, 0)
    assert got == [P.CHOL_E_TIMEOUT] * 3
    batch.factorize([A.vals for A, _ in mats], use_graph=False)
    for f, (A, perm) in zip(nums, mats):
        assert f.status()[0] == P.CHOL_OK
        b = A.to_scipy_full() @ inputs.rhs_block(9, A.n, 1)[:, 0]
        if precision == P.CHOL_FP64:
            lp, _, lx = f.export()
            assert column_error(lp, lx, oracle.cholesky(A, perm).lx) <= 1e-12
            assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, b, f.solve(b)) <= 1e-13
        else:
            assert f.refine(b)[1]["residual"] <= 1e-12
