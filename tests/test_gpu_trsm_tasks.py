"""GPU tests of the tensor-core TRSM's CTAs with several tasks: levels of one task per CTA, of many per CTA
with the same and with another supernode's inverse, and batches whose members' tasks follow one
another, against the FP64 TRSM of the same matrices (each within 1e-12 of the exact factor per
column)."""
import pytest

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


def symbolic(ctx, name, rows):
    A, perm = inputs.workload(name)
    sym = P.Symbolic(ctx, A, perm)
    P.chol_sym_set_tile_policy(sym.handle, {"min_rows_trsm_tc": rows})
    return A, sym


@pytest.mark.parametrize("names", [["st27x3_12"], ["st27x3_32"], ["diff3d7_40"],
                                   ["st27x3_16", "diff3d7_24", "st27x3_16", "st27x3_20"] * 3])
def test_against_fp64_trsm(torch, names):
    ctx = P.Context()
    exports = []
    for rows in (1, 1 << 30):
        parts = [symbolic(ctx, n, rows) for n in names]
        nums = [P.Factor(ctx, s, A.vals) for A, s in parts]
        if len(nums) > 1:
            P.Batch(ctx, nums).factorize([A.vals for A, _ in parts])
        assert all(n.status()[0] == P.CHOL_OK for n in nums)
        exports.append([n.export() for n in nums])
    for (lp, li, lx), (_, _, ref) in zip(*exports):
        assert column_error(lp, lx, ref) <= 2e-12
