"""GPU test of the solves by substitution (factors wider than 64 columns, which keep no inverse) with
every number of right-hand sides per pass and its remainders."""
import numpy as np
import pytest

import oracle
import paper_2202_09288_gb300 as P
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("width", [65, 128])
@pytest.mark.parametrize("owner", [False, True])
def test_right_hand_sides(torch, width, owner):
    A, perm = inputs.workload("st27x3_10")
    ctx = P.Context(width_cap=width,
                    assembly=P.CHOL_ASSEMBLY_OWNER if owner else P.CHOL_ASSEMBLY_ATOMIC)
    sym = P.Symbolic(ctx, A, perm)
    assert sym.info["max_width"] == width
    num = P.Factor(ctx, sym, A.vals)
    mixed = P.Factor(ctx, sym, A.vals, P.CHOL_MIXED)
    full = A.to_scipy_full()
    for k in (1, 3, 4, 7, 8, 9, 15, 16, 17, 31, 32, 33):
        B = np.asfortranarray(full @ inputs.rhs_block(k, A.n, k))
        assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, B, num.solve(B)) <= 1e-13, k
        X, info = mixed.refine(B)
        assert info["fell_back"] is False and info["residual"] <= 1e-12, k
