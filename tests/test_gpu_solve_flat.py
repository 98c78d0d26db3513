"""GPU tests of the solves on flat elimination trees: levels of one wave that hold nearly all
supernodes, with 17 to 32 right-hand sides (two groups), where the backward solve has fewer
arrival counters than tasks times groups (see test_solve_shape.py)."""
import numpy as np
import pytest

import oracle
import paper_2202_09288_gb300 as P
from flat_trees import FLAT, flat
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("name", FLAT)
@pytest.mark.parametrize("owner", [False, True])
def test_two_groups(torch, name, owner):
    A, perm = flat(name)
    ctx = P.Context(assembly=P.CHOL_ASSEMBLY_OWNER if owner else P.CHOL_ASSEMBLY_ATOMIC)
    sym = P.Symbolic(ctx, A, perm)
    num = P.Factor(ctx, sym, A.vals)
    mixed = P.Factor(ctx, sym, A.vals, P.CHOL_MIXED)
    full = A.to_scipy_full()
    for k in (16, 17, 24, 25, 32):
        B = np.asfortranarray(full @ inputs.rhs_block(k, A.n, k))
        X = num.solve(B)
        assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, B, X) <= 1e-13, k
        if owner:  # a fixed order of every sum: the same bits again
            assert np.array_equal(X, num.solve(B)), k
        Bd = torch.from_numpy(np.ascontiguousarray(B.T)).cuda()
        Xd = torch.full_like(Bd, float("nan"))
        P.chol_solve_noalloc(ctx.handle, num.handle, Bd, Xd)
        torch.cuda.synchronize()
        assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, B, Xd.cpu().numpy().T) <= 1e-13, k
        X, info = mixed.refine(B)
        assert info["fell_back"] is False and info["residual"] <= 1e-12, k
        assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, B, X) <= 1e-12, k
    # the stored values the residuals come from are untouched
    num.refactor(A.vals)
    assert num.status()[0] == P.CHOL_OK
