"""GPU test of the owner-ordered assembly with more sources per target than one look-up batch
(32), targets of several column blocks and partial last blocks."""
import numpy as np
import pytest

import oracle
import paper_2202_09288_gb300 as P
from conftest import column_error
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu


def arrow(leaves, tail, seed):
    """`leaves` unknowns coupled only to a random half of the last `tail`, which are dense."""
    n = leaves + tail
    u = inputs.uniform(seed, 9, n * n).reshape(n, n)
    a = np.tril(u, -1)
    a[:leaves, :leaves] = 0
    a[leaves:, :leaves][inputs.uniform(seed, 10, tail * leaves).reshape(tail, leaves) < 0] = 0
    a = a + a.T
    return inputs.from_dense(a + np.diag(np.abs(a).sum(axis=1) + 1))


@pytest.mark.parametrize("leaves,tail", [(1, 5), (31, 33), (32, 64), (33, 70), (100, 40), (150, 97)])
@pytest.mark.parametrize("precision", [P.CHOL_FP64, P.CHOL_MIXED])
def test_many_sources(leaves, tail, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = arrow(leaves, tail, leaves)
    perm = np.arange(A.n, dtype=np.int32)
    ref = oracle.cholesky(A, perm)
    ctx = P.Context(assembly=P.CHOL_ASSEMBLY_OWNER, relax=-1.0)
    sym = P.Symbolic(ctx, A, perm)
    num = P.Factor(ctx, sym, A.vals, precision)
    assert num.status()[0] == P.CHOL_OK
    lp, li, lx = num.export()
    scale = np.sqrt(A.vals[A.colptr[:-1]])[li] if precision == P.CHOL_MIXED else 1.0
    tol = 1e-12 if precision == P.CHOL_FP64 else A.n * 2.0 ** -24
    assert column_error(lp, lx * scale, ref.lx) <= tol
    num.refactor(A.vals)
    assert np.array_equal(num.export()[2], lx)  # a fixed order: the same bits
