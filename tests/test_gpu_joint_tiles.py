"""GPU tests of FP64 Schur tiles that sum two merged chunks in tensor memory: many tiles, chunks of one and of two units of 32 columns with whole and cut
16-column steps, last chunks narrower than the first, and rows whose entries in the two chunks
differ by many binary orders (one exponent serves both)."""
import numpy as np
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


@pytest.mark.parametrize("n,width,graded", [(1536, 64, False), (1800, 64, False), (1800, 64, True),
                                            (1700, 56, False), (1700, 40, False), (1700, 24, True),
                                            (1657, 8, False), (2600, 64, True)])
def test_against_dense(torch, n, width, graded):
    rng = np.random.default_rng(n + width)
    M = rng.standard_normal((n, n))
    if graded:  # columns of L of very different sizes next to one another
        M *= np.exp2(rng.integers(-30, 1, n // 16 + 1))[np.arange(n) // 16][None, :]
    full = np.tril(M, -1) / np.sqrt(n) + np.diag(1.0 + rng.random(n))
    full = full @ full.T
    full = (full + full.T) / 2
    A = inputs.from_dense(full)
    ctx = P.Context(width_cap=width)
    sym = P.Symbolic(ctx, A, np.arange(n, dtype=np.int32))
    num = P.Factor(ctx, sym, A.vals)
    assert num.status()[0] == P.CHOL_OK
    lp, li, lx = num.export()
    ref = np.linalg.cholesky(full)
    # errors of n products of at most 1 each are about n 2^-53 of a column's norm times the
    # condition of the leading blocks (the factor's diagonal is at least 1): 1e-12 at n = 2600
    assert column_error(lp, lx, np.concatenate([ref[j:, j] for j in range(n)])) <= 1e-12
    x = rng.standard_normal(n)
    b = full @ x
    r = b - full @ num.solve(b)
    assert np.linalg.norm(r) <= 1e-13 * np.linalg.norm(full, 2) * np.linalg.norm(x) * n ** 0.5
