"""GPU test of the FP64 POTRF's backward error on ill-conditioned diagonal blocks: columns of a
block dependent to eps, so that 8 x 8 diagonal blocks have condition numbers up to 1 / eps.
|A - L L^T| <= (n + 1) u |L||L^T| for substitution (Higham, Accuracy and Stability, Thm 10.3;
u = 2^-53), and |L||L^T|_ij <= d_i d_j with d_i^2 = a_ii; four times that allows for the
8 x 8 quotients' refinement."""
import numpy as np
import pytest

import paper_2202_09288_gb300 as P
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("n", [10, 16, 24, 43, 64])
@pytest.mark.parametrize("eps", [1e-1, 1e-2, 1e-3, 1e-4, 1e-5])
@pytest.mark.parametrize("border", [0, 130])  # 130: with the whole inverse, tensor-core TRSM
def test_dependent_columns(torch, n, eps, border):
    g = inputs.uniform(n, 11, 4 * n * n).reshape(4, n, n)
    m = g[0].copy()
    for near, to in ((1, 0), (5, 2), (9, 4)) + (((n - 2, n - 5), (n // 2 + 1, 3)) if n > 16 else ()):
        m[near] = m[to] + eps * g[1][near]
    # the smallest eigenvalue of the block, scaled to a unit diagonal, is above 4 n (n + 1) u
    a = m @ m.T + eps * eps * np.eye(n)
    full = np.zeros((n + border, n + border))
    full[:n, :n] = (a + a.T) / 2
    if border:  # rows below within the span of the block's, and their own part
        c = inputs.uniform(n, 12, border * n).reshape(border, n)
        full[n:, :n] = c @ full[:n, :n]
        full[n:, n:] = full[n:, :n] @ c.T + n * np.eye(border)
        full[:n, n:] = full[n:, :n].T
    full = (full + full.T) / 2
    A = inputs.from_dense(full)
    ctx = P.Context(width_cap=n)
    sym = P.Symbolic(ctx, A, np.arange(A.n, dtype=np.int32))
    if border:
        P.chol_sym_set_tile_policy(sym.handle, {"min_rows_trsm_tc": 1})
    num = P.Factor(ctx, sym, A.vals)
    assert num.status()[0] == P.CHOL_OK
    lp, li, lx = num.export()
    L = np.zeros((n, n), np.longdouble)
    for j in range(n):
        L[:, j][li[lp[j]:lp[j] + n - j]] = lx[lp[j]:lp[j] + n - j]
    d = np.sqrt(np.diag(full)[:n])
    err = np.abs(np.tril(L @ L.T - full[:n, :n])) / np.outer(d, d)
    assert err.max() <= 4 * (n + 1) * 2.0 ** -53, float(err.max())
    # the solves apply the block's inverse: a residual of cond(L) n u at most
    b = full @ inputs.rhs_block(n, A.n, 1)[:, 0]
    x = num.solve(b)
    r = np.abs(b - full @ x).max() / (np.abs(full).sum(axis=1).max() * np.abs(x).max())
    assert r <= A.n * 2.0 ** -53 * np.linalg.cond(np.asarray(L, np.float64)), r
