"""GPU tests of the diagonal-block kernels at the edges of their 8 x 8 and 16 x 16 blocks (POTRF
in FP64 and FP32, with and without the whole inverse), over the exponent range, and of the
TRSM's row splits."""
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


def bordered(n, u, scale=None):
    """Dense first n columns coupled to u more unknowns (dense as well), optionally D A D."""
    a = inputs.uniform(n + 100 * u, 6, (n + u) ** 2).reshape(n + u, n + u)
    a = a @ a.T + (n + u) * np.eye(n + u)
    if scale is not None:
        a = a * scale[:, None] * scale[None, :]
    return inputs.from_dense(a)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 24, 33, 48, 57, 63, 64, 65])
@pytest.mark.parametrize("tc", [False, True])  # tc: the whole inverse, tensor-core TRSM
def test_block_sizes(torch, n, tc):
    A = bordered(n, 130)
    perm = np.arange(A.n, dtype=np.int32)
    ref = oracle.cholesky(A, perm)
    ctx = P.Context(width_cap=min(n, 64))
    sym = P.Symbolic(ctx, A, perm)
    if tc:
        P.chol_sym_set_tile_policy(sym.handle, {"min_rows_trsm_tc": 1})
    num = P.Factor(ctx, sym, A.vals)
    assert num.status()[0] == P.CHOL_OK
    lp, li, lx = num.export()
    assert column_error(lp, lx, ref.lx) <= 1e-12
    b = A.to_scipy_full() @ inputs.rhs_block(1, A.n, 1)[:, 0]
    assert oracle.residual(A.n, A.colptr, A.rowind, A.vals, b, num.solve(b)) <= 1e-13
    mixed = P.Factor(ctx, sym, A.vals, P.CHOL_MIXED)
    lp, li, lx = mixed.export()
    # panels of S A S in FP32: undo S = diag(A)^-1/2; n products and sums of 2^-24 each
    diag = A.vals[A.colptr[:-1]]
    lx = lx * np.sqrt(diag)[li]
    assert column_error(lp, lx, ref.lx) <= 200 * 2.0 ** -24
    x, info = mixed.refine(b)
    assert info["residual"] <= 1e-12 and not info["fell_back"]


# D A D with powers of two: the factor is D L exactly, whatever path the pivots take (the
# reciprocal by integers in the middle of the exponent range, square roots beyond)
@pytest.mark.parametrize("span", [0, 150, 210, 400])
def test_scaled_blocks(torch, span):
    n, u = 40, 20
    d = np.ldexp(1.0, np.round(span * inputs.uniform(9, 7, n + u)).astype(np.int64))
    A, S = bordered(n, u), bordered(n, u, d)
    perm = np.arange(A.n, dtype=np.int32)
    ref = oracle.cholesky(A, perm)
    ctx = P.Context(width_cap=n)
    num = P.Factor(ctx, P.Symbolic(ctx, S, perm), S.vals)
    assert num.status()[0] == P.CHOL_OK
    lp, li, lx = num.export()
    assert column_error(lp, lx / d[li], ref.lx) <= 1e-12


@pytest.mark.parametrize("col", [0, 6, 7, 8, 31, 40, 63])
@pytest.mark.parametrize("precision", [P.CHOL_FP64, P.CHOL_MIXED])
def test_bad_pivot_column(torch, col, precision):
    a = inputs.uniform(3, 8, 64 * 64).reshape(64, 64)
    a = a @ a.T + np.eye(64)
    L = np.linalg.cholesky(a)
    a[col, col] -= 1.05 * L[col, col] ** 2  # pivot col becomes -0.05 of itself
    A = inputs.from_dense(a)
    if a[col, col] <= 0 and precision == P.CHOL_MIXED:
        pytest.skip("rejected by the equilibration")
    ctx = P.Context()
    num = P.Factor(ctx, P.Symbolic(ctx, A, np.arange(64, dtype=np.int32)), A.vals, precision)
    assert num.status() == (P.CHOL_E_NOT_SPD, col)


# 32-row TRSM tasks of a level: 1-38 (8 rows per CTA), 39-76 (16), more, and four per CTA
@pytest.mark.parametrize("name", ["st27x3_6", "st27x3_10", "st27x3_14", "lap2d_160"])
@pytest.mark.parametrize("precision", [P.CHOL_FP64, P.CHOL_MIXED])
def test_trsm_splits(torch, name, precision):
    A, perm = inputs.workload(name)
    ctx = P.Context()
    sym = P.Symbolic(ctx, A, perm)
    num = P.Factor(ctx, sym, A.vals, precision)
    if precision == P.CHOL_FP64:
        ref = oracle.cholesky(A, perm)
        lp, li, lx = num.export()
        assert column_error(lp, lx, ref.lx) <= 1e-12
    b = A.to_scipy_full() @ inputs.rhs_block(2, A.n, 2)
    x, info = num.refine(np.asfortranarray(b))
    assert info["residual"] <= 1e-12 and not info["fell_back"]
