"""GPU test of the FP64 tensor-core Schur tiles entry by entry, at the accuracy of their slices.

The matrix is [[I, B^T], [B, C]] with B = L21 exact: S_ij = C_ij - sum_k b_ik b_jk is read from the factor, whose
trailing block is S = diag(s^2) up to rounding errors (L_ij = S_ij / s_j off the diagonal, products
of two such entries are below 2^-90).  C_ij is the rounded sum of products (plus s_i^2 on the
diagonal), known to the last bit, so S_ij carries the tile's error alone.  The leading columns
are one chunk (its update of the next chunk's columns, K = width) or two merged ones (K = twice
that, one exponent per row).

Tolerance, in units of the rows' scales 2^(e_i + e_j): for uniform digits and K = 128 the omitted
slice pairs p + q >= 7 have a standard deviation of sqrt(6 K) 2^16 / 12 2^-70 = 2^-52.8, the
entries' rounding at 2^-56 sqrt(2 K / 3) / sqrt(3) 2^-56 = 2^-53.6, the rounding of the
sum, below 8, to 53 bits 2^-51.8: 2^-51.0 in all, and eight times that for the largest of
50,000 entries.  A digit lost (2^-48 of a row's scale) is 2^-46.6."""
import numpy as np
import pytest

import paper_2202_09288_gb300 as P
from paper_2202_09288_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 2.0 ** -48


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def exact_products(b):
    """b b^T in integers: (sums, bits) with every sum exact at 2^-bits."""
    bits = 120
    m, e = np.frexp(b)
    ints = np.array([[int(v) << int(s) if s >= 0 else int(v) >> int(-s) for v, s in zip(mr, sr)]
                     for mr, sr in zip((m * 2.0 ** 53).astype(np.int64), e.astype(np.int64) - 53 + bits)],
                    dtype=object)
    return ints @ ints.T, 2 * bits


# width: columns of a chunk; chunks: of the identity block; grade: the second half of the columns
# smaller by that many binary orders; scale: rows of B over that many
@pytest.mark.parametrize("width,chunks,u,grade,scale", [
    (64, 2, 300, 0, 0), (64, 1, 300, 0, 0), (64, 2, 257, 0, 30), (64, 2, 300, 25, 0), (40, 2, 200, 0, 0),
    (24, 2, 160, 0, 20)])
@pytest.mark.parametrize("owner", [False, True])
def test_entries(torch, width, chunks, u, grade, scale, owner):
    k, n = width * chunks, width * chunks + u
    b = inputs.uniform(width + u, 13, u * k).reshape(u, k)
    b[:, k // 2:] *= 2.0 ** -grade
    s = np.ldexp(1.0, np.round(scale * inputs.uniform(u, 14, u)).astype(np.int64))
    b = b * s[:, None]
    sums, bits = exact_products(b)
    c = np.zeros((u, u))
    d = np.zeros((u, u))  # C - the exact sum, off the diagonal
    for i in range(u):
        for j in range(i + 1):
            c[i, j] = np.ldexp(float(sums[i, j] >> 40), 40 - bits)
            m, e = np.frexp(c[i, j])
            d[i, j] = np.ldexp(float((int(m * 2.0 ** 53) << (int(e) - 53 + bits)) - sums[i, j]), -bits)
        c[i, i] += s[i] ** 2
    full = np.zeros((n, n))
    full[:k, :k] = np.eye(k)
    full[k:, :k], full[k:, k:] = b, c
    colptr = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    A = inputs.SpdMatrix(n, colptr, np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32),
                         np.concatenate([full[j:, j] for j in range(n)]), (), 1)
    ctx = P.Context(width_cap=width,
                    assembly=P.CHOL_ASSEMBLY_OWNER if owner else P.CHOL_ASSEMBLY_ATOMIC)
    sym = P.Symbolic(ctx, A, np.arange(n, dtype=np.int32))
    num = P.Factor(ctx, sym, A.vals)
    assert num.status()[0] == P.CHOL_OK
    lp, _, lx = num.export()
    L = np.zeros((n, n))
    for j in range(n):
        L[j:, j] = lx[lp[j]:lp[j + 1]]
    assert np.array_equal(L[k:, :k], b)
    S = L[k:, k:] * s[None, :]
    e = np.exp2(np.frexp(np.abs(b).max(axis=1))[1].astype(float))
    err = np.abs(np.tril(S - d, -1)) / np.outer(e, e)
    assert err.max() <= TOL, np.log2(err.max())
