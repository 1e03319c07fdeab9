"""Matrix rows with more columns than the assembly's accumulators hold (32 in D,
64 in M): collected in windows of 64 columns.  Coarse slaves on fine masters
have rows of a few hundred columns in M, coarse slave fans long rows in D; the
lengths lie on both sides of a window's ends.  The assembled matrices equal the
pair blocks' sums: the same columns, and values summed in pair order, so to the
last bit where the sum is formed in that order.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2202_03933_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_03933_gb300 import build, mortar
    build()
    return mortar


def _sums(rows, cols, vals):
    """{(row, col): sum in order}"""
    out = {}
    for r, c, v in zip(rows, cols, vals):
        out[(r, c)] = out[(r, c)] + v if (r, c) in out else v
    return out


def _check(A: sp.csr_matrix, want):
    got = {(r, c): v for r, (b, e) in enumerate(zip(A.indptr, A.indptr[1:])) for c, v in zip(A.indices[b:e], A.data[b:e])}
    assert all(np.all(np.diff(A.indices[b:e]) > 0) for b, e in zip(A.indptr, A.indptr[1:]))
    assert got == want


def _fan(n):
    """n triangles about one node, a fan of unit radius."""
    t = 2 * np.pi * np.arange(n) / n
    x = np.vstack([[0.0, 0.0, 0.0], np.c_[np.cos(t), np.sin(t), np.zeros(n)]])
    return x, np.array([[0, 1 + k, 1 + (k + 1) % n] for k in range(n)], np.int32)


@pytest.mark.parametrize("nm", [6, 7, 8, 15, 22])
def test_rows_of_m(mt, nm):
    itf = inputs.planar_noisy(1, nm, 0, 31, "long")
    m = mt.Mortar(lm=0, d_domain=1, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    M, _, flag = m.pair_blocks(with_D=True)
    p = np.flatnonzero(flag)
    rows = itf.conn_s[s[p]][:, :, None].repeat(4, 2).ravel()
    cols = itf.conn_m[mm[p]][:, None, :].repeat(4, 1).ravel()
    A = m.scipy(mt.MATRIX_M)
    assert max(np.diff(A.indptr)) == (nm + 1) ** 2
    _check(A, _sums(rows, cols, M[p].ravel()))


@pytest.mark.parametrize("n", [31, 32, 62, 63, 64, 100, 127, 128, 200])
def test_rows_of_d(mt, n):
    x, c = _fan(n)
    xm = np.array([[-2.0, -2.0, 0.0], [2.0, -2.0, 0.0], [2.0, 2.0, 0.0], [-2.0, 2.0, 0.0]])
    m = mt.Mortar(lm=0, d_domain=1, delta=1e-9)
    m.set_interface(x, c, xm, np.array([[0, 1, 2, 3]], np.int32))
    m.evaluate()
    s, _ = m.pairs()
    _, D, flag = m.pair_blocks(with_D=True)
    p = np.flatnonzero(flag)
    rows = c[s[p]][:, :, None].repeat(3, 2).ravel()
    cols = c[s[p]][:, None, :].repeat(3, 1).ravel()
    A = m.scipy(mt.MATRIX_D)
    assert max(np.diff(A.indptr)) == n + 1
    _check(A, _sums(rows, cols, D[p][:, :3, :3].ravel()))
