"""Runs of more than one chunk of pairs (4 M pairs; 1 M with quadratic slaves):
quadratic slave elements against the oracle on sampled pairs of every chunk, and
the gradient with segment D against the one-pair-per-thread FP64 kernels.
"""
import numpy as np
import pytest

from paper_2202_03933_gb300 import inputs
from gpu_util import blocks_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_03933_gb300 import build, mortar
    build()
    return mortar


def test_quadratic_chunks(mt, orc):
    itf = inputs.quadratic_planar(600, 520, "quad8", warp=0.1, name="chunks")
    m = mt.Mortar(lm=0, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    chunk = 1 << 20
    assert s.size > chunk
    M, _, flag = m.pair_blocks()
    rng = np.random.default_rng(15)
    pick = np.unique(np.concatenate([rng.integers(0, s.size, 4000), rng.integers(chunk, s.size, 2000),
                                     np.arange(chunk - 40, chunk + 40), np.arange(s.size - 70, s.size)]))
    rM, rflag = orc.quadratic_pair_blocks(itf, s[pick], mm[pick], orc.make_opts(lm=0, delta=itf.delta))[:2]
    assert np.array_equal(flag[pick], np.asarray(rflag, bool))
    blocks_parity(M[pick], rM)


def test_gradient_chunks_with_segment_d(mt):
    itf = inputs.planar_noisy(1200, 1040, 1, 92, "chunks")
    lam = np.random.default_rng(16).uniform(-1, 1, itf.xs.shape)
    m = mt.Mortar(lm=1, d_domain=1, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    J, gs, gm = m.weighted_gap_grad(lam)
    st = m.stats()
    assert st["n_pairs"] > 1 << 22
    D, M = m.scipy(mt.MATRIX_D), m.scipy(mt.MATRIX_M)
    m.set_launch(variant=1)
    J1, gs1, gm1 = m.weighted_gap_grad(lam)
    st1 = m.stats()
    for k in ("n_pairs", "n_nonempty", "n_cells", "n_gauss_points"):
        assert st[k] == st1[k]
    for A, B in ((D, m.scipy(mt.MATRIX_D)), (M, m.scipy(mt.MATRIX_M))):
        assert np.array_equal(A.indptr, B.indptr) and np.array_equal(A.indices, B.indices)
        assert np.abs(A.data - B.data).max() <= 1e-12 * np.abs(B.data).max()
    # x_s and x_m cancel (coplanar surfaces); either term's gradient is lam . x d(weights)/dX, about |lam| |x| h
    scale = np.abs(lam).max() * np.abs(itf.xs).max() / 1200
    assert max(np.abs(gs - gs1).max(), np.abs(gm - gm1).max()) <= 1e-12 * scale
