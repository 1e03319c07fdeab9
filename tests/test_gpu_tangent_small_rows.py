"""Linearisation where a pair touches a slave element near one of its corners.

There the shape function of the opposite node, and with it that node's row of
K, is small; every row is compared with its own largest entry.  A factor
1 -+ xi of size d is known to 2^-53 / d of itself (the back-projected point, in
the reference and in the kernel), and a reverse sweep is a few dozen roundings:
64 2^-53 / d.
"""
import numpy as np
import pytest

from paper_2202_03933_gb300 import inputs

pytestmark = pytest.mark.gpu

QUAD = np.array([[0.0, 0.0, 0.0], [1.1, 0.1, 0.05], [1.0, 1.2, 0.0], [-0.1, 0.9, 0.03]])
TRI = np.array([[0.0, 0.0, 0.0], [1.1, 0.1, 0.05], [0.2, 1.2, 0.0]])


@pytest.fixture(scope="module")
def mt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_03933_gb300 import build, mortar
    build()
    return mortar


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("xs", [QUAD, TRI], ids=["quad4", "tri3"])
@pytest.mark.parametrize("d", [0.3, 0.1, 0.03, 0.01, 0.003])
def test_rows_of_far_nodes(mt, orc, d, xs, d_domain):
    n = xs.shape[0]
    for corner in range(n):
        for seed in (1, 2, 3):
            rng = np.random.default_rng(seed)
            xm = xs[corner] + d * np.array([[a, b, 0.02 * rng.standard_normal()]
                                            for a, b in ((-1.3, -1.0), (1.2, -1.1), (1.0, 1.3), (-1.0, 0.9))])
            itf = inputs.Interface("corner", xs, np.arange(n, dtype=np.int32)[None], n, xm,
                                   np.array([[0, 1, 2, 3]], np.int32), 4, lm=0, delta=0.2)
            ys, ym = rng.uniform(-1, 1, xs.shape), rng.uniform(-1, 1, xm.shape)
            if d_domain == 0:
                ys[:] = 0.0   # the element's D has no small rows
            m = mt.Mortar(lm=0, d_domain=d_domain, delta=itf.delta)
            m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
            m.evaluate()
            s, mm = m.pairs()
            assert m.pair_blocks()[2].all()
            rp, ci, v = m.tangent(ys, ym)
            rrp, rci, rv = orc.tangent(itf, s, mm, ys, ym, orc.make_opts(lm=0, d_domain=d_domain, delta=itf.delta))
            assert np.array_equal(rp, rrp) and np.array_equal(ci, rci)
            for i in range(n):
                row = slice(rp[i], rp[i + 1])
                assert np.abs(v[row] - rv[row]).max() <= 64 * 2.0 ** -53 / d * np.abs(rv[row]).max(), (corner, seed, i)
