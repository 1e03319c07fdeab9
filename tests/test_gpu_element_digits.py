"""Element-based integration: entries made of a rule's smallest products.

A small master over a corner point of the n x n rule owns that point alone, so
a block's entries are single products W N_a N_l, the smallest of them
w_n^2 (1 - x_n)^2 / 4 of the element's weight (2^-17 at n = 8, 2^-22 at n = 12).
Every entry is as accurate relative to itself as FP64 gives it.  In units of
2^-53 / (1 - x_n): a factor 1 -+ x_n is rounded to one, there are two of them in
N_a, two weights 2 / ((1 - x_n^2) P_n'^2) with two each, all that in the
reference and in the kernel; 16 in all with the rounded products, twice as much
where both factors are the slave's (D).
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("tri", [False, True])
@pytest.mark.parametrize("n", [8, 10, 12])
def test_corner_points(mt, orc, n, tri, d_domain):
    x, w = np.polynomial.legendre.leggauss(n)
    gap = 0.5 * (x[-1] - x[-2])
    size = min(0.9 * gap, 0.05)      # half a master's side: the neighbouring points stay outside
    xm, cm = [], []
    for cx, cy in ((x[0], x[0]), (x[-1], x[0]), (x[-1], x[-1]), (x[0], x[-1])):
        c = np.array([0.5 * (cx + 1.0), 0.5 * (cy + 1.0), 0.0])
        corners = ((-0.9, -0.8), (1.1, -0.8), (-0.9, 1.2)) if tri else ((-1, -1), (1, -1.1), (1.1, 1), (-1, 0.9))
        cm.append([len(xm) + k for k in range(len(corners))])
        xm += [c + 0.5 * size * np.array([*p, 0.0]) for p in corners]
    itf = inputs.Interface("corners", inputs.grid_nodes(1, 1), inputs.grid_quad4(1, 1), 4, np.array(xm),
                           np.array(cm, np.int32), 3 if tri else 4, lm=0, delta=1e-9)
    m = mt.Mortar(lm=0, d_domain=d_domain, delta=itf.delta, integration=mt.INTEGRATE_ELEMENT, element_rule_n=n)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    M, D, flags = m.pair_blocks(with_D=d_domain == 1)
    assert flags.all() and m.stats()["n_gauss_points"] == 4
    s, mm = m.pairs()
    rM, rD, _ = orc.element_based_blocks(itf, s, mm, n, orc.make_opts(lm=0, d_domain=d_domain, delta=itf.delta))
    tol = 16 * 2.0 ** -53 / (1.0 - x[-1])
    nm = 3 if tri else 4
    assert (np.abs(M - rM)[:, :, :nm] <= tol * np.abs(rM)[:, :, :nm]).all(), np.nanmax(np.abs(M / rM - 1)[:, :, :nm])
    if d_domain == 1:
        assert (np.abs(D - rD) <= 2 * tol * np.abs(rD)).all()
