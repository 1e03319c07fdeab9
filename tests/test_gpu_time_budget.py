"""A time budget that runs out in any of the pair kernels.

The kernels of a chunk hand each other an order and records; after one of them
has stopped early the later ones take no work, the call returns
MORTAR_ERR_TIMEOUT and the context stays usable.  The candidate lists are
mostly empty, so that the kernels' times differ: the clip looks at every
pair, the cell and finish kernels have next to nothing to do, and budgets
between those times stop one kernel and not the next.  A call that returns in
time gives the results of a call without a budget, bit for bit.
"""
import numpy as np
import pytest

from paper_2202_03933_gb300 import inputs

pytestmark = pytest.mark.gpu

BUDGETS = (3, 12, 30, 60, 100, 150, 220, 330, 500, 1000, 10000000)   # microseconds


@pytest.fixture(scope="module")
def mt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_03933_gb300 import build, mortar
    build()
    return mortar


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("form", ["forward", "forward_segment", "gradient", "quadratic"])
def test_budgets_between_the_kernels(mt, form):
    if form == "quadratic":
        itf, lm = inputs.quadratic_planar(40, 36, "quad8", warp=0.1, name="tb"), 0
    else:
        itf, lm = inputs.planar_noisy(110, 96, 1, 87, "tb"), 1
    dom = 1 if form == "forward_segment" else 0
    lam = np.random.default_rng(8).uniform(-1, 1, itf.xs.shape)
    m = mt.Mortar(lm=lm, d_domain=dom, delta=0.04)   # some forty candidates for each slave element
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)

    def call():
        out = list(m.weighted_gap_grad(lam)[1:]) if form == "gradient" else (m.evaluate(), [])[1]
        return out + [m.scipy(w).data for w in (mt.MATRIX_D, mt.MATRIX_M)]
    ref = call()
    timeouts = 0
    for us in BUDGETS:
        for _ in range(2):
            m.set_watchdog(us)
            try:
                got = call()
            except mt._native.MortarError as e:
                assert "TIMEOUT" in str(e)
                timeouts += 1
                continue
            assert _same(got, ref)
    assert 2 <= timeouts < 2 * len(BUDGETS)   # the least budget cannot do, the last one does
    m.set_watchdog(0)
    assert _same(call(), ref)


def test_budget_of_a_captured_run(mt):
    itf = inputs.planar_noisy(300, 260, 1, 88, "tbg")
    lam = np.random.default_rng(9).uniform(-1, 1, itf.xs.shape)
    m = mt.Mortar(lm=1, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.run_graph(lam)
    ref = list(m.gradient()[1:]) + [m.scipy(w).data for w in (mt.MATRIX_D, mt.MATRIX_M)]
    away = itf.xm + np.array([0.0, 0.0, 5.0])
    m.set_coordinates(itf.xs, away)
    m.set_watchdog(40)
    m.run_graph(lam)          # captured without pairs, within the budget
    m.set_coordinates(itf.xs, itf.xm)
    for _ in range(2):        # replayed with them
        with pytest.raises(mt._native.MortarError, match="TIMEOUT"):
            m.run_graph(lam)
    m.set_coordinates(itf.xs, away)
    m.run_graph(lam)
    assert not m.gradient()[2].any()
    m.set_watchdog(0)
    m.set_coordinates(itf.xs, itf.xm)
    for _ in range(2):
        m.run_graph(lam)
        assert _same(list(m.gradient()[1:]) + [m.scipy(w).data for w in (mt.MATRIX_D, mt.MATRIX_M)], ref)


def test_budget_of_the_linearisation(mt):
    itf = inputs.planar_noisy(120, 104, 1, 89, "tbt")
    rng = np.random.default_rng(10)
    ys, ym = rng.uniform(-1, 1, itf.xs.shape), rng.uniform(-1, 1, itf.xm.shape)
    m = mt.Mortar(lm=1, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    ref = m.tangent(ys, ym)
    m.set_watchdog(20)
    with pytest.raises(mt._native.MortarError, match="TIMEOUT"):
        m.tangent(ys, ym)
    m.set_watchdog(0)
    assert _same(m.tangent(ys, ym), ref)
