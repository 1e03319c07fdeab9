"""Statistics of gradient runs whose pairs leave the fixed-point kernels.

A pair can leave them twice: the clip kernel keeps it for FP64 (sizes far
apart, maps out of range), or the cell kernel hands it back (a point of a
strongly distorted element did not settle).  Either way it is counted once.
The counts are whole numbers and equal the oracle's.  The kites' corner angles
approach 180 degrees as d -> 0.5; their Jacobian at that corner is about
2 (1 - 2 d) of the centre's.  Needles that cross at an angle are what the cell
kernel hands back; on them the counts are those of the forward run, whose clip
takes the same decisions.
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


CASES = {
    "kite_470": lambda: inputs.kite_master(12, 10, 0.47, lm=1),
    "kite_490": lambda: inputs.kite_master(12, 10, 0.49, lm=1),
    "kite_495": lambda: inputs.kite_master(13, 10, 0.495, lm=0),
    "kite_499": lambda: inputs.kite_master(12, 11, 0.499, lm=1),
    "kite_4995": lambda: inputs.kite_master(12, 11, 0.4995, lm=0),
    "ratio_75": lambda: inputs.planar_noisy(75, 1, 1, 76, "r75", noise=0.0),
    "ratio_75_distorted": lambda: inputs.planar_noisy(1, 75, 0, 77, "r75d"),
}


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_counts_of_a_gradient_run(mt, orc, name, d_domain):
    itf = CASES[name]()
    lam = np.random.default_rng(12).uniform(-1, 1, itf.xs.shape)
    m = mt.Mortar(lm=itf.lm, d_domain=d_domain, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.weighted_gap_grad(lam)
    st = m.stats()
    ref = orc.evaluate(itf, orc.make_opts(lm=itf.lm, d_domain=d_domain, delta=itf.delta), search="bruteforce")
    assert (st["n_nonempty"], st["n_cells"], st["n_gauss_points"]) == \
        (ref.stats["nonempty"], ref.stats["cells"], ref.stats["gauss_points"])


def _needles(aspect, angle, noise, lm):
    """Distorted grids of 1 : aspect elements, the master's turned by angle."""
    def grid(n, seed):
        x = inputs.perturb_grid_inplane(inputs.grid_nodes(n, n, -0.5, -0.5, 0.5, 0.5), n, noise / n, seed, 3)
        return x * np.array([1.0, 1.0 / aspect, 0.0])
    xs, xm = grid(30, 5), grid(27, 6)
    c, s = np.cos(angle), np.sin(angle)
    xm = xm @ np.array([[c, s, 0.0], [-s, c, 0.0], [0.0, 0.0, 1.0]])
    return inputs.Interface("needles", xs, inputs.grid_quad4(30, 30), 4, xm, inputs.grid_quad4(27, 27), 4, lm=lm,
                            delta=1e-9)


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("aspect,angle,noise,lm", [(100, 0.02, 0.4, 1), (100, 0.6, 0.4, 0), (1000, 0.003, 0.3, 1),
                                                   (1000, 0.1, 0.4, 1), (10000, 0.0005, 0.3, 0)])
def test_counts_on_crossing_needles(mt, aspect, angle, noise, lm, d_domain):
    itf = _needles(aspect, angle, noise, lm)
    m = mt.Mortar(lm=lm, d_domain=d_domain, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    ref = m.stats()
    m.weighted_gap_grad(np.random.default_rng(13).uniform(-1, 1, itf.xs.shape))
    st = m.stats()
    assert ref["n_nonempty"] > 0
    for k in ("n_pairs", "n_nonempty", "n_cells", "n_gauss_points", "n_newton_fail", "n_clip_overflow"):
        assert st[k] == ref[k], k
