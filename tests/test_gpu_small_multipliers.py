"""Gradient for multipliers far below and above FP32's range: J and both gradients
are linear in the multipliers, so a power of two times the multipliers gives
that power of two times the results.  Multipliers of different size meet in one
pair's forms, which may then take another path: 1e-12 of the largest entry, the
bound of either path.
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
@pytest.mark.parametrize("power", [-300, -200, -160, -130, -100, 100, 130, 300])
def test_linear_in_the_multipliers(mt, power, d_domain):
    itf = inputs.planar_noisy(9, 8, 1, 91, "small")
    itf.xs = inputs.perturb_grid_inplane(itf.xs, 9, 0.1 / 9, 91, 7)
    lam = np.random.default_rng(14).uniform(-1, 1, itf.xs.shape)
    lam[::3] = 0.0
    m = mt.Mortar(lm=1, d_domain=d_domain, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    J, gs, gm = m.weighted_gap_grad(lam)
    J2, gs2, gm2 = m.weighted_gap_grad(np.ldexp(lam, power))
    scale = max(np.abs(gs).max(), np.abs(gm).max())
    assert np.abs(np.ldexp(gs2, -power) - gs).max() <= 1e-12 * scale
    assert np.abs(np.ldexp(gm2, -power) - gm).max() <= 1e-12 * scale
    assert abs(np.ldexp(J2, -power) - J) <= 1e-12 * scale
