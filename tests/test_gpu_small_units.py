"""Meshes in units so small that the clip's thresholds leave FP32's range: the
decisions (which polygons are dropped, which vertices merge) are those of the
same mesh in ordinary units.  A power of two times all coordinates moves no
rounding, so the flags are equal and the blocks are that power's square.
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


def _specks(power):
    """One slave element; masters of 1e-9 .. 1e-5 of its size at its centre, on
    both sides of the least area (1e-14 of the slave's), and slivers of the merge distance."""
    xm, cm = [], []
    for k, d in enumerate(np.geomspace(1e-9, 1e-5, 17)):
        for w in (d, 1e-10, 3e-10):
            cm.append(len(xm) + np.arange(4))
            xm += [[0.5 + 0.3 * d + a * d, 0.5 - 0.2 * d + b * w, 0.0] for a, b in ((-1, -1), (1, -1), (1, 1), (-1, 1))]
    f = 2.0 ** power
    return inputs.Interface("specks", f * inputs.grid_nodes(1, 1), inputs.grid_quad4(1, 1), 4, f * np.array(xm),
                            np.array(cm, np.int32), 4, lm=0, delta=f * 1e-9)


@pytest.mark.parametrize("power", [-30, -40, -50, -60, -70])
def test_decisions_do_not_depend_on_the_unit(mt, power):
    out = []
    for p in (0, power):
        itf = _specks(p)
        m = mt.Mortar(lm=0, delta=itf.delta)
        m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
        m.evaluate()
        M, _, flag = m.pair_blocks()
        m.weighted_gap_grad(np.ones_like(itf.xs))
        out.append((m.pairs(), flag, M, m.pair_blocks()[2]))
    (p0, f0, M0, g0), (p1, f1, M1, g1) = out
    assert np.array_equal(p0[1], p1[1])
    assert 0 < f0.sum() < f0.size
    assert np.array_equal(f0, f1) and np.array_equal(g0, g1) and np.array_equal(f0, g0)
    assert np.array_equal(np.ldexp(M1, -2 * power), M0)
