"""Fixed-point quadrature at the edges of its range, against the oracle.

A pair runs in fixed point when its elements are within a factor 2^6 in size
and its polygon fits; others run in FP64.  The cases lie on both sides of that
line and at the group sizes (32 pairs) of the kernels.  Tolerances: the
parity tolerances of the FP64 path (1e-12 of the matrix, rows and entries as in
gpu_util), since either path rounds at the FP64 level at most.
"""
import numpy as np
import pytest

from paper_2202_03933_gb300 import inputs
from gpu_util import forward_parity, grad_parity, grad_sensitivity, grad_term_scale

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_03933_gb300 import build, mortar
    build()
    return mortar


def _scaled(itf, f, shift=0.0):
    itf.xs, itf.xm = itf.xs * f + shift, itf.xm * f + shift
    itf.delta *= f
    return itf


def _corner_master(nm, part):
    """One slave element against a fine master mesh over a corner of it."""
    itf = inputs.planar_noisy(1, nm, 0, 77, "corner")
    itf.xm = itf.xm * part
    return itf


def _both_noisy(ns, nm, lm, seed):
    itf = inputs.planar_noisy(ns, nm, lm, seed, "both")
    itf.xs = inputs.perturb_grid_inplane(itf.xs, ns, 0.1 / ns, seed, 7)
    return itf


CASES = {
    "one_pair": lambda: inputs.planar_noisy(1, 1, 0, 71, "one", noise=0.0),
    "one_to_many": lambda: inputs.planar_noisy(1, 5, 1, 72, "otm"),
    "pairs_32": lambda: inputs.planar_noisy(4, 2, 0, 73, "p32", noise=0.0),
    "ratio_20": lambda: inputs.planar_noisy(40, 2, 1, 74, "r20", noise=0.0),
    "ratio_20_small_master": lambda: inputs.planar_noisy(2, 40, 0, 75, "r20m"),
    "ratio_150_beyond_limit": lambda: inputs.planar_noisy(150, 1, 1, 76, "r150", noise=0.0),
    "ratio_75_small_master": lambda: _corner_master(6, 0.08),
    "both_distorted": lambda: _both_noisy(14, 13, 1, 78),
    "both_distorted_std": lambda: _both_noisy(9, 16, 0, 79),
    "tiny_units": lambda: _scaled(_both_noisy(7, 6, 0, 80), 2.0 ** -40),
    "huge_units": lambda: _scaled(_both_noisy(7, 6, 1, 81), 2.0 ** 40),
    "tri_both": lambda: _tri_both(),
    "kite": lambda: inputs.kite_master(12, 10, 0.47, lm=1),
}


def _tri_both():
    a, b = inputs.mixed_tri(4, 9, seed=5), inputs.mixed_tri(4, 8, seed=6, angle_deg=0.0, offset=(0.0, 0.0))
    return inputs.Interface("tt", b.xm, b.conn_m, 3, a.xm, a.conn_m, 3, lm=0, delta=1e-9)


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_forward_at_the_edges(mt, orc, name, d_domain):
    itf = CASES[name]()
    o = orc.make_opts(lm=itf.lm, d_domain=d_domain, delta=itf.delta)
    ref = orc.evaluate(itf, o, search="bruteforce")
    m = mt.Mortar(lm=itf.lm, d_domain=d_domain, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    assert np.array_equal(s, ref.s) and np.array_equal(mm, ref.m)
    assert np.array_equal(m.pair_blocks()[2], ref.nonempty)

    def again(x):
        r = orc.evaluate(x, o, pairs=(ref.s, ref.m))
        return r.D, r.M
    forward_parity(m.scipy(mt.MATRIX_D), m.scipy(mt.MATRIX_M), ref.D, ref.M, again, itf)
    st = m.stats()
    assert st["n_gauss_points"] == ref.stats["gauss_points"] and st["n_nonempty"] == ref.stats["nonempty"]


# multipliers: ordinary, none, and far from 1 in size
LAMBDA = {"one_pair": 1.0, "one_to_many": 1e-30, "pairs_32": 0.0, "both_distorted": 1e30}


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_adjoint_at_the_edges(mt, orc, name, d_domain):
    itf = CASES[name]()
    lam = LAMBDA.get(name, 1.0) * np.random.default_rng(11).uniform(-1, 1, itf.xs.shape)
    m = mt.Mortar(lm=itf.lm, d_domain=d_domain, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    J, gs, gm = m.weighted_gap_grad(lam)
    s, mm = m.pairs()
    o = orc.make_opts(lm=itf.lm, d_domain=d_domain, delta=itf.delta)
    _, rs, rm = orc.weighted_gap_grad(itf, lam, s, mm, o)
    if not lam.any():
        assert J == 0.0 and not gs.any() and not gm.any()
        return
    scale = grad_term_scale(orc, itf, lam, s, mm, o)
    grad_parity(gs, gm, rs, rm, scale, lambda: grad_sensitivity(orc, itf, lam, s, mm, o))


@pytest.mark.parametrize("kind,ns,nm", [("quad8", 1, 1), ("quad8", 3, 17), ("quad8", 20, 1), ("quad8", 45, 1),
                                        ("tri6", 1, 1), ("tri6", 3, 17), ("tri6", 20, 1)])
def test_quadratic_at_the_edges(mt, orc, kind, ns, nm):
    itf = inputs.quadratic_planar(ns, nm, kind, warp=0.2, name="qe")
    o = orc.make_opts(lm=0, d_domain=0, delta=itf.delta)
    ref = orc.evaluate(itf, o, search="bruteforce")
    m = mt.Mortar(lm=0, d_domain=0, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    assert np.array_equal(s, ref.s) and np.array_equal(mm, ref.m)
    assert np.array_equal(m.pair_blocks()[2], ref.nonempty)

    def again(x):
        r = orc.evaluate(x, o, pairs=(ref.s, ref.m))
        return r.D, r.M
    forward_parity(m.scipy(mt.MATRIX_D), m.scipy(mt.MATRIX_M), ref.D, ref.M, again, itf)


def _tri_slave(seed):
    a = inputs.mixed_tri(5, 6, seed=seed)
    return inputs.Interface("ts", a.xm, a.conn_m, 3, a.xs, a.conn_s, 4, lm=1, delta=a.delta)


# element-based: rules on both sides of the FP64 lines (12 on quad4, 8 on tri3),
# elements with more pairs than a chunk (12), sizes beyond 2^6, units
ELEMENT = {
    "n1": (lambda: inputs.planar_noisy(6, 5, 0, 90, "e1"), 1),
    "n12": (lambda: _both_noisy(5, 6, 1, 91), 12),
    "n13": (lambda: _both_noisy(5, 6, 1, 92), 13),
    "tri_n8": (lambda: _tri_slave(3), 8),
    "tri_n9": (lambda: _tri_slave(4), 9),
    "tri_both_n7": (lambda: _tri_both(), 7),
    "affine_masters": (lambda: inputs.planar_noisy(33, 27, 0, 93, "ea", noise=0.0), 8),
    "many_pairs": (lambda: _both_noisy(3, 11, 1, 94), 8),
    "mixed_counts": (lambda: _both_noisy(7, 13, 0, 95), 5),
    "beyond_ratio": (lambda: inputs.planar_noisy(140, 1, 0, 96, "er", noise=0.0), 2),
    "kite": (lambda: inputs.kite_master(9, 7, 0.47, lm=1), 8),
    "tiny_units": (lambda: _scaled(_both_noisy(7, 6, 1, 97), 2.0 ** -40), 8),
    "huge_units": (lambda: _scaled(_both_noisy(7, 6, 0, 98), 2.0 ** 40), 8),
}


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("name", list(ELEMENT))
def test_element_based_at_the_edges(mt, orc, name, d_domain):
    make, n = ELEMENT[name]
    itf = make()
    m = mt.Mortar(lm=itf.lm, d_domain=d_domain, delta=itf.delta, integration=mt.INTEGRATE_ELEMENT, element_rule_n=n)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    o = orc.make_opts(lm=itf.lm, d_domain=d_domain, delta=itf.delta)
    D, M, _, fl = orc.evaluate_element_based(itf, n, o, pairs=(s, mm))
    assert np.array_equal(m.pair_blocks()[2], fl)
    forward_parity(m.scipy(mt.MATRIX_D), m.scipy(mt.MATRIX_M), D, M,
                   lambda x: orc.evaluate_element_based(x, n, o, pairs=(s, mm))[:2], itf)
    assert m.stats()["n_nonempty"] == int(fl.sum())
