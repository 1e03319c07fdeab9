"""Stretched elements, and elements that overlap by a sliver.

The pair kernels hold a pair's in-plane coordinates in a frame with one
exponent for each direction, and scale shape functions that stay small over a
pair; both have to hold whatever the aspect and however thin the overlap.

Blocks of axis-parallel rectangles are products of two integrals of products of
linear functions, taken here from the nodes in extended precision.  Bound of an
entry: n elements of size h = 1/n on a side hold their parameters to about
d = 4 n 2^-53 in either arithmetic (two rounded end points, two rounded plane
coordinates), which moves an integral of a factor f by d / f of itself where f
is small, and the overlap of w elements by d / w of itself; and a few dozen
rounded products and sums, 1e-14.  A thin overlap of 1e-4 element widths has
factors of 1e-4.
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


def _grid(n, aspect, along, shift=(0.0, 0.0), noise=0.0, seed=1):
    """n x n grid of the unit square moved by `shift` elements, then squeezed to 1 : aspect along axis `along`."""
    x = inputs.grid_nodes(n, n)
    if noise:
        x = inputs.perturb_grid_inplane(x, n, noise / n, seed, 5)
    x[:, :2] += np.asarray(shift) / n
    x[:, along] /= aspect
    return x


def _interface(n, aspect, along, shift, lm=0, noise=0.0):
    xs, xm = _grid(n, aspect, along, noise=noise, seed=2), _grid(n, aspect, along, shift, noise, 3)
    return inputs.Interface("stretched", xs, inputs.grid_quad4(n, n), 4, xm, inputs.grid_quad4(n, n), 4, lm=lm,
                            delta=1e-12)


def _hat_integrals(s0, s1, m0, m1):
    """[[int Na Nl]] of the linear functions of the intervals s and m over their
    overlap, the largest values of each there, and the overlap."""
    s0, s1, m0, m1 = (np.longdouble(v) for v in (s0, s1, m0, m1))
    a, b = max(s0, m0), min(s1, m1)
    f = lambda x0, x1, x: ((x1 - x) / (x1 - x0), (x - x0) / (x1 - x0))
    sa, sb, ma, mb = f(s0, s1, a), f(s0, s1, b), f(m0, m1, a), f(m0, m1, b)
    I = [[(b - a) / 6 * (sa[i] * (2 * ma[j] + mb[j]) + sb[i] * (2 * mb[j] + ma[j])) for j in (0, 1)] for i in (0, 1)]
    top = lambda p, q: [max(p[k], q[k]) for k in (0, 1)]
    return I, top(sa, sb), top(ma, mb), b - a


@pytest.mark.parametrize("thin", [0.3, 1e-4])
@pytest.mark.parametrize("along", [0, 1])
@pytest.mark.parametrize("aspect", [1, 30, 1000, 60000, 100000])
def test_rectangles(mt, aspect, along, thin):
    n = 6
    shift = (0.4, thin) if along == 1 else (thin, 0.4)
    itf = _interface(n, aspect, along, shift)
    m = mt.Mortar(lm=0, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    blocks, flags = m.pair_blocks()[0], m.pair_blocks()[2]
    assert flags.sum() >= (n - 1) ** 2
    corner = ((0, 0), (1, 0), (1, 1), (0, 1))
    d = 4 * n * 2.0 ** -53
    for p in np.flatnonzero(flags):
        S, M = itf.xs[itf.conn_s[s[p]]], itf.xm[itf.conn_m[mm[p]]]
        ix, sx, mx, wx = _hat_integrals(S[0, 0], S[1, 0], M[0, 0], M[1, 0])
        iy, sy, my, wy = _hat_integrals(S[0, 1], S[3, 1], M[0, 1], M[3, 1])
        for a, (ax, ay) in enumerate(corner):
            for l, (lx, ly) in enumerate(corner):
                ref = ix[ax][lx] * iy[ay][ly]
                moved = d * ref * ((S[1, 0] - S[0, 0]) / wx + (S[3, 1] - S[0, 1]) / wy)
                moved += d * wx * wy * ((sx[ax] + mx[lx]) * sy[ay] * my[ly] + (sy[ay] + my[ly]) * sx[ax] * mx[lx])
                assert abs(blocks[p][a][l] - ref) <= 1e-14 * ref + moved, (p, a, l, float(ref), blocks[p][a][l])


@pytest.mark.parametrize("d_domain", [0, 1])
@pytest.mark.parametrize("thin", [0.3, 1e-4])
@pytest.mark.parametrize("aspect,along,noise", [(30, 1, 0.0), (30, 1, 0.15), (30, 0, 0.0), (30, 0, 0.15), (1000, 1, 0.0),
                                                (1000, 1, 0.15), (100000, 1, 0.0), (100000, 1, 0.15), (100000, 0, 0.0)])
def test_against_the_oracle(mt, orc, aspect, along, thin, noise, d_domain):
    itf = _interface(6, aspect, along, (0.4, thin) if along == 1 else (thin, 0.4), lm=1, noise=noise)
    lam = np.random.default_rng(21).uniform(-1, 1, itf.xs.shape)
    o = orc.make_opts(lm=1, d_domain=d_domain, delta=itf.delta)
    ref = orc.evaluate(itf, o, search="bruteforce")
    m = mt.Mortar(lm=1, d_domain=d_domain, delta=itf.delta)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    assert np.array_equal(s, ref.s) and np.array_equal(mm, ref.m)
    assert np.array_equal(m.pair_blocks()[2], ref.nonempty)

    def again(x):
        r = orc.evaluate(x, o, pairs=(ref.s, ref.m))
        return r.D, r.M
    forward_parity(m.scipy(mt.MATRIX_D), m.scipy(mt.MATRIX_M), ref.D, ref.M, again, itf)
    J, gs, gm = m.weighted_gap_grad(lam)
    _, rs, rm = orc.weighted_gap_grad(itf, lam, s, mm, o)
    scale = grad_term_scale(orc, itf, lam, s, mm, o)
    grad_parity(gs, gm, rs, rm, scale, lambda: grad_sensitivity(orc, itf, lam, s, mm, o))


@pytest.mark.parametrize("aspect,thin,n", [(30, 0.3, 4), (1000, 1e-4, 8), (100000, 0.3, 8), (100000, 1e-4, 5)])
def test_element_based(mt, orc, aspect, thin, n):
    itf = _interface(6, aspect, 1, (0.4, thin), lm=1, noise=0.1)
    o = orc.make_opts(lm=1, delta=itf.delta)
    m = mt.Mortar(lm=1, delta=itf.delta, integration=mt.INTEGRATE_ELEMENT, element_rule_n=n)
    m.set_interface(itf.xs, itf.conn_s, itf.xm, itf.conn_m)
    m.evaluate()
    s, mm = m.pairs()
    D, M, _, fl = orc.evaluate_element_based(itf, n, o, pairs=(s, mm))
    assert np.array_equal(m.pair_blocks()[2], fl)
    forward_parity(m.scipy(mt.MATRIX_D), m.scipy(mt.MATRIX_M), D, M,
                   lambda x: orc.evaluate_element_based(x, n, o, pairs=(s, mm))[:2], itf)
