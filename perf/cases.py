"""Performance cases of the mortar library: what a user's program has it do.

Every case is one call sequence of the public binding (``Mortar`` and
``integrate_pairs_static``) on a synthetic interface of the families in
``paper_2202_03933_gb300.inputs``: planar grids with in-plane node noise, a
cylinder patch with a rough master, rotated grids of random triangles,
batches of uneven interfaces and serendipity slave elements.  Meshes are made
on the GPU from the seed; the context (``Mortar``) is the handle a program
keeps over the steps of a simulation.  Passes that a simulation repeats with
moved nodes upload the coordinates in every pass.

Operations (``op``):

* ``step``     search, integration, assembly of D and M, and the gradient of the
               weighted gap: one evaluation of a nonlinear iteration.  ``graph``:
               replayed as a CUDA graph, gradient read to the host; otherwise the
               eager call with device outputs.
* ``forward``  search, integration and assembly only (``graph`` as above).
* ``tangent``  the consistent linearisation as a 3x3-block sparse matrix.
* ``element``  element-based integration (n x n points per slave element).
* ``contact``  nodal normals, weighted gap, active set and residual.
* ``static``   per-pair blocks through the no-allocation entry point.

``exact`` restates the method in plain FP64 torch (search, clip, quadrature,
dual basis; gradients by automatic differentiation) without this package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2202_03933_gb300 import inputs, mortar

LM = {"standard": mortar.LM_STANDARD, "dual": mortar.LM_DUAL}
DOMAIN = {"element": mortar.D_ELEMENT, "segment": mortar.D_SEGMENT}
NEN = {"quad4": 4, "tri3": 3, "quad8": 8}
_GAP = 1e-4   # largest gap of a batch's interfaces, and their search inflation


def _case(op, mesh, ns, nm, slave="quad4", master="quad4", lm="dual", domain="element", slave_noise=0.0,
          noise=0.1, graph=False, rule=0, count=1):
    return {"op": op, "mesh": mesh, "ns": ns, "nm": nm, "slave": slave, "master": master, "lm": lm,
            "domain": domain, "slave_noise": slave_noise, "noise": noise, "graph": graph, "rule": rule,
            "count": count}


def listed():
    cases = {
        # the smallest interface of the benchmark: launches and latency
        "planar_8x7_step": _case("step", "planar", 8, 7, lm="standard", graph=True),
        # a pair list of a caller that may not allocate, in one small call
        "static_64x56": _case("static", "planar", 64, 56),
        # curved contact surface with a rough counterpart, one iteration's evaluation
        "cylinder_200x173_step": _case("step", "cylinder", 200, 173, graph=True),
        # hexahedra against tetrahedra: quad4 slave, tri3 master
        "mixed_300x400_step": _case("step", "planar", 300, 400, master="tri3", lm="standard", noise=0.0, graph=True),
        # many uneven interfaces of one model, integrated as one batch
        "batched_128_step": _case("step", "batch", 128, 128, lm="standard", noise=0.0, graph=True, count=128),
        # meshtying set-up on unstructured meshes: both sides distorted, D over the covered part
        "planar_600x520_forward_segment": _case("forward", "planar", 600, 520, lm="standard", domain="segment",
                                                slave_noise=0.1),
        # a large sliding interface, re-searched and re-integrated every step
        "planar_1000x866_forward": _case("forward", "planar", 1000, 866, graph=True),
        # the benchmark's workload, the largest: 14.9 M pairs with the gradient
        "planar_2000x1733_step": _case("step", "planar", 2000, 1733),
        # Newton matrix of a nonlinear iteration on distorted meshes
        "tangent_300x260": _case("tangent", "planar", 300, 260, slave_noise=0.1),
        # the cheap rule for early iterations
        "element_600x520_n8": _case("element", "planar", 600, 520, rule=8),
        # higher-order slave elements
        "quad8_450x390_forward": _case("forward", "planar", 450, 390, slave="quad8", lm="standard"),
        # contact iteration on a triangulated surface: terms of the active-set strategy
        "contact_tri3_300x347": _case("contact", "planar", 300, 347, slave="tri3", slave_noise=0.1),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def draw(rng):
    """One more case: sizes log-uniform, mesh ratios 0.7 to 1.3, options as listed."""
    op = rng.choice(["step", "step", "step", "forward", "forward", "tangent", "element", "contact", "static"])
    hi = {"step": 1600, "forward": 1600, "tangent": 400, "element": 800, "contact": 800, "static": 90}[op]
    ns = int(round(math.exp(rng.uniform(math.log(8), math.log(hi)))))
    nm = max(3, int(round(ns * rng.uniform(0.7, 1.3))))
    mesh = "planar" if op == "static" else rng.choice(["planar", "planar", "planar", "cylinder"])
    c = _case(op, mesh, ns, nm, lm=rng.choice(["standard", "dual"]), graph=op in ("step", "forward") and rng.random() < 0.5)
    if mesh == "planar":
        c["slave_noise"] = rng.choice([0.0, 0.1])
        c["noise"] = rng.choice([0.05, 0.1, 0.15])
        c["slave"] = rng.choice(["quad4", "quad4", "tri3"])
        c["master"] = rng.choice(["quad4", "quad4", "tri3"])
        # two triangles a square: as many pairs on a coarser grid
        f = 0.7 ** ((c["slave"] == "tri3") + (c["master"] == "tri3"))
        c["ns"], c["nm"] = max(5, int(ns * f)), max(3, int(nm * f))
    if op in ("step", "forward", "tangent"):
        c["domain"] = rng.choice(["element", "element", "segment"])
    if op == "element":
        c["rule"] = rng.choice([4, 8])
    if op == "forward" and mesh == "planar" and rng.random() < 0.3:
        c.update(slave="quad8", lm="standard", domain="element", ns=min(c["ns"], 600), nm=min(c["nm"], 600))
    if op == "step" and rng.random() < 0.25:
        c.update(mesh="batch", slave="quad4", master="quad4", lm="standard", domain="element", noise=0.0,
                 slave_noise=0.0, graph=True, ns=min(max(ns, 16), 128), nm=min(max(ns, 16), 128), count=rng.randint(8, 200))
    return c


# ------------------------------------------------------------------ meshes
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grid(n, dev):
    t = torch.arange(n + 1, dtype=torch.float64, device=dev) / n
    y, x = torch.meshgrid(t, t, indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), torch.zeros_like(x).reshape(-1)], 1).contiguous()


def _quads(n, dev):
    j, i = torch.meshgrid(torch.arange(n, device=dev), torch.arange(n, device=dev), indexing="ij")
    a = (j * (n + 1) + i).reshape(-1)
    return torch.stack([a, a + 1, a + n + 2, a + n + 1], 1)


def _uniform(shape, gen, dev):
    return 2.0 * torch.rand(shape, dtype=torch.float64, device=dev, generator=gen) - 1.0


def _jitter(x, n, amp, gen):
    """In-plane node noise of +-amp h; nodes on the square's edges stay on them."""
    if amp == 0.0:
        return x
    d = _uniform((x.shape[0], 2), gen, x.device) * (amp / n)
    ids = torch.arange(x.shape[0], device=x.device)
    i, j = ids % (n + 1), ids // (n + 1)
    x = x.clone()
    x[:, 0] += torch.where((i > 0) & (i < n), d[:, 0], 0.0)
    x[:, 1] += torch.where((j > 0) & (j < n), d[:, 1], 0.0)
    return x


def _triangles(q, gen):
    flip = (torch.rand(q.shape[0], device=q.device, generator=gen) < 0.5)[:, None]
    a = torch.where(flip, q[:, [0, 1, 3]], q[:, [0, 1, 2]])
    b = torch.where(flip, q[:, [1, 2, 3]], q[:, [0, 2, 3]])
    return torch.stack([a, b], 1).reshape(-1, 3)


def _cylinder(n, radius, dev):
    g = _grid(n, dev)
    th, z = 0.5 * math.pi * g[:, 0], 2.0 * g[:, 1]
    return torch.stack([radius * torch.cos(th), radius * torch.sin(th), z], 1).contiguous()


def _mesh(case, seed):
    """(xs, conn_s, xm, conn_m, delta) on the device; connectivity int32.

    The node noise and the diagonals belong to the case, so that every seed has the same sparsity; the seed
    stretches the interface, sets the gap and tilts the master in it."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(40_009 * case["ns"] + case["nm"])
    own = torch.Generator(device=dev).manual_seed(1000003 * int(seed) + 17)
    stretch = 1.0 + 0.2 * _uniform((3,), own, dev)
    ns, nm = case["ns"], case["nm"]
    if case["mesh"] == "cylinder":
        h_m = max(2.0 * math.sin(0.25 * math.pi / nm), 2.0 / nm)
        h_s = max(2.0 * math.sin(0.25 * math.pi / ns), 2.0 / ns)
        r = 1.0 + 0.01 * h_m * torch.randn((nm + 1) ** 2, dtype=torch.float64, device=dev, generator=gen)
        f = stretch[0]
        return (_cylinder(ns, 1.0, dev) * f, _quads(ns, dev).int(), _cylinder(nm, r, dev) * f, _quads(nm, dev).int(),
                0.05 * h_s * float(f))
    if case["slave"] == "quad8":
        x, c = inputs.quadratic_grid(ns, "quad8")
        xs, cs = torch.from_numpy(x).to(dev), torch.from_numpy(c).to(dev)
    else:
        xs, cs = _jitter(_grid(ns, dev), ns, case["slave_noise"], gen), _quads(ns, dev)
        if case["slave"] == "tri3":
            cs = _triangles(cs, gen)
    xm, cm = _jitter(_grid(nm, dev), nm, case["noise"], gen), _quads(nm, dev)
    if case["master"] == "tri3":   # rotated and shifted against the slave, as volumes meshed apart are
        cm = _triangles(cm, gen)
        a = math.radians(7.0)
        u, v = xm[:, 0] - 0.5, xm[:, 1] - 0.5
        xm = torch.stack([0.513 + math.cos(a) * u - math.sin(a) * v, 0.529 + math.sin(a) * u + math.cos(a) * v,
                          torch.zeros_like(u)], 1)
    # a gap of 0.005 to 0.055 h: the master lies above the slave, slightly tilted
    xm = xm.clone()
    xm[:, 2] = (0.01 + xm[:, :2] @ (0.01 + 0.01 * _uniform((2,), own, dev))) / ns
    xm[:, 2].clamp_(min=0.005 / ns, max=0.055 / ns)
    stretch[2] = 1.0
    xs, xm = xs * stretch, xm * stretch
    return xs.contiguous(), cs.int().contiguous(), xm.contiguous(), cm.int().contiguous(), 0.03 / ns


def _batch(case, seed):
    """`count` interfaces of n x n slave quads, n log-uniform in [4, ns], ratio 0.7 to 1.3, shifted."""
    rng = np.random.default_rng(seed)
    k = np.random.default_rng(case["count"])   # sizes and shifts belong to the case
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(k.uniform(math.log(4.0), math.log(case["ns"])))))
        m = max(2, int(round(n * k.uniform(0.7, 1.3))))
        dx, dy = k.uniform(-0.05, 0.05, 2)
        f = np.append(rng.uniform(0.8, 1.2, 2), 1.0)
        xm = inputs.grid_nodes(m, m, dx, dy, 1.0 + dx, 1.0 + dy)
        xm[:, 2] = _GAP * (0.5 + 0.5 * rng.random())
        out.append(inputs.Interface(f"i{i}", inputs.grid_nodes(n, n) * f, inputs.grid_quad4(n, n), 4, xm * f,
                                    inputs.grid_quad4(m, m), 4))
    return out


def _lambda(n, seed, width=3):
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(7000001 * int(seed) + 5)
    return _uniform((n, width), gen, dev)


# ------------------------------------------------------------------ the library's side
_STREAM = []


def prepare(case, seed):
    op = case["op"]
    if not _STREAM:   # one stream for all: calls of the no-allocation entry point share its scratch
        _STREAM.append(torch.cuda.Stream())
    st = {"op": op, "graph": case["graph"], "stream": _STREAM[0]}
    with torch.cuda.stream(st["stream"]):
        if op == "static":
            xs, cs, xm, cm, delta = _mesh(case, seed)
            ps, pm = _static_pairs(case)
            st.update(args=(xs, cs, xm, cm, ps.int().contiguous(), pm.int().contiguous()), lm=LM[case["lm"]],
                      domain=DOMAIN[case["domain"]], delta=delta)
            st["stream"].synchronize()
            return st
        more = {}
        if op == "element":
            more = {"integration": mortar.INTEGRATE_ELEMENT, "element_rule_n": case["rule"]}
        if case["mesh"] == "batch":
            itf = _batch(case, seed)
            m = mortar.Mortar(lm=LM[case["lm"]], d_domain=DOMAIN[case["domain"]], delta=_GAP, **more).set_batch(itf)
            dev = _device()
            xs = torch.from_numpy(np.concatenate([i.xs for i in itf])).to(dev)
            xm = torch.from_numpy(np.concatenate([i.xm for i in itf])).to(dev)
        else:
            xs, cs, xm, cm, delta = _mesh(case, seed)
            st["stream"].synchronize()
            m = mortar.Mortar(lm=LM[case["lm"]], d_domain=DOMAIN[case["domain"]], delta=delta, **more)
            m.set_interface(xs, cs, xm, cm)
        st.update(m=m, xs=xs, xm=xm)
        if op in ("step", "contact"):
            st["lam"] = _lambda(xs.shape[0], seed)
        if op == "contact":
            st["lam_n"] = st["lam"][:, 0].cpu().numpy()
        st["stream"].synchronize()
    return st


def _static_pairs(case):
    """The caller's pair list: it keeps one list while the interface is stretched."""
    xs, cs, xm, cm, delta = _mesh(case, 0)
    return _candidates(_boxes(xs, cs, delta), _boxes(xm, cm, delta))


def _csr(t):
    return [t.crow_indices(), t.col_indices(), t.values()]


def run(st):
    with torch.cuda.stream(st["stream"]):
        if st["op"] == "static":
            M, D, ne = mortar.integrate_pairs_static(*st["args"], lm=st["lm"], d_domain=st["domain"],
                                                     delta=st["delta"], stream=st["stream"].cuda_stream)
            return {"M": M, "nonempty": ne}
        m = st["m"]
        m.set_coordinates(st["xs"], st["xm"])   # the nodes have moved
        if st["op"] == "tangent":
            rp, ci, va = m.tangent(st["xs"], st["xm"], add_direct=True, out_device=True)
            return {"K": [rp, ci, va]}
        if st["op"] == "contact":
            return dict(m.contact_terms(st["lam_n"], c=50.0))
        out = {}
        if st["op"] == "step":
            if st["graph"]:
                m.run_graph(st["lam"])
                out["J"], out["gs"], out["gm"] = m.gradient()
            else:
                out["J"], out["gs"], out["gm"] = m.weighted_gap_grad(st["lam"], out_device=True)
        elif st["graph"]:
            m.run_graph()
        else:
            m.evaluate()
        out["D"] = _csr(m.torch_csr(mortar.MATRIX_D))
        out["M"] = _csr(m.torch_csr(mortar.MATRIX_M))
        return out


def _sizes(case):
    """(slave elements, slave nodes, master elements, master nodes, pairs), pairs for uniform grids."""
    if case["mesh"] == "batch":
        k = np.random.default_rng(case["count"])
        es = sn = em = mn = p = 0
        for _ in range(case["count"]):
            n = int(round(math.exp(k.uniform(math.log(4.0), math.log(case["ns"])))))
            m = max(2, int(round(n * k.uniform(0.7, 1.3))))
            k.uniform(-0.05, 0.05, 2)
            es, sn, em, mn, p = es + n * n, sn + (n + 1) ** 2, em + m * m, mn + (m + 1) ** 2, p + (n + m) ** 2
        return es, sn, em, mn, p
    ns, nm = case["ns"], case["nm"]
    es, em = ns * ns * (2 if case["slave"] == "tri3" else 1), nm * nm * (2 if case["master"] == "tri3" else 1)
    sn = (ns + 1) ** 2 + (2 * ns * (ns + 1) if case["slave"] == "quad8" else 0)
    p = (ns + nm) ** 2 * (es // (ns * ns)) * (em // (nm * nm))
    return es, sn, em, (nm + 1) ** 2, p


def work(case):
    """Inputs read once and outputs written once; FP64 operations of a pair as this method needs them
    (clip, about four cells of seven points, two element-map inversions per point, the products)."""
    es, sn, em, mn, p = _sizes(case)
    read = 24 * (sn + mn) + 4 * (NEN[case["slave"]] * es + NEN[case["master"]] * em)
    ratio = 2.0 * case["nm"] / case["ns"] + 2.0
    csr = 8 * 2 * (sn + 1) + 12 * (sn * (1 if case["lm"] == "dual" else 9) + sn * ratio * ratio)
    flops = {"step": 8500, "forward": 3000, "tangent": 35000, "element": 40 * case["rule"] ** 2 * es / p,
             "contact": 3000, "static": 3000}[case["op"]]
    if case["slave"] == "quad8":
        flops = 11000
    out = {"step": csr + 24 * (sn + mn), "forward": csr, "element": csr, "contact": 41 * sn, "static": 129 * p,
           "tangent": 76 * (9 * sn + sn * ratio * ratio)}[case["op"]]
    return {"bytes": read + out, "flops": flops * p}


# ------------------------------------------------------------------ plain FP64 restatement
_CHUNK = 400_000   # pairs per chunk
_CORNER = ((-1.0, -1.0), (1.0, -1.0), (1.0, 1.0), (-1.0, 1.0))
_G3 = math.sqrt(0.6)
_s15 = math.sqrt(15.0)


def _boxes(x, conn, delta):
    X = x[conn.long()]
    return X.amin(1) - delta, X.amax(1) + delta


def _candidates(bs, bm):
    """All (s, m) with overlapping boxes (closed), sorted, by a uniform grid of box centres."""
    size = torch.maximum((bs[1] - bs[0]).amax(0), (bm[1] - bm[0]).amax(0)) * 1.0001 + 1e-12
    org = torch.minimum(bs[0].amin(0), bm[0].amin(0))
    cell = lambda b: ((0.5 * (b[0] + b[1]) - org) / size).floor().long() + 1  # noqa: E731
    cs, cm = cell(bs), cell(bm)
    nb = torch.maximum(cs.amax(0), cm.amax(0)) + 2
    key = lambda c: (c[:, 0] * nb[1] + c[:, 1]) * nb[2] + c[:, 2]  # noqa: E731
    km, order = key(cm).sort()
    found = []
    for off in range(27):
        o = torch.tensor([off // 9 - 1, off // 3 % 3 - 1, off % 3 - 1], device=cs.device)
        k = key(cs + o)
        lo, hi = torch.searchsorted(km, k), torch.searchsorted(km, k, right=True)
        n = hi - lo
        if int(n.sum()) == 0:
            continue
        s = torch.repeat_interleave(torch.arange(cs.shape[0], device=cs.device), n)
        at = torch.arange(s.shape[0], device=s.device) - torch.repeat_interleave(n.cumsum(0) - n, n)
        m = order[torch.repeat_interleave(lo, n) + at]
        ok = ((bs[0][s] <= bm[1][m]) & (bm[0][m] <= bs[1][s])).all(1)
        found.append(torch.stack([s[ok], m[ok]]))
    p = torch.cat(found, 1)
    p = p[:, (p[0] * bm[0].shape[0] + p[1]).argsort()]
    return p[0], p[1]


def _shape(nen, xi, eta):
    if nen == 4:
        return torch.stack([0.25 * (1 + a * xi) * (1 + b * eta) for a, b in _CORNER], -1)
    if nen == 3:
        return torch.stack([1 - xi - eta, xi, eta], -1)
    N = [0.25 * (1 + a * xi) * (1 + b * eta) * (a * xi + b * eta - 1) for a, b in _CORNER]
    N += [0.5 * (1 - xi * xi) * (1 - eta), 0.5 * (1 + xi) * (1 - eta * eta), 0.5 * (1 - xi * xi) * (1 + eta),
          0.5 * (1 - xi) * (1 - eta * eta)]
    return torch.stack(N, -1)


def _tri_rule(ref):
    a, b = (6 - _s15) / 21, (6 + _s15) / 21
    wa, wb = (155 - _s15) / 1200, (155 + _s15) / 1200
    l = [(1 / 3, 1 / 3)] + [p for c in (a, b) for p in ((c, 1 - 2 * c), (1 - 2 * c, c), (c, c))]
    new = lambda v: torch.tensor(v, dtype=torch.float64, device=ref.device)  # noqa: E731
    l = new(l)
    return l[:, 0], l[:, 1], new([0.225] + 3 * [wa] + 3 * [wb])


def _element_integrals(X, nen):
    """Me = int N N^T, Dh = int N over elements X (E, nen, 3) in their own surface measure."""
    if nen == 3:
        l1, l2, w = _tri_rule(X)
        w = 0.5 * w
    else:
        g = torch.tensor([-_G3, 0.0, _G3], dtype=torch.float64, device=X.device)
        ww = torch.tensor([5 / 9, 8 / 9, 5 / 9], dtype=torch.float64, device=X.device)
        l1, l2, w = g.repeat_interleave(3), g.repeat(3), (ww[:, None] * ww).reshape(-1)
    a, b = l1.clone().requires_grad_(), l2.clone().requires_grad_()
    with torch.enable_grad():
        N = _shape(nen, a, b)
        d1 = torch.stack([torch.autograd.grad(N[:, k].sum(), a, retain_graph=True)[0] if nen > 3 else
                          torch.full_like(l1, (-1.0, 1.0, 0.0)[k]) for k in range(nen)], -1)
        d2 = torch.stack([torch.autograd.grad(N[:, k].sum(), b, retain_graph=True)[0] if nen > 3 else
                          torch.full_like(l1, (-1.0, 0.0, 1.0)[k]) for k in range(nen)], -1)
    N = N.detach()
    g1, g2 = torch.einsum("qa,eak->eqk", d1, X), torch.einsum("qa,eak->eqk", d2, X)
    wj = w * torch.linalg.cross(g1, g2).norm(dim=-1)
    return torch.einsum("eq,qa,qb->eab", wj, N, N), wj @ N


def _multipliers(X, nen, lm):
    """LM coefficients A (Phi = A N) and the element block of D."""
    Me, Dh = _element_integrals(X, nen)
    if lm == "standard":
        return None, Me
    return torch.linalg.solve(Me, torch.diag_embed(Dh)).transpose(1, 2), torch.diag_embed(Dh)


def _coeffs(p, nen):
    """Map coefficients (.., 4, 2) of x = c0 + c1 xi + c2 eta + c3 xi eta from nodes (.., nen, 2)."""
    if nen == 3:
        return torch.stack([p[..., 0, :], p[..., 1, :] - p[..., 0, :], p[..., 2, :] - p[..., 0, :],
                            torch.zeros_like(p[..., 0, :])], -2)
    s = [[1, 1, 1, 1], [-1, 1, 1, -1], [-1, -1, 1, 1], [1, -1, 1, -1]]
    return torch.einsum("ia,...ak->...ik", 0.25 * torch.tensor(s, dtype=torch.float64, device=p.device), p)


def _invert(c, x, steps=12):
    """xi with x(xi) = x for c (B, 4, 2), x (B, Q, 2): Newton, then one differentiable step."""
    def step(c, x, xi, eta):
        j0 = c[:, None, 1] + c[:, None, 3] * eta[..., None]
        j1 = c[:, None, 2] + c[:, None, 3] * xi[..., None]
        r = c[:, None, 0] + j0 * xi[..., None] + c[:, None, 2] * eta[..., None] - x
        det = j0[..., 0] * j1[..., 1] - j1[..., 0] * j0[..., 1]
        return (xi - (j1[..., 1] * r[..., 0] - j1[..., 0] * r[..., 1]) / det,
                eta - (j0[..., 0] * r[..., 1] - j0[..., 1] * r[..., 0]) / det)
    with torch.no_grad():
        xi = torch.zeros_like(x[..., 0])
        eta = torch.zeros_like(xi)
        for _ in range(steps):
            xi, eta = step(c, x, xi, eta)
    return step(c, x, xi, eta)


def _cross(a, b):
    return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]


def _plane(X, nen):
    """x0, t1, t2 of the auxiliary planes of linear elements X (E, nen, 3)."""
    if nen == 4:
        g1, g2 = 0.25 * (X[:, 1] - X[:, 0] + X[:, 2] - X[:, 3]), 0.25 * (X[:, 2] - X[:, 1] + X[:, 3] - X[:, 0])
    else:
        g1, g2 = X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]
    n = torch.linalg.cross(g1, g2)
    n = n / n.norm(dim=1, keepdim=True)
    e = X[:, 1] - X[:, 0]
    e = e - (e * n).sum(1, keepdim=True) * n
    t1 = e / e.norm(dim=1, keepdim=True)
    return X.mean(1), t1, torch.linalg.cross(n, t1)


def _project(Y, plane):
    d = Y - plane[0][:, None]
    return torch.stack([(d * plane[1][:, None]).sum(-1), (d * plane[2][:, None]).sum(-1)], -1)


def _take(v, i):
    return v.gather(1, i[..., None].expand(*i.shape, 2))


def _ccw(p):
    a = _cross(p, p.roll(-1, 1)).sum(1)
    return torch.where((a < 0)[:, None, None], p.flip(1), p), a


def _clip(ps, pm, h):
    """Clip polygons of projected slaves ps and masters pm: vertices (P, K, 2) and counts."""
    P, ns, nm = ps.shape[0], ps.shape[1], pm.shape[1]
    K = ns + nm
    eps = (1e-12 * h * h)[:, None]
    win, area = _ccw(ps)
    v = torch.cat([_ccw(pm)[0], pm.new_zeros(P, K - nm, 2)], 1)
    n = torch.full((P,), nm, device=ps.device)
    ks = torch.arange(K, device=ps.device)[None]
    for i in range(ns):
        a, e = win[:, i], win[:, (i + 1) % ns] - win[:, i]
        live = ks < n[:, None]
        nxt = torch.where(ks + 1 == n[:, None], 0, (ks + 1).clamp(max=K - 1))
        q = _take(v, nxt)
        dp, dq = _cross(e[:, None], v - a[:, None]), _cross(e[:, None], q - a[:, None])
        cut = live & (((dp > eps) & (dq < -eps)) | ((dp < -eps) & (dq > eps)))
        t = dp / torch.where(cut, dp - dq, torch.ones_like(dp))
        x = v + torch.where(cut, t, torch.zeros_like(t))[..., None] * (q - v)
        keep = live & (dq >= -eps)
        put = torch.stack([cut, keep], 2).reshape(P, 2 * K)
        at = torch.where(put, put.long().cumsum(1) - 1, K).clamp(max=K)
        both = torch.stack([x, q], 2).reshape(P, 2 * K, 2)
        v = v.new_zeros(P, K + 1, 2).scatter(1, at[..., None].expand(-1, -1, 2), both)[:, :K]
        n = put.sum(1)
    m2 = (1e-10 * h) ** 2
    idx, nr = torch.zeros((P, K), dtype=torch.long, device=ps.device), torch.zeros_like(n)
    dist = lambda a, b: ((a - b) ** 2).sum(-1)  # noqa: E731
    with torch.no_grad():
        rows = torch.arange(P, device=ps.device)
        for k in range(K):
            last = v[rows, idx[rows, (nr - 1).clamp(min=0)]]
            add = (k < n) & ((nr == 0) | ~(dist(v[:, k], last) < m2))
            idx[rows[add], nr[add]] = k
            nr = nr + add.long()
        for _ in range(K):
            last, first = v[rows, idx[rows, (nr - 1).clamp(min=0)]], v[rows, idx[:, 0]]
            nr = nr - ((nr > 1) & (dist(last, first) < m2)).long()
    v = _take(v, idx)
    live = ks < nr[:, None]
    nxt = _take(v, torch.where(ks + 1 == nr[:, None], 0, (ks + 1).clamp(max=K - 1)))
    a2 = torch.where(live, _cross(v, nxt), 0.0).sum(1)
    return v, torch.where((nr >= 3) & ~(0.5 * a2.abs() < 1e-14 * 0.5 * area.abs()), nr, 0)


def _integrals(Xs, Xm, segment, parent=None):
    """G = int N_s N_m^T, H = int N_s N_s^T over the clip polygons of element pairs (Xs, Xm), and which are
    not empty.  parent: the quadrant (P,) of a serendipity element that the linear slave element is."""
    ns, nm = Xs.shape[1], Xm.shape[1]
    h = (Xs[:, :, None] - Xs[:, None]).norm(dim=-1).amax((1, 2)).detach()
    plane = _plane(Xs, ns)
    ps, pm = _project(Xs, plane), _project(Xm, plane)
    v, n = _clip(ps, pm, h)
    K = v.shape[1]
    ks = torch.arange(K, device=v.device)[None]
    live = ks < n[:, None]
    cen = torch.where(live[..., None], v, 0.0).sum(1) / n.clamp(min=1)[:, None]
    p, k = torch.where((n == 3)[:, None], ks == 0, live).nonzero(as_tuple=True)
    tri = n[p] == 3
    a = torch.where(tri[:, None], v[p, 0], cen[p])
    b = v[p, torch.where(tri, 1, k)]
    c = v[p, torch.where(tri, 2, torch.where(k + 1 == n[p], 0, (k + 1).clamp(max=K - 1)))]
    l1, l2, w = _tri_rule(v)
    x = a[:, None] + l1[None, :, None] * (b - a)[:, None] + l2[None, :, None] * (c - a)[:, None]
    W = w * (0.5 * _cross(b - a, c - a).abs())[:, None]
    s1, s2 = _invert(_coeffs(ps, ns)[p], x, 1 if ns == 3 else 12)
    m1, m2 = _invert(_coeffs(pm, nm)[p], x, 1 if nm == 3 else 12)
    if parent is not None:
        ox = torch.tensor([-1.0, 1.0, 1.0, -1.0], dtype=torch.float64, device=v.device)[parent[p]][:, None]
        oy = torch.tensor([-1.0, -1.0, 1.0, 1.0], dtype=torch.float64, device=v.device)[parent[p]][:, None]
        s1, s2, ns = 0.5 * (s1 + ox), 0.5 * (s2 + oy), 8
    Ns, Nm = _shape(ns, s1, s2), _shape(nm, m1, m2)
    G = v.new_zeros(Xs.shape[0], ns, nm).index_add(0, p, torch.einsum("cq,cqa,cqb->cab", W, Ns, Nm))
    H = v.new_zeros(Xs.shape[0], ns, ns).index_add(0, p, torch.einsum("cq,cqa,cqb->cab", W, Ns, Ns)) if segment else None
    return G, H, n > 0


def _pair_terms(Xs, Xm, case):
    """M and (segment) D blocks of element pairs, and which are not empty."""
    G, H, live = _integrals(Xs, Xm, case["domain"] == "segment")
    if case["lm"] == "dual":
        A = _multipliers(Xs, Xs.shape[1], "dual")[0]
        G, H = A @ G, (A @ H if H is not None else None)
    return G, H, live


def _sparse(rows, cols, vals, ncol):
    """Values of the sparse matrix that sums (rows, cols, vals), in row-column order."""
    keys, at = torch.unique(rows * ncol + cols, return_inverse=True)
    out = torch.zeros((keys.shape[0],) + vals.shape[1:], dtype=torch.float64, device=vals.device)
    return keys, out.index_add(0, at, vals)


def _outer(a, b):
    return a[:, :, None].expand(-1, -1, b.shape[1]).reshape(-1), b[:, None].expand(-1, a.shape[1], -1).reshape(-1)


def _quadratic_pairs(X8, Xm):
    """M blocks (P, 8, 4) of serendipity slave elements by their four linear sub-elements."""
    c = -0.25 * X8[:, :4].sum(1) + 0.5 * X8[:, 4:].sum(1)
    X9 = torch.cat([X8, c[:, None]], 1)
    G, live = 0.0, False
    for k, sub in enumerate(((0, 4, 8, 7), (4, 1, 5, 8), (8, 5, 2, 6), (7, 8, 6, 3))):
        q = torch.full((X8.shape[0],), k, device=X8.device)
        g, _, l = _integrals(X9[:, list(sub)], Xm, False, q)
        G, live = G + g, live | l
    return G, None, live


def _element_based(xs, cs, xm, cm, ps, pm, case):
    """M blocks of the element-based rule: every point goes to the first covering master in pair order."""
    n, ns, nm = case["rule"], cs.shape[1], cm.shape[1]
    g, gw = (torch.from_numpy(t).to(xs.device) for t in np.polynomial.legendre.leggauss(n))
    xi, eta, w = g.repeat_interleave(n), g.repeat(n), (gw[:, None] * gw).reshape(-1)
    if ns == 3:
        xi, eta, w = 0.5 * (xi + 1), 0.5 * (eta + 1), 0.25 * w
        eta, w = eta * (1 - xi), w * (1 - xi)
    c = _coeffs(_project(xs[cs], _plane(xs[cs], ns)), ns)
    mono = torch.stack([torch.ones_like(xi), xi, eta, xi * eta], -1)
    x = torch.einsum("qi,eik->eqk", mono, c)
    W = w * _cross(c[:, None, 1] + c[:, None, 3] * eta[:, None], c[:, None, 2] + c[:, None, 3] * xi[:, None]).abs()
    owner = torch.full(W.shape, ps.shape[0], dtype=torch.long, device=xs.device)
    held = []
    for b in range(0, ps.shape[0], _CHUNK):
        s, m = ps[b:b + _CHUNK], pm[b:b + _CHUNK]
        plane = _plane(xs[cs[s]], ns)
        a1, a2 = _invert(_coeffs(_project(xm[cm[m]], plane), nm), x[s], 1 if nm == 3 else 12)
        lim = 1 + 1e-10
        inside = ((a1.abs() <= lim) & (a2.abs() <= lim)) if nm == 4 else \
            ((a1 >= -1e-10) & (a2 >= -1e-10) & (a1 + a2 <= lim))
        ids = torch.arange(b, b + s.shape[0], device=xs.device)[:, None]
        owner.scatter_reduce_(0, s[:, None].expand(-1, W.shape[1]), torch.where(inside, ids, ps.shape[0]), "amin")
        held.append((s, ids, a1, a2))
    N = _shape(ns, xi, eta)
    blocks, live = [], []
    for s, ids, a1, a2 in held:
        mine = owner[s] == ids
        Nm = _shape(nm, torch.where(mine, a1, 0.0), torch.where(mine, a2, 0.0))
        blocks.append(torch.einsum("pq,qa,pql->pal", torch.where(mine, W[s], 0.0), N, Nm))
        live.append(mine.any(1))
    M = torch.cat(blocks)
    if case["lm"] == "dual":
        M = _multipliers(xs[cs], ns, "dual")[0][ps] @ M
    return M, None, torch.cat(live)


def _normals(xs, cs):
    X, nen = xs[cs], cs.shape[1]
    if nen == 3:
        n = torch.linalg.cross(X[:, 1] - X[:, 0], X[:, 2] - X[:, 0])[:, None].expand(-1, 3, -1)
    else:
        d1 = torch.stack([X[:, 1] - X[:, 0], X[:, 1] - X[:, 0], X[:, 2] - X[:, 3], X[:, 2] - X[:, 3]], 1)
        d2 = torch.stack([X[:, 3] - X[:, 0], X[:, 2] - X[:, 1], X[:, 2] - X[:, 1], X[:, 3] - X[:, 0]], 1)
        n = torch.linalg.cross(d1, d2)
    n = n / n.norm(dim=-1, keepdim=True)
    s = torch.zeros_like(xs).index_add(0, cs.reshape(-1), n.reshape(-1, 3))
    return s / s.norm(dim=1, keepdim=True)


def _exact_mesh(case, seed):
    if case["mesh"] != "batch":
        xs, cs, xm, cm, delta = _mesh(case, seed)
        cs, cm = cs.long(), cm.long()
        if case["op"] == "static":
            return (xs, cs, xm, cm) + _static_pairs(case)
        return (xs, cs, xm, cm) + _candidates(_boxes(xs, cs, delta), _boxes(xm, cm, delta))
    parts, off = [], [0, 0, 0, 0]
    for i in _batch(case, seed):
        xs, cs, xm, cm = (torch.from_numpy(np.ascontiguousarray(a)).to(_device()) for a in (i.xs, i.conn_s, i.xm, i.conn_m))
        s, m = _candidates(_boxes(xs, cs, _GAP), _boxes(xm, cm, _GAP))
        parts.append((xs, cs.long() + off[0], xm, cm.long() + off[1], s + off[2], m + off[3]))
        off = [off[0] + len(xs), off[1] + len(xm), off[2] + len(cs), off[3] + len(cm)]
    return tuple(torch.cat(t) for t in zip(*parts))


def exact(case, seed):
    op = case["op"]
    xs, cs, xm, cm, ps, pm = _exact_mesh(case, seed)
    Ns, Nm, ns, nm = xs.shape[0], xm.shape[0], cs.shape[1], cm.shape[1]
    if op == "static":
        out = torch.cat([_pair_terms(xs[cs[ps[b:b + _CHUNK]]], xm[cm[pm[b:b + _CHUNK]]], case)[0]
                         for b in range(0, ps.shape[0], _CHUNK)])
        pad = out.new_zeros(ps.shape[0], 4, 4)
        pad[:, :ns, :nm] = out
        return {"M": pad, "nonempty": None}
    lam = _lambda(Ns, seed) if op in ("step", "contact") else None
    per_elem = case["domain"] == "element"
    Xe = xs[cs].requires_grad_(op in ("step", "tangent"))
    De = _multipliers(Xe, ns, case["lm"])[1] if per_elem else None
    gs, gm, J = torch.zeros_like(xs), torch.zeros_like(xm), 0.0
    K = []
    if op == "step" and per_elem:
        je = (lam[cs] * (De @ Xe)).sum()
        gs.index_add_(0, cs.reshape(-1), torch.autograd.grad(je, Xe)[0].reshape(-1, 3))
        J += float(je.detach())
    if op == "tangent" and per_elem:
        K.append(_jacobian_blocks(De @ xs[cs], [Xe], [De]) + (cs, cs))
    Ms, Ds, live = [], [], []
    for b in range(0, ps.shape[0], _CHUNK):
        s, m = ps[b:b + _CHUNK], pm[b:b + _CHUNK]
        Xs, Xm = xs[cs[s]], xm[cm[m]]
        if op == "element":
            M, D, l = _element_based(xs, cs, xm, cm, ps, pm, case)
        elif ns == 8:
            M, D, l = _quadratic_pairs(Xs, Xm)
        else:
            grad = op in ("step", "tangent")
            Xs.requires_grad_(grad), Xm.requires_grad_(grad)
            M, D, l = _pair_terms(Xs, Xm, case)
        if op == "step":
            j = ((lam[cs[s]] * ((D @ Xs if D is not None else 0.0) - M @ Xm)) * l[:, None, None]).sum()
            a, c = torch.autograd.grad(j, [Xs, Xm])
            gs.index_add_(0, cs[s].reshape(-1), a.reshape(-1, 3))
            gm.index_add_(0, cm[m].reshape(-1), c.reshape(-1, 3))
            J += float(j.detach())
        if op == "tangent":
            f = (D @ xs[cs[s]] if D is not None else 0.0) - M @ xm[cm[m]]
            k = _jacobian_blocks(f, [Xs, Xm], [D, -M])[0][l]
            K.append((k, cs[s][l], torch.cat([cs[s], cm[m] + Ns], 1)[l]))
        Ms.append(M.detach()), live.append(l)
        Ds.append(D.detach() if D is not None else None)
        if op == "element":
            break
    if op == "tangent":
        rows, cols = zip(*(_outer(r, c) for _, r, c in K))
        _, v = _sparse(torch.cat(rows), torch.cat(cols), torch.cat([k.reshape(-1, 3, 3) for k, _, _ in K]), Ns + Nm)
        return {"K": [None, None, v]}
    live = torch.cat(live)
    sl, ml = cs[ps[live]], cm[pm[live]]
    M = _sparse(*_outer(sl, ml), torch.cat(Ms)[live].reshape(-1), Nm)
    if not per_elem:
        D = _sparse(*_outer(sl, sl), torch.cat(Ds)[live].reshape(-1), Ns)
    elif case["lm"] == "dual":
        D = _sparse(cs.reshape(-1), cs.reshape(-1), De.detach().diagonal(dim1=1, dim2=2).reshape(-1), Ns)
    else:
        D = _sparse(*_outer(cs, cs), De.detach().reshape(-1), Ns)
    if op == "contact":
        n = _normals(xs, cs)
        v = torch.zeros_like(xs).index_add_(0, D[0] // Ns, D[1][:, None] * xs[D[0] % Ns])
        v.index_add_(0, M[0] // Nm, -M[1][:, None] * xm[M[0] % Nm])
        gap = -(n * v).sum(1)
        t = lam[:, 0] + 50.0 * gap
        return {"normals": n, "gap": gap, "active": None, "ncp": lam[:, 0] - t.clamp(max=0.0)}
    out = {"D": [None, None, D[1]], "M": [None, None, M[1]]}
    if op == "step":
        out.update(J=J, gs=gs, gm=gm)
    return out


def _jacobian_blocks(f, xs, direct):
    """(P, rows, cols, 3, 3) derivatives of f (P, rows, 3) by the nodes in xs, plus direct (x) I3."""
    got = []
    for a in range(f.shape[1]):
        for c in range(3):
            g = torch.autograd.grad(f[:, a, c].sum(), xs, retain_graph=True)
            got.append(torch.cat(g, 1))
    k = torch.stack(got, 1).reshape(f.shape[0], f.shape[1], 3, -1, 3).transpose(2, 3)
    d = torch.cat([t if t is not None else torch.zeros(f.shape[0], f.shape[1], f.shape[1], dtype=f.dtype, device=f.device)
                   for t in direct], 2).detach()
    return (k + d[..., None, None] * torch.eye(3, dtype=f.dtype, device=f.device),)
