"""Rounding error of the float64 difference operator against extended precision,
point by point: the bound of a stencil that is formed axis by axis from small
differences.  (Taking the neighbours from one large diagonal product costs two
to three times as much.)"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _problem(n, cplx):
    d = len(n)
    return W.problem(d, n, (-2.0,) * d, (2.0,) * d, "fd", beta=10.0, is_complex=cplx)


def _field(p, kind):
    rng = np.random.default_rng(11)
    xs = W._mesh(p)
    f = np.exp(-sum((x - 0.1) ** 2 for x in xs)) if kind == "smooth" else rng.standard_normal(W.array_shape(p))
    if p["is_complex"]:
        f = f * np.exp(1j * (0.7 * xs[0] + (rng.standard_normal(W.array_shape(p)) if kind == "noise" else 0.0)))
    return np.broadcast_to(f, W.array_shape(p)).copy()


def exact_and_bound(p, f):
    """H_lin f in extended precision (real f) and the bound, in units of 2^-53: for every axis the rounding of the sum of
    the neighbours (half of |sum|) and of the difference from it, both times 1/h^2, then one rounding per addition to
    the sum over the axes and for V f (V itself: four)."""
    g = f.astype(LD)
    lin, err = LD(0) * g, LD(0) * g
    for a in range(p["dim"]):
        h = (p["hi"][a] - p["lo"][a]) / p["n"][a]
        c = LD(1.0 / (h * h))
        ax = f.ndim - 1 - a
        pad = [(1, 1) if i == ax else (0, 0) for i in range(f.ndim)]
        q = np.pad(g, pad)
        n = f.shape[ax]
        t = np.take(q, range(0, n), ax) + np.take(q, range(2, n + 2), ax)
        d = g - t / 2
        lin = lin + c * d
        err = err + c * (abs(t) / 2 + abs(d)) + abs(lin)
    v = sum(LD(0.5) * x.astype(LD) ** 2 for x in W._mesh(p)) * g
    lin = lin + v
    return lin, err + 4 * abs(v) + abs(lin)


@pytest.mark.parametrize("kind", ["smooth", "noise"])
@pytest.mark.parametrize("n,cplx", [((400,), False), ((90, 71), True), ((64, 50, 41), False), ((33, 40, 27), True)])
def test_fd_operator_rounding(n, cplx, kind):
    import torch
    import paper_1504_02891_gb300 as G
    p = _problem(n, cplx)
    f = _field(p, kind)
    with G.Plan(p) as plan:
        t = G.to_device(f)
        out = plan.hessvec(torch.zeros_like(t), t, 0.0).cpu().numpy()
    for part in ((np.real, np.imag) if cplx else (np.real,)):
        ref, err = exact_and_bound(p, part(f))
        # one per cent for the products of two roundings
        assert np.all(abs(part(out).astype(LD) - ref) <= LD(1.01) * LD(2.0) ** -53 * err)
