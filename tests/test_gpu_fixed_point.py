"""The float64 line operator in 64-bit fixed point (csrc/fixfft.cuh) against
circulant sums in extended precision, at the edges of its line lengths and
input ranges."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def _kernel(F, L):
    """(1/F) sum_p lam_p^2/2 e^{2 pi i p m/F} (real part) and (1/F) sum_p lam_p e^{...}: the circulant rows of the
    kinetic and the first-derivative symbol, p = -F/2 .. F/2-1 (the Nyquist mode at -F/2)."""
    p = np.array([k if k < F // 2 else k - F for k in range(F)]).astype(LD)
    lam = 2 * PI * p / LD(L)
    ang = 2 * PI / LD(F) * np.arange(F).astype(LD)
    ct, st = np.cos(ang), np.sin(ang)
    idx = np.outer(np.arange(F), np.arange(F)) % F
    return (ct[idx] @ (lam * lam / 2)) / F, (ct[idx] @ lam) / F, (st[idx] @ lam) / F


def _field(p, kind, seed=3):
    rng = np.random.default_rng(seed)
    shape = W.array_shape(p)
    r2 = sum(x * x for x in W._mesh(p))
    if kind == "smooth":
        f = np.exp(-r2 / 8)
    elif kind == "noise":
        f = rng.standard_normal(shape)
    else:   # one large value above a small state
        f = 1e-3 * np.exp(-r2)
        f[tuple(s // 3 for s in shape)] = 1.0
    if p["is_complex"]:
        f = f * np.exp(1j * (0.3 * W._mesh(p)[0] + 0.01 * rng.standard_normal(shape)))
    return np.broadcast_to(f, shape).copy()


def _apply(p, f):
    """H_lin f (the Hessian at psi = 0)."""
    import torch
    import paper_1504_02891_gb300 as G
    with G.Plan(p) as plan:
        t = G.to_device(f)
        return plan.hessvec(torch.zeros_like(t), t, 0.0).cpu().numpy()


def _problem(n, omega=0.0, cplx=False):
    d = len(n)
    return W.problem(d, n, (-16.0,) * d, (16.0,) * d, "fourier", beta=100.0, omega=omega, is_complex=cplx)


@pytest.mark.parametrize("kind", ["smooth", "noise", "spike"])
@pytest.mark.parametrize("n,omega,cplx", [((64, 64), 0.0, False), ((128, 256), 0.6, True), ((512, 64), 0.0, False),
                                          ((64, 1024), 0.9, True), ((1024, 512), 0.9, True)])
def test_against_extended_precision(n, omega, cplx, kind):
    """Errors below 2^-52 of (largest value) x (sum over the axes of the largest symbol): a unit of the spectrum is
    2^-61 of a line's L1 norm (at most 2 F max), it is rounded a few times, and the inverse transform averages F such
    errors down by sqrt(F)."""
    p = _problem(n, omega, cplx)
    f = _field(p, kind)
    out = _apply(p, f)
    xs = [W.axis_nodes(p, a) for a in range(2)]
    ks = [_kernel(N, 32.0) for N in n]
    lmax = [np.pi * N / 32.0 for N in n]
    bound = 2.0 ** -52 * np.max(np.abs(f)) * sum(l * l / 2 + omega * 16.0 * l for l in lmax)
    # V f and the sum of the parts are rounded in float64 too
    bound += 2.0 ** -50 * np.max(np.abs(out))
    rng = np.random.default_rng(7)
    fr, fi = np.real(f).astype(LD), np.imag(f).astype(LD)
    for _ in range(40):
        j, i = int(rng.integers(n[1])), int(rng.integers(n[0]))
        re = im = LD(0)
        for a, (lr, li, at) in enumerate(((fr[j], fi[j], i), (fr[:, i], fi[:, i], j))):
            t2, c, s = (k[(at - np.arange(n[a])) % n[a]] for k in ks[a])
            re, im = re + np.sum(t2 * lr), im + np.sum(t2 * li)
            w = LD(omega) * (LD(xs[1][j]) if a == 0 else -LD(xs[0][i]))
            re, im = re + w * np.sum(c * lr - s * li), im + w * np.sum(c * li + s * lr)
        v = LD(0.5) * (LD(xs[0][i]) ** 2 + LD(xs[1][j]) ** 2)
        re, im = re + v * fr[j, i], im + v * fi[j, i]
        assert abs(LD(np.real(out[j, i])) - re) <= bound
        assert abs(LD(np.imag(out[j, i])) - im) <= bound


@pytest.mark.parametrize("n,cplx", [((64, 128), False), ((512, 256), True)])
def test_scale_zero_and_nonfinite_lines(n, cplx):
    """Powers of two scale exactly (the level of a line is its own), zero stays zero, and a NaN or an infinity reaches
    its own row and column and nothing else."""
    p = _problem(n, 0.0, cplx)
    f = _field(p, "smooth")
    f[3, :] = 0.0
    ref = _apply(p, f)
    for e in (-600, 700):
        np.testing.assert_array_equal(_apply(p, f * 2.0 ** e), ref * 2.0 ** e)
    assert not np.any(_apply(p, np.zeros_like(f)))
    for bad in (np.nan, np.inf):
        g = f.copy()
        g[10, 20] = bad
        out = _apply(p, g)
        fin = np.isfinite(out)
        assert not fin[10, :].any() and not fin[:, 20].any()
        # a real grid packs two rows (and columns) into one line: the partner shares the line
        rows = [10] if cplx else [10, 11]
        cols = [20] if cplx else [20, 21]
        fin[rows, :] = True
        fin[:, cols] = True
        assert fin.all()
