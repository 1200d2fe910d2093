"""Lines built against the partial sums of the fixed-point line operator
(csrc/fixfft.cuh): the pure Nyquist line, and lines that align with the symbol's
partial sum over every F/n-th frequency, with rotation of either sign.  An
overflow in any stage would be an error of the size of the values."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_point import LD, _apply, _kernel

pytestmark = pytest.mark.gpu
OMEGA = 4.0   # |a| = |c| of the symbol a p^2 + c p within the box for up to 1024 points


def _problem(n, cplx):
    return W.problem(2, n, (-16.0, -16.0), (16.0, 16.0), "fourier", beta=100.0, omega=OMEGA if cplx else 0.0,
                     is_complex=cplx)


def _lines(p, kind):
    """Complex x-lines, one per row (real grids: one per pair of rows), of entries at most 1 in size."""
    F, rows = p["n"][0], p["n"][1] if p["is_complex"] else p["n"][1] // 2
    m = np.arange(F)
    if kind == "nyquist":
        return np.tile((-1.0) ** m, (rows, 1)) * np.exp(1j * np.arange(rows))[:, None]
    freq = np.where(m < F // 2, m, m - F)
    lam = 2 * np.pi * freq / 32.0
    y = W.axis_nodes(p, 1)
    out = np.zeros((rows, F), complex)
    steps = [n for n in (4, 8, 64, 512, F) if n <= F]
    for j in range(rows):
        sym = 0.5 * lam ** 2 + (OMEGA * y[j] * lam if p["is_complex"] else 0.0)
        n = steps[j % len(steps)]
        # the offset that holds the Nyquist frequency, then others
        C = np.arange((j // len(steps)) % (F // n), F, F // n)
        K = np.exp(-2j * np.pi * np.outer(m, C) / F) @ sym[C]
        out[j] = np.conj(K) / (np.max(np.abs(K)) if kind == "kernel" else np.maximum(np.abs(K), 1e-300))
    return out


@pytest.mark.parametrize("kind", ["nyquist", "kernel", "phase"])
@pytest.mark.parametrize("n,cplx", [((32, 32), True), ((64, 128), True), ((128, 64), False), ((256, 64), True),
                                    ((512, 128), True), ((1024, 64), True), ((1024, 128), False)])
def test_partial_sums_do_not_overflow(n, cplx, kind):
    """The bound of test_against_extended_precision: 2^-52 of (largest value) x (sum over the axes of the largest
    symbol), and the rounding of the parts in float64."""
    p = _problem(n, cplx)
    x = _lines(p, kind)
    f = x if cplx else np.stack([x.real, x.imag], axis=1).reshape(n[1], n[0])
    out = _apply(p, np.ascontiguousarray(f))
    om = OMEGA if cplx else 0.0
    xs = [W.axis_nodes(p, a) for a in range(2)]
    ks = [_kernel(N, 32.0) for N in n]
    lmax = [np.pi * N / 32.0 for N in n]
    bound = 2.0 ** -52 * np.max(np.abs(f)) * sum(l * l / 2 + om * 16.0 * l for l in lmax)
    bound += 2.0 ** -50 * np.max(np.abs(out))
    rng = np.random.default_rng(3)
    fr, fi = np.real(f).astype(LD), np.imag(f).astype(LD)
    for _ in range(40):
        j, i = int(rng.integers(n[1])), int(rng.integers(n[0]))
        re = im = LD(0)
        for a, (lr, li, at) in enumerate(((fr[j], fi[j], i), (fr[:, i], fi[:, i], j))):
            t2, c, s = (k[(at - np.arange(n[a])) % n[a]] for k in ks[a])
            re, im = re + np.sum(t2 * lr), im + np.sum(t2 * li)
            w = LD(om) * (LD(xs[1][j]) if a == 0 else -LD(xs[0][i]))
            re, im = re + w * np.sum(c * lr - s * li), im + w * np.sum(c * li + s * lr)
        v = LD(0.5) * (LD(xs[0][i]) ** 2 + LD(xs[1][j]) ** 2)
        assert abs(LD(np.real(out[j, i])) - (re + v * fr[j, i])) <= bound
        assert abs(LD(np.imag(out[j, i])) - (im + v * fi[j, i])) <= bound
