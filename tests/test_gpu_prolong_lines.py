"""The line prolongation (csrc/prolong.cuh) at its edges: every coarse line
length, mixes with axes too short for it, real and complex lines, batches.
The transfer of the oracle is the reference."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1504_02891_gb300 as G  # noqa: E402

SHAPES = [((32,), "fourier"), ((512,), "fourier"), ((16,), "sine"), ((256,), "sine"), ((64, 32), "fourier"),
          ((16, 64), "fourier"), ((128, 16), "sine"), ((8, 32), "sine"), ((32, 16, 64), "fourier"),
          ((8, 32, 32), "fourier"), ((16, 32, 64), "sine"), ((32, 16, 8), "sine")]


def _pad(u, axis, n, disc):
    """Spectral interpolation to twice the mesh along one axis in plain numpy (float64)."""
    u = np.moveaxis(u, axis, -1)
    if disc == "sine":
        m, f = np.arange(1, n), np.arange(1, 2 * n)
        fwd = np.sin(np.pi / n * (np.outer(m, m) % (2 * n))) * (2.0 / n)
        out = u @ fwd @ np.sin(np.pi / (2 * n) * (np.outer(m, f) % (4 * n)))
    else:
        w = np.fft.fft(u, axis=-1) * 2.0
        p = np.zeros(u.shape[:-1] + (2 * n,), complex)
        p[..., : n // 2] = w[..., : n // 2]
        p[..., 2 * n - n // 2 + 1:] = w[..., n // 2 + 1:]
        p[..., n // 2] = p[..., 2 * n - n // 2] = 0.5 * w[..., n // 2]
        out = np.fft.ifft(p, axis=-1)
        out = out if np.iscomplexobj(u) else out.real
    return np.moveaxis(out, -1, axis)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("prec,tol", [(G.F32, 2e-5), (G.F64, 1e-12)])
@pytest.mark.parametrize("n,disc", SHAPES)
def test_prolongation_matches_padded_spectrum(n, disc, prec, tol, cplx):
    d, nb = len(n), 2
    box = dict(beta=10.0, is_complex=cplx)
    pc = W.problem(d, n, (-8.0,) * d, (8.0,) * d, disc, **box)
    pf = W.problem(d, tuple(2 * v for v in n), (-8.0,) * d, (8.0,) * d, disc, **box)
    dt = np.complex128 if cplx else np.float64
    f32 = np.complex64 if cplx else np.float32
    psi = np.stack([W.random_field(pc, seed=5 + i) for i in range(nb)]).astype(f32 if prec == G.F32 else dt)
    with G.Plan(pc, nbatch=nb, prec=prec) as coarse, G.Plan(pf, nbatch=nb, prec=prec) as fine:
        out = coarse.prolong_to(fine, G.to_device(psi, prec)).cpu().numpy().astype(dt)
    for b in range(nb):
        u = psi[b].astype(dt)
        for a in range(d):
            u = _pad(u, d - 1 - a, n[a], disc)
        u = W.normalise(pf, u)
        assert np.max(np.abs(out[b] - u)) <= tol * np.max(np.abs(u))
        assert abs(O.norm2(O.build_grid(pf), out[b]) - 1.0) <= tol
