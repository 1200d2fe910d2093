"""The per-axis line kernels of 1D, 3D and sine grids (csrc/lines3.cuh) against
the oracle: every line length, mixes with axes too short for them, packed line
pairs without a partner, odd row lengths, batches."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1504_02891_gb300 as G  # noqa: E402

SHAPES = [((32,), "fourier"), ((1024,), "fourier"), ((16,), "sine"), ((512,), "sine"), ((32, 64), "fourier"),
          ((16, 32), "fourier"), ((256, 16), "sine"), ((8, 64), "sine"), ((32, 32, 32), "fourier"),
          ((64, 16, 128), "fourier"), ((8, 32, 64), "fourier"), ((64, 8, 8), "fourier"), ((16, 32, 64), "sine"),
          ((32, 8, 16), "sine"), ((8, 16, 16), "sine"), ((64, 128, 16), "sine"), ((16, 16, 256), "fourier")]


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("prec,tol", [(G.F32, 2e-5), (G.F64, 1e-12)])
@pytest.mark.parametrize("n,disc", SHAPES)
def test_operator_matches_oracle(n, disc, prec, tol, cplx):
    d, nb = len(n), 3
    omega = 0.5 if cplx and d > 1 and disc == "fourier" else 0.0
    p = W.problem(d, n, (-8.0,) * d, (8.0, 7.0, 6.0)[:d], disc, beta=50.0, omega=omega, is_complex=cplx,
                  potential={"kind": "harmonic", "gamma": (1.0, 1.2, 1.5)[:d]})
    g = O.build_grid(p)
    dt = np.complex128 if cplx else np.float64
    f32 = np.complex64 if cplx else np.float32
    psi, dd = (np.stack([W.random_field(p, seed=s + i) for i in range(nb)]).astype(f32 if prec == G.F32 else dt)
               for s in (1, 11))
    with G.Plan(p, nbatch=nb, prec=prec) as plan:
        tp, td = G.to_device(psi, prec), G.to_device(dd, prec)
        out, (E, mu) = plan.grad(tp, with_energy=True)
        hv = plan.hessvec(tp, td, 0.25)
        out, hv = out.cpu().numpy().astype(dt), hv.cpu().numpy().astype(dt)
    for b in range(nb):
        x, e = psi[b].astype(dt), dd[b].astype(dt)
        ref = O.apply_hlin(g, x) + g.beta * np.abs(x) ** 2 * x
        assert np.max(np.abs(out[b] - ref)) <= tol * np.max(np.abs(ref))
        assert abs(E[b] - O.energy(g, x)) <= tol * abs(E[b])
        ref = O.apply_hlin(g, e) + g.beta * (np.abs(x) ** 2 * e + 2 * np.real(np.conj(x) * e) * x) + 0.25 * e
        assert np.max(np.abs(hv[b] - ref)) <= tol * np.max(np.abs(ref))


# A batch of more than two waves of line groups per device: float64 x-kernels
# then load the epilogue's operands after the transforms, and a CTA of the
# float32 2D y-kernel takes several groups.  The arithmetic of a point does not
# depend on the batch: the same bits as one instance alone.
@pytest.mark.parametrize("n,disc,cplx,prec,nb", [
    ((32, 32, 32), "fourier", False, G.F64, 97), ((32, 32, 32), "fourier", True, G.F64, 49),
    ((16, 16, 16), "sine", False, G.F64, 401), ((64,), "fourier", True, G.F64, 2603),
    ((512,), "fourier", False, G.F64, 1601), ((64, 128), "fourier", True, G.F32, 401),
    ((128, 64), "fourier", False, G.F32, 801)])
def test_large_batches_repeat_single_instances(n, disc, cplx, prec, nb):
    d = len(n)
    p = W.problem(d, n, (-8.0,) * d, (8.0, 7.0, 6.0)[:d], disc, beta=50.0, omega=0.5 if cplx and d > 1 else 0.0,
                  is_complex=cplx, potential={"kind": "harmonic", "gamma": (1.0, 1.2, 1.5)[:d]})
    psi = G.to_device(np.stack([W.random_field(p, seed=s % 7) * (1.0 + 0.01 * s) for s in range(nb)]), prec)
    dd = G.to_device(np.stack([W.random_field(p, seed=20 + s % 5) for s in range(nb)]), prec)
    with G.Plan(p, nbatch=nb, prec=prec) as plan:
        out, hv = plan.grad(psi), plan.hessvec(psi, dd, 0.25)
    with G.Plan(p, nbatch=1, prec=prec) as plan:
        for b in (0, 1, nb // 2, nb - 1):
            assert torch.equal(out[b], plan.grad(psi[b:b + 1].contiguous()).reshape(out[b].shape))
            assert torch.equal(hv[b], plan.hessvec(psi[b:b + 1].contiguous(), dd[b:b + 1].contiguous(), 0.25).reshape(hv[b].shape))
