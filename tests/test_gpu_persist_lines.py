"""The persistent float32 Algorithm 1 launch with line transforms
(csrc/persist_lines.cuh): the same ground state as with per-iteration launches
at the edges of its line lengths and line kinds, and an expired barrier wait
that ends in an error and leaves the plan usable."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1504_02891_gb300 as G  # noqa: E402


def _problem(n, disc, cplx):
    d = len(n)
    return W.problem(d, n, (-8.0,) * d, (8.0,) * d, disc, beta=100.0, omega=0.1 if cplx else 0.0, is_complex=cplx,
                     potential={"kind": "harmonic", "gamma": (1.0, 1.2, 1.5)[:d]})


@pytest.mark.parametrize("n,disc,cplx", [((32, 32), "sine", False), ((256, 256), "sine", False),
                                         ((256, 256), "fourier", True), ((512, 512), "fourier", False),
                                         ((32, 32, 32), "sine", False), ((64, 64, 64), "fourier", False),
                                         ((64, 64, 64), "fourier", True)])
def test_same_state_as_per_iteration_launches(n, disc, cplx):
    """Both runs refine to ||H psi - mu psi||_h <= 1e-9: energies agree to 1e-11 and states to the residual over the
    smallest excitation (about 1), and the oracle finds the residual."""
    p = _problem(n, disc, cplx)
    g = O.build_grid(p)
    out = []
    for persistent in (1, 0):
        with G.Plan(p) as plan:
            t = G.to_device(W.gaussian(p, dtype=None))
            rep = plan.solve(t, mode=1, levels=1, res_tol=1e-9, delta_stop=1e-14, persistent=persistent, cluster=0)
            assert rep["status"] == 0, rep
            out.append((rep["E"], t.cpu().numpy()))
    (Ea, a), (Eb, b) = out
    assert abs(Ea - Eb) <= 1e-11 * abs(Eb)
    a = a * np.exp(-1j * np.angle(np.vdot(b, a))) if cplx else a
    assert np.linalg.norm(a - b) <= 2e-8 * np.linalg.norm(b)
    h = O.apply_hlin(g, b) + g.beta * np.abs(b) ** 2 * b
    mu = g.h_vol * np.real(np.vdot(b, h))
    assert np.sqrt(g.h_vol) * np.linalg.norm(h - mu * b) <= 1.5e-9


def test_expired_wait_then_solve_succeeds():
    p = _problem((32, 32, 32), "sine", False)
    with G.Plan(p) as plan:
        t = G.to_device(W.gaussian(p))
        G.set_wait_limit(1)
        try:
            with pytest.raises(G.GPEError) as ei:
                plan.solve(t, mode=1, levels=1, res_tol=1e-9)
            assert ei.value.status == G.ETIMEOUT
        finally:
            G.set_wait_limit(0)
        t = G.to_device(W.gaussian(p))
        rep = plan.solve(t, mode=1, levels=1, res_tol=1e-9)
    assert rep["status"] == 0
