"""Chains of entry points without a wait between them.  Their kernels are
launched as programmatic dependents, so each is resident while the one ahead
still writes the very buffers it reads; every buffer is written again in every
turn.  The chain must give the bits of the same calls with a wait after each."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1504_02891_gb300 as G  # noqa: E402

CASES = [
    # disc, n, complex, precision, batch: two line kernels, fused kernel, axis kernels, float32 passes, stencil
    ("fourier", (128, 64), True, G.F64, 1),
    ("fourier", (512, 512), False, G.F32, 2),
    ("fourier", (64, 64), True, G.F32, 20),
    ("sine", (64, 64, 32), False, G.F64, 1),
    ("sine", (128, 128, 128), False, G.F64, 1),
    ("fourier", (64, 32, 32), True, G.F32, 2),
    ("fourier", (256,), False, G.F32, 3),
    ("fd", (50, 41, 33), True, G.F64, 2),
    ("fd", (90, 70), False, G.F32, 1),
]


def _run(p, prec, nb, wait):
    with G.Plan(p, nbatch=nb, prec=prec) as plan:
        rng = np.random.default_rng(5)
        shape = ((nb,) if nb > 1 else ()) + plan.shape
        a = rng.standard_normal(shape)
        if p["is_complex"]:
            a = a + 1j * rng.standard_normal(shape)
        a /= np.sqrt(plan.h_vol * np.sum(np.abs(a) ** 2) / nb)
        psi = [torch.from_numpy(a).to(plan.dtype).cuda(), plan.empty()]
        h, d = plan.empty(), plan.empty()
        done = torch.cuda.synchronize if wait else (lambda: None)
        done()
        for k in range(12):
            x, y = psi[k & 1], psi[1 - (k & 1)]
            plan.grad(x, out=h)
            done()
            plan.feasible_step(x, h, 1e-3, out=y)     # y is the next turn's psi
            done()
            plan.hessvec(y, h, 0.5, out=d)            # psi just written, direction just read
            done()
            plan.feasible_step(y, d, 1e-4, out=x)     # and written again
            done()
            plan.hessvec(x, d, -0.5, out=h)
            done()
        torch.cuda.synchronize()
        return [t.cpu() for t in (*psi, h, d)]


@pytest.mark.parametrize("disc,n,cplx,prec,nb", CASES)
def test_chain_is_the_waited_chain(disc, n, cplx, prec, nb):
    dim = len(n)
    p = W.problem(dim, n, (-8.0,) * dim, (8.0,) * dim, disc, beta=50.0, is_complex=cplx)
    for a, b in zip(_run(p, prec, nb, False), _run(p, prec, nb, True)):
        assert torch.equal(a, b) and torch.isfinite(torch.view_as_real(a) if cplx else a).all()
