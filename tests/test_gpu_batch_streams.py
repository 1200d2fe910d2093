"""gpe_solve_batch with other streams at work: its groups and refinement lanes
run on streams of their own, so everything they read (cleared counters, tables,
potentials on their way from host memory) has to be in place whatever the
default stream and the caller's stream are doing."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1504_02891_gb300 as G  # noqa: E402


def _problems():
    """Two grids, rotating and real instances, four potentials."""
    ps = [p for p in W.batched_sweep(64) if p["n"][0] <= 128][:4]
    real = dict(ps[0], omega=0.0, is_complex=False)
    return ps + [real, dict(real, beta=2.0 * real["beta"])]


def _initial(ps):
    out = []
    for i, p in enumerate(ps):
        a = W.sweep_initial(p, i)
        if not p["is_complex"]:
            a = W.normalise(p, np.abs(a))
        out.append(a.astype(np.complex64 if p["is_complex"] else np.float32))
    return out


OPTS = dict(max_iter=300, res_tol=1e-7, mode=1, max_outer=4)


def _solve(ps, start, stream, ahead=0):
    """`ahead` matrix products are queued on the caller's stream before the call."""
    with torch.cuda.stream(stream):
        psi = [torch.from_numpy(a).cuda() for a in start]
        if ahead:
            m = torch.eye(4096, device="cuda") + 0.01
            _work(m, 2)
            stream.synchronize()
            _work(m, ahead)
        reps = G.solve_batch(ps, psi, stream=stream, **OPTS)
        stream.synchronize()
    return psi, reps


def _same(a, b):
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x, y)
    for r, s in zip(a[1], b[1]):
        for k in ("E", "mu", "res", "inner_f32", "inner_f64", "nfe", "status"):
            assert r[k] == s[k], k


def _work(m, n):
    for _ in range(n):
        m = torch.mm(m, m)
        m = m / m.norm()
    return m


def test_default_stream_busy():
    """Another host thread keeps the default stream busy: same states, bit for bit, and a plan made meanwhile on a
    stream of its own gives the same energies."""
    ps = _problems()
    start = _initial(ps)
    side = torch.cuda.Stream()
    quiet = _solve(ps, start, side)
    with G.Plan(ps[0], prec=G.F32, stream=side) as plan:
        E0 = plan.energy(quiet[0][0])
    stop = threading.Event()

    def busy():
        m = torch.eye(2048, device="cuda") + 0.01
        torch.cuda.current_stream().synchronize()
        while not stop.is_set():
            _work(m, 50)
            torch.cuda.current_stream().synchronize()   # the queue stays short

    t = threading.Thread(target=busy)
    t.start()
    try:
        loud = _solve(ps, start, side)
        with torch.cuda.stream(side):
            with G.Plan(ps[0], prec=G.F32, stream=side) as plan:
                E1 = plan.energy(loud[0][0])
    finally:
        stop.set()
        t.join()
    _same(quiet, loud)
    assert E0 == E1


def test_caller_stream_busy():
    """The copies from host memory are queued behind the caller's work, long before they run."""
    ps = _problems()
    start = _initial(ps)
    side = torch.cuda.Stream()
    _same(_solve(ps, start, side), _solve(ps, start, side, ahead=100))
