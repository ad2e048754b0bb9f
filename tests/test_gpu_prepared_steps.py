"""The post-pair launch forms the slot tables and source vectors of the step after it. A run whose every step carries
its own set-up launch (here: after a call that spends what was prepared) gives the same state bit for bit, at the
edges of the launch's blocks (8, 16 or 32 particles), with rings of two slots, wrapped rings and rings longer than the
blocks' threads together; also when the caller's own graph of a step is replayed from another state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402

DT = 1e-15


def _solver(N, D, precision, proposal, adaptive, bunches=None, **kw):
    s = emppp.Solver(N, D, DT, precision=precision, proposal=proposal, bunches=bunches, **kw)
    if adaptive:
        s.set_adaptive_dt()
    return s


def _run(s, b, steps, spend):
    s.set_particles(b.x.copy(), b.u.copy())
    if spend:
        for _ in range(steps):
            s.step(1, emppp.bext_uniform((5e-5, 0.0, 0.0)))
            s.sample_delays(np.array([[0, 1]], dtype=np.int32))
    else:
        s.step(steps, emppp.bext_uniform((5e-5, 0.0, 0.0)))
    x, u, t, n = s.get_state()
    E, B = s.get_fields()
    return x, u, np.array([t, n]), E, B


@pytest.mark.parametrize("N,D,gamma0,bunches", [
    (7, 2, 3.0, None), (9, 700, 3.0, None), (257, 5, 30.0, None), (2433, 3, 3.0, None), (4865, 4, 3.0, None),
    (130, 6, 12.0, [1, 8, 121]),
])
@pytest.mark.parametrize("precision,proposal,adaptive", [
    ("fp64", "bisect", False), ("fp64", "closed_form", True), ("mixed", "closed_form", False), ("mixed", "bisect", True),
])
def test_prepared_steps_equal_steps_with_their_own_set_up(N, D, gamma0, bunches, precision, proposal, adaptive):
    b = inputs.gaussian_bunch(N, 8e-6, gamma0, seed=N)
    out = []
    for spend in (False, True):
        with _solver(N, D, precision, proposal, adaptive, bunches) as s:
            out.append(_run(s, b, 6, spend))
    for p, q in zip(*out):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_captured_step_carries_its_set_up(precision):
    b, c = (inputs.gaussian_bunch(300, 8e-6, 3.0, seed=k) for k in (1, 2))
    stream = torch.cuda.Stream()
    out = []
    for capture in (False, True):
        with _solver(300, 8, precision, "closed_form", False, stream=stream, graphs=False) as s:
            s.set_particles(b.x.copy(), b.u.copy())
            s.step(3)  # the next step is prepared
            if capture:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
                    s.step(1)
            s.set_particles(c.x.copy(), c.u.copy())
            for _ in range(4):
                if capture:
                    with torch.cuda.stream(stream):
                        g.replay()
                else:
                    s.step(1)
            stream.synchronize()
            out.append(s.get_state()[:2])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
