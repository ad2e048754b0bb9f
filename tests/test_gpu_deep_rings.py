"""Few particles with a deep history: their steps' slot tables come from the set-up launch, with a thread per slot, where
the post-pair launch has few threads for them. Around the rule (8 slots per thread, 64 threads for up to 8 particles) the
state is that of steps with their own set-up bit for bit, and a step with 65536 slots takes not much longer than one with
64 (1.5 times; with the tables in the post-pair launch 50 times)."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402

DT = 1e-15


@pytest.mark.parametrize("D", [511, 512, 513, 1025])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_state_around_the_rule(D, precision):
    b = inputs.gaussian_bunch(8, 8e-6, 3.0, seed=6)
    out = []
    for spend in (False, True):
        with emppp.Solver(8, D, DT, precision=precision, proposal="closed_form") as s:
            s.set_particles(b.x.copy(), b.u.copy())
            for _ in range(5):
                s.step(1)
                if spend:
                    s.sample_delays(np.array([[0, 1]], dtype=np.int32))
            out.append(s.get_state()[:2] + s.get_fields())
    for p, q in zip(*out):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_time_of_a_step_with_a_deep_ring(precision):
    h = inputs.gaussian_bunch(2, 8e-6, 3.0, seed=7)
    best = {}
    for D in (64, 65536):
        v = h.u / np.sqrt(1.0 + np.sum(h.u ** 2, axis=1, keepdims=True) / inputs.C_LIGHT ** 2)
        T = np.arange(D) * DT
        W = h.x[None] + v[None] * (T - T[-1])[:, None, None]
        args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (T, W, np.broadcast_to(v, W.shape), h.u)]
        with emppp.Solver(2, D, DT, precision=precision, proposal="closed_form", stream=torch.cuda.Stream()) as s:
            torch.cuda.synchronize()
            s.set_history(D - 1, *args)
            ts = []
            for _ in range(6):
                t = time.perf_counter()
                s.step(32)
                s.synchronize()
                ts.append(time.perf_counter() - t)
            best[D] = min(ts)
    assert best[65536] < 8 * best[64], best
