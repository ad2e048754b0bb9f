"""Steps after a replay of a graph that the caller captured from the same handle: the host cannot see the replay, so such a
step brings its own set-up. Every sequence is compared bit for bit with the same steps taken by calls, the handle's
options set to what each replayed step was captured with."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402

DT, N, D = 1e-15, 300, 64


def _capture(s, stream, call):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        call(s)
    return g


def _run(stream, first, then, captured, replayed):
    """Three steps, `captured` captured (or not), the options of `then`, two steps, the captured call replayed (or made
    with the options of `first`), two steps, by one call each and by a call that replays the library's graph."""
    b = inputs.gaussian_bunch(N, 8e-6, 3.0, seed=1)
    with emppp.Solver(N, D, DT, stream=stream, **first) as s:
        s.set_particles(b.x.copy(), b.u.copy())
        g = _capture(s, stream, captured) if replayed else None
        s.set_particles(b.x.copy(), b.u.copy())
        s.step(3)
        for k in (1, 2):
            s.set_options(**then)
            s.step(1)
            s.step(1)
            if replayed:
                with torch.cuda.stream(stream):
                    g.replay()
            else:
                s.set_options(**first)
                captured(s)
                s.set_options(**then)
            s.step(k)
        s.step(1)
        return s.get_state()[:2] + s.get_fields()


# source_split: one work split for both precisions, which a captured step keeps
FIELDS = dict(precision="fp64", pair_fields=True, proposal="closed_form", field_point="present", source_split=1)


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("first,then", [
    (dict(pair_fields=False), dict(pair_fields=True)),
    (dict(precision="mixed"), dict(precision="fp64")),
    (dict(precision="fp64"), dict(precision="mixed")),
    (dict(field_point="half_step"), dict(field_point="present")),
    (dict(), dict()),
])
def test_step_after_a_replayed_step(first, then, graphs):
    stream = torch.cuda.Stream()
    first, then = {**FIELDS, **first, "graphs": graphs}, {**FIELDS, **then, "graphs": graphs}
    out = [_run(stream, first, then, lambda s: s.step(1), replayed) for replayed in (False, True)]
    for p, q in zip(*out):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_step_after_a_replayed_transport(precision):
    """The captured transport carries the time it ends at, so the time stamps, and with them the light-travel distances of
    the steps after it, differ in their last places (2^-53 of 20 steps over one): 64 * 2^-53 of each."""
    stream = torch.cuda.Stream()
    opts = {**FIELDS, "precision": precision, "graphs": False}
    ext = emppp.bext_uniform((0.1, -0.2, 0.3))
    out = [_run(stream, opts, opts, lambda s: s.transport(3, DT, ext), replayed) for replayed in (False, True)]
    for p, q in zip(*out):
        assert np.max(np.abs(p - q)) <= 64 * 2.0 ** -53 * np.max(np.abs(p))


@pytest.mark.parametrize("N,precision", [(300, "fp64"), (2100, "mixed")])
def test_step_after_a_capture_that_is_not_replayed(N, precision):
    """The captured step's target order is not there before a replay: the step after it forms its own. (Before, it read
    whatever the order's memory held as particle indices, which is why this is not shown on the code before the change.)"""
    b = inputs.gaussian_bunch(N, 8e-6, 3.0, seed=2)
    stream = torch.cuda.Stream()
    out = []
    for capture in (False, True):
        with emppp.Solver(N, D, DT, stream=stream, precision=precision, proposal="closed_form", graphs=False) as s:
            s.set_particles(b.x.copy(), b.u.copy())
            if capture:
                _capture(s, stream, lambda s: s.step(2))
            s.step(1)
            s.step(1)
            out.append(s.get_state()[:2] + s.get_fields())
    for p, q in zip(*out):
        assert np.array_equal(p, q)
