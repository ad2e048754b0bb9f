"""The spatial target order is a permutation of each bunch at the edges of its sort (64 particles, windows of 2048), for
one bunch, several, and particles that coincide in all but one place or lie on a line: fields with the order equal fields
without it bit for bit, since a target's sum runs over the sources in one order whichever thread evaluates it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402


@pytest.mark.parametrize("sizes,shape", [
    ([2], "gauss"), ([63], "gauss"), ([64], "gauss"), ([65], "gauss"), ([2047], "gauss"), ([2048], "gauss"),
    ([2049], "gauss"), ([4097], "gauss"), ([5, 64, 2050, 129], "gauss"), ([300], "line"), ([2100], "pile"),
])
def test_order_is_a_permutation(sizes, shape):
    parts = [inputs.gaussian_bunch(n, 8e-6, 3.0, seed=n) for n in sizes]
    x, u = (np.concatenate([getattr(p, k) for p in parts]) for k in ("x", "u"))
    if shape == "line":
        x[:, :2] = x[0, :2]
    elif shape == "pile":  # all but one within a cell of the key
        x = x[0] + 1e-9 * (x - x[0]) / 8e-6
        x[-1] += 1e-3
    out = []
    for order in (0, 1):
        with emppp.Solver(0, 6, 1e-15, precision="fp64", proposal="bisect", bunches=sizes) as s:
            s.set_particles(x.copy(), u.copy())
            s.set_tuning(items_per_block=16, target_order=order)
            s.step(2)
            out.append(s.get_state()[:2] + s.get_fields())
    for a, b in zip(*out):
        assert np.array_equal(a, b) and np.all(np.isfinite(a))


@pytest.mark.parametrize("N", [1024, 1025, 2048, 2049])
@pytest.mark.parametrize("adaptive,graphs", [(False, False), (False, True), (True, True)])
def test_order_from_the_second_step(N, adaptive, graphs):
    """Middle systems on the mixed path form the order in their second step, and again after a new state."""
    b = inputs.gaussian_bunch(N, 8e-6, 3.0, seed=N)
    out = []
    for order in (0, 1):
        with emppp.Solver(N, 8, 1e-15, precision="mixed", proposal="closed_form", graphs=graphs,
                          stream=torch.cuda.Stream()) as s:
            if adaptive:
                s.set_adaptive_dt()
            s.set_tuning(items_per_block=16, target_order=order)
            for _ in range(2):
                s.set_particles(b.x.copy(), b.u.copy())
                s.step(1)
                s.step(18)
            out.append(s.get_state()[:2] + s.get_fields())
    for a, c in zip(*out):
        assert np.array_equal(a, c)
