"""The rounding error of the stage-2 transport over many steps does not grow in proportion to them. A step rounds each
component of u once, by at most 2^-53 of |u| and independently of the steps before, and what it adds to u is small, so
after n steps the error is a random walk: its standard deviation is below 2^-53 sqrt(n) |u| (a rounding's is 0.29 of its
range of two such), and eight of those bound every particle. A kick that scales u by 1 / (1 + t^2) and back rounds it
several times a step with a bias, 1.6e-16 a step, and is beyond that bound from 512 steps on."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)
if np.finfo(np.longdouble).nmant < 100:
    pytest.skip("needs a quadruple-precision long double", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402
from test_gpu_transport import reference  # noqa: E402

R_E = 6.371e6
M0 = 3.1e-5 * R_E ** 3 / 1e-7


@pytest.mark.parametrize("gamma0", [3.0, 20.0])
@pytest.mark.parametrize("steps", [512, 2048])
def test_error_is_a_random_walk(steps, gamma0):
    b = inputs.gaussian_bunch(64, 50e-6, gamma0, seed=5, center=(-4 * R_E, 0, 0))
    with emppp.Solver(64, 2, 1e-15) as s:
        s.set_particles(b.x.copy(), b.u.copy())
        s.transport(steps, 1e-9, emppp.bext_dipole(M0))
        u = s.get_state()[1]
    _, ur, _ = reference(b.x, b.u, 1e-9, steps, "dipole", (M0, (0.0, 0.0, 0.0)))
    e = np.abs(u - ur).max(axis=1) / np.linalg.norm(b.u, axis=1)
    assert e.max() <= 8 * 2.0 ** -53 * np.sqrt(steps), float(e.max())
