"""Stage-2 transport against the Higuera-Cary push written out in extended precision (numpy longdouble), for the three
background fields, at the edges of its one-warp blocks and of its chunks of 4096 steps, with weak and strong rotation
per step.

Tolerance: a step rounds u, v and the rotation a few dozen times, each below 2^-53 of the value, and x by 2^-53 of the
distance from the origin twice; the errors add at most linearly: 48 * 2^-53 * steps of |u|, and of |x| for the position
plus what that error of v has moved it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402

L = np.longdouble
C, QE, ME = L(299792458), L(1.602176634e-19), L(9.1093837015e-31)
MU0_4PI = L(1.25663706212e-6) / (4 * L(np.pi))


def reference(x, u, dt, steps, kind, par):
    x, u, dt = x.astype(L), u.astype(L), L(dt)
    h = -QE * dt / (2 * ME)
    dot = lambda a, b: (a * b).sum(1, keepdims=True)  # noqa: E731
    gam = lambda a: np.sqrt(1 + dot(a, a) / C ** 2)  # noqa: E731
    for _ in range(steps):
        xh = x + dt / 2 * u / gam(u)
        B = np.zeros_like(x)
        if kind == "uniform":
            B = B + np.array(par, dtype=L)
        elif kind == "dipole":
            d = xh - np.array(par[1], dtype=L)
            r = np.sqrt(dot(d, d))
            n = d / r
            B = 3 * L(par[0]) * n[:, 2:3] * n
            B[:, 2] -= L(par[0])
            B = MU0_4PI * B / r ** 3
        tau = h * B
        sig = gam(u) ** 2 - dot(tau, tau)
        gp = np.sqrt((sig + np.sqrt(sig ** 2 + 4 * (dot(tau, tau) + (dot(u, tau) / C) ** 2))) / 2)
        t = tau / gp
        up = (u + dot(u, t) * t + np.cross(u, t)) / (1 + dot(t, t))
        u = up + np.cross(up, t)
        x = xh + dt / 2 * u / gam(u)
    return x, u, B


@pytest.mark.parametrize("N,steps,dt,kind,par", [
    (1, 1, 1e-9, "none", None), (33, 7, 1e-9, "none", None),
    (31, 3, 1e-9, "uniform", (5e-5, 0.0, 0.0)), (32, 40, 1e-9, "uniform", (0.1, -0.2, 0.3)),  # 0.4 rad per step
    (65, 200, 1e-9, "dipole", (8e22, (0.0, 0.0, 0.0))), (2, 4097, 1e-9, "dipole", (8e22, (3e6, -2e6, 1e6))),
    (40, 20, 1e-8, "dipole", (3e24, (1e4, 2e4, -3e4))),
])
def test_transport_matches_extended_precision(N, steps, dt, kind, par):
    b = inputs.gaussian_bunch(N, 1e-4, 4.0, seed=N)
    u0 = b.u.copy()
    u0[::3, 0] += 3e8  # part of the particles across the field
    x0 = b.x + (np.array([2e7, 1e6, -3e6]) if kind == "dipole" and N != 40 else np.array([1e6, 0.0, 0.0]))
    bext = {"none": emppp.bext_none, "uniform": lambda: emppp.bext_uniform(par),
            "dipole": lambda: emppp.bext_dipole(*par)}[kind]()
    with emppp.Solver(N, 4, 1e-15) as s:
        s.set_particles(x0.copy(), u0.copy())
        s.transport(steps, dt, bext)
        x, u, t, n = s.get_state()
        E, B = s.get_fields()
    xr, ur, Br = reference(x0, u0, dt, steps, kind, par)
    assert n == steps and np.all(E == 0.0)
    e = 48 * 2.0 ** -53 * steps
    un, xn = np.linalg.norm(u0, axis=1).max(), np.linalg.norm(x0, axis=1).max()
    assert np.max(np.abs(u - ur)) <= e * un
    assert np.max(np.abs(x - xr)) <= e * (xn + float(C) * dt * steps)
    assert np.max(np.abs(B - Br)) <= 64 * 2.0 ** -53 * max(np.abs(Br).max(), 1e-300) * max(1.0, steps)
