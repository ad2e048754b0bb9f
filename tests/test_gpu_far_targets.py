"""Brackets of targets that the FP32 split cannot hold (more than 0.5 m from the bunch's split origin): their node tests
are FP64 ones, so no FP32 bound may settle one. Targets on the light sphere of one of their source's stored slots, 1e4 to
7e5 m from the bunch's first particle, where the split's low part rounds by 1e-11 to 1e-9 m: every bracket is the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import DT, light_sphere_case  # noqa: E402
from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402


def far_case(nb, n, R, oldest):
    """Bunches of three: a particle at rest at the origin, then a pair of light_sphere_case moved to R along x."""
    T, W2, V2, u2 = light_sphere_case(nb, n, seed=71, oldest=oldest)
    W, V, u = np.zeros((n + 1, 3 * nb, 3)), np.zeros((n + 1, 3 * nb, 3)), np.zeros((3 * nb, 3))
    for k in (0, 1):
        W[:, 1 + k::3], V[:, 1 + k::3], u[1 + k::3] = W2[:, k::2] + np.array([R, 0.0, 0.0]), V2[:, k::2], u2[k::2]
    return T, W, V, u


@pytest.mark.parametrize("proposal", ["bisect", "closed_form", "mlp"])
@pytest.mark.parametrize("R,oldest", [(1.2345678901e4, False), (9.87654321e4, False), (6.54321987e5, False), (9.87654321e4, True)])
def test_brackets_far_from_the_split_origin(R, oldest, proposal):
    nb, n, D = 256, 40, 64
    T, W, V, u = far_case(nb, n, R, oldest)
    with emppp.Solver(0, D, DT, precision="mixed", proposal=proposal, bunches=[3] * nb) as s:
        s.set_history(n, T, W, V, u)
        if proposal == "mlp":
            s.set_proposal(0.05 * inputs.mlp_init_params(5))
        got, _ = s.bracket_dump()
    bad = 0
    for b in range(nb):
        sl = slice(3 * b, 3 * b + 3)
        bad += int((got[sl, sl] != oracle.bracket_table(T, W[:, sl], n, D)).sum())
    assert bad == 0, bad
