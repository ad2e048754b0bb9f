"""Adaptive steps of the mixed path at sizes whose work items fill one round of eight blocks to an SM but not of seven,
which an instance of their own takes, and beside them: the guessed search gives the state of the paper's bisection bit
for bit, since every search leads to the same bracket and the same forms. At gamma 3 no source needs its line in FP64, at
gamma 100 a warp's list of them overflows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import DT, history_case, window  # noqa: E402
from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402


@pytest.mark.parametrize("proposal", ["closed_form", "mlp"])
@pytest.mark.parametrize("N,gamma0", [(700, 100.0), (750, 3.0), (750, 100.0), (3000, 100.0), (3500, 3.0)])
def test_guessed_search_equals_bisection(N, gamma0, proposal):
    h = history_case(N, 60, sigma=20e-6, gamma0=gamma0, seed=N, wiggle=1e-5)
    T, W, V, u = window(h, 48)
    out = []
    for prop in ("bisect", proposal):
        with emppp.Solver(N, 48, DT, precision="mixed", proposal=prop) as s:
            s.set_adaptive_dt()
            if prop == "mlp":
                s.set_proposal(0.05 * inputs.mlp_init_params(5))
            s.set_history(h.n, T, W, V, u)
            s.step(3)
            out.append(s.get_state() + s.get_fields())
    for a, b in zip(*out):
        assert np.array_equal(a, b)
