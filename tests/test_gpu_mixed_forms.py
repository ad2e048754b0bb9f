"""The mixed pair kernel's fields from the source's line at t_n against the FP64 oracle where that form is most
exposed: high gamma with a fixed step (its FP64 guard), pairs in the last segment with R far below c dt, and
ragged tiles. Tolerance: the mixed path's stated 1e-5 of each target's sum of field magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import field_errors, gpu_fields_from_history, history_case  # noqa: E402
from paper_2605_05543_gb300.emppp import Solver  # noqa: E402


@pytest.mark.parametrize("proposal", ["bisect", "closed_form"])
@pytest.mark.parametrize("N,n,D,sigma,gamma0,dt,guarded", [
    (300, 200, 256, 10e-6, 20.0, 1e-15, True),
    (129, 60, 64, 2e-4, 60.0, 1e-13, True),
    (257, 30, 64, 1e-6, 3.0, 1e-13, False),  # c dt = 30 um: nearly every pair in the last segment
    (65, 90, 32, 20e-6, 3.0, 1e-15, False),  # a tile of one source, wrapped ring
])
def test_line_form_against_oracle(proposal, N, n, D, sigma, gamma0, dt, guarded):
    h = history_case(N, n, sigma=sigma, gamma0=gamma0, seed=3 + N, dt=dt, wiggle=1e-5)
    E, B, st, _, _ = gpu_fields_from_history(Solver, h, D, dt=dt, precision="mixed", proposal=proposal, source_split=2)
    E_ref, B_ref, _, M = oracle.self_fields(h.T, h.W, h.V, h.n, D, mags=True)
    eE, eB = field_errors(E, B, E_ref, B_ref, M)
    assert eE <= 1e-5 and eB <= 1e-5, (eE, eB)
    br = oracle.bracket_table(h.T, h.W, h.n, D) % 4
    off = ~np.eye(N, dtype=bool)
    assert (st["out_of_history"], st["shortcut"], st["bisection"]) == tuple(int((br[off] == k).sum()) for k in range(3))
    if guarded:
        assert st["guard_fallbacks"] > 0
