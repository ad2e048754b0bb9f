"""Precision of the mixed path where a source moves nearly towards its target: the separation from the source's line is
formed in FP64 where its FP32 rounding would move tau by 1e-6 of itself. Below that kappa moves by 2e-6, a field, which goes
with its inverse cube, by 6e-6 of the pair's, and the dozen FP32 operations after it add at most 1e-6: c B of every
target within 7e-6 of its sum of magnitudes. (E of such pairs cancels further, with gamma^2, and has the path's 1e-5.)
The seeds are those whose largest error was 8e-6 to 1e-5 with the bound at 2e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import field_errors, gpu_fields_from_history, history_case  # noqa: E402
from paper_2605_05543_gb300.emppp import Solver  # noqa: E402


@pytest.mark.parametrize("gamma0,N,n,D,sigma,seed", [
    (20.0, 300, 63, 64, 30e-6, 21), (40.0, 100, 200, 256, 8e-6, 1), (40.0, 300, 63, 64, 30e-6, 22),
    (6.0, 300, 63, 64, 10e-6, 11), (6.0, 300, 63, 64, 10e-6, 3), (20.0, 100, 200, 256, 8e-6, 53),
])
def test_forward_pairs(gamma0, N, n, D, sigma, seed):
    h = history_case(N, n, sigma=sigma, gamma0=gamma0, seed=seed, wiggle=1e-5)
    E, B, _, _, _ = gpu_fields_from_history(Solver, h, D, precision="mixed", proposal="closed_form")
    E_ref, B_ref, _, M = oracle.self_fields(h.T, h.W, h.V, n, D, mags=True)
    eE, eB = field_errors(E, B, E_ref, B_ref, M)
    assert eE <= 1e-5 and eB <= 7e-6, (eE, eB)
