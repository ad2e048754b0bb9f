"""emppp_fields_noalloc at the edges of its launch: one slice that writes the fields itself (n <= 32) and several, tiles
of 64 sources with a remainder, target blocks of 128 with a ragged tail, unevenly spaced slots (the guess assumes even
ones), high gamma, and far from the origin. Against the oracle within the file's bar of test_zz_no_alloc.py, 1e-12 of
each target's sum of magnitudes, times (gamma0 / 3)^2 for the retarded solve's conditioning; the shifted case against
the unshifted oracle, with the shift's rounding of the inputs (2^-53 of 1e-3 m against distances of a micrometre)."""
import numpy as np
import pytest

import oracle
from gpu_helpers import field_errors, history_case

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp  # noqa: E402


def _fields(T, W, V):
    t, w, v = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (T, W, V))
    E, B = (torch.full((W.shape[1], 3), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    emppp.fields_noalloc(t, w, v, E, B, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    return E.cpu().numpy(), B.cpu().numpy()


@pytest.mark.parametrize("N,nslots,sigma,gamma0", [
    (2, 5, 3e-6, 3.0), (20, 40, 3e-6, 3.0), (33, 3, 1e-6, 3.0), (64, 30, 5e-6, 3.0), (65, 70, 5e-6, 20.0),
    (129, 120, 10e-6, 3.0), (700, 250, 10e-6, 3.0),
])
def test_sizes_match_the_oracle(N, nslots, sigma, gamma0):
    h = history_case(N, nslots - 1, sigma=sigma, gamma0=gamma0, seed=40 + N)
    E, B = _fields(h.T, h.W, h.V)
    E_ref, B_ref, _, M = oracle.self_fields(h.T, h.W, h.V, h.n, nslots, mags=True)
    assert max(field_errors(E, B, E_ref, B_ref, M)) <= 1e-12 * (gamma0 / 3.0) ** 2


def test_uneven_slots_match_the_oracle():
    h = history_case(200, 160, sigma=8e-6, seed=50)
    keep = np.unique(np.concatenate([[0, 1, 2, 50, 51, 90], np.arange(120, 161)]))  # wide steps, then fine ones
    T, W, V = h.T[keep], np.ascontiguousarray(h.W[keep]), np.ascontiguousarray(h.V[keep])
    E, B = _fields(T, W, V)
    E_ref, B_ref, _, M = oracle.self_fields(T, W, V, len(keep) - 1, len(keep), mags=True)
    assert max(field_errors(E, B, E_ref, B_ref, M)) <= 1e-12


def test_far_from_the_origin():
    h = history_case(150, 100, sigma=5e-6, seed=51)
    E_ref, B_ref, _, M = oracle.self_fields(h.T, h.W, h.V, h.n, 101, mags=True)
    E, B = _fields(h.T, h.W + np.array([1e-3, 0.0, -1e-3]), h.V)
    d = h.W[-1][:, None] - h.W[-1][None]
    near = np.sqrt((d ** 2).sum(-1) + np.eye(150)).min()
    # positions rounded by 2^-53 * 1e-3 m move a pair's field by gamma^2 times that over the nearest distance
    assert max(field_errors(E, B, E_ref, B_ref, M)) <= 9 * 8 * 2.0 ** -53 * 1e-3 / near
