"""Mixed path, batches of many small bunches: from one and a half rounds of target tiles on, a bunch of at most 128 is one
chunk that writes its fields itself, a larger one beside it keeps chunks. Fields of sampled bunches against the oracle
within the mixed path's 1e-5, around the rule, with bunches of 128 and 129."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import DT, field_errors, history_case, window  # noqa: E402
from paper_2605_05543_gb300 import emppp  # noqa: E402

TILES = 3 * 8 * torch.cuda.get_device_properties(0).multi_processor_count // 2  # one and a half rounds


@pytest.mark.parametrize("tiles", [TILES - 1, TILES, TILES + 700])
def test_fields_of_small_bunches(tiles):
    sizes = [40, 129, 128, 1, 300] + [33] * (tiles - 8)
    n, D = 40, 32
    N = sum(sizes)
    h = history_case(N, n, sigma=5e-6, seed=12)
    T, W, V, u = window(h, D)
    with emppp.Solver(N, D, DT, precision="mixed", proposal="closed_form", bunches=sizes) as s:
        s.set_history(n, T, W, V, u)
        s.step(1)
        E, B = s.get_fields()
    off = np.concatenate([[0], np.cumsum(sizes)])
    for b in (0, 1, 2, 4, 5, len(sizes) - 1):
        sl = slice(off[b], off[b + 1])
        E_ref, B_ref, _, M = oracle.self_fields(h.T, np.ascontiguousarray(h.W[:, sl]), np.ascontiguousarray(h.V[:, sl]), n, D,
                                                mags=True)
        assert max(field_errors(E[sl], B[sl], E_ref, B_ref, M)) <= 1e-5
    assert np.all(E[off[3]] == 0.0)
