"""emppp_set_history from device arrays (one launch over all slots) against the same history from host arrays (a launch
per slot): the stored history comes back bit for bit, every pair's bracket is the oracle's, the FP64 fields are equal, and the mixed ones agree within its
FP32 records' last place (their 1 / gamma^2 is formed without a division). Slot counts around the launch's groups of
8 slots, rings that wrap and rings that do not fill, two bunches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import DT, field_errors, history_case, window  # noqa: E402
from paper_2605_05543_gb300.emppp import Solver  # noqa: E402


@pytest.mark.parametrize("N,n,D,bunches", [
    (33, 0, 8, None), (257, 6, 16, None), (256, 7, 16, None), (300, 8, 16, None), (129, 40, 17, None),
    (300, 63, 64, [130, 170]), (65, 100, 24, None),
])
def test_device_history_equals_host_history(N, n, D, bunches):
    h = history_case(N, n, seed=N + n)
    T, W, V, u = window(h, D)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (T, W, V, u)]
    out = {}
    for precision in ("fp64", "mixed"):
        for where, args in (("host", (T, W, V, u)), ("device", dev)):
            with Solver(N, D, DT, precision=precision, proposal="closed_form", bunches=bunches) as s:
                s.set_history(n, *args)
                _, T2, W2, V2, u2 = s.get_history()
                for a, b in ((T, T2), (W, W2), (V, V2), (u, u2)):
                    assert np.array_equal(a, b)
                if bunches is None:
                    assert np.array_equal(s.bracket_dump()[0], oracle.bracket_table(h.T, h.W, h.n, D))
                s.step(1)
                out[precision, where] = s.get_fields()
    for a, b in zip(out["fp64", "host"], out["fp64", "device"]):
        assert np.array_equal(a, b)
    if bunches is None:
        _, _, _, M = oracle.self_fields(h.T, h.W, h.V, h.n, D, mags=True)
        # a last place of 1 / gamma^2 or gamma^2 (u = 2^-24) moves a pair's field by at most 8 gamma^2 u, gamma = 3
        eE, eB = field_errors(*out["mixed", "device"], *out["mixed", "host"], M)
        assert max(eE, eB) <= 8 * 9 * 2.0 ** -24
