"""The FP32 records of a history set from device arrays are those of the same history set from host arrays, bit for bit:
mixed fields, fixed and adaptive steps, up to a gamma where forming 1 / gamma^2 in two ways shows in its last place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import history_case, window  # noqa: E402
from paper_2605_05543_gb300 import emppp  # noqa: E402


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("N,n,D,gamma0,dt", [(700, 300, 256, 197.0, 1e-14), (300, 100, 64, 3.0, 1e-15),
                                             (700, 300, 256, 5000.0, 1e-14), (1500, 0, 4, 60.0, 1e-14)])
def test_mixed_steps_from_device_and_host_histories(N, n, D, gamma0, dt, adaptive):
    h = history_case(N, n, sigma=20e-6, gamma0=gamma0, seed=9, dt=dt, wiggle=1e-5 / gamma0)
    T, W, V, u = window(h, D)
    out = []
    for args in ((T, W, V, u), [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (T, W, V, u)]):
        with emppp.Solver(N, D, dt, precision="mixed", proposal="closed_form") as s:
            if adaptive:
                s.set_adaptive_dt()
            s.set_history(n, *args)
            s.step(2)
            out.append(s.get_state() + s.get_fields())
    for p, q in zip(*out):
        assert np.array_equal(p, q)
