"""A call that reports a device error leaves the caller's arrays as they were, host arrays (small and large ones) and device
arrays alike, and time and step too; a good call fills them, also where only one array is asked for, and device arrays
that start off a multiple of eight bytes."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402


def _arrays(N, device):
    if device:
        return [torch.full((N, 3), -7.0, dtype=torch.float64, device="cuda") for _ in range(2)]
    return [np.full((N, 3), -7.0) for _ in range(2)]


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("N", [2, 1365, 1366, 5000])
def test_arrays_after_an_error(N, device):
    b = inputs.gaussian_bunch(N, 8e-6, 3.0, seed=8)
    x = b.x.copy()
    x[1] = x[0]  # coincident particles
    with emppp.Solver(N, 4, 1e-15) as s:
        s.set_particles(x, b.u.copy())
        s.step(1)
        for call in (s.get_state, s.get_fields):
            a = _arrays(N, device)
            with pytest.raises(emppp.EmpppError) as e:
                call(*a)
            assert e.value.status == emppp.ERR_NUMERIC
            assert all(bool((q == -7.0).all()) for q in a)
        t, n = ctypes.c_double(-7.0), ctypes.c_int64(-7)
        assert s.lib.emppp_get_state(s.handle, None, None, ctypes.byref(t), ctypes.byref(n), 0) == emppp.ERR_NUMERIC
        assert (t.value, n.value) == (-7.0, -7)


@pytest.mark.parametrize("N", [2, 1365, 1366, 5000])
def test_arrays_of_a_good_call(N):
    b = inputs.gaussian_bunch(N, 8e-6, 3.0, seed=8)
    with emppp.Solver(N, 4, 1e-15) as s:
        s.set_particles(b.x.copy(), b.u.copy())
        s.step(2)
        x, u, _, _ = s.get_state()
        E, B = s.get_fields()
        W = s.get_history()[2]
        assert np.array_equal(x, W[-1]) and np.all(np.isfinite(u)) and np.any(E != 0.0) and np.any(B != 0.0)
        for call, ref in ((s.get_state, (x, u)), (s.get_fields, (E, B))):
            for device in (False, True):
                for only in (0, 1, None):
                    a = _arrays(N, device)
                    call(*[q if only in (k, None) else None for k, q in enumerate(a)])
                    for k, q in enumerate(a):
                        got = q.cpu().numpy() if device else q
                        assert np.array_equal(got, ref[k] if only in (k, None) else np.full((N, 3), -7.0))
        raw = torch.zeros(24 * N + 8, dtype=torch.uint8, device="cuda")
        assert s.lib.emppp_get_fields(s.handle, raw.data_ptr() + 4, None, 1) == emppp.OK
        assert np.array_equal(raw[4:4 + 24 * N].cpu().numpy().view(np.float64).reshape(N, 3), E)
