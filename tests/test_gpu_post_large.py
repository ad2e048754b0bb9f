"""The post-pair launch with a thread per particle (large systems without partial sums), at sizes around its rule (32
particles in each of four blocks an SM) and the edges of its 256-thread blocks: without pair fields every particle moves
as it does in a smaller system (bit for bit); a step with pair fields after such steps agrees with the oracle on a sample
of targets; steps that it prepared equal steps with their own set-up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import DT, field_errors  # noqa: E402
from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402

FIRST = 32 * 4 * torch.cuda.get_device_properties(0).multi_processor_count + 1
EXT = (0.1, -0.2, 0.3)


@pytest.mark.parametrize("N", [FIRST - 1, FIRST, 256 * 77, 256 * 77 + 1])
def test_steps_without_pair_fields_do_not_depend_on_the_size(N):
    b = inputs.gaussian_bunch(N, 8e-6, 12.0, seed=3)
    out = []
    for n in (N, 300):
        with emppp.Solver(n, 3, DT, precision="mixed", pair_fields=False) as s:
            s.set_particles(b.x[-n:].copy(), b.u[-n:].copy())
            s.step(5, emppp.bext_uniform(EXT))
            out.append([a[-300:] for a in s.get_state()[:2] + s.get_fields() + tuple(s.get_history()[2:4][k][j] for k in (0, 1) for j in (0, 1, 2))])
    for p, q in zip(*out):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_pair_fields_after_steps_without(precision):
    N, D = FIRST, 8
    b = inputs.gaussian_bunch(N, 8e-6, 3.0, seed=4)
    with emppp.Solver(N, D, DT, precision=precision, proposal="closed_form", pair_fields=False) as s:
        s.set_particles(b.x.copy(), b.u.copy())
        s.step(4, emppp.bext_uniform(EXT))
        n, T, W, V, u = s.get_history()
        s.set_options(pair_fields=True)
        s.step(1)
        E, B = s.get_fields()
    tg = np.arange(0, N, N // 40, dtype=np.int64)
    E_ref, B_ref, _, M = oracle.self_fields(T, W, V, n, D, targets=tg, mags=True)
    bar = 1e-12 if precision == "fp64" else 1e-5
    assert max(field_errors(E[tg], B[tg], E_ref, B_ref, M)) <= bar


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_prepared_steps_equal_steps_with_their_own_set_up(precision):
    N = FIRST + 200
    b = inputs.gaussian_bunch(N, 8e-6, 12.0, seed=5)
    out = []
    for spend in (False, True):
        with emppp.Solver(N, 5, DT, precision=precision, proposal="closed_form", source_split=1) as s:
            s.set_particles(b.x.copy(), b.u.copy())
            for _ in range(7):
                s.step(1)
                if spend:
                    s.sample_delays(np.array([[0, 1]], dtype=np.int32))
            out.append(s.get_state()[:2] + s.get_fields())
    for p, q in zip(*out):
        assert np.array_equal(p, q)
