"""The FP64 pair kernel's forms of the retarded solve and the fields against the textbook formulas in extended
precision (numpy longdouble, at least 64 mantissa bits), at the edges of its 64-source tiles and where the
quadratic about the bracket's older node cancels.

Tolerances, of each target's sum of field magnitudes: the separation from the source's line at t_n carries a
rounding of 2u of the distance c (t_n - t1), which the solve amplifies by at most 1 / (1 - beta) < 2 gamma^2, and a
dozen further roundings follow, each amplified by as much: 16 u * 2 gamma^2 * max(1, c dt / R_min).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_helpers import gpu_fields_from_history, history_case  # noqa: E402
from paper_2605_05543_gb300 import inputs  # noqa: E402
from paper_2605_05543_gb300.emppp import Solver  # noqa: E402

L = np.longdouble
C = L(299792458)
KQ = L(-1.602176634e-19) / (4 * L(np.pi) * L(8.8541878128e-12))
U = 2.0 ** -53


def extended_fields(h, D):
    """Self fields, sums of magnitudes and the smallest |eta| at slot h.n, in extended precision."""
    k0 = max(0, h.n - D + 1)
    T, W, V = h.T[k0:], h.W[k0:], h.V[k0:]
    br = oracle.bracket_table(h.T, h.W, h.n, D)  # 4 (k1 - k0) + branch
    N = W.shape[1]
    j = np.arange(N)
    E, B, M = np.zeros((N, 3), L), np.zeros((N, 3), L), np.zeros((N, 2))
    rmin = np.inf
    for i in range(N):
        o = j != i
        k1, ooh = br[i, o] // 4, br[i, o] % 4 == 0
        w1, v1, T1 = W[k1, j[o]].astype(L), V[k1, j[o]].astype(L), (L(T[-1]) - T[k1].astype(L))[:, None]
        up = np.minimum(k1 + 1, len(T) - 1)
        dT = np.where(ooh, L(1), T[up].astype(L) - T[k1].astype(L))[:, None]
        a = np.where(ooh[:, None], L(0), (V[up, j[o]].astype(L) - v1) / dT)
        p = W[-1, i].astype(L) - w1 - v1 * T1
        c2, pv, pp = C * C - (v1 * v1).sum(1), (p * v1).sum(1), (p * p).sum(1)
        sq = np.sqrt(pv * pv + c2 * pp)
        tau = np.where(pv >= 0, (pv + sq) / c2, pp / (sq - pv))[:, None]
        eta, v = p + v1 * tau, v1 + a * (T1 - tau)
        R = np.sqrt((eta * eta).sum(1))[:, None]
        u = C * eta / R - v
        F = (C * C - (v * v).sum(1)[:, None]) * u + np.cross(eta, np.cross(u, a))
        F = F * KQ * R / ((eta * u).sum(1)[:, None]) ** 3
        G = np.cross(eta / R, F) / C
        E[i], B[i] = F.sum(0), G.sum(0)
        M[i] = np.sqrt((F * F).sum(1)).sum(), np.sqrt((G * G).sum(1)).sum()
        rmin = min(rmin, float(R.min()))
    return E, B, M, rmin


@pytest.mark.parametrize("proposal", ["bisect", "closed_form"])
@pytest.mark.parametrize("N,n,D,sigma,gamma0,dt,split", [
    (63, 20, 64, 10e-6, 3.0, 1e-15, 1),   # one source short of a tile
    (64, 70, 32, 10e-6, 3.0, 1e-15, 1),   # a whole tile, wrapped ring
    (65, 70, 128, 10e-6, 3.0, 1e-15, 1),  # a tile of one source
    (193, 40, 64, 10e-6, 20.0, 1e-15, 2),  # chunks of 98 and 95: a tile and a remainder each
    (130, 0, 8, 10e-6, 3.0, 1e-15, 1),    # the present slot alone
    (150, 30, 64, 1e-6, 3.0, 1e-13, 1),   # c dt = 30 um, pairs down to a few nm: the last segment
])
def test_forms_against_extended_precision(proposal, N, n, D, sigma, gamma0, dt, split):
    h = history_case(N, n, sigma=sigma, gamma0=gamma0, seed=5 + N, dt=dt)
    E, B, _, _, _ = gpu_fields_from_history(Solver, h, D, dt=dt, proposal=proposal, source_split=split)
    Er, Br, M, rmin = extended_fields(h, D)
    tol = 16 * U * 2 * gamma0 ** 2 * max(1.0, inputs.C_LIGHT * dt / rmin)
    assert np.max(np.abs(E - Er) / M[:, :1]) <= tol
    assert np.max(np.abs(B - Br) / M[:, 1:]) <= tol
