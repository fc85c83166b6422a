"""NaN, infinities and terms of 2^67 and more (which the fixed-point sums cannot
hold) stay visible: the energy, the flux and the adjoint sums of a field that
holds one are NaN, not a finite sum of the rest."""
import math

import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


def _solver(lattice, nx, ny, precision, method, walls=None):
    from paper_2505_13097_gb300 import solver
    kw = {"newton_tol": 1e-12, "newton_max_iter": 50} if method == "ILFBM" else {}
    S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, precision, walls or {}, **kw)
    S.set_method(method)
    return S


@pytest.mark.parametrize("lattice,nx,ny,precision,method,timed", [
    (1, 64, 1, 0, "EEBM", False), (1, 64, 1, 1, "EEBM", False), (1, 5000, 1, 0, "EEBM", False), (1, 64, 1, 0, "ILFBM", False),
    (2, 64, 40, 0, "EEBM", False), (2, 700, 300, 0, "EEBM", False), (2, 64, 40, 0, "EEBM", True), (2, 64, 40, 0, "ILFBM", False),
    (3, 64, 40, 0, "EEBM", False), (3, 64, 40, 0, "EEBM", True), (3, 64, 40, 0, "ILFBM", False)])
@pytest.mark.parametrize("value", [math.nan, math.inf, -math.inf, 1e21])
def test_energy(lattice, nx, ny, precision, method, timed, value):
    S = _solver(lattice, nx, ny, precision, method)
    th0 = np.full((ny, nx), 1.0)
    th0[ny // 2, 0] = value
    S.set_ic(th0)
    assert math.isnan(S.stats()["energy"])
    (S.step_timed if timed else S.step)(2)
    st = S.stats()
    S.sync()
    assert st["steps"] == 2 and st["error"] == 0
    assert math.isnan(st["energy"]) and math.isnan(st["energy_prev"]) and math.isnan(st["imbalance"])
    # the wall's flux as well (a finite value bounces back and cancels)
    assert math.isnan(st["flux"]) or value == 1e21
    # nothing of it is left for the next field: the statistics are those of a fresh handle
    out = []
    for T in (S, _solver(lattice, nx, ny, precision, method)):
        T.set_ic(np.full((ny, nx), 1.0))
        (T.step_timed if timed else T.step)(2)
        out.append(T.stats())
        T.close()
    assert math.isfinite(out[0]["energy"]) and out[0] == out[1]


@pytest.mark.parametrize("lattice", [2, 3])
def test_shift_of_large_fields(lattice):
    # the shift of an FP32 state is half the mean, beyond the fixed-point range too
    S = _solver(lattice, 64, 40, 1, "EEBM")
    S.set_ic(np.full((40, 64), 1e21))
    S.step(2)
    th = S.theta()
    S.close()
    assert np.max(np.abs(th / 1e21 - 1.0)) <= 2 * 10 * 2.0 ** -24


@pytest.mark.parametrize("value", [math.nan, math.inf])
def test_shift_of_nonfinite_fields(value):
    S = _solver(2, 64, 40, 1, "EEBM")
    th0 = np.full((40, 64), 1.0)
    th0[7, 9] = value
    S.set_ic(th0)
    th = S.theta()
    S.close()
    assert not np.any(np.isfinite(th))   # stored less a shift that is not finite


@pytest.mark.parametrize("lattice,nx,ny,precision", [(1, 64, 1, 0), (2, 64, 40, 0), (2, 64, 40, 1)])
def test_adjoint_sums(lattice, nx, ny, precision):
    import torch
    S = _solver(lattice, nx, ny, precision, "IREBM", {"W": (1, 0.5)})
    planes = S.new_theta_planes(2)
    planes.zero_()
    planes[1] = 1e-3
    target = torch.full((ny, nx), 0.2, dtype=torch.float64, device="cuda")
    a, b = S.new_state_buffer(), S.new_state_buffer()
    for bad in (True, False):
        if bad:
            target[ny // 2, 0] = target[ny // 2, nx // 2] = math.nan
        else:
            target.fill_(0.2)
        loss = S.adjoint_seed(planes[1], target, a)
        S.adjoint_step(planes[0], planes[1], a, b)
        g0 = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
        gw, gs = S.adjoint_finish(b, g0)
        assert math.isnan(loss) == math.isnan(gw[0]) == math.isnan(gs) == bad
        assert gw[1:] == [0.0, 0.0, 0.0]
    S.close()
