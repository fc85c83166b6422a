"""ILFBM on D1Q3 at the edges of its segments of 32 nodes, with a front whose
surroundings alone are evaluated, one and many steps per call.  Tolerances as in
test_gpu_ilfbm.py: 1e-12 of the largest temperature, or ten times the problem's
own rounding floor (the oracle started one ulp away); liquid fraction 1e-10."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import _abi, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,steps,calls", [(31, 200, 1), (32, 200, 1), (33, 200, 50), (64, 300, 1), (513, 300, 3), (801, 100, 1),
                                           (2844, 40, 1)])
@pytest.mark.parametrize("walls,bb_mode", [({"W": (1, 1.0), "E": (1, -0.5)}, 0), ({"W": (1, 1.0)}, 0), ({"E": (1, -0.7)}, 1), ({}, 1)])
def test_ilfbm_line_parity(orc, n, steps, calls, walls, bb_mode):
    from paper_2505_13097_gb300 import solver
    x = np.arange(n)
    th0 = np.where(x < 9.4, 1.0 - x / 9.4, -0.5 * (1 - np.exp(-(x - 9.4) / 8.0)))[None, :]
    th0 = th0 + workloads.random_field((1, n), -1e-3, 1e-3, seed=n)
    S = solver.Stefan(_abi.LBM_D1Q3, n, 1, 0.62, 0.01, 0.3, _abi.LBM_FP64, walls, newton_tol=1e-12, newton_max_iter=200,
                      bb_mode=bb_mode)
    S.set_method("ILFBM")
    S.set_ic(th0)
    for _ in range(calls):
        S.step(steps // calls)
    th, l, _ = S.fields()
    st = S.stats()
    S.close()
    P = orc.Problem(1, n, 1, tau=0.62, delta=0.01, ste=0.3, walls=walls, bb_mode=bb_mode)
    _, lo, tho, failed, mx = P.ilfbm_run(th0, steps, tol=1e-12, maxit=200)
    rng = np.random.Generator(np.random.PCG64(12345))
    _, lp, thp, _, _ = P.ilfbm_run(th0 + np.spacing(th0) * rng.choice([-1, 0, 1], size=th0.shape), steps, tol=1e-12, maxit=200)
    assert failed == 0 and st["error"] == 0 and st["steps"] == steps
    assert np.max(np.abs(th - tho)) <= max(1e-12 * np.max(np.abs(tho)), 10 * np.max(np.abs(thp - tho)))
    assert np.max(np.abs(l - lo)) <= max(1e-10, 10 * np.max(np.abs(lp - lo)))
    assert 1 <= st["newton_max_iter"] <= mx
