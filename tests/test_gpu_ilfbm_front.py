"""ILFBM in 2D on fields with a front, where most units of 32 nodes lie still in
an inner iteration and are passed over: columns at the edges of a unit, a call
longer than one launch (256 steps), and calls of one step.  Tolerances as in
test_gpu_ilfbm.py: 1e-12 of the largest temperature, or ten times the
problem's own rounding floor (the oracle started one ulp away); the liquid
fraction 1e-10, the inner loop's tolerance 1e-12 times its contraction 1/(1 - 8/9)
and ten for the steps' accumulation."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import _abi, workloads

pytestmark = pytest.mark.gpu


def _front(nx, ny, seed):
    d = np.minimum(np.arange(nx)[None, :], np.arange(ny)[:, None] + 3.0)
    th = np.where(d < 7.3, -1.0 * (1 - d / 7.3), 0.3 * (1 - np.exp(-(d - 7.3) / 6.0)))
    return th + workloads.random_field((ny, nx), -1e-3, 1e-3, seed=seed)


@pytest.mark.parametrize("nx,ny,steps,calls", [(31, 40, 40, 1), (32, 33, 40, 1), (33, 20, 40, 8), (64, 64, 30, 1),
                                               (97, 35, 300, 1), (200, 150, 12, 12)])
def test_ilfbm_front_parity(orc, nx, ny, steps, calls):
    from paper_2505_13097_gb300 import solver
    tau, ste, walls = 0.84, 0.05, {"W": (1, -1.0), "S": (1, -1.0)}
    th0 = _front(nx, ny, nx)
    S = solver.Stefan(_abi.LBM_D2Q9, nx, ny, tau, 0.01, ste, _abi.LBM_FP64, walls, newton_tol=1e-12, newton_max_iter=400)
    S.set_method("ILFBM")
    S.set_ic(th0)
    for _ in range(calls):
        S.step(steps // calls)
    th, l, _ = S.fields()
    st = S.stats()
    S.close()
    P = orc.Problem(2, nx, ny, tau=tau, delta=0.01, ste=ste, walls=walls)
    _, lo, tho, failed, mx = P.ilfbm_run(th0, steps, tol=1e-12, maxit=400)
    rng = np.random.Generator(np.random.PCG64(12345))
    pert = th0 + np.spacing(th0) * rng.choice([-1, 0, 1], size=th0.shape)
    _, lp, thp, _, _ = P.ilfbm_run(pert, steps, tol=1e-12, maxit=400)
    assert failed == 0 and st["error"] == 0 and st["steps"] == steps
    assert np.max(np.abs(th - tho)) <= max(1e-12 * np.max(np.abs(tho)), 10 * np.max(np.abs(thp - tho)))
    assert np.max(np.abs(l - lo)) <= max(1e-10, 10 * np.max(np.abs(lp - lo)))
    assert 1 < st["newton_max_iter"] <= mx
