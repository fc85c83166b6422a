"""dL/dSte and dL/dtheta_wall of one reverse step, FP32 flat kernel against the FP64
marching kernel, on inputs whose terms all have one sign: nothing cancels, so a
node left out or counted twice shows (the terms are within a factor of a few of
one another, and the largest lattice has some 5,000).

Bound: theta is taken to 20 bits; below 0.1 that is 1e-7, 5e-6 of theta/delta, twice
in phi(theta(t+1)) - phi(theta(t)) (arguments 0.25 to 0.5 apart: 4e-5), in the two
cosh and in F' (1e-5 each), and some 30 FP32 roundings: 1e-4; 2e-4 here."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu

WALLS = [{}, {"W": (1, 0.9)}, {"W": (1, 0.9), "S": (1, -0.5)}, {"E": (1, -0.5), "N": (1, 0.9)}]


@pytest.mark.parametrize("shape", [(2, 2), (3, 3), (5, 4), (6, 6), (67, 19), (68, 20), (69, 21), (133, 37), (200, 5)])
@pytest.mark.parametrize("bb_mode", [0, 1])
@pytest.mark.parametrize("wi", range(len(WALLS)))
def test_sums_of_one_sign(shape, bb_mode, wi):
    import torch
    from paper_2505_13097_gb300 import solver
    nx, ny = shape
    rng = np.random.Generator(np.random.PCG64(nx * 100 + ny))
    th = [rng.uniform(-0.04, 0.03, (ny, nx))]
    th.append(th[0] + rng.uniform(0.005, 0.01, (ny, nx)))
    # Dirichlet nodes hold their wall's value: no term in dL/dSte
    side = {"W": np.s_[:, 0], "E": np.s_[:, -1], "S": np.s_[0, :], "N": np.s_[-1, :]}
    for name in "NSEW":
        if name in WALLS[wi]:
            for t in th:
                t[side[name]] = WALLS[wi][name][1]
    lam = rng.uniform(0.5, 1.0, (9, ny, nx))
    res = []
    for prec in (workloads.FP32, workloads.FP64):
        # tau = 1.25: 1 - omega > 0, and so is every factor of a wall node's terms
        S = solver.Stefan(2, nx, ny, 1.25, 0.02, 0.2, prec, WALLS[wi], bb_mode=bb_mode)
        planes = S.new_theta_planes(2)
        planes.zero_()
        for k in range(2):
            planes[k, :, :nx] = torch.tensor(th[k], device="cuda")
        a, b = S.new_state_buffer(), S.new_state_buffer()
        n = 9 * (ny + 2) * S.row_stride * (4 if prec else 8)
        # clears the sums
        S.adjoint_seed(planes[1], torch.zeros((ny, nx), dtype=torch.float64, device="cuda"), a, want_loss=False)
        view = a[:n].view(torch.float32 if prec else torch.float64).view(9, ny + 2, S.row_stride)
        view[:, 1:-1, :nx] = torch.tensor(lam, device="cuda").to(view.dtype)
        torch.cuda.synchronize()
        S.adjoint_step(planes[0], planes[1], a, b)
        g0 = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
        b.zero_()   # adjoint_finish adds the initial field's part to the walls: none here
        res.append(S.adjoint_finish(b, g0))
        S.close()
    (gw, gs), (hw, hs) = res
    free = np.ones((ny, nx), dtype=bool)
    for name in WALLS[wi]:
        free[side[name]] = False
    assert (hs != 0.0) == bool(free.any())
    assert abs(gs - hs) <= 2e-4 * abs(hs)
    for k, name in enumerate("WESN"):
        assert (hw[k] != 0.0) == (name in WALLS[wi])
        assert abs(gw[k] - hw[k]) <= 2e-4 * abs(hw[k])
