"""Nodes in equilibrium (m0 = theta) take one iteration of the local solve: a
uniform field inside the mushy band steps with newton_max_iter = 1."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,nx,ny", [(1, 64, 1), (2, 64, 40), (3, 64, 40), (2, 700, 300)])
@pytest.mark.parametrize("precision", [workloads.FP64, workloads.FP32])
def test_one_iteration_in_equilibrium(lattice, nx, ny, precision):
    from paper_2505_13097_gb300 import solver
    for v in np.linspace(-0.02, 0.02, 20):   # (without 0, where FP32 resolves any update)
        S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, precision, {}, newton_max_iter=1)
        S.set_ic(np.full((ny, nx), v))
        S.step(1)
        st = S.stats()
        S.close()
        assert st["error"] == 0 and st["newton_nodes"] == nx * ny
        assert st["newton_iters"] == nx * ny and st["newton_max_iter"] == 1
