"""Populations in the subnormal range of FP32: a uniform field in equilibrium
keeps its value (to the rounding of a few subnormal operations, 2^-149 each; the
stored populations carry up to half of that each, theta of nine)."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,nx,ny", [(1, 64, 1), (1, 9000, 1), (2, 64, 40), (3, 64, 40), (2, 700, 300)])
@pytest.mark.parametrize("value", [1e-39, -3e-40])
def test_uniform_field_keeps_its_value(lattice, nx, ny, value):
    from paper_2505_13097_gb300 import solver
    S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, workloads.FP32, {}, bb_mode=1)
    S.set_ic(np.full((ny, nx), value))
    before = S.theta()
    S.step(2)
    th, st = S.theta(), S.stats()
    S.close()
    assert st["error"] == 0 and st["newton_nodes"] == nx * ny
    assert np.max(np.abs(before - value)) <= 9 * 2.0 ** -149
    assert np.max(np.abs(th - value)) <= 2 * 60 * 2.0 ** -149
