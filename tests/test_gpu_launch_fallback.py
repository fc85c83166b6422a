"""Calls whose resident grid the device refuses (the hook's max_blocks), and calls
cut into several launches (max_steps), give what a normal call gives."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


def _field(nx, ny, seed=0):
    return 0.3 * np.sin(np.arange(nx) / 9.0)[None, :] + workloads.random_field((ny, nx), -0.02, 0.02, seed=seed)


@pytest.mark.parametrize("lattice", [2, 3])
@pytest.mark.parametrize("max_blocks,max_steps", [(0, 0), (20, 0), (3, 0), (2, 3)])
def test_ilfbm_grids(lattice, max_blocks, max_steps):
    """2D ILFBM: any grid gives the same bits and statistics."""
    import torch
    from paper_2505_13097_gb300 import _abi, solver
    out = []
    for blocks, steps in ((0, 0), (max_blocks, max_steps)):
        S = solver.Stefan(lattice, 130, 90, 0.84, 0.01, 0.1, 0, {"W": (1, 1.0)}, stream=torch.cuda.Stream(), newton_tol=1e-12,
                          newton_max_iter=20000)
        S.set_method("ILFBM")
        S.set_launch_test(max_blocks=blocks, max_steps=steps)
        S.set_ic(_field(130, 90))
        S.step(7)
        out.append((S.stats(), S.theta()))
        S.close()
    assert out[0][0] == out[1][0] and out[0][0]["steps"] == 7
    assert np.array_equal(out[0][1], out[1][1])
    S = solver.Stefan(lattice, 130, 90, 0.84, 0.01, 0.1, 0, {"W": (1, 1.0)}, stream=torch.cuda.Stream())
    S.set_method("ILFBM")
    S.set_launch_test(max_blocks=1)
    S.set_ic(_field(130, 90))
    with pytest.raises(_abi.LBMError) as ei:
        S.step(1)
    assert ei.value.status == _abi.LBM_ERR_CUDA
    S.close()
