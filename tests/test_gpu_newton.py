"""The liquid fraction and the local Newton solve of Eq. (14) at the edges of
their ranges: next to 0, at the saturation bound 19.5 delta, and on fields
whose nodes jump across the front in one step.

Bounds.  phi = 1/(1 + exp(-2x/delta)) with FP64 rounding in its argument
(error of phi at most 0.3 units of 2^-53), its exponential (0.8), its
reciprocal (1) and product (0.5), and exactly 0 or 1 from 19.5 delta on (0.1):
4 units of 2^-53.  theta' = m0 + (phi(theta) - phi(root))/Ste: two phi on each
side of the comparison, 16 units of 2^-53 over Ste, and 1e-14 for the solve's
tolerance and the sums of nine populations.
"""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("delta", [0.005, 0.01, 1.0])
def test_phi_field(delta):
    from paper_2505_13097_gb300 import solver
    rng = np.random.Generator(np.random.PCG64(7))
    z = np.concatenate([rng.uniform(-25, 25, 4000), rng.uniform(-1, 1, 1000), [0.0, 1e-300, -1e-300, 1e-17, -1e-17, 1e3, -1e3],
                        19.5 * (1 + np.arange(-40, 41) * 2.0 ** -50), -19.5 * (1 + np.arange(-40, 41) * 2.0 ** -50)])
    th0 = np.zeros((2, z.size))
    th0[:] = z * delta
    S = solver.Stefan(2, z.size, 2, 1.0, delta, 0.1, workloads.FP64)
    S.set_ic(th0)
    th, ph, H = S.fields()
    S.close()
    x = th.astype(np.longdouble) / np.longdouble(delta)
    ref = 1 / (1 + np.exp(-2 * x))
    assert np.max(np.abs(ph.astype(np.longdouble) - ref)) <= 4 * U
    assert np.all(ph[th >= 19.6 * delta] == 1.0) and np.all(ph[th <= -19.6 * delta] == 0.0)


@pytest.mark.parametrize("lattice", [1, 2, 3])
@pytest.mark.parametrize("ste", [0.01, 0.1, 1.0])
@pytest.mark.parametrize("delta", [0.005, 0.01])
@pytest.mark.parametrize("spread", [0.3, 3.0, 30.0])
def test_one_step_roots(orc, lattice, ste, delta, spread):
    from paper_2505_13097_gb300 import solver
    nx, ny = (1201, 1) if lattice == 1 else (67, 35)
    th0 = workloads.random_field((ny, nx), -spread * delta, spread * delta, seed=11)
    walls = {"W": (1, 0.5)}
    S = solver.Stefan(lattice, nx, ny, 0.9, delta, ste, workloads.FP64, walls)
    S.set_ic(th0)
    S.step(1)
    th, st = S.theta(), S.stats()
    S.close()
    P = orc.Problem(lattice, nx, ny, tau=0.9, delta=delta, ste=ste, walls=walls)
    _, ref = P.run(th0, 1)
    assert st["newton_nodes"] > 0
    assert np.max(np.abs(th - ref)) <= 16 * U / ste + 1e-14
