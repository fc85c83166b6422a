"""FP64 collision of saturated nodes, bit for bit: M0 rounded once, c = omega M0
(D1Q3: M0 - (1 - omega) M0), w_i c and (1 - omega) q_i + w_i c rounded once each,
restated with fractions.

A constant omega w_i rounded ahead of the step would save a multiplication, but
its error is the same at every node and step: the field's sum would drift by it
(tau = 0.62: 2.2e-16 of itself per step on D1Q3 and D2Q5).
"""
from fractions import Fraction as F

import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu

EX = {1: (0, 1, -1), 3: (0, 1, 0, -1, 0), 2: (0, 1, 0, -1, 0, 1, -1, -1, 1)}
EY = {1: (0, 0, 0), 3: (0, 0, 1, 0, -1), 2: (0, 0, 1, 0, -1, 1, 1, -1, -1)}
W = {1: (2 / 3, 1 / 6, 1 / 6), 3: (1 / 3,) + (1 / 6,) * 4, 2: (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4}


def _rn(x):
    return F(float(x))   # a fraction's float is correctly rounded


# the resident and the separate kernels; D1Q3: one block, and one launch per step
@pytest.mark.parametrize("lattice,nx,ny,timed", [(1, 300, 1, False), (1, 5000, 1, False), (2, 40, 37, False), (2, 700, 300, False),
                                                 (2, 131, 35, True), (3, 40, 37, False), (3, 700, 300, False), (3, 131, 35, True)])
@pytest.mark.parametrize("tau", [0.55, 0.62, 0.84, 1.3, 2.5])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_saturated_collision(lattice, nx, ny, timed, tau, sign):
    from paper_2505_13097_gb300 import solver
    th = sign * workloads.random_field((ny, nx), 1.0, 2.0, seed=nx)
    S = solver.Stefan(lattice, nx, ny, tau, 0.01, 0.1, workloads.FP64, {}, bb_mode=1)
    S.set_ic(th)
    (S.step_timed if timed else S.step)(1)
    q = len(W[lattice])
    buf = np.empty(S.state_bytes, dtype=np.uint8)
    S.get_state(buf)
    got = buf[:q * (ny + 2) * S.row_stride * 8].view(np.float64).reshape(q, ny + 2, S.row_stride)[:, 1:-1, :nx]
    S.close()
    omega = 1.0 / tau
    omc = F(1.0 - omega)
    rng = np.random.Generator(np.random.PCG64(1))
    for _ in range(60):
        x = int(rng.integers(1, nx - 1))
        y = int(rng.integers(1, ny - 1)) if ny > 1 else 0
        qs = [F(W[lattice][i] * th[y - EY[lattice][i], x - EX[lattice][i]]) for i in range(q)]
        m0 = _rn(sum(qs))   # terms within 2^6 of one another: the moment's integer sum is exact
        c = _rn(m0 - omc * m0) if lattice == 1 else _rn(F(omega) * m0)
        for i in range(q):
            assert got[i, y, x] == float(omc * qs[i] + _rn(F(W[lattice][i]) * c)), (x, y, i)
