"""Nodes that leave the mushy band in one step: the root lies at an end of the
solve's bracket [m0 + (phi(theta) - 1)/Ste, m0 + phi(theta)/Ste], to within its
rounding.  Each solve stays within the iteration limit, and theta' is m0 plus the
latent heat released: rounding of phi and of terms below 8 (16 u over Ste at
most), and 1e-14 for the solve's tolerance."""
import math

import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("delta", [0.005, 0.01])
def test_roots_at_the_bracket(sign, delta):
    from paper_2505_13097_gb300 import solver
    n, ste = 4001, 0.3
    for seed in range(20):
        rng = np.random.Generator(np.random.PCG64(seed))
        th0 = np.empty((1, n))
        th0[0, ::2] = sign * rng.uniform(7.0, 10.0, (n + 1) // 2)
        th0[0, 1::2] = sign * rng.uniform(5 * delta, 9 * delta, n // 2)
        S = solver.Stefan(1, n, 1, 1.0, delta, ste, workloads.FP64, {})
        S.set_ic(th0)
        S.step(1)
        th, st = S.theta()[0], S.stats()
        S.close()
        assert st["error"] == 0 and st["newton_nodes"] >= n // 2 - 1
        x = np.arange(3, n - 3, 2)
        m0 = np.array([math.fsum((2 / 3 * th0[0, k], 1 / 6 * th0[0, k - 1], 1 / 6 * th0[0, k + 1])) for k in x])
        phi = 1 / (1 + np.exp(-2 * th0[0, x] / delta))
        ref = m0 + (phi - (1.0 if sign > 0 else 0.0)) / ste
        assert np.max(np.abs(th[x] - ref)) <= 16 * 2.0 ** -53 / ste + 1e-14
