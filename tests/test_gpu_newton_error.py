"""Rounding error of the local Newton solve, theta' = m0 + (phi(theta) - phi(root))/Ste,
in units u = 2^-53.

phi = r or 1 - r, r = 1/(1 + E), E = exp(-2|x|/delta).  An error of r is half an
ulp (0.5 u) and E r^2 <= 0.25 times the relative error of E: 1.1 u of table and
product, and (at most 0.22 of) half an ulp of the argument: 0.9 u at most.  Two
phi and their difference: 2.5 u over Ste at most.  Their standard deviation:
0.289 u of r, 0.25 x 0.35 u and 0.06 u of E, twice, and 0.14 u of the difference:
0.46 u over Ste; 0.5 here.
"""
import math

import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
L = np.longdouble


def _phi(x, inv_delta):
    return 1 / (1 + np.exp(-2 * x * inv_delta))


def _root(m0, theta, inv_ste, inv_delta):
    """Bracketed Newton in long double (64 bits or more)."""
    pt = _phi(theta, inv_delta)
    lo, hi = m0 + (pt - 1) * inv_ste, m0 + pt * inv_ste
    x, old = (lo + hi) / 2, hi - lo
    for _ in range(300):
        p = _phi(x, inv_delta)
        f = (x - m0) + (p - pt) * inv_ste
        lo, hi = np.where(f < 0, x, lo), np.where(f > 0, x, hi)
        step = f / (1 + 2 * p * (1 - p) * inv_delta * inv_ste)
        xn = x - step
        out = (~((xn > lo) & (xn < hi)) | (np.abs(step) > old / 2)) & (np.abs(step) > 1e-18)
        xn = np.where(out, (lo + hi) / 2, xn)
        x, old = xn, np.abs(xn - x)
    assert np.all(old <= 1e-17)
    return x


@pytest.mark.parametrize("ste", [0.01, 0.1])
@pytest.mark.parametrize("delta", [0.005, 0.01])
@pytest.mark.parametrize("lo,hi", [(-6, 6), (6, 12), (-12, -6)])
def test_error_of_theta(ste, delta, lo, hi):
    # at the tails, where F' is near 1, an error of phi shows undamped.  D1Q3 at tau = 1 (1 - omega = 0): theta' is the sum of the populations after the step,
    # and theta and m0 are correctly rounded sums of three
    from paper_2505_13097_gb300 import solver
    n, errs = 4000, []
    for seed in range(1):
        th0 = workloads.random_field((1, n), lo * delta, hi * delta, seed=seed)
        S = solver.Stefan(1, n, 1, 1.0, delta, ste, workloads.FP64, {})
        S.set_ic(th0)
        S.step(1)
        th, st = S.theta()[0], S.stats()
        S.close()
        assert st["error"] == 0 and st["newton_nodes"] == n
        f0, f1 = (2 / 3) * th0[0], (1 / 6) * th0[0]
        theta = np.array([math.fsum((f0[x], f1[x], f1[x])) for x in range(1, n - 1)])
        m0 = np.array([math.fsum((f0[x], f1[x - 1], f1[x + 1])) for x in range(1, n - 1)])
        ref = _root(m0.astype(L), theta.astype(L), L(1.0 / ste), L(1.0 / delta))
        errs.append((th[1:-1].astype(L) - ref).astype(np.float64) / U)
    e = np.concatenate(errs)
    # the solve's own tolerance, 0.1 newton_tol, and the sum of three below 1/8
    assert np.max(np.abs(e)) <= 2.5 / ste + 1e-15 / U + 0.5
    assert np.sqrt(np.mean(e ** 2)) <= 0.5 / ste


@pytest.mark.parametrize("sea", [4.1, -3.9, 5.3, 6.7])
def test_error_with_a_shift(sea):
    # mushy nodes in a hot (cold) sea, which an FP32 state stores less half the mean: the sums
    # of its populations are exact in float pairs, and theta is their sum plus the shift
    import torch
    from paper_2505_13097_gb300 import solver
    delta, ste, nx, ny = 0.007, 1.0, 120, 90   # 2/delta has all its bits
    rng = np.random.Generator(np.random.PCG64(5))
    th0 = np.full((ny, nx), sea)
    th0[2:-2:3, 2:-2:3] = rng.uniform(-delta, delta, th0[2:-2:3, 2:-2:3].shape)
    S = solver.Stefan(2, nx, ny, 1.0, delta, ste, workloads.FP32, {}, stream=torch.cuda.Stream())
    S.set_ic(th0)
    buf = np.empty(S.state_bytes, dtype=np.uint8)
    S.get_state(buf)
    f = buf[:9 * (ny + 2) * S.row_stride * 4].view(np.float32).reshape(9, ny + 2, S.row_stride)[:, 1:-1, :nx].astype(np.float64)
    shift = float(buf[-256:-252].view(np.float32)[0])
    traj = S.new_theta_planes(1)
    torch.cuda.synchronize()
    S.step_record(1, traj)
    S.sync()
    got = traj[0, :, :nx].cpu().numpy()
    S.close()
    ex, ey = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    q = np.stack([np.roll(f[i], (ey[i], ex[i]), (0, 1)) for i in range(9)])
    at = (slice(2, -2, 3), slice(2, -2, 3))
    theta = (f.sum(0) + shift)[at].astype(L)      # multiples of 2^-28 below 8: exact
    m0 = (q.sum(0).astype(L) + L(shift))[at]
    ref = _root(m0, theta, L(1.0), L(1.0 / delta))
    e = (got[at].astype(L) - ref).astype(np.float64) / U
    # 2.5 u over Ste, the solve's tolerance, and theta' less the shift and itself, below 8: 4 u each
    assert np.max(np.abs(e)) <= 2.5 / ste + 1e-15 / U + 8.0
