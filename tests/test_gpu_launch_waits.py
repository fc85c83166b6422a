"""Bounded waits of the resident launches, without a GPU fault: one block does not
arrive at a barrier, the waits for it run out after 20 ms, every block leaves, the
launch ends normally and the next synchronizing call returns LBM_ERR_TIMEOUT.
The handle then takes a new initial field and gives the bits and the statistics of
a fresh one: barrier and sums are clean."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


def _field(nx, ny, seed=0):
    return 0.3 * np.sin(np.arange(nx) / 9.0)[None, :] + workloads.random_field((ny, nx), -0.02, 0.02, seed=seed)


# a lattice of items alone, one with a first pass; ILFBM: barriers of the inner iterations
@pytest.mark.parametrize("lattice,nx,ny,precision,method", [
    (2, 40, 37, 1, "IREBM"), (2, 700, 300, 1, "IREBM"), (2, 700, 300, 0, "IREBM"), (3, 700, 300, 1, "IREBM"),
    (2, 700, 300, 1, "EEBM"), (2, 90, 70, 0, "ILFBM")])
@pytest.mark.parametrize("withhold", [0, 2, 4])
def test_withheld_arrival_times_out(lattice, nx, ny, precision, method, withhold):
    import torch
    from paper_2505_13097_gb300 import _abi, solver
    kw = {"newton_tol": 1e-12, "newton_max_iter": 400} if method == "ILFBM" else {}

    def make():
        S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, precision, {"W": (1, 1.0)}, stream=torch.cuda.Stream(), **kw)
        S.set_method(method)
        return S
    S, T = make(), make()
    S.set_launch_test(wait_limit_s=0.02, withhold=withhold)
    S.set_ic(_field(nx, ny))
    S.step(5)   # barrier 4: after the last step, where the statistics alone wait
    with pytest.raises(_abi.LBMError) as ei:
        S.sync()
    assert ei.value.status == _abi.LBM_ERR_TIMEOUT
    S.set_launch_test()
    out = []
    for h in (S, T):
        h.set_ic(_field(nx, ny))
        h.step(6)
        out.append((h.stats(), h.theta()))
        h.close()
    assert out[0][0]["error"] == 0
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("withhold", [0, 1, 2, 4])
def test_batch_after_a_timeout(withhold):
    import torch
    from paper_2505_13097_gb300 import _abi, solver
    cases = [workloads.Case("b%d" % k, 2, 33 + 60 * k, 200 - 30 * k, 1.0, 0.01, 0.1, {"W": (1, 1.0)}, 0, workloads.FP32)
             for k in range(5)]
    B = solver.StefanBatch(cases, stream=torch.cuda.Stream())
    F = solver.StefanBatch(cases, stream=torch.cuda.Stream())
    B.set_launch_test(wait_limit_s=0.02, withhold=withhold)
    for k, c in enumerate(cases):
        B.set_ic(k, _field(c.nx, c.ny, k))
    B.step(6 if withhold != 4 else 5)
    for k in range(len(cases)):
        with pytest.raises(_abi.LBMError) as ei:
            B.theta(k)
        assert ei.value.status == _abi.LBM_ERR_TIMEOUT
    B.set_launch_test()
    if withhold == 4:
        B.step(1)   # set_ic wants an even number of steps
    for b in (B, F):
        for k, c in enumerate(cases):
            b.set_ic(k, _field(c.nx, c.ny, k))
        b.step(1)
        first = [b.stats(k) for k in range(len(cases))]
        b.step(5)
        b.out = [(first[k], b.stats(k), b.theta(k)) for k in range(len(cases))]
        b.close()
    for x, y in zip(B.out, F.out):
        assert x[0] == y[0] and x[1] == y[1]
        assert np.array_equal(x[2], y[2])


@pytest.mark.parametrize("lattice,limit,steps,maxit", [(2, 0.002, 100, 400), (3, 0.005, 2, 20000)])
def test_a_long_step_is_no_timeout(lattice, limit, steps, maxit):
    """The bound counts from the last arrival of any block: a launch whose steps (D2Q5: many
    inner iterations) or whose statistics' waits (16 steps ahead) last longer runs to its end."""
    import torch
    from paper_2505_13097_gb300 import solver
    out = []
    for w in (limit, 5.0):
        S = solver.Stefan(lattice, 200, 150, 0.84, 0.01, 0.0521, 0, {"W": (1, -2.0), "S": (1, -2.0)},
                          stream=torch.cuda.Stream(), newton_tol=1e-12, newton_max_iter=maxit)
        S.set_method("ILFBM")
        S.set_launch_test(wait_limit_s=w)
        S.set_ic(_field(200, 150) + 0.7)
        S.step(steps)
        out.append((S.stats(), S.theta()))
        S.close()
    assert out[0][0]["newton_max_iter"] > 20 and out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])


def test_hook_rejects_bad_values():
    from paper_2505_13097_gb300 import _abi, solver
    c = workloads.melt_2d(n=64, steps=1)
    S, B = solver.Stefan.from_case(c), solver.StefanBatch([c])
    for bad in ((0.0, -1, 0, 0), (61.0, -1, 0, 0), (float("nan"), -1, 0, 0), (1.0, -2, 0, 0), (1.0, -1, -1, 0), (1.0, -1, 0, -1)):
        for h in (S, B):
            with pytest.raises(_abi.LBMError) as ei:
                h.set_launch_test(*bad)
            assert ei.value.status == _abi.LBM_ERR_ARG
    S.close()
    B.close()
