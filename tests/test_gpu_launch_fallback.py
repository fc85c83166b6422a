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


def _run(lattice, nx, ny, precision, method, calls, **hook):
    import torch
    from paper_2505_13097_gb300 import solver
    S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, precision, {"W": (1, 1.0), "N": (1, -0.3)}, stream=torch.cuda.Stream())
    S.set_method(method)
    S.set_launch_test(**hook)
    S.set_ic(_field(nx, ny))
    for n in calls:
        S.step(n)
    out = S.theta(), S.stats()
    S.close()
    return out


# 41 and 70 steps: replays of the separate kernels' graph between single steps
@pytest.mark.parametrize("lattice,nx,ny", [(2, 40, 37), (2, 700, 90), (3, 515, 60)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("method", ["IREBM", "EEBM"])
@pytest.mark.parametrize("hook", [{"max_blocks": 1}, {"max_steps": 7}])
def test_steps(lattice, nx, ny, precision, method, hook):
    th, st = _run(lattice, nx, ny, precision, method, (111,))
    t2, s2 = _run(lattice, nx, ny, precision, method, (41, 70), **hook)
    if precision or "max_steps" in hook:
        assert np.array_equal(th, t2)   # the same kernels, or kernels that round alike
    else:
        # FP64 routes round differently at walls: a node in the mushy zone carries that over with
        # gain phi'/Ste at most 500 a step, and relaxes it by its neighbours: 111 steps of 8 units
        assert np.max(np.abs(th - t2)) <= 111 * 8 * 500 * 2.0 ** -53
    for f in ("steps", "newton_nodes", "error"):
        assert st[f] == s2[f]
    tol = 1e-6 + 1e-9 * abs(st["energy"])
    if precision and method == "EEBM":
        tol = nx * ny * 10 * 12 * 2.0 ** -24   # plain FP32 sums of nine populations: ten half-ulps of 12
    assert abs(st["energy"] - s2["energy"]) <= tol


@pytest.mark.parametrize("lattice,nx,ny,max_steps", [(2, 1021, 777, 3), (2, 40, 37, 1), (3, 515, 60, 2)])
def test_recorded_steps_across_launches(lattice, nx, ny, max_steps):
    """Recorded planes advance with each launch of a call."""
    import torch
    from paper_2505_13097_gb300 import solver
    out = []
    for hook in ({}, {"max_steps": max_steps}):
        S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, 1, {"W": (1, 1.0)}, stream=torch.cuda.Stream())
        S.set_launch_test(**hook)
        S.set_ic(_field(nx, ny))
        traj = S.new_theta_planes(7)
        torch.cuda.synchronize()
        S.step_record(7, traj)
        S.step(1)
        S.sync()
        out.append((traj[:, :, :nx].cpu().numpy(), S.theta()))
        S.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("hook", [{"max_blocks": 1}, {"max_steps": 3}])
def test_adjoint_segment(hook):
    import torch
    from paper_2505_13097_gb300 import solver
    nx, ny, n = 200, 90, 10
    out = []
    for h in ({}, hook):
        S = solver.Stefan(2, nx, ny, 0.84, 0.01, 0.1, 1, {"W": (1, 1.0)}, stream=torch.cuda.Stream())
        S.set_launch_test(**h)
        S.set_ic(_field(nx, ny))
        cp, a, b = S.new_state_buffer(), S.new_state_buffer(), S.new_state_buffer()
        traj = S.new_theta_planes(n + 1)
        last = S.new_theta_planes(1)
        target = torch.full((ny, nx), 0.3, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        S.get_state(cp)
        S.step(n)
        S.theta_plane(last)
        S.adjoint_seed(last, target, a, want_loss=False)
        lam, _ = S.adjoint_segment(cp, n, traj, a, b)
        g0 = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
        gw, gs = S.adjoint_finish(lam, g0)
        out.append((g0.cpu().numpy(), S.theta()))
        S.close()
    assert np.array_equal(out[0][1], out[1][1])
    # the recorded temperatures of solved nodes are FP64 and may differ in their last bits between
    # the two routes: the FP32 adjoint's own accuracy
    assert np.max(np.abs(out[0][0] - out[1][0])) <= 1e-4 * np.max(np.abs(out[0][0]))


@pytest.mark.parametrize("own_stream", [False, True])
def test_batches(own_stream):
    """The separate kernels of a batch, on a stream of its own the split step."""
    import torch
    from paper_2505_13097_gb300 import solver
    cases = [workloads.Case("b%d" % k, 2, 33 + 90 * k, 240 - 40 * k, 1.0, 0.01, 0.1, {"W": (1, 1.0)}, 0, workloads.FP32)
             for k in range(5)]
    out = []
    for hook in ({}, {"max_blocks": 1}, {"max_steps": 7}):
        B = solver.StefanBatch(cases, stream=torch.cuda.Stream() if own_stream else None)
        B.set_launch_test(**hook)
        for k, c in enumerate(cases):
            B.set_ic(k, _field(c.nx, c.ny, k))
        B.step(41)
        B.step(70)
        out.append([(B.theta(k), B.stats(k)) for k in range(len(cases))])
        B.close()
    for other in out[1:]:
        for (th, st), (t2, s2) in zip(out[0], other):
            assert np.array_equal(th, t2)
            for f in ("steps", "newton_nodes", "newton_iters", "newton_max_iter", "error"):
                assert st[f] == s2[f]
            assert abs(st["energy"] - s2["energy"]) <= 1e-6 + 1e-9 * abs(st["energy"])


def test_handles_side_by_side():
    """Resident launches of several handles, on streams and threads of their own."""
    import threading
    import torch
    from paper_2505_13097_gb300 import solver
    jobs = [(2, 700, 300, 1, "IREBM"), (2, 130, 64, 1, "IREBM"), (3, 515, 260, 0, "IREBM"), (2, 300, 200, 1, "EEBM")]
    alone = [_run(*j, (30, 31)) for j in jobs]
    got = [None] * len(jobs)

    def work(i):
        for _ in range(3):
            got[i] = _run(*jobs[i], (30, 31))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (th, st), (t2, s2) in zip(alone, got):
        assert np.array_equal(th, t2) and st == s2


def test_launch_counts():
    """What bench.py reports as launches: counted where they are made."""
    import torch
    from paper_2505_13097_gb300 import solver
    S = solver.Stefan(2, 1021, 777, 1.0, 0.01, 0.1, 1, {"W": (1, 1.0)}, stream=torch.cuda.Stream())
    S.set_ic(_field(1021, 777))
    assert S.resident_launches() == (0, 0)
    S.step(6000)   # 2^32 node updates, 5,413 steps, in a launch
    assert S.resident_launches() == (2, 6000)
    S.set_launch_test(max_steps=4)
    S.step(10)
    assert S.resident_launches() == (5, 6010)
    S.set_launch_test(max_blocks=1)
    S.step(40)
    S.sync()
    assert S.resident_launches() == (5, 6010) and S.stats()["steps"] == 6050
    S.close()
