"""A caller's own CUDA graph of lbm_stefan_step / _step_record: its replays see the
walls and the Stefan number of their time, as the library's calls do."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu


def _field(nx, ny):
    return workloads.random_field((ny, nx), -0.25, -0.15, seed=nx)


@pytest.mark.parametrize("lattice,nx,ny,precision,method", [
    (1, 200, 1, 0, "IREBM"), (1, 200, 1, 1, "IREBM"), (1, 200, 1, 0, "EEBM"), (1, 200, 1, 0, "ILFBM"), (1, 5000, 1, 0, "IREBM"),
    (2, 150, 64, 0, "IREBM"), (2, 150, 64, 1, "IREBM"), (2, 700, 300, 1, "IREBM"), (2, 150, 64, 1, "EEBM"), (3, 150, 64, 1, "IREBM"),
    (3, 150, 64, 0, "EEBM")])
@pytest.mark.parametrize("steps", [6, 40])
def test_replay_after_new_walls(lattice, nx, ny, precision, method, steps):
    import torch
    from paper_2505_13097_gb300 import solver
    s = torch.cuda.Stream()
    S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, precision, {"W": (1, 1.0)}, stream=s,
                      **({"newton_tol": 1e-12, "newton_max_iter": 200} if method == "ILFBM" else {}))
    S.set_method(method)
    S.set_ic(_field(nx, ny))
    S.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        S.step(steps)   # an even number: the replay starts from the state that the capture did
    S.set_bc("W", 1, 2.0)
    S.set_ste(0.2)
    S.set_ic(_field(nx, ny))
    with torch.cuda.stream(s):
        g.replay()
    th, st = S.theta(), S.stats()
    S.set_ic(_field(nx, ny))
    S.step(steps)
    ref, sr = S.theta(), S.stats()
    S.close()
    assert st["steps"] == sr["steps"] == steps and st["error"] == sr["error"] == 0
    assert np.max(ref) > 1.5
    # FP32: the same bits by either route; FP64: sums of a few nodes' terms, gain phi'/Ste at most 250 per step
    assert np.max(np.abs(th - ref)) <= (0.0 if precision else 1e-11)
    assert abs(st["energy"] - sr["energy"]) <= 1e-5 + 1e-9 * abs(sr["energy"])


@pytest.mark.parametrize("lattice,nx,ny", [(1, 200, 1), (2, 150, 64)])
def test_recorded_replay(lattice, nx, ny):
    """A graph captured before the wall changed records what one captured after does, bit for bit."""
    import torch
    from paper_2505_13097_gb300 import solver
    s = torch.cuda.Stream()
    S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, 1, {"W": (1, 1.0)}, stream=s)
    traj = S.new_theta_planes(4)
    graphs, out = [], []
    for wall in (1.0, 2.0):
        S.set_bc("W", 1, wall)
        S.set_ic(_field(nx, ny))
        S.sync()
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1], stream=s):
            S.step_record(4, traj)
    for g in graphs:
        S.set_ic(_field(nx, ny))
        with torch.cuda.stream(s):
            g.replay()
        S.sync()
        out.append(traj[:, :, :nx].cpu().numpy())
    S.close()
    assert np.max(out[1]) == 2.0
    assert np.array_equal(out[0], out[1])
