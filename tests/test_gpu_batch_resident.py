"""FP32 batches in resident launches: every problem gives the bits it gives alone
(the kernels share their arithmetic), over sides at the edges of the 128 x 8
tiles and of the wall units, mushy tiles that fill their queue, calls of one and
many steps, and both schedules."""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (3, 5), (5, 3), (31, 34), (33, 8), (64, 66), (127, 9), (128, 10), (129, 65), (130, 97), (257, 40), (400, 35), (700, 20)]
WALLS = [{}, {"W": (1, 1.0)}, {"S": (1, -1.0), "W": (1, -0.4), "N": (1, 0.3)}, {"E": (1, 0.2), "N": (1, -0.1)}]


def _cases():
    return [workloads.Case("b%d" % k, 2, nx, ny, (0.84, 1.0, 0.62)[k % 3], 0.01, (0.1, 0.01, 0.5)[k % 3], WALLS[k % 4], 0,
                           workloads.FP32) for k, (nx, ny) in enumerate(SIZES)]


def _field(c, k):
    # every third problem is mushy all over
    if k % 3 == 0:
        return workloads.random_field((c.ny, c.nx), -0.03, 0.03, seed=k)
    return 0.3 * np.sin(np.arange(c.nx) / 9.0)[None, :] + workloads.random_field((c.ny, c.nx), -0.02, 0.02, seed=k)


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("calls", [(40,), (1, 2, 33, 4)])
def test_batch_equals_single(own_stream, calls):
    import torch
    from paper_2505_13097_gb300 import solver
    cases = _cases()
    stream = torch.cuda.Stream() if own_stream else None
    B = solver.StefanBatch(cases, stream=stream)
    for schedule in (1, 0):
        B.set_schedule(8, schedule)
        for k, c in enumerate(cases):
            B.set_ic(k, _field(c, k))
        for n in calls:
            B.step(n)
        for k, c in enumerate(cases):
            S = solver.Stefan.from_case(c, stream=stream)
            S.set_ic(_field(c, k))
            S.step(sum(calls))
            th, st, sb = S.theta(), S.stats(), B.stats(k)
            S.close()
            assert np.array_equal(B.theta(k), th), (k, c.nx, c.ny)
            for f in ("steps", "newton_nodes", "newton_iters", "newton_max_iter", "error"):
                assert sb[f] == st[f], (k, f)
            # FP32 pair sums of at most 16,800 terms below 101 (theta + phi/Ste)
            assert abs(sb["energy"] - st["energy"]) <= 1e-6 + 1e-9 * abs(st["energy"])
            assert abs(sb["flux"] - st["flux"]) <= 1e-6 + 1e-9 * abs(st["flux"])
    B.close()
