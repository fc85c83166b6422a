"""Steps in one resident launch (lbm_stefan_step, _step_record) against the same
steps kernel by kernel (lbm_stefan_step_timed), over lattices at the edges of
the resident kernel's tiles: sides around 32, 128 and the thinnest lattices,
lattices with and without a first pass, and one whose mushy nodes fill the
queue several times over.

FP32: the same bits.  FP64: the zeroth moment is summed in another order, so a
node's theta differs by a few units of 2^-53, which a node leaving the mushy
zone carries over with gain phi'/Ste (up to 1/(2 delta Ste) = 500 here): 20
steps of 8 units with that gain, 1e-11.
"""
import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu

WALLS = [{}, {"W": (1, 1.0)}, {"S": (1, -1.0), "W": (1, -0.4), "N": (1, 0.3)}, {"E": (1, 0.2), "N": (1, -0.1)}]
SHAPES = [(3, 3), (4, 7), (5, 3), (31, 33), (33, 4), (128, 5), (129, 65), (257, 31), (700, 90), (1025, 130)]


def _field(nx, ny, seed):
    th = 0.3 * np.sin(np.arange(nx) / 9.0)[None, :] + 0.1 * np.cos(np.arange(ny) / 7.0)[:, None]
    return th + workloads.random_field((ny, nx), -0.02, 0.02, seed=seed)


def _pair(lattice, nx, ny, precision, method, walls, bb_mode, steps, th0):
    import torch
    from paper_2505_13097_gb300 import solver
    out = []
    for timed in (False, True):
        S = solver.Stefan(lattice, nx, ny, 0.84, 0.01, 0.1, precision, walls, bb_mode=bb_mode, stream=torch.cuda.Stream())
        S.set_method(method)
        S.set_ic(th0)
        (S.step_timed if timed else S.step)(steps)
        buf = np.empty(S.state_bytes, dtype=np.uint8)
        S.get_state(buf)
        # the populations of the nodes (EEBM's separate kernels leave values in the padding columns)
        q, elem = (9 if lattice == 2 else 5), np.float32 if precision else np.float64
        n = q * (ny + 2) * S.row_stride
        planes = buf[:n * np.dtype(elem).itemsize].view(elem).reshape(q, ny + 2, S.row_stride)[:, 1:-1, :nx]
        out.append((S.theta(), S.stats(), planes))
        S.close()
    return out


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("lattice", [2, 3])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("method", ["IREBM", "EEBM"])
def test_resident_equals_separate_kernels(shape, lattice, precision, method):
    nx, ny = shape
    for wi, walls in enumerate(WALLS):
        for bb in ((0, 1) if lattice == 2 else (0, 1, 2)):
            (ta, sa, ba), (tb, sb, bb_) = _pair(lattice, nx, ny, precision, method, walls, bb, 21, _field(nx, ny, wi))
            if precision == 1:
                assert np.array_equal(ba, bb_), (walls, bb)
            else:
                assert np.max(np.abs(ta - tb)) <= 1e-11, (walls, bb)
            assert sa["error"] == sb["error"] == 0
            assert sa["steps"] == sb["steps"] == 21
            assert sa["newton_nodes"] == sb["newton_nodes"]
            # sums of up to 133,000 terms below 12 (theta + phi/Ste), in FP32 pairs or exact
            tol = 1e-6 + 1e-9 * abs(sb["energy"])
            if precision == 1 and method == "EEBM":
                # each term is a plain FP32 sum of nine populations: ten half-ulps of 12
                tol = nx * ny * 10 * 12 * 2.0 ** -24
            assert abs(sa["energy"] - sb["energy"]) <= tol
            assert abs(sa["flux"] - sb["flux"]) <= 1e-6 + 1e-9 * abs(sb["flux"])


@pytest.mark.parametrize("precision", [0, 1])
def test_resident_mushy_everywhere(precision):
    # 2,050^2 nodes, all of them solved: several queues per step
    n = 2050 if precision else 1100
    th0 = workloads.random_field((n, n), -0.03, 0.03, seed=5)
    (ta, sa, ba), (tb, sb, bb) = _pair(2, n, n, precision, "IREBM", {"W": (1, 1.0)}, 0, 3, th0)
    assert sa["newton_nodes"] == sb["newton_nodes"] > 0.9 * n * n
    if precision:
        assert np.array_equal(ba, bb)
    else:
        assert np.max(np.abs(ta - tb)) <= 1e-11


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", [(40, 37), (515, 140)])
def test_resident_record(precision, shape):
    """Recorded planes are the fields after each step."""
    import torch
    from paper_2505_13097_gb300 import solver
    nx, ny = shape
    th0 = _field(nx, ny, 3)
    S = solver.Stefan(2, nx, ny, 0.9, 0.01, 0.1, precision, {"W": (1, 0.5)}, stream=torch.cuda.Stream())
    S.set_ic(th0)
    traj = S.new_theta_planes(4)
    torch.cuda.synchronize()
    S.step_record(4, traj)
    S.sync()
    S.set_ic(th0)
    for k in range(4):
        S.step(1)
        # theta' against the sum of the stored populations: their rounding
        tol = 1e-14 if precision == 0 else 9 * 2.0 ** -25
        assert np.max(np.abs(traj[k, :, :nx].cpu().numpy() - S.theta())) <= tol
    S.close()


def test_resident_many_steps():
    """More steps than sets of sums in flight; the energy balance of every step holds."""
    from paper_2505_13097_gb300 import solver
    S = solver.Stefan(2, 130, 64, 1.0, 0.01, 0.1, 0, {"W": (1, 1.0)})
    S.set_ic(_field(130, 64, 1))
    S.step(300)
    st = S.stats()
    assert st["steps"] == 300 and st["error"] == 0
    # E and the flux: 8,320 terms below 12 with relative rounding 2^-53 each
    assert st["imbalance_max"] <= 8320 * 12 * 4 * 2.0 ** -53
    S.close()
