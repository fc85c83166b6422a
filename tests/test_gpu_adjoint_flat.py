"""One reverse step of the FP32 flat adjoint kernel against the FP64 marching
kernel on the same adjoint state and temperatures, over lattices at the edges
of its 64 x 16 tiles and of the ring of two nodes along the walls.

Bound: the FP32 form takes theta to 20 bits, an error of 2 x 13 x 2^-20 =
2.5e-5 in exp(-2 theta/delta) at the edge of the band; mu and nu hold two such
factors, and some 30 FP32 roundings add 2e-6: 1e-4 of the largest value."""
import ctypes

import numpy as np
import pytest

from paper_2505_13097_gb300 import workloads

pytestmark = pytest.mark.gpu

WALLS = [{}, {"W": (1, 0.9)}, {"W": (1, 0.2), "S": (1, -0.3)}, {"E": (1, -0.1), "N": (1, 0.4)}]


@pytest.mark.parametrize("shape", [(2, 2), (3, 3), (4, 5), (5, 4), (6, 6), (67, 19), (68, 20), (69, 21), (133, 37), (200, 5)])
@pytest.mark.parametrize("bb_mode", [0, 1])
@pytest.mark.parametrize("wi", range(len(WALLS)))
def test_flat_reverse_step(shape, bb_mode, wi):
    import torch
    from paper_2505_13097_gb300 import solver
    nx, ny = shape
    rng = np.random.Generator(np.random.PCG64(nx * 100 + ny))
    th = [rng.uniform(-0.2, 0.2, (ny, nx)) for _ in range(1)]
    th.append(th[0] + rng.uniform(-0.01, 0.01, (ny, nx)))
    lam = rng.uniform(-1, 1, (9, ny, nx))
    res = []
    for prec in (workloads.FP32, workloads.FP64):
        S = solver.Stefan(2, nx, ny, 0.8, 0.02, 0.2, prec, WALLS[wi], bb_mode=bb_mode)
        dt = torch.float32 if prec else torch.float64
        es = 4 if prec else 8
        planes = S.new_theta_planes(2)
        planes.zero_()
        for k in range(2):
            planes[k, :, :nx] = torch.tensor(th[k], device="cuda")
        a, b = S.new_state_buffer(), S.new_state_buffer()
        n = 9 * (ny + 2) * S.row_stride

        def view(buf):
            return buf[:n * es].view(dt).view(9, ny + 2, S.row_stride)[:, 1:-1, :nx]
        view(a)[:] = torch.tensor(lam, device="cuda").to(dt)
        # clears the gradient accumulators
        S.adjoint_seed(planes[1], torch.zeros((ny, nx), dtype=torch.float64, device="cuda"), b, want_loss=False)
        S.adjoint_step(planes[0], planes[1], a, b)
        g0 = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
        gw, gs = S.adjoint_finish(b, g0)
        res.append((view(b).double().cpu().numpy(), np.array(gw), gs))
        S.close()
    (x, gw, gs), (y, hw, hs) = res
    assert np.max(np.abs(x - y)) <= 1e-4 * np.max(np.abs(y))
    # sums over the nodes of terms of the same accuracy (Ste's up to 1/Ste^2 each)
    assert np.max(np.abs(gw - hw)) <= 1e-4 * (np.max(np.abs(y)) * nx * ny)
    assert abs(gs - hs) <= 1e-4 * nx * ny / 0.2 ** 2


@pytest.mark.parametrize("shape", [(67, 19), (133, 37)])
def test_state_buffers_on_8_bytes(shape):
    """Adjoint states that are not on 16 bytes take the marching kernel: the same
    function in other FP32 roundings, 2e-6 of the largest value (above)."""
    import torch
    from paper_2505_13097_gb300 import solver
    nx, ny = shape
    rng = np.random.Generator(np.random.PCG64(nx))
    S = solver.Stefan(2, nx, ny, 0.8, 0.02, 0.2, workloads.FP32, {"W": (1, 0.9)})
    planes = S.new_theta_planes(2)
    planes.zero_()
    th = rng.uniform(-0.2, 0.2, (ny, nx))
    planes[0, :, :nx] = torch.tensor(th, device="cuda")
    planes[1, :, :nx] = torch.tensor(th + rng.uniform(-0.01, 0.01, (ny, nx)), device="cuda")
    lam = torch.tensor(rng.uniform(-1, 1, (9, ny, nx)), device="cuda").float()
    n, out = 9 * (ny + 2) * S.row_stride, []
    for off in (0, 8):
        size = S.new_state_buffer().numel()
        a, b = (torch.zeros(size + 16, dtype=torch.uint8, device="cuda")[off:off + size] for _ in range(2))
        assert a.data_ptr() % 16 == off and b.data_ptr() % 16 == off

        def view(buf):
            return buf[:4 * n].view(torch.float32).view(9, ny + 2, S.row_stride)[:, 1:-1, :nx]
        view(a)[:] = lam
        S.adjoint_step(planes[0], planes[1], a, b)
        S.sync()
        out.append(view(b).double().cpu().numpy())
    S.close()
    assert np.max(np.abs(out[0] - out[1])) <= 2e-6 * np.max(np.abs(out[0]))
