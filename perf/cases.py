"""Measured cases of the library: what a user has it do, through its public entry points.

A case is a plain dict.  ``prepare`` builds what a user's program holds before
the call (solver handle, initial field, checkpoint, buffers), ``run`` is one
pass from a known start: restart or initial field, a number of time steps,
read-out.  ``exact`` repeats the pass in plain torch, in 64 bits.

Initial fields are developed fronts (a molten or frozen layer along the
Dirichlet walls with a diffusive tail, front position and noise from the
seed), as a run meets them in its middle, at the temperatures, Stefan numbers,
widths and relaxation times of the workloads in
``paper_2505_13097_gb300.workloads``.

Outputs of the FP32 form are FP32 (its populations; batch temperatures and
gradients collected in FP32, the accuracy of the form), those of the FP64 form
the FP64 fields.
"""
from __future__ import annotations

import ctypes
import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_2505_13097_gb300 import _abi
from paper_2505_13097_gb300.autograd import misfit
from paper_2505_13097_gb300.solver import Stefan, StefanBatch
from paper_2505_13097_gb300.workloads import CAVITY_STE, Case

D1Q3, D2Q9, D2Q5 = _abi.LBM_D1Q3, _abi.LBM_D2Q9, _abi.LBM_D2Q5
FP64, FP32 = _abi.LBM_FP64, _abi.LBM_FP32

EX = {D1Q3: (0, 1, -1), D2Q5: (0, 1, 0, -1, 0), D2Q9: (0, 1, 0, -1, 0, 1, -1, -1, 1)}
EY = {D1Q3: (0, 0, 0), D2Q5: (0, 0, 1, 0, -1), D2Q9: (0, 0, 1, 0, -1, 1, 1, -1, -1)}
W = {D1Q3: (2 / 3, 1 / 6, 1 / 6), D2Q5: (1 / 3,) + (1 / 6,) * 4, D2Q9: (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4}
OPP = {D1Q3: (0, 2, 1), D2Q5: (0, 3, 4, 1, 2), D2Q9: (0, 3, 4, 1, 2, 7, 8, 5, 6)}

# scenes: Dirichlet walls with their temperature, and the temperature far from them
SCENES = {
    "melt": ({"W": 1.0}, -0.2),                  # melting from the west wall
    "melt_1d": ({"W": 1.0}, -0.5),               # the 1D melting run
    "bar": ({"W": 1.0, "E": -0.5}, -0.5),        # the 1D bar, both ends held
    "corner": ({"W": -1.0, "S": -1.0}, 0.3),     # freezing from a corner
    "cavity": ({"W": -2.0, "S": -2.0}, 1.0),     # the 2D cavity frozen from two walls
}


def _single(name, lattice, nx, ny, precision, method, scene, steps, tau, delta, ste, bb_mode=0, start="ic"):
    c = dict(kind="single", lattice=lattice, nx=nx, ny=ny, precision=precision, method=method, scene=scene, steps=steps,
             tau=tau, delta=delta, ste=ste, bb_mode=bb_mode, start=start)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the large production run: a restart from a checkpoint, 64 steps, the next checkpoint
        _single("melt_2d_4096_fp32", D2Q9, 4096, 4096, FP32, "IREBM", "melt", 64, 1.0, 0.01, 0.1, start="state"),
        # an ordinary lattice of odd sides, run from a field
        _single("melt_2d_1021x777_fp32", D2Q9, 1021, 777, FP32, "IREBM", "melt", 200, 1.0, 0.01, 0.1),
        # a small lattice, where launches and latency count
        _single("melt_2d_130x64_fp32", D2Q9, 130, 64, FP32, "IREBM", "melt", 300, 1.0, 0.01, 0.1),
        # full precision on the corner freezing problem, fields read back
        _single("corner_2d_2048_fp64", D2Q9, 2048, 2048, FP64, "IREBM", "corner", 32, 0.84, 0.005, 0.1),
        # the paper's 2D case on its own lattice with the Neumann closure, large
        _single("cavity_d2q5_4096_fp32", D2Q5, 4096, 4096, FP32, "IREBM", "cavity", 64, 0.84, 0.01, CAVITY_STE, 2, "state"),
        # the same in full precision at one of the paper's sizes
        _single("cavity_d2q5_401_fp64", D2Q5, 401, 401, FP64, "IREBM", "cavity", 200, 0.84, 0.01, CAVITY_STE, 2),
        # the explicit comparison scheme
        _single("eebm_2d_2048_fp32", D2Q9, 2048, 2048, FP32, "EEBM", "melt", 64, 1.0, 0.01, 0.1, start="state"),
        # the 1D melting run
        _single("melt_1d_512_fp64", D1Q3, 512, 1, FP64, "IREBM", "melt_1d", 2000, 1.0, 0.01, 0.1),
        # the implicit liquid-fraction comparison scheme on the paper's 1D bar
        _single("ilfbm_bar_801_fp64", D1Q3, 801, 1, FP64, "ILFBM", "bar", 400, 0.62, 0.01, 100.0 / 350.0),
        # and on its 2D case
        _single("ilfbm_cavity_401_fp64", D2Q9, 401, 401, FP64, "ILFBM", "cavity", 8, 0.84, 0.01, CAVITY_STE),
        # a parameter study: many problems of uneven size advanced together
        dict(name="batch_2d_256_fp32", kind="batch", count=256, lo=64, hi=1024, steps=64, precision=FP32),
        # one iteration of an optimisation: misfit and its gradients
        dict(name="adjoint_2d_1024_fp32", kind="adjoint", lattice=D2Q9, nx=1024, ny=1024, precision=FP32, scene="melt",
             steps=200, tau=1.0, delta=0.01, ste=0.1, bb_mode=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["melt32", "melt32", "d2q9_64", "d2q5_32", "d2q5_64", "eebm", "d1q3", "ilfbm1", "ilfbm2", "batch",
                       "adjoint"])
    ste = math.exp(rng.uniform(math.log(0.01), math.log(1.0)))
    tau = rng.choice([0.62, 0.84, 1.0, rng.uniform(0.6, 1.4)])
    delta = rng.choice([0.005, 0.01])
    scene = rng.choice(["melt", "corner", "cavity"])
    bb = rng.choice([0, 1])

    def sides(lo, hi):
        # the two sides of a lattice differ by at most a factor of four
        nx = _log_int(rng, lo, hi)
        return nx, max(lo, min(hi, int(nx * math.exp(rng.uniform(-1.3, 1.3)))))

    def steps(nx, ny, most, lo=24, hi=300):
        # passes of at most `most` node updates
        return max(lo, min(hi, int(most / (nx * ny)))) // 2 * 2

    if kind == "melt32":
        nx, ny = sides(64, 4096)
        return _single(None, D2Q9, nx, ny, FP32, "IREBM", scene, steps(nx, ny, 6e8), tau, delta, ste, bb,
                       rng.choice(["ic", "state"]))
    if kind == "d2q9_64":
        nx, ny = sides(64, 2048)
        return _single(None, D2Q9, nx, ny, FP64, rng.choice(["IREBM", "IREBM", "EEBM"]), scene, steps(nx, ny, 1.2e8), tau,
                       delta, ste, bb)
    if kind in ("d2q5_32", "d2q5_64"):
        p = FP32 if kind == "d2q5_32" else FP64
        nx, ny = sides(64, 4096 if p == FP32 else 1024)
        return _single(None, D2Q5, nx, ny, p, rng.choice(["IREBM", "IREBM", "EEBM"]), scene,
                       steps(nx, ny, 6e8 if p == FP32 else 6e7), tau, delta, ste, rng.choice([0, 1, 2, 2]),
                       rng.choice(["ic", "state"]) if p == FP32 else "ic")
    if kind == "eebm":
        nx, ny = sides(64, 4096)
        return _single(None, D2Q9, nx, ny, FP32, "EEBM", scene, steps(nx, ny, 6e8), tau, delta, ste, bb,
                       rng.choice(["ic", "state"]))
    if kind == "d1q3":
        return _single(None, D1Q3, _log_int(rng, 200, 1601), 1, FP64, rng.choice(["IREBM", "IREBM", "EEBM"]),
                       rng.choice(["melt_1d", "bar"]), rng.randrange(400, 2001), tau, delta, ste, bb)
    if kind == "ilfbm1":
        return _single(None, D1Q3, _log_int(rng, 200, 1601), 1, FP64, "ILFBM", "bar", rng.randrange(50, 301), 0.62, 0.01,
                       100.0 / 350.0, bb)
    if kind == "ilfbm2":
        nx, ny = sides(64, 401)
        return _single(None, D2Q9, nx, ny, FP64, "ILFBM", "cavity", rng.randrange(2, 9), 0.84, 0.01, CAVITY_STE)
    if kind == "batch":
        hi = rng.choice([256, 512, 1024])
        return dict(kind="batch", count=_log_int(rng, 16, 256), lo=64, hi=hi, steps=2 * rng.randrange(16, 33),
                    precision=rng.choice([FP32, FP32, FP32, FP64]) if hi < 1024 else FP32)
    nx, ny = sides(64, 1024)
    return dict(kind="adjoint", lattice=D2Q9, nx=nx, ny=ny, precision=FP32, scene=rng.choice(["melt", "corner"]),
                steps=rng.randrange(60, 201), tau=tau, delta=0.01, ste=max(0.05, ste), bb_mode=0)


# ------------------------------------------------------------------ inputs
def _walls(scene):
    return {k: (_abi.LBM_DIRICHLET, t) for k, t in SCENES[scene][0].items()}


def _front_field(nx, ny, walls, far, gen, x_front=24.0, tail=40.0):
    """A developed front: linear from the wall value to 0 over x_front nodes,
    then an exponential tail to `far`; the position wavers along the wall and
    with the seed, and the field carries noise of 1e-3."""
    dev = "cuda"
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, :].expand(ny, nx)
    y = torch.arange(ny, dtype=torch.float64, device=dev)[:, None].expand(ny, nx)
    dist = {"W": x, "E": nx - 1 - x, "S": y, "N": ny - 1 - y}
    r = torch.rand(3, generator=gen, dtype=torch.float64, device=dev).tolist()
    x_front = min(x_front, nx / 6.0) * (0.9 + 0.2 * r[0])
    tail = min(tail, nx / 4.0) * (0.9 + 0.2 * r[1])
    names = [k for k, t in walls.items() if t * far < 0]   # the walls the front starts from
    d = dist[names[0]]
    for k in names[1:]:
        d = torch.minimum(d, dist[k])
    along = y if names[0] in "WE" else x
    xf = x_front * (1.0 + 0.1 * torch.sin(2 * math.pi * (along / max(ny, 2) * 3.0 + r[2])))
    tw = walls[names[0]]
    th = torch.where(d < xf, tw * (1.0 - d / xf), far * (1.0 - torch.exp(-(d - xf) / tail)))
    th = th + 1e-3 * (2.0 * torch.rand((ny, nx), generator=gen, dtype=torch.float64, device=dev) - 1.0)
    return th.contiguous()


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _theta0(case, seed):
    walls, far = SCENES[case["scene"]]
    one_d = case["lattice"] == D1Q3
    return _front_field(case["nx"], case["ny"], walls, far, _generator(seed), 40.0 if one_d else 24.0,
                        80.0 if one_d else 40.0)


def _batch_inputs(case, seed):
    """Sides log-uniform in [lo, hi] (from the sizes of the case alone), Stefan
    numbers log-uniform in [0.01, 1], west wall uniform in [0.5, 2]."""
    g = torch.Generator().manual_seed(case["count"] * 4099 + case["hi"])
    s = torch.rand(case["count"], generator=g, dtype=torch.float64)
    g = torch.Generator().manual_seed(int(seed))
    u = torch.rand((case["count"], 2), generator=g, dtype=torch.float64)
    cases = []
    for k in range(case["count"]):
        n = int(round(math.exp(math.log(case["lo"]) + float(s[k]) * math.log(case["hi"] / case["lo"]))))
        ste = math.exp(math.log(0.01) * (1.0 - float(u[k, 0])))
        tw = 0.5 + 1.5 * float(u[k, 1])
        cases.append(Case("batch%d" % k, D2Q9, n, n, 1.0, 0.01, ste, {"W": (_abi.LBM_DIRICHLET, tw)}, case["steps"],
                          case["precision"]))
    gen = _generator(seed)
    return cases, [_front_field(c.nx, c.ny, {"W": c.walls["W"][1]}, -0.2, gen) for c in cases]


def _adjoint_inputs(case, seed):
    """A FP32 parameter field and the liquid fraction of a displaced front as target."""
    walls, far = SCENES[case["scene"]]
    p = _theta0(case, seed).float()
    t = _front_field(case["nx"], case["ny"], walls, far, _generator(seed + 7919), 27.0, 44.0)
    return p, 0.5 + 0.5 * torch.tanh(t / case["delta"])


def _solver_args(case):
    # the inner loop of ILFBM: its tolerance on the liquid fraction and its limit
    if case["method"] == "ILFBM":
        return {"newton_tol": 1e-12, "newton_max_iter": 200 if case["lattice"] == D1Q3 else 400}
    return {}


class _State:
    """What a user's program holds between passes."""


def prepare(case, seed):
    s = _State()
    s.case = case
    s.kind = case["kind"]
    s.stream = torch.cuda.Stream()
    if s.kind == "single":
        s.theta0 = _theta0(case, seed)
        s.stream.wait_stream(torch.cuda.current_stream())
        s.solver = Stefan(case["lattice"], case["nx"], case["ny"], case["tau"], case["delta"], case["ste"],
                          case["precision"], _walls(case["scene"]), bb_mode=case["bb_mode"], stream=s.stream,
                          **_solver_args(case))
        if case["method"] != "IREBM":
            s.solver.set_method(case["method"])
        s.solver.set_ic(s.theta0)
        if case["precision"] == FP32:
            s.out = s.solver.new_state_buffer()
            q, ny, pitch = len(W[case["lattice"]]), case["ny"], s.solver.row_stride
            planes = s.out[:4 * q * (ny + 2) * pitch].view(torch.float32).view(q, ny + 2, pitch)
            s.populations = planes[:, 1:ny + 1, :case["nx"]]
        if case["start"] == "state":
            s.checkpoint = s.solver.new_state_buffer()
            s.stream.wait_stream(torch.cuda.current_stream())
            s.solver.get_state(s.checkpoint)
    elif s.kind == "batch":
        cases, s.fields = _batch_inputs(case, seed)
        s.batch = StefanBatch(cases, precision=case["precision"], stream=s.stream)
        s.theta = torch.empty(max(c.nx * c.ny for c in cases), dtype=torch.float64, device="cuda")
        s.out = torch.empty(sum(c.nx * c.ny for c in cases), device="cuda",
                            dtype=torch.float32 if case["precision"] == FP32 else torch.float64)
    else:
        s.theta0, s.target = _adjoint_inputs(case, seed)
        s.theta0.requires_grad_(True)
        walls = _walls(case["scene"])
        s.walls = torch.tensor([walls.get(k, (0, 0.0))[1] for k in "WESN"], device="cuda", requires_grad=True)
        s.ste = torch.tensor(case["ste"], device="cuda", requires_grad=True)
        s.problem = Case("adjoint", case["lattice"], case["nx"], case["ny"], case["tau"], case["delta"], case["ste"], walls,
                         case["steps"], case["precision"])
    return s


def run(s):
    here = torch.cuda.current_stream()
    if s.kind == "single":
        s.stream.wait_stream(here)
        if s.case["start"] == "state":
            s.solver.set_state(s.checkpoint)
        else:
            s.solver.set_ic(s.theta0)
        s.solver.step(s.case["steps"])
        if s.case["precision"] == FP64:
            theta, phi, H = s.solver.fields(device=True)
            return {"theta": theta, "phi": phi, "H": H}
        s.solver.get_state(s.out)
        here.wait_stream(s.stream)
        return {"populations": s.populations}
    if s.kind == "batch":
        s.stream.wait_stream(here)
        for k, f in enumerate(s.fields):
            s.batch.set_ic(k, f)
        s.batch.step(s.case["steps"])
        at = 0
        for k, f in enumerate(s.fields):
            n = f.numel()
            _abi.check(s.batch.lib.lbm_stefan_batch_get_fields(s.batch.h, k, ctypes.c_void_p(s.theta.data_ptr()), 1))
            with torch.cuda.stream(s.stream):
                s.out[at:at + n] = s.theta[:n]
            at += n
        here.wait_stream(s.stream)
        return {"theta": s.out}
    s.theta0.grad = s.walls.grad = s.ste.grad = None
    loss = misfit(s.theta0.double(), s.walls.double(), s.ste.double(), s.problem, s.case["steps"], s.target,
                  bb_mode=s.case["bb_mode"])
    loss.backward()
    return {"loss": loss.detach().float(), "g_theta0": s.theta0.grad, "g_walls": s.walls.grad, "g_ste": s.ste.grad}


def _nodes(case):
    if case["kind"] != "batch":
        return case["nx"] * case["ny"]
    g = torch.Generator().manual_seed(case["count"] * 4099 + case["hi"])
    s = torch.rand(case["count"], generator=g, dtype=torch.float64)
    r = math.log(case["hi"] / case["lo"])
    return sum(int(round(math.exp(math.log(case["lo"]) + float(v) * r))) ** 2 for v in s)


def work(case):
    """Each population read once and written once per step, and about five
    operations per population; a reverse step moves the adjoint populations and
    two recorded temperatures, and its segment is recomputed once (recording a
    temperature).  ILFBM: a step's populations and liquid fraction, whatever
    its inner iterations cost."""
    n, steps = _nodes(case), case["steps"]
    q = len(W[case.get("lattice", D2Q9)])
    elem = 4 if case["precision"] == FP32 else 8
    step = 2 * q * elem
    if case.get("method") == "ILFBM":
        step += 2 * elem
    if case["kind"] == "adjoint":
        return {"bytes": float(n) * steps * (3 * step + 8 + 16), "flops": 15.0 * q * n * steps}
    return {"bytes": float(n) * steps * step, "flops": 5.0 * q * n * steps}


# ------------------------------------------------------------------ the passes in 64 bits
class _Exact:
    """Problems of one lattice in plain torch, FP64, populations stored after the
    collision (Eq. 12), their nodes one after the other in flat vectors.

    problems: (nx, ny, ste, {wall: temperature}) each; ste and temperatures are
    floats, or 0-d tensors that gradients reach."""

    def __init__(self, lattice, problems, tau, delta, bb_mode, method):
        self.omega, self.delta, self.bb, self.method = 1.0 / tau, delta, bb_mode, method
        self.w, self.opp = W[lattice], OPP[lattice]
        dev, Q, at = "cuda", len(W[lattice]), 0
        source, edge, unknown, inward = [[] for _ in range(Q)], [], [[] for _ in range(Q)], []
        values, which = [torch.zeros((), dtype=torch.float64, device=dev)], []
        two_d = lattice != D1Q3
        for nx, ny, _, walls in problems:
            x = torch.arange(nx, device=dev).repeat(ny)
            y = torch.arange(ny, device=dev).repeat_interleave(nx)
            on = {"W": x == 0, "E": x == nx - 1, "S": (y == 0) & two_d, "N": (y == ny - 1) & two_d}
            here = (on["W"] | on["E"] | on["S"] | on["N"]).nonzero().squeeze(1)   # the boundary nodes
            for i in range(Q):
                sx, sy = x - EX[lattice][i], y - EY[lattice][i]
                out = (sx < 0) | (sx >= nx) | (sy < 0) | (sy >= ny)
                source[i].append(at + sy.clamp(0, ny - 1) * nx + sx.clamp(0, nx - 1))
                unknown[i].append(out[here])
            wall = torch.zeros(here.shape, dtype=torch.long, device=dev)
            for k in reversed([k for k in "WESN" if k in walls]):   # the first of W, E, S, N wins
                wall[on[k][here]] = len(values)
                values.append(torch.as_tensor(walls[k], dtype=torch.float64, device=dev))
            which.append(wall)
            ex, ey = x[here], y[here]
            step_y = ((ey == 0).long() - (ey == ny - 1).long()) * two_d
            inward.append(at + (ey + step_y) * nx + ex + (ex == 0).long() - (ex == nx - 1).long())   # one step inwards
            edge.append(at + here)
            at += nx * ny
        self.source = [torch.cat(v) for v in source]
        self.unknown = [torch.cat(v) for v in unknown]
        self.edge, self.inward, wall = torch.cat(edge), torch.cat(inward), torch.cat(which)
        self.dirichlet = wall > 0
        self.td = torch.stack(values)[wall]
        ste = [torch.as_tensor(p[2], dtype=torch.float64, device=dev) for p in problems]
        # the Stefan number: one value, or one per node
        self.ste = ste[0] if len(ste) == 1 else torch.cat([v.expand(p[0] * p[1]) for v, p in zip(ste, problems)])

    def ste_at(self, idx):
        return self.ste if self.ste.dim() == 0 else self.ste[idx]

    def phi(self, t):
        return 0.5 + 0.5 * torch.tanh(t / self.delta)

    def enthalpy(self, t, ste):
        return t + (t > 0).double() / ste

    def temperature(self, H):
        return torch.where(H < 0, H, torch.where(H > 1 / self.ste, H - 1 / self.ste, torch.zeros_like(H)))

    def start(self, theta0):
        th = theta0.reshape(-1).clone()
        th = th.index_copy(0, self.edge, torch.where(self.dirichlet, self.td, th[self.edge]))
        if self.method == "EEBM":
            H = self.enthalpy(th, self.ste)
            return [H - (1 - self.w[0]) * th] + [w * th for w in self.w[1:]]
        return [w * th for w in self.w]

    def pull(self, f):
        return [v[i] for v, i in zip(f, self.source)]

    def close(self, q, f, target):
        """The unknown q of the boundary nodes: `target` is M0(q) on Dirichlet nodes."""
        e, Q = self.edge, len(q)
        qe, fe = [v[e] for v in q], [v[e] for v in f]
        unk = self.unknown
        known = sum(torch.where(unk[i], torch.zeros_like(qe[i]), qe[i]) for i in range(Q))
        wu = sum(unk[i].double() * self.w[i] for i in range(Q))
        if self.bb == 2:
            # Eq. (17): M0(q) of the node one step inwards
            inner = sum(v[self.inward] for v in q)
            target = torch.where(self.dirichlet, target, inner)
        share = (target - known) / wu
        new = []
        for i in range(Q):
            o = self.opp[i]
            back = torch.where(unk[o], fe[o], qe[o]) if self.bb == 0 else fe[o]
            v = self.w[i] * share if self.bb == 2 else torch.where(self.dirichlet, self.w[i] * share, back)
            new.append(q[i].index_copy(0, e, torch.where(unk[i], v, qe[i])))
        return new

    def root(self, m0, theta, ph, ste):
        """The root of Eq. (14) by bracketed Newton steps."""
        lo, hi = m0 + (ph - 1) / ste, m0 + ph / ste
        x = torch.minimum(torch.maximum(theta, lo), hi)
        for k in range(100):
            t = torch.tanh(x / self.delta)
            F = (x - m0) + (0.5 + 0.5 * t - ph) / ste
            lo, hi = torch.where(F < 0, x, lo), torch.where(F > 0, x, hi)
            xn = x - F / (1 + 0.5 * (1 - t) * (1 + t) / self.delta / ste)
            # a step out of the bracket bisects; a node that is late does so every other time
            bad = (xn < lo) | (xn > hi)
            if k >= 12 and k % 2:
                bad = bad | ((xn - x).abs() > 1e-10)
            xn = torch.where(bad, 0.5 * (lo + hi), xn)
            if k >= 4 and k % 2 == 0 and bool(((xn - x).abs() <= 1e-10 * (1 + x.abs())).all()):
                return xn
            x = xn
        return x

    def new_theta(self, m0, theta):
        band = 19.5 * self.delta   # tanh is +-1 in FP64 beyond it: theta' = m0
        idx = (~((theta > band) & (m0 > band)) & ~((theta < -band) & (m0 < -band))).nonzero().squeeze(1)
        m, t, ste = m0[idx], theta[idx], self.ste_at(idx)
        ph = self.phi(t)
        with torch.no_grad():
            x = self.root(m, t, ph, ste)
            d = torch.tanh(x / self.delta)
            slope = 1 + 0.5 * (1 - d) * (1 + d) / self.delta / ste
        # one Newton step with the slope held: the root's value and its derivatives
        x = x - ((x - m) + (self.phi(x) - ph) / ste) / slope
        return m0.index_copy(0, idx, x)

    def step(self, f):
        om, td, ste = self.omega, self.td, self.ste_at(self.edge)
        q = self.pull(f)
        theta = sum(f)
        if self.method == "EEBM":
            target = self.enthalpy(td, ste)
        else:
            target = td + (self.phi(td) - self.phi(theta[self.edge])) / ste
        q = self.close(q, f, target)
        m0 = sum(q)
        if self.method == "EEBM":
            th = self.temperature(m0)
            return [(1 - om) * q[0] + om * (m0 - (1 - self.w[0]) * th)] + [
                (1 - om) * v + om * w * th for v, w in zip(q[1:], self.w[1:])]
        th = self.new_theta(m0, theta)
        th = th.index_copy(0, self.edge, torch.where(self.dirichlet, td, th[self.edge]))
        c = th - (1 - om) * m0
        return [(1 - om) * v + w * c for v, w in zip(q, self.w)]

    def step_ilfbm(self, f, l, tol, most):
        om, theta = self.omega, sum(f)
        f0 = [v - (v - w * theta) * om for v, w in zip(f, self.w)]
        td = self.td
        wall_l = (td > 0).double()
        lp = l
        for _ in range(most):
            g = [v + w / self.ste * (l - lp) for v, w in zip(f0, self.w)]
            q = self.close(self.pull(g), g, td)
            H = sum(q) + lp / self.ste
            ln = torch.where(H < 0, torch.zeros_like(H), torch.where(H > 1 / self.ste, torch.ones_like(H), self.ste * H))
            ln = ln.index_copy(0, self.edge, torch.where(self.dirichlet, wall_l, ln[self.edge]))
            done = not bool(((ln - lp).abs() > tol).any())
            lp = ln
            if done:
                break
        return q, ln


def _exact_single(case, seed):
    walls = SCENES[case["scene"]][0]
    e = _Exact(case["lattice"], [(case["nx"], case["ny"], case["ste"], walls)], case["tau"], case["delta"],
               case["bb_mode"], case["method"])
    theta0 = _theta0(case, seed)
    f = e.start(theta0)
    shape = (case["ny"], case["nx"])
    if case["method"] == "ILFBM":
        l = (sum(f) > 0).double()
        a = _solver_args(case)
        for _ in range(case["steps"]):
            f, l = e.step_ilfbm(f, l, a["newton_tol"], a["newton_max_iter"])
        th = sum(f)
        return {"theta": th.view(shape), "phi": l.view(shape), "H": (th + l / e.ste).view(shape)}
    for _ in range(case["steps"]):
        f = e.step(f)
    if case["precision"] == FP64:
        m = sum(f)
        if case["method"] == "EEBM":
            th, ph, H = e.temperature(m), (e.ste * m).clamp(0, 1), m
        else:
            th, ph = m, e.phi(m)
            H = th + ph / e.ste
        return {"theta": th.view(shape), "phi": ph.view(shape), "H": H.view(shape)}
    # the FP32 state holds Omega_i - w_i s, s half the mean of the initial M0
    start = e.enthalpy(theta0, e.ste) if case["method"] == "EEBM" else theta0
    s = float((0.5 * start.mean()).float())
    return {"populations": torch.stack([(v - w * s).view(shape) for v, w in zip(f, e.w)])}


def exact(case, seed):
    if case["kind"] == "single":
        with torch.no_grad():
            return _exact_single(case, seed)
    if case["kind"] == "batch":
        cases, fields = _batch_inputs(case, seed)
        with torch.no_grad():
            e = _Exact(D2Q9, [(c.nx, c.ny, c.ste, {k: t for k, (_, t) in c.walls.items()}) for c in cases], cases[0].tau,
                       cases[0].delta, 0, "IREBM")
            f = e.start(torch.cat([v.reshape(-1) for v in fields]))
            for _ in range(case["steps"]):
                f = e.step(f)
            return {"theta": sum(f)}
    p, target = _adjoint_inputs(case, seed)
    p.requires_grad_(True)
    walls = SCENES[case["scene"]][0]
    leaves = {k: torch.tensor(t, device="cuda", requires_grad=True) for k, t in walls.items()}
    ste = torch.tensor(case["ste"], device="cuda", requires_grad=True)
    e = _Exact(case["lattice"], [(case["nx"], case["ny"], ste.double(), {k: v.double() for k, v in leaves.items()})],
               case["tau"], case["delta"], case["bb_mode"], "IREBM")

    def advance(n, *f):
        f = list(f)
        for _ in range(n):
            f = e.step(f)
        return tuple(f)

    f = tuple(e.start(p.double()))
    every, left = 14, case["steps"]
    while left > 0:
        n = min(every, left)
        f = checkpoint(advance, n, *f, use_reentrant=False)
        left -= n
    loss = 0.5 * ((e.phi(sum(f)) - target.reshape(-1)) ** 2).sum()
    loss.backward()
    g = [leaves[k].grad.double() if k in leaves else torch.zeros((), dtype=torch.float64, device="cuda") for k in "WESN"]
    return {"loss": loss.detach(), "g_theta0": p.grad.double(), "g_walls": torch.stack(g), "g_ste": ste.grad.double()}
