"""The work a user of this package has it do, as cases that can be timed.

A case is a run of time steps of one cavity (its sizes, storage and number of
steps), of a batch of cavities, or the gradient of the mean Nusselt number, each
through the package's public calls: ``Cavity2D.step`` / ``fields`` /
``nusselt``, ``Batch.step``, ``nusselt_objective`` with ``backward``.

``prepare`` gives each cavity a developed state (smooth convection rolls over
the conduction profile, a perturbed hot wall), uploaded as a program that goes
on with a saved flow does it; ``run`` advances it and reads what such a program
reads: the fields on the GPU and the Nusselt history. Nusselt numbers are
differences of float32 temperatures, so the history is kept as float32.

``exact`` is the double-MRT step of arXiv:1601.04633 in 64 bits with dense
matrices, plain torch (its gradient by autograd).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1601_04633_gb300 import dmrt as D
from paper_1601_04633_gb300 import inputs

STORAGE = {"float32": D.DMRT_FP32, "float16": D.DMRT_FP16, "bfloat16": D.DMRT_BF16, "mixed": D.DMRT_MIXED,
           "theta32": D.DMRT_THETA32}
STATE_BYTES = {"float32": 56, "float16": 28, "bfloat16": 28, "mixed": 38, "theta32": 30}  # per node
STEP_FLOPS = 160     # both collisions of one node, additions and multiplications
REVERSE_FLOPS = 420  # the transposed collision of one node with its force derivatives


def _cavity(name, nx, ny, steps, storage="float32", Ra=1e5, Pr=0.01, nusselt=True):
    return {"name": name, "kind": "cavity", "nx": nx, "ny": ny, "steps": steps, "storage": storage, "Ra": Ra, "Pr": Pr,
            "nusselt": nusselt}


def listed():
    return [
        # One step and its fields, as an interactive view or a coupling loop asks for them.
        _cavity("frame_64", 64, 64, 1, Ra=1e4, nusselt=False),
        # The paper's first case on the usual small grid.
        _cavity("cavity_64", 64, 64, 2000, Ra=1e4),
        # The grid on which the paper's cases are compared with its Nusselt numbers.
        _cavity("cavity_128", 128, 128, 1000),
        # The oscillatory workload, float32 and the reduced-precision storage that is meant for it.
        _cavity("cavity_256", 256, 256, 1000, Pr=0.005),
        _cavity("cavity_256_mixed", 256, 256, 1000, "mixed", Pr=0.005),
        # A middle-sized grid of odd sizes, as a grid-refinement study has them.
        _cavity("ragged_383x389", 383, 389, 500, Ra=1e6),
        # The large single cavity that the throughput is quoted on.
        _cavity("large_4096", 4096, 4096, 64, Ra=1e7, Pr=0.001),
        # Large cavities in the two accurate reduced-precision storages (stochastic rounding), the second of odd sizes.
        _cavity("large_2048_mixed", 2048, 2048, 64, "mixed", Ra=1e7, Pr=0.001),
        _cavity("ragged_1999x1531_theta32", 1999, 1531, 64, "theta32", Ra=1e7, Pr=0.001),
        # A parameter sweep: 64 cavities of sides 128 to 384 stepped together.
        {"name": "sweep_64", "kind": "batch", "n": 64, "low": 128, "high": 384, "steps": 256, "storage": "float32"},
        {"name": "sweep_64_mixed", "kind": "batch", "n": 64, "low": 128, "high": 384, "steps": 256, "storage": "mixed"},
        # Design by gradient: d(mean Nu)/d(hot-wall profile, Ra).
        {"name": "adjoint_128", "kind": "adjoint", "nx": 128, "ny": 128, "steps": 2000, "last": 400, "Ra": 1e5, "Pr": 0.01},
    ]


def _resolved(Ra, Pr, ny, cell):
    """Ra as far as a grid of ny rows resolves it: a Mach number of at most 0.05 and
    at most `cell` for the free-fall velocity times the node spacing over the viscosity
    (beyond these a run of many thousand steps does not stay bounded)."""
    return min(Ra, (0.3 * ny) ** 2 / Pr, Pr * (cell * ny) ** 2)


def draw(rng):
    """Cavities of 16 to 2048 nodes a side in every storage, batches, gradients."""
    kind = rng.choice(["cavity", "cavity", "cavity", "cavity", "batch", "adjoint"])
    Ra, Pr = 10.0 ** rng.uniform(4, 6), rng.choice([0.005, 0.01])
    if kind == "batch":
        low = rng.randint(40, 200)
        return {"kind": "batch", "n": rng.randint(3, 48), "low": low, "high": low + rng.randint(1, 200),
                "steps": rng.randint(16, 256), "storage": rng.choice(["float32", "mixed"])}
    if kind == "adjoint":
        n = int(2.0 ** rng.uniform(5, 8))
        steps = rng.randint(200, 1000)
        return {"kind": "adjoint", "nx": n, "ny": n + rng.randint(0, 9), "steps": steps, "last": steps // 5,
                "Ra": _resolved(Ra, Pr, n, 12), "Pr": Pr}
    nx = int(2.0 ** rng.uniform(4, 11))
    ny = max(8, int(nx * 2.0 ** rng.uniform(-1, 0.5)))
    # Enough steps to be a run, fewer the larger the cavity is.
    steps = max(16, min(rng.randint(200, 2000), int(3e8 / (nx * ny))))
    case = _cavity("", nx, ny, steps, rng.choice(["float32", "float32", "mixed", "theta32", "float16", "bfloat16"]),
                   _resolved(Ra, Pr, ny, 12), Pr)
    del case["name"]
    return case


# ---- inputs -------------------------------------------------------------------


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _members(case):
    """The sides, Ra and Pr of a batch's cavities (they belong to the case, not to the seed)."""
    rng = np.random.default_rng(3)
    sides = [128, 192, 256, 384] if (case["low"], case["high"]) == (128, 384) else None
    out = []
    for _ in range(case["n"]):
        nx = int(rng.choice(sides)) if sides else int(rng.integers(case["low"], case["high"] + 1))
        ny = nx if sides else int(rng.integers(case["low"], case["high"] + 1))
        Ra, Pr = 10.0 ** rng.uniform(4, 6), float(rng.choice([0.001, 0.005, 0.01]))
        out.append((nx, ny, _resolved(Ra, Pr, ny, 30), Pr))
    return out


ALPHA = 0.1
A5 = 20.0 * math.sqrt(3.0) * ALPHA - 4.0  # the free D2Q5 parameter
EX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
EY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def _hot_profile(ny, seed):
    return 0.5 + 0.01 * np.random.default_rng(seed).standard_normal(ny)


def _state(nx, ny, Ra, Pr, seed):
    """Populations [14][ny][nx] (float32, host) of a developed flow: rolls of the
    buoyant velocity scale, the conduction profile bent by them, equilibrium populations."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(seed)
    X = (torch.arange(nx, device=dev, dtype=torch.float64)[None, :] + 0.5) / nx
    Y = (torch.arange(ny, device=dev, dtype=torch.float64)[:, None] + 0.5) / ny
    U = 0.4 * math.sqrt(Ra * Pr) * ALPHA / ny  # below the free-fall velocity
    r = torch.rand(4, generator=gen, device=dev, dtype=torch.float64).tolist()
    u = torch.zeros(ny, nx, device=dev, dtype=torch.float64)
    v = torch.zeros_like(u)
    for m, n, amp in ((1, 1, 1.0), (1, 2, 0.3 * (r[0] - 0.5)), (2, 1, 0.3 * (r[1] - 0.5)), (2, 2, 0.2 * (r[2] - 0.5))):
        # Stream function amp sin^2(m pi X) sin^2(n pi Y) / pi: velocities vanish at every wall.
        u -= U * amp * n * torch.sin(m * math.pi * X) ** 2 * torch.sin(2 * n * math.pi * Y)
        v += U * amp * m * torch.sin(2 * m * math.pi * X) * torch.sin(n * math.pi * Y) ** 2
    # The main roll rises along the hot wall, so the top is warmer than the bottom.
    theta = 0.5 - X - 0.15 * (1 + 0.2 * r[3]) * torch.sin(math.pi * X) * torch.cos(math.pi * Y)
    theta = theta + 1e-3 * (2 * torch.rand(ny, nx, generator=gen, device=dev, dtype=torch.float64) - 1)
    uu = u * u + v * v
    out = torch.empty(14, ny, nx, dtype=torch.float32, device=dev)
    for i in range(9):
        eu = EX[i] * u + EY[i] * v
        out[i] = W9[i] * (3 * eu + 4.5 * eu * eu - 1.5 * uu)
    out[9] = (1 - A5) / 5 * theta
    for i in range(1, 5):
        out[9 + i] = (4 + A5) / 20 * theta + 0.5 * (EX[i] * u + EY[i] * v) * theta
    return out.cpu().numpy()


def prepare(case, seed):
    if case["kind"] == "adjoint":
        cav = inputs.Cavity(case["nx"], case["ny"], case["Ra"], case["Pr"], alpha=ALPHA, seed=seed)
        theta_w = torch.tensor(_hot_profile(case["ny"], seed), dtype=torch.float32, device="cuda", requires_grad=True)
        Ra = torch.tensor(case["Ra"], dtype=torch.float32, device="cuda", requires_grad=True)
        return {"case": case, "cavity": cav, "theta_w": theta_w, "Ra": Ra}
    if case["kind"] == "batch":
        members = _members(case)
        cavs = [inputs.Cavity(nx, ny, Ra, Pr, alpha=ALPHA, noise_amp=0.0) for nx, ny, Ra, Pr in members]
        batch = D.Batch.from_inputs(cavs, nu_capacity=1 << 12, storage=STORAGE[case["storage"]])
        for k, (m, (nx, ny, Ra, Pr)) in enumerate(zip(batch.members, members)):
            m.set_state(_state(nx, ny, Ra, Pr, 1000 * seed + k))
        return {"case": case, "batch": batch}
    cav = inputs.Cavity(case["nx"], case["ny"], case["Ra"], case["Pr"], alpha=ALPHA, noise_amp=0.0,
                        theta_hot_profile=_hot_profile(case["ny"], seed))
    sim = D.Cavity2D.from_inputs(cav, nu_capacity=1 << 12, storage=STORAGE[case["storage"]])
    sim.set_state(_state(case["nx"], case["ny"], case["Ra"], case["Pr"], seed))
    return {"case": case, "sim": sim}


# ---- one pass -----------------------------------------------------------------


def run(state):
    case = state["case"]
    steps = case["steps"]
    if case["kind"] == "adjoint":
        theta_w, Ra = state["theta_w"], state["Ra"]
        theta_w.grad = Ra.grad = None
        J = D.nusselt_objective(theta_w, Ra, state["cavity"], steps, case["last"])
        J.backward()
        return {"J": J.detach(), "theta_w": theta_w.grad, "Ra": Ra.grad}
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(steps)
        # The fields of all cavities in three flat arrays, one cavity after another.
        out = [torch.empty(batch.nodes, dtype=torch.float32, device="cuda") for _ in range(3)]
        at = 0
        for m in batch.members:
            D.dmrt_fields(m.h, *[t.data_ptr() + 4 * at for t in out], True)
            at += m.nx * m.ny
        nu = np.stack([m.nusselt(steps)[2] for m in batch.members]).astype(np.float32)
        return {"u": out[0], "v": out[1], "theta": out[2], "nu": nu}
    sim = state["sim"]
    sim.step(steps)
    u, v, theta = sim.fields()
    out = {"u": u, "v": v, "theta": theta}
    if case["nusselt"]:
        _, local, series = sim.nusselt(steps)
        out["nu_rows"], out["nu"] = local.astype(np.float32), series.astype(np.float32)
    return out


def work(case):
    """Each state read and written once in a pass and the fields written; the gradient
    also keeps every forward state for the reverse steps."""
    steps = case["steps"]
    if case["kind"] == "adjoint":
        nodes = case["nx"] * case["ny"]
        return {"bytes": 2 * 56 * nodes * steps, "flops": (STEP_FLOPS + REVERSE_FLOPS) * nodes * steps}
    nodes = sum(nx * ny for nx, ny, _, _ in _members(case)) if case["kind"] == "batch" else case["nx"] * case["ny"]
    return {"bytes": (2 * STATE_BYTES[case["storage"]] + 12) * nodes, "flops": STEP_FLOPS * nodes * steps}


# ---- the same in 64 bits ---------------------------------------------------------

M9 = [[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
      [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
      [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]
N5 = [[1, 1, 1, 1, 1], [0, 1, 0, -1, 0], [0, 0, 1, 0, -1], [-4, 1, 1, 1, 1], [0, 1, -1, 1, -1]]


class _Exact:
    """The step of cavities of one size (axis 1 of f [9][B][ny][nx] and g [5][B][ny][nx])."""

    def __init__(self, nx, ny, Ra, Pr, dev):
        t = lambda x: torch.tensor(x, dtype=torch.float64, device=dev)  # noqa: E731
        self.nx, self.ny = nx, ny
        Ra = (Ra if torch.is_tensor(Ra) else t(Ra)).reshape(-1, 1, 1)
        nu = ALPHA * t(Pr).reshape(-1, 1, 1)
        self.gbeta = Ra * nu * ALPHA / ny ** 3
        s_nu = 2 / (6 * nu + 1)
        s_q = 8 * (2 - s_nu) / (8 - s_nu)
        zero = torch.zeros_like(s_nu)
        self.S = torch.stack([zero, s_nu, s_nu, zero, s_q, zero, s_q, s_nu, s_nu])
        sk, se = 1 / (0.5 + math.sqrt(3) / 6), 1 / (0.5 + math.sqrt(3) / 3)
        self.Q = t([0, sk, sk, se, se]).reshape(5, 1, 1, 1)
        self.M, self.N = t(M9), t(N5)
        self.Mi, self.Ni = torch.linalg.inv(self.M), torch.linalg.inv(self.N)
        ones = torch.ones(ny, nx, device=dev)
        self.out = []  # nodes whose pull along direction i crosses a wall
        for ex, ey in zip(EX, EY):
            m = torch.zeros_like(ones, dtype=torch.bool)
            if ex:
                m[:, 0 if ex > 0 else -1] = True
            if ey:
                m[0 if ey > 0 else -1, :] = True
            self.out.append(m)

    @staticmethod
    def _mat(A, f):
        return (A @ f.reshape(f.shape[0], -1)).reshape(f.shape)

    def step(self, f, g, hot):
        """One step; also the pre-collision u, v, theta and the rows' Nusselt numbers. hot: [B][ny]."""
        pull = lambda p, i: torch.roll(p[i], (EY[i], EX[i]), (-2, -1))  # noqa: E731
        f = torch.stack([f[0]] + [torch.where(self.out[i], f[OPP[i]], pull(f, i)) for i in range(1, 9)])
        abb = 2 * math.sqrt(3) * ALPHA
        gs = [g[0]]
        for i in range(1, 5):
            wall = g[OPP[i]]
            if EX[i]:
                wall = abb * (hot[:, :, None] if EX[i] > 0 else -0.5) - wall
            gs.append(torch.where(self.out[i], wall, pull(g, i)))
        g = torch.stack(gs)
        m = self._mat(self.M, f)
        rho, u, v = m[0], m[3], m[5]
        uu = u * u + v * v
        theta = g.sum(0)
        Gy = self.gbeta * theta
        meq = torch.stack([rho, -2 * rho + 3 * uu, rho - 3 * uu, u, -u, v, -v, u * u - v * v, u * v])
        F = []
        for i in range(9):
            eu = EX[i] * u + EY[i] * v
            F.append(3 * W9[i] * (EY[i] - v) * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu))
        f2 = f - self._mat(self.Mi, self.S * (m - meq)) + Gy * torch.stack(F)
        n = self._mat(self.N, g)
        neq = torch.stack([theta, u * theta, v * theta, A5 * theta, torch.zeros_like(theta)])
        g2 = g - self._mat(self.Ni, self.Q * (n - neq))
        rows = self.ny / 3.0 * (8 * hot - 9 * theta[..., 0] + theta[..., 1])
        return f2, g2, u, v, theta, rows


def _exact_run(nx, ny, Ra, Pr, states, hot, steps):
    dev = _device()
    E = _Exact(nx, ny, Ra, Pr, dev)
    s = torch.stack([torch.from_numpy(x) for x in states], 1).to(dev).double()
    f, g = s[:9], s[9:]
    nu = []
    for _ in range(steps):
        f, g, u, v, theta, rows = E.step(f, g, hot)
        nu.append(rows.mean(-1))
    return u, v, theta, rows, torch.stack(nu, 1)


def exact(case, seed):
    dev = _device()
    steps = case["steps"]
    with torch.set_grad_enabled(case["kind"] == "adjoint"):
        if case["kind"] == "adjoint":
            if case["nx"] * case["ny"] * steps > 4e7:
                return None  # autograd's record of the whole run would be too large
            nx, ny = case["nx"], case["ny"]
            cav = inputs.Cavity(nx, ny, case["Ra"], case["Pr"], alpha=ALPHA, seed=seed)
            theta = torch.from_numpy(cav.theta0()).to(dev).reshape(1, ny, nx)
            # What the call gets: float32 values.
            hot = torch.tensor(_hot_profile(ny, seed), dtype=torch.float32, device=dev).double().requires_grad_()
            Ra = torch.tensor(float(np.float32(case["Ra"])), dtype=torch.float64, device=dev, requires_grad=True)
            E = _Exact(nx, ny, Ra, case["Pr"], dev)
            f = torch.zeros(9, 1, ny, nx, dtype=torch.float64, device=dev)
            g = torch.stack([(1 - A5) / 5 * theta] + [(4 + A5) / 20 * theta] * 4)
            J = 0.0
            for k in range(steps):
                f, g, _, _, _, rows = E.step(f, g, hot[None])
                if k >= steps - case["last"]:
                    J = J + rows.mean() / case["last"]
            J.backward()
            return {"J": J.detach(), "theta_w": hot.grad, "Ra": Ra.grad}
        if case["kind"] == "batch":
            members = _members(case)
            out = [None] * len(members)
            for size in {m[:2] for m in members}:
                idx = [k for k, m in enumerate(members) if m[:2] == size]
                nx, ny = size
                hot = torch.full((len(idx), ny), 0.5, dtype=torch.float64, device=dev)
                got = _exact_run(nx, ny, [members[k][2] for k in idx], [members[k][3] for k in idx],
                                 [_state(*members[k], 1000 * seed + k) for k in idx], hot, steps)
                for q, k in enumerate(idx):
                    out[k] = [x[q].reshape(-1) for x in got]
            u, v, theta = (torch.cat([o[i] for o in out]) for i in range(3))
            return {"u": u, "v": v, "theta": theta, "nu": torch.stack([o[4] for o in out])}
        nx, ny = case["nx"], case["ny"]
        hot = torch.tensor(_hot_profile(ny, seed), dtype=torch.float32, device=dev).double()[None]
        u, v, theta, rows, nu = _exact_run(nx, ny, case["Ra"], case["Pr"],
                                           [_state(nx, ny, case["Ra"], case["Pr"], seed)], hot, steps)
        res = {"u": u[0], "v": v[0], "theta": theta[0]}
        if case["nusselt"]:
            # With the temperature itself in 16 bits its differences at the wall are rounding: no such value.
            thermal16 = case["storage"] in ("float16", "bfloat16")
            res["nu_rows"], res["nu"] = (None, None) if thermal16 else (rows[0], nu[0])
        return res
