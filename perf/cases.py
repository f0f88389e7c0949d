"""The work whose speed is measured, through the package's public entry points.

Kinds of case, by the call that a user's program makes:
  host     Controller.step_host: one MPPI iteration from host arrays, as a control loop does it
  step     Controller.step: one MPPI iteration on device tensors; with "elite" the full Eq. 8 update and
           its covariance blocks, with "qp" the smoothing projection of every sample, with "task" the
           ball-task cost suite
  batch    Batch.step(graph=True): one iteration of many controllers of different sizes
  rollout  Controller.rollout_batch: explicit controls from many start states, costs and final states
  sim      Controller.sim_step: one simulator step of many states
  project  qp_project: the smoothing projection of stored sequences
Scenes, sample counts, horizons, boxes, sigma and iteration counts are those of the repository's five
configurations, its pools and its benchmark options.  The temperature of the whole-iteration cases is about
the standard deviation of the sample costs, a common rule for MPPI (planar 1, transfer 2, its task costs 20;
the lift's 0.05 is the configuration's own).
"""
import functools
import math

import numpy as np
import torch

from paper_2511_21264_gb300 import flops, native, scenes

DEV = "cuda"


def listed():
    return [
        # the smallest plan: the two planar arms of configuration 1 inside a host control loop (latency, launches, copies)
        {"name": "host planar K64 H20", "kind": "host", "scene": "planar", "boxes": 0, "K": 64, "H": 20, "lam": 1.0},
        # the ball lift of configuration 2
        {"name": "step lift K1024 H32", "kind": "step", "scene": "lift", "boxes": 0, "K": 1024, "H": 32, "lam": 0.05},
        # the transfer past eight boxes of configuration 3: the largest single controller
        {"name": "step transfer K4096 H64", "kind": "step", "scene": "transfer", "boxes": 8, "K": 4096, "H": 64, "lam": 2.0},
        # the paper's complete optimiser: elite set, learning rate, covariance blocks, projected samples
        {"name": "step eq8 qp K1024 H32", "kind": "step", "scene": "lift", "boxes": 0, "K": 1024, "H": 32, "lam": 0.05,
         "elite": 64, "qp": 30},
        # the paper's ball-task costs on the transfer scene, move phase
        {"name": "step task K4096 H64", "kind": "step", "scene": "transfer", "boxes": 8, "K": 4096, "H": 64, "lam": 20.0,
         "task": 1},
        # configuration 4: 64 controllers, K 256-4096, H 16-64, 0-16 boxes, in one launch
        {"name": "batch 64", "kind": "batch", "count": 64, "pool": 0, "lam": 2.0},
        # a batch below one full wave of the chip: what a server has at a moderate load
        {"name": "batch 5", "kind": "batch", "count": 5, "pool": 3, "lam": 2.0},
        # explicit controls: candidate plans scored from perturbed states, planar (ragged count)
        {"name": "rollout planar n777 H20", "kind": "rollout", "scene": "planar", "boxes": 0, "n": 777, "H": 20},
        # the same for the transfer, with the pick phase's task costs
        {"name": "rollout task n2048 H32", "kind": "rollout", "scene": "transfer", "boxes": 8, "n": 2048, "H": 32, "task": 0},
        # stepping a large set of simulator states once, as a data generator does
        {"name": "sim transfer n16384", "kind": "sim", "scene": "transfer", "boxes": 8, "n": 16384},
        # smoothing of stored sequences: configuration 3's 4096 x 14, and a short ragged horizon
        {"name": "project n57344 H64", "kind": "project", "n": 57344, "H": 64, "iters": 30},
        {"name": "project n5000 H27", "kind": "project", "n": 5000, "H": 27, "iters": 30},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["host", "step", "step", "step", "batch", "rollout", "rollout", "sim", "project", "project"])
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 2, 48), "pool": rng.randrange(50), "lam": 2.0}
    if kind == "project":
        return {"kind": kind, "n": _log(rng, 200, 50000), "H": rng.choice([rng.randint(2, 32), rng.randint(33, 128)]),
                "iters": rng.choice([20, 30, 50])}
    scene = rng.choice(["planar", "lift", "transfer", "transfer"])
    case = {"kind": kind, "scene": scene, "boxes": rng.randint(1, 16) if scene == "transfer" else 0}
    if kind == "host":
        return case | {"K": _log(rng, 32, 1024), "H": rng.randint(8, 48), "lam": {"planar": 1.0, "lift": 0.05, "transfer": 2.0}[scene]}
    if kind == "sim":
        return case | {"n": _log(rng, 64, 16384)}
    if kind == "rollout":
        case |= {"n": _log(rng, 64, 4096), "H": rng.randint(4, 32)}
        return case | ({"task": rng.randrange(2)} if rng.random() < 0.3 else {})
    case |= {"K": _log(rng, 64, 4096), "H": rng.randint(8, 64), "lam": {"planar": 1.0, "lift": 0.05, "transfer": 2.0}[scene]}
    option = rng.choice(["", "", "elite", "qp", "task"])
    if option == "elite":
        case |= {"elite": max(2, case["K"] // 16)}
    elif option == "qp":
        case |= {"qp": 30}
    elif option == "task":
        case |= {"task": rng.randrange(2), "lam": 20.0}
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _scene(kind, boxes):
    if kind == "planar":
        return scenes.planar_scene()
    return scenes.dh_scene(seed=0, n_boxes=boxes, task="lift" if kind == "lift" else "transfer")


@functools.lru_cache(maxsize=None)
def _pool(count, pool):
    return scenes.batched_pool(count, seed=pool)


def _warm_start(rng, H, nu, n=None):
    """A nominal sequence in the middle of a run: smooth joint velocities of a few tenths of a rad/s."""
    shape = (nu,) if n is None else (n, nu)
    t = np.arange(H)[:, None] * 0.01
    amp, freq, ph = rng.uniform(-0.4, 0.4, shape), rng.uniform(0.2, 1.0, shape), rng.uniform(0, 2 * np.pi, shape)
    if n is not None:
        amp, freq, ph = amp[:, None], freq[:, None], ph[:, None]
    return (amp * np.sin(2 * np.pi * freq * t + ph)).astype(np.float32)


def _start(sc, n, seed):
    """States of a run: the arms within a tenth of a radian of the home pose and moving, the ball at rest on the floor."""
    x = scenes.random_states(sc, n, seed, q_spread=0.1, v_spread=0.1)
    x[:, sc.nq + sc.nu:] = 0.0
    return x.astype(np.float32)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "batch":
        pool = _pool(case["count"], case["pool"])
        models = [native.Model(sc.to_blob()) for sc in pool]
        batch = native.Batch([(m, sc.K, sc.H, case["lam"], sc.sigma_vec(), scenes.controller_key(seed, i))
                              for i, (m, sc) in enumerate(zip(models, pool))])
        xs = [_gpu(_start(sc, 1, seed + i)[0]) for i, sc in enumerate(pool)]
        us = [_gpu(_warm_start(rng, sc.H, sc.nu)) for sc in pool]
        return {"kind": kind, "batch": batch, "models": models, "xs": xs, "us": us, "stream": torch.cuda.Stream()}
    if kind == "project":
        n, H = case["n"], case["H"]
        g = torch.Generator(DEV).manual_seed(seed)
        base = 0.5 * torch.randn(n, 1, device=DEV, generator=g)
        v = (base + 0.2 * torch.randn(n, H, device=DEV, generator=g)).contiguous()
        q0 = 0.3 * (2 * torch.rand(n, device=DEV, generator=g) - 1)
        qd0 = 0.3 * (2 * torch.rand(n, device=DEV, generator=g) - 1)
        return {"kind": kind, "v": v, "q0": q0, "qd0": qd0, "out": torch.empty_like(v), "iters": case["iters"],
                "bounds": _bounds()}
    sc = _scene(case["scene"], case["boxes"])
    model = native.Model(sc.to_blob())
    if kind in ("rollout", "sim"):
        n, H = case["n"], case.get("H", 1)
        x = _gpu(_start(sc, n, seed))
        ctl = native.Controller(model, n, H, 1.0, sc.sigma_vec(), seed)
        u = _gpu(_warm_start(rng, H, sc.nu, n) + rng.normal(0.0, sc.sigma, (n, H, sc.nu)).astype(np.float32))
        if "task" in case:
            ctl.set_task_cost(scenes.ball_task(sc, case["task"]))
        if kind == "sim":
            return {"kind": kind, "ctl": ctl, "start": x, "x": torch.empty_like(x), "u": u.reshape(n, sc.nu)}
        return {"kind": kind, "ctl": ctl, "x": x, "u": u, "costs": torch.empty(n, device=DEV), "end": torch.empty_like(x)}
    x, u = _start(sc, 1, seed)[0], _warm_start(rng, case["H"], sc.nu)
    ctl = native.Controller(model, case["K"], case["H"], case["lam"], sc.sigma_vec(), scenes.controller_key(seed, 0))
    state = {"kind": kind, "ctl": ctl}
    if kind == "host":
        return state | {"x": x, "u": u}
    if "elite" in case:
        ctl.set_update(case["elite"], eta=0.7, update_cov=True, cov_floor=0.01)
        state |= {"cov": torch.empty(case["H"], sc.nu, sc.nu, device=DEV), "best": torch.empty(case["H"], sc.nu, device=DEV)}
    if "qp" in case:
        ctl.set_projection(scenes.projection_bounds(sc), iters=case["qp"])
    if "task" in case:
        ctl.set_task_cost(scenes.ball_task(sc, case["task"]))
    return state | {"x": _gpu(x), "u": _gpu(u), "out": torch.empty(case["H"], sc.nu, device=DEV)}


def _bounds():
    return np.array([-1.0, 1.0, -math.pi, math.pi, -10.0, 10.0, -300.0, 300.0], dtype=np.float32)


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].step(state["xs"], state["us"], stream=state["stream"], graph=True)
        return state["us"]
    if kind == "project":
        return native.qp_project(state["v"], state["bounds"], state["q0"], state["qd0"], 0.01, iters=state["iters"],
                                 v_out=state["out"])
    ctl = state["ctl"]
    if kind == "host":
        return ctl.step_host(state["x"], state["u"])
    if kind == "rollout":
        ctl.rollout_batch(state["x"], state["u"], state["costs"], state["end"])
        return {"costs": state["costs"], "end": state["end"]}
    if kind == "sim":
        state["x"].copy_(state["start"])
        return ctl.sim_step(state["x"], state["u"])
    out = {"u": ctl.step(state["x"], state["u"], state["out"])}
    if "cov" in state:
        out |= {"cov": ctl.covariance(state["cov"]), "best": ctl.best_controls(state["best"])}
    return out


def work(case):
    """Operations and bytes that the result needs: simulator, task costs, sampling, projection and update by the
    package's operation counts with one ball contact and no exact box test a step; inputs and outputs once."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work({"kind": "step", "K": sc.K, "H": sc.H, "pool_scene": sc}) for sc in _pool(case["count"], case["pool"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "project":
        n, H = case["n"], case["H"]
        return {"bytes": 4.0 * (2 * n * H + 2 * n), "flops": n * flops.qp_flops(H, case["iters"])}
    sc = case["pool_scene"] if "pool_scene" in case else _scene(case["scene"], case["boxes"])
    n, H = case.get("K", case.get("n")), case.get("H", 1)
    nx = sc.nq + sc.nv
    f = n * H * flops.per_sample_step(sc, 1.0, 0.0, 1.0)
    if "task" in case:
        f += n * (H + 1) * flops.task_flops(sc, case["task"])
    if kind in ("rollout", "sim"):
        return {"bytes": 4.0 * (2 * n * nx + n * H * sc.nu + n), "flops": f}
    if "qp" in case:
        f += n * sc.nu * flops.qp_flops(H, case["qp"])
    cov = 2 * H * sc.nu * sc.nu if "elite" in case else 0
    return {"bytes": 4.0 * (nx + 2 * H * sc.nu + cov), "flops": f + flops.update_flops(n, H, sc.nu)}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None  # dozens of controllers: minutes in 64 bits
    if kind == "project":
        s = prepare(case, seed)
        b = torch.from_numpy(s["bounds"]).to(DEV).double()
        return _admm(s["v"].double(), b, s["q0"].double(), s["qd0"].double(), 0.01, case["iters"])
    sc = _scene(case["scene"], case["boxes"])
    sim = _Sim(sc, scenes.ball_task(sc, case["task"]) if "task" in case else None)
    if kind in ("rollout", "sim"):
        s = prepare(case, seed)
        if kind == "sim":
            return sim.rollout(s["start"].double(), s["u"].double()[:, None])[1]
        cost, end = sim.rollout(s["x"].double(), s["u"].double())
        return {"costs": cost, "end": end}
    rng = np.random.default_rng(seed)
    K, H = case["K"], case["H"]
    x = _gpu(_start(sc, 1, seed)[0]).double()
    nom = _gpu(_warm_start(rng, H, sc.nu)).double()
    U = nom + float(np.float32(sc.sigma)) * _normals(scenes.controller_key(seed, 0), K, H, sc.nu)
    if "qp" in case:
        b = scenes.projection_bounds(sc).astype(np.float32).astype(np.float64)
        for j in range(sc.nu):
            U[:, :, j] = _admm(U[:, :, j], torch.from_numpy(b[j]).to(DEV), x[j].expand(K), x[sc.nq + j].expand(K), sc.dt,
                               case["qp"])
    else:
        U = torch.minimum(torch.maximum(U, sim.u_lo), sim.u_hi)
    cost = sim.rollout(x.expand(K, -1), U)[0]
    if "elite" not in case:
        u = torch.einsum("k,khj->hj", torch.softmax(-cost / case["lam"], 0), U)
        return u.cpu().numpy() if kind == "host" else {"u": u}
    pick = torch.argsort(cost, stable=True)[: case["elite"]]
    w = torch.softmax(-cost[pick] / case["lam"], 0)
    eta, Ue = float(np.float32(0.7)), U[pick]
    u = (1 - eta) * nom + eta * torch.einsum("k,khj->hj", w, Ue)
    d = Ue - u
    eye = torch.eye(sc.nu, device=DEV, dtype=torch.float64)
    cov = (1 - eta) * sc.sigma ** 2 * eye + eta * torch.einsum("k,khi,khj->hij", w, d, d) + 0.01 * eye
    return {"u": u, "cov": cov, "best": Ue[0]}


def _normals(key, K, H, nu):
    """Standard normals K x H x nu: Philox4x32-10 words (key = seed, counter = (j/4, h, k, 0)), Box-Muller on the pairs."""
    nb = (nu + 3) // 4
    k, h, b = np.meshgrid(np.arange(K), np.arange(H), np.arange(nb), indexing="ij")
    c = [a.astype(np.uint64) for a in (b, h, k, np.zeros_like(b))]
    k0, k1, m = key & 0xFFFFFFFF, key >> 32, np.uint64(0xFFFFFFFF)
    for r in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    w = [(((a >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23) for a in c]
    z = np.empty((K, H, nb, 4))
    for p in range(2):
        r, a = np.sqrt(-2.0 * np.log(w[2 * p])), 2.0 * np.pi * w[2 * p + 1]
        z[..., 2 * p], z[..., 2 * p + 1] = r * np.cos(a), r * np.sin(a)
    return torch.from_numpy(z.reshape(K, H, 4 * nb)[:, :, :nu].copy()).to(DEV)


def _admm(v, b, q, qd, dt, iters, rho=1.0):
    """`iters` ADMM iterations on the rows position/dt, velocity, acceleration dt and jerk dt^2, scaled by 0.1, 1, 2, 4."""
    n, H = v.shape
    f8 = {"device": DEV, "dtype": torch.float64}
    dt, I = float(np.float32(dt)), torch.eye(H, **f8)
    B = I - torch.diag(torch.ones(H - 1, **f8), -1)
    rows = [torch.tril(torch.ones(H, H, **f8)), I, B, (B @ B)[1:]]
    first = torch.zeros(n, H, **f8)
    first[:, 0] = qd  # the present velocity enters the first difference, and the second one of step 1
    lo = [((b[0] - q) / dt)[:, None].expand(n, H), b[2].expand(n, H), b[4] * dt + first, b[6] * dt * dt - first[:, : H - 1]]
    hi = [((b[1] - q) / dt)[:, None].expand(n, H), b[3].expand(n, H), b[5] * dt + first, b[7] * dt * dt - first[:, : H - 1]]
    s = [float(np.float32(t)) for t in (0.1, 1.0, 2.0, 4.0)]
    D = torch.cat([t * r for t, r in zip(s, rows)])
    lo, hi = (torch.cat([t * g for t, g in zip(s, a)], 1) for a in (lo, hi))
    inv = torch.linalg.inv(I + rho * D.T @ D)
    y, x = torch.zeros_like(lo), v
    for _ in range(iters):
        a = x @ D.T + y
        w = torch.minimum(torch.maximum(a, lo), hi)
        y = a - w
        x = (v + rho * (w - y) @ D) @ inv
    return x


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


class _Sim:
    """The contact simulator and its costs over a batch of states, from the definitions: link Jacobians, dense blocks,
    box distances by bisection on the slope along the segment."""

    def __init__(self, sc, task=None):
        t = lambda f: torch.tensor(np.array([[f(l) for l in arm] for arm in sc.links], dtype=np.float64), device=DEV)  # noqa: E731
        self.sc, self.na, self.nl, self.nb = sc, sc.n_a, 2 * sc.n_a, sc.n_boxes
        self.FR, self.Fp, self.com, self.I = t(lambda l: l.F_R), t(lambda l: l.F_p), t(lambda l: l.com), t(lambda l: l.inertia)
        self.s0, self.s1, self.rc, self.mass = t(lambda l: l.s0), t(lambda l: l.s1), t(lambda l: l.radius), t(lambda l: l.mass)
        self.D, self.gear, self.tau = t(lambda l: l.damping + l.kv), t(lambda l: l.gear), t(lambda l: l.tau_max)
        self.gw = t(lambda l: 1.0 - l.gravcomp)
        self.u_lo, self.u_hi = t(lambda l: l.u_lo).reshape(-1), t(lambda l: l.u_hi).reshape(-1)
        self.bR, self.bp, self.g, self.goal, self.bc, self.bh = (
            torch.tensor(np.array(a, dtype=np.float64), device=DEV)
            for a in (sc.base_R, sc.base_p, sc.gravity, sc.goal, sc.boxes_c, sc.boxes_h))
        self.below = torch.tril(torch.ones(self.na, self.na, device=DEV, dtype=torch.float64))  # joint j moves link l
        reach = torch.zeros(self.nl + 1, self.nl, device=DEV, dtype=torch.float64)
        reach[: self.na, : self.na] = reach[self.na: self.nl, self.na:] = self.below
        self.reach = reach  # last row: no link
        P = [(-1, -1)] + [(-1, l) for l in range(self.nl)] + [(-1, -1)] * self.nb
        P += [(l, -1) for l in range(self.nl) for _ in range(self.nb)]
        self.linkA, self.linkB = (torch.tensor([p[i] for p in P], device=DEV) for i in (0, 1))
        self.ballA = torch.tensor([1.0] * (1 + self.nl + self.nb) + [0.0] * (self.nl * self.nb), device=DEV, dtype=torch.float64)
        self.task = None if task is None else torch.tensor(task, device=DEV, dtype=torch.float64)

    def fk(self, q):
        n = q.shape[0]
        R, p = self.bR.expand(n, 2, 3, 3), self.bp.expand(n, 2, 3)
        q = q.reshape(n, 2, self.na)
        z, o, Rs, ps = [], [], [], []
        for i in range(self.na):
            z.append(R[..., 2])
            o.append(p)
            c, s, l0, l1 = torch.cos(q[..., i]), torch.sin(q[..., i]), torch.zeros_like(q[..., i]), torch.ones_like(q[..., i])
            Rz = torch.stack([c, -s, l0, s, c, l0, l0, l0, l1], -1).reshape(n, 2, 3, 3)
            Rq = R @ Rz
            p = (Rq @ self.Fp[:, i, :, None])[..., 0] + p
            R = Rq @ self.FR[:, i]
            Rs.append(R)
            ps.append(p)
        z, o, R, p = (torch.stack(a, 2) for a in (z, o, Rs, ps))
        at = lambda s: (R @ s[..., None])[..., 0] + p  # noqa: E731
        return z, o, R, at(self.com), at(self.s0), at(self.s1)

    def arms(self, z, o, R, c, qd, u):
        """(M + dt D) of each arm, and the right-hand side drive - bias - D qd."""
        n, dt = z.shape[0], self.sc.dt
        J = _cross(z[:, :, None].expand(-1, -1, self.na, -1, -1), c[:, :, :, None] - o[:, :, None]) * self.below[..., None]
        Iw = R @ self.I @ R.transpose(-1, -2)
        zl = z[:, :, None] * self.below[..., None]
        M = torch.einsum("bl,nbljx,nblkx->nbjk", self.mass, J, J) + torch.einsum("nbljx,nblxy,nblky->nbjk", zl, Iw, zl)
        qd = qd.reshape(n, 2, self.na)
        w = torch.zeros(n, 2, 3, device=DEV, dtype=torch.float64)
        al, ao = w, w
        F, N = [], []
        for i in range(self.na):
            zi = z[:, :, i] * qd[:, :, i, None]
            al = al + _cross(w, zi)
            w = w + zi
            acc = lambda r: ao + _cross(al, r) + _cross(w, _cross(w, r))  # noqa: E731, B023
            F.append(self.mass[:, i, None] * (acc(c[:, :, i] - o[:, :, i]) - self.gw[:, i, None] * self.g))
            Iwi = Iw[:, :, i]
            N.append((Iwi @ al[..., None])[..., 0] + _cross(w, (Iwi @ w[..., None])[..., 0]))
            if i + 1 < self.na:
                ao = acc(o[:, :, i + 1] - o[:, :, i])
        bias = torch.einsum("nbljx,nblx->nbj", J, torch.stack(F, 2)) + torch.einsum("nbljx,nblx->nbj", zl, torch.stack(N, 2))
        drive = torch.minimum(torch.maximum(self.gear * u.reshape(n, 2, self.na), -self.tau), self.tau)
        return M + torch.diag_embed(dt * self.D), drive - bias - self.D * qd

    @staticmethod
    def box(x, c, h):
        """Signed distance, outward normal and closest surface point (inside: nearest face, ties within 1e-5)."""
        d = x - c
        cl = torch.minimum(torch.maximum(d, -h), h)
        q = d - cl
        ln = torch.linalg.norm(q, dim=-1)
        inside = (d.abs() <= h).all(-1)
        face = torch.stack([h - d, h + d], -1).flatten(-2)
        best = face.min(-1).values
        f = (face <= best[..., None] + 1e-5).to(torch.int8).argmax(-1)
        nf = torch.nn.functional.one_hot(f // 2, 3).double() * (1.0 - 2.0 * (f % 2))[..., None]
        sf = torch.where(nf != 0, nf * h, d)
        n = torch.where(inside[..., None], nf, q / ln.clamp_min(1e-300)[..., None])
        return torch.where(inside, -best, ln), n, torch.where(inside[..., None], sf, cl) + c

    def segment_box(self, a, b, c, h):
        """Point of the segment with the lowest signed distance: bisection on the sign of its slope (a convex function)."""
        d = b - a
        lo, hi = torch.zeros_like(a[..., :1]), torch.ones_like(a[..., :1])
        for _ in range(54):
            m = 0.5 * (lo + hi)
            x = a + m * d - c
            e = x.abs() - h
            out = e.clamp_min(0.0)
            inside = (e <= 0).all(-1, keepdim=True)
            g = torch.where(inside, torch.nn.functional.one_hot(e.argmax(-1), 3).double(), out) * torch.sign(x)
            up = (g * d).sum(-1, keepdim=True) > 0
            lo, hi = torch.where(up, lo, m), torch.where(up, m, hi)
        cand = torch.stack([a + 0.5 * (lo + hi) * d, a, b])
        f = self.box(cand, c, h)[0].argmin(0)
        return torch.gather(cand, 0, f[None, ..., None].expand(1, *a.shape))[0]

    def collide(self, ball, a0, a1):
        sc, n, nl, nb = self.sc, ball.shape[0], self.nl, self.nb
        a0, a1, rc = a0.reshape(n, nl, 3), a1.reshape(n, nl, 3), self.rc.reshape(-1)
        up = torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=torch.float64)
        fp = torch.cat([ball[:, :2], 0.5 * (ball[:, 2:] - sc.ball_r + sc.floor_z)], 1)
        dist, pt, nn = [(ball[:, 2:] - sc.floor_z) - sc.ball_r], [fp[:, None]], [up.expand(n, 1, 3)]
        d = a1 - a0
        t = (((ball[:, None] - a0) * d).sum(-1) / (d * d).sum(-1)).clamp(0.0, 1.0)
        s = a0 + t[..., None] * d
        df = ball[:, None] - s
        ln = torch.linalg.norm(df, dim=-1)
        nv = df / ln[..., None]
        dist.append(ln - sc.ball_r - rc)
        pt.append(0.5 * ((ball[:, None] - sc.ball_r * nv) + (s + rc[:, None] * nv)))
        nn.append(nv)
        if nb:
            f, nv, surf = self.box(ball[:, None].expand(n, nb, 3), self.bc, self.bh)
            dist.append(f - sc.ball_r)
            pt.append(0.5 * ((ball[:, None] - sc.ball_r * nv) + surf))
            nn.append(nv)
            near = ((0.5 * (a0 + a1))[:, :, None] - self.bc).abs() <= self.bh + (0.5 * d.abs())[:, :, None] + rc[:, None, None] + 1e-6
            i, l, b = torch.nonzero(near.all(-1), as_tuple=True)
            x = self.segment_box(a0[i, l], a1[i, l], self.bc[b], self.bh[b])
            f, nv, surf = self.box(x, self.bc[b], self.bh[b])
            dl = torch.ones(n, nl, nb, device=DEV, dtype=torch.float64)
            pl = torch.zeros(n, nl, nb, 3, device=DEV, dtype=torch.float64)
            ql = up.expand(n, nl, nb, 3).clone()
            dl[i, l, b] = f - rc[l]
            pl[i, l, b] = 0.5 * ((x - rc[l, None] * nv) + surf)
            ql[i, l, b] = nv
            dist.append(dl.reshape(n, -1))
            pt.append(pl.reshape(n, -1, 3))
            nn.append(ql.reshape(n, -1, 3))
        return torch.cat(dist, 1), torch.cat(pt, 1), torch.cat(nn, 1)

    def solve(self, L, vf, ball, z, o, dist, pt, nn):
        """Impulses by projected Gauss-Seidel over the first max_contacts active pairs, and the velocities after them."""
        sc, n, na, nl = self.sc, vf.shape[0], self.na, self.nl
        act = dist < 0
        rank = torch.cumsum(act, 1) - 1
        C = int((act & (rank < sc.max_contacts)).sum(1).max())
        if C == 0:
            return vf
        slots = [(act & (rank == s)) for s in range(C)]
        idx = torch.stack([m.to(torch.int8).argmax(1) for m in slots], 1)
        on = torch.stack([m.any(1) for m in slots], 1).double()
        take = lambda a: torch.gather(a, 1, idx[..., None].expand(-1, -1, 3))  # noqa: E731
        p, nv, dep = take(pt), take(nn), -torch.gather(dist, 1, idx)
        ax = torch.nn.functional.one_hot(nv.abs().argmin(-1), 3).double()
        t1 = _cross(nv, ax)
        t1 = t1 / torch.linalg.norm(t1, dim=-1, keepdim=True)
        e = torch.stack([nv, t1, _cross(nv, t1)], 2)  # n x C x 3 rows x 3
        zl, ol = z.reshape(n, 1, nl, 3), o.reshape(n, 1, nl, 3)
        lever = _cross(zl.expand(n, C, nl, 3), p[:, :, None] - ol)
        side = self.reach[self.linkA[idx]] * (self.linkA[idx] >= 0)[..., None] - self.reach[self.linkB[idx]] * (self.linkB[idx] >= 0)[..., None]
        Ja = torch.einsum("ncrx,ncjx->ncrj", e, lever) * side[:, :, None]
        bs = self.ballA[idx][..., None, None]
        Jb = bs * torch.cat([e, _cross((p - ball[:, None])[:, :, None].expand_as(e), e)], -1)
        J = (torch.cat([Ja, Jb], -1) * on[..., None, None]).reshape(n, 3 * C, nl + 6)
        X = [torch.cholesky_solve(J[:, :, a * na: (a + 1) * na].transpose(1, 2), L[:, a]) for a in range(2)]
        im = torch.tensor([1 / sc.ball_m] * 3 + [1 / sc.ball_I] * 3, device=DEV, dtype=torch.float64)
        X = torch.cat(X + [im[:, None] * J[:, :, nl:].transpose(1, 2)], 1)
        A = J @ X
        b = (J @ vf[..., None])[..., 0]
        diag = torch.diagonal(A, dim1=1, dim2=2)
        R = (1 - sc.impedance) / sc.impedance * diag
        den = torch.where(diag > 0, diag + R, torch.ones_like(diag))
        lam = torch.zeros_like(b)
        for _ in range(sc.sweeps):
            for c in range(C):
                i = 3 * c
                r = b[:, i] + R[:, i] * lam[:, i] - sc.erp / sc.dt * dep[:, c] + (A[:, i] * lam).sum(1)
                ln = (lam[:, i] - r / den[:, i]).clamp_min(0.0) * on[:, c]
                lam = torch.cat([lam[:, :i], ln[:, None], lam[:, i + 1:]], 1)
                rt = b[:, i + 1: i + 3] + R[:, i + 1: i + 3] * lam[:, i + 1: i + 3] + (A[:, i + 1: i + 3] * lam[:, None]).sum(2)
                lt = lam[:, i + 1: i + 3] - rt / den[:, i + 1: i + 3]
                m, lim = torch.linalg.norm(lt, dim=1), sc.mu * ln
                lt = lt * torch.where(m > lim, lim / m.clamp_min(1e-300), torch.ones_like(m))[:, None]
                lam = torch.cat([lam[:, : i + 1], lt, lam[:, i + 3:]], 1)
        return vf + (X @ lam[..., None])[..., 0]

    def distances(self, ball, a0, a1):
        """The task's collision pairs: links x boxes, links x ball (pick phase), left x right links."""
        n, nl, na = ball.shape[0], self.nl, self.na
        a0, a1, rc = a0.reshape(n, nl, 3), a1.reshape(n, nl, 3), self.rc.reshape(-1)
        out = []
        if self.nb:
            shape = (n, nl, self.nb, 3)
            c, h = self.bc.expand(shape), self.bh.expand(shape)
            x = self.segment_box(a0[:, :, None].expand(shape), a1[:, :, None].expand(shape), c, h)
            out.append((self.box(x, c, h)[0] - rc[:, None]).reshape(n, -1))
        if self.task[0] == 0:
            out.append(self.segments(a0, a1, ball[:, None], ball[:, None]) - rc - self.sc.ball_r)
        d = self.segments(a0[:, :na, None], a1[:, :na, None], a0[:, None, na:], a1[:, None, na:])
        out.append((d - rc[:na, None] - rc[na:]).reshape(n, -1))
        return torch.cat(out, 1)

    @staticmethod
    def segments(a0, a1, b0, b1):
        """Distance of two segments: the lowest over the interior stationary point and the four ends' projections."""
        u, v, w = a1 - a0, b1 - b0, a0 - b0
        dot = lambda x, y: (x * y).sum(-1, keepdim=True)  # noqa: E731
        A, B, C, D, E = dot(u, u), dot(u, v), dot(v, v), dot(u, w), dot(v, w)
        den = A * C - B * B
        ok = den > 1e-14 * A * C
        safe = torch.where(ok, den, torch.ones_like(den))
        s, t = (B * E - C * D) / safe, (A * E - B * D) / safe
        ok = ok & (s >= 0) & (s <= 1) & (t >= 0) & (t <= 1)
        gap = lambda s, t: torch.linalg.norm(w + s * u - t * v, dim=-1)  # noqa: E731
        best = torch.where(ok[..., 0], gap(s, t), torch.full_like(gap(s, t), math.inf))
        pos = lambda x, y: torch.where(y > 0, x / y.clamp_min(1e-300), torch.zeros_like(x)).clamp(0.0, 1.0)  # noqa: E731
        for k in (0.0, 1.0):
            k = torch.full_like(A, k)
            best = torch.minimum(best, gap(k, pos(E + k * B, C)))
            best = torch.minimum(best, gap(pos(k * B - D, A), k))
        return best

    def rollout(self, x, U):
        """Summed costs and final states of the controls U (n x H x nu) from the states x."""
        sc, nl, nq = self.sc, self.nl, self.sc.nq
        dt, q, v = sc.dt, x[:, :nq].clone(), x[:, nq:].clone()
        cost = torch.zeros(x.shape[0], device=DEV, dtype=torch.float64)
        terms = _Task(self) if self.task is not None else None
        geom = self.fk(q[:, :nl])
        if terms:
            terms.state(q, v, geom, True)
        for h in range(U.shape[1]):
            z, o, R, c, a0, a1 = geom
            ball = q[:, nl: nl + 3]
            M, rhs = self.arms(z, o, R, c, v[:, :nl], U[:, h])
            L = torch.linalg.cholesky(M)
            vf = v.clone()
            vf[:, :nl] += dt * torch.cholesky_solve(rhs[..., None], L)[..., 0].reshape(-1, nl)
            vf[:, nl: nl + 3] += dt * self.g
            dist, pt, nn = self.collide(ball, a0, a1)
            v = self.solve(L, vf, ball, z, o, dist, pt, nn)
            pen = (-dist).clamp_min(0.0)
            boxed = pen[:, 1 + nl:].sum(1)
            w = v[:, nl + 3:] * dt
            ang = torch.linalg.norm(w, dim=1, keepdim=True)
            k = torch.where(ang > 0, torch.sin(0.5 * ang) / ang.clamp_min(1e-300), torch.full_like(ang, 0.5))
            a, b = torch.cos(0.5 * ang), w * k
            s, r = q[:, nl + 3: nl + 4], q[:, nl + 4:]
            quat = torch.cat([a * s - (b * r).sum(1, keepdim=True), a * r + s * b + _cross(b, r)], 1)
            quat = quat / torch.linalg.norm(quat, dim=1, keepdim=True)
            q = torch.cat([q[:, : nl + 3] + dt * v[:, : nl + 3], quat], 1)
            geom = self.fk(q[:, :nl])
            if terms:
                terms.state(q, v, geom, False)
                continue
            e = q[:, nl: nl + 3] - self.goal
            cost = cost + sc.w_goal * (e * e).sum(1) + sc.w_u * (U[:, h] ** 2).sum(1) + sc.w_pen * pen.sum(1) + sc.w_obst * boxed
            if sc.w_grasp:
                e = geom[5][:, 0, -1] + geom[5][:, 1, -1] - 2 * q[:, nl: nl + 3]
                cost = cost + sc.w_grasp * (e * e).sum(1)
        return terms.total() if terms else cost, torch.cat([q, v], 1)


class _Task:
    """The ball-task cost suite (Sec. IV-B) summed over the states of a rollout."""

    def __init__(self, sim):
        self.sim, self.p = sim, sim.task
        self.sums, self.before = {}, None

    def add(self, name, v):
        self.sums[name] = self.sums.get(name, 0.0) + v

    def state(self, q, v, geom, first):
        sim, p, nl, na = self.sim, self.p, self.sim.nl, self.sim.na
        z, o, R, _, a0, a1 = geom
        d = sim.distances(q[:, nl: nl + 3], a0, a1)
        before, self.before = self.before, d
        if first:
            return
        self.add("c", ((1 - p[2]) * before - d).clamp_min(0.0).sum(1) + (d < 0).sum(1))
        ee = a1[:, :, -1]
        vel = (_cross(z, ee[:, :, None] - o) * v[:, :nl].reshape(-1, 2, na, 1)).sum(2)
        dp, dv, mid = ee[:, 0] - ee[:, 1], vel[:, 0] - vel[:, 1], 0.5 * (ee[:, 0] + ee[:, 1])
        norm = lambda x: torch.linalg.norm(x, dim=1)  # noqa: E731
        self.add("th", norm(q[:, :nl] - p[26:]))
        self.add("yz", norm(dp[:, 1:]))
        self.add("v2", (dp * dv).sum(1) ** 2)
        for a, at in ((0, 18), (1, 22)):  # half of the angle between the two rotations, each as |<q, q*>|
            w, x, y, k = p[at: at + 4]
            T = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                             2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                             2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)]).reshape(3, 3)
            tr = (R[:, a, -1] * T).sum((1, 2))
            self.add("r", 0.5 * torch.acos((0.5 * (tr - 1)).clamp(-1.0, 1.0)))
        self.add("l", (norm(dp) - p[8]) ** 2)
        off = torch.stack([torch.zeros_like(p[11]), torch.zeros_like(p[11]), p[11]])
        self.add("eo", norm(mid - p[12:15] + off))
        self.add("ot", norm(mid + off - p[15:18]))

    def total(self):
        p, s = self.p, self.sums
        reach = p[9] * s["eo"] if p[0] == 0 else p[10] * s["ot"]
        return (p[1] * s["c"] + reach + p[3] * s["th"] + p[4] * s["yz"] + p[5] * torch.sqrt(s["v2"]) + p[6] * s["r"]
                + p[7] * s["l"])
