"""Performance cases of the q-LSKUM solver and its warm-start network.

Each case is one call sequence that a user's program makes through the public
entry points (``lskum.Solver``, ``surrogate.MLP``): pseudo-time iterations in
FP64 and in mixed precision, on one cloud, on many conditions at once and on
packed clouds; the evaluation of a residual and its derivatives; the network's
prediction on a whole cloud and its loss and gradients on a training batch.
Clouds are the library's NACA 0012 generator's, in shuffled input order; the
flow is a seeded smooth perturbation of the free stream at every point, so
every neighbour pair does its full work. A pass of the solver sets the state
from pinned host memory, iterates, and reads residue, forces and state back.

``exact`` evaluates the same inputs in 64 bits with plain torch.
"""

import functools
import math
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2108_07031_gb300 import cloud as Cl  # noqa: E402
from paper_2108_07031_gb300 import lskum as L  # noqa: E402
from paper_2108_07031_gb300 import surrogate as S  # noqa: E402

GAMMA = 1.4
CFL = 0.2
ENTRIES = 13.9  # mean neighbours of a point


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest configuration: 5,120 points in FP64, latency counts
        dict(name="fp64-5k", kind="solve", points=5120, precision="fp64", steps=10, inner=2,
             conditions=1, members=1, mach=0.63, alpha=2.0),
        # the next study size with the paper's three inner iterations
        dict(name="fp64-46k-inner3", kind="solve", points=46080, precision="fp64", steps=4, inner=3,
             conditions=1, members=1, mach=0.63, alpha=2.0),
        # the benchmark family in FP64: 0.6M and 2.5M points
        dict(name="fp64-600k", kind="solve", points=600_000, precision="fp64", steps=2, inner=2,
             conditions=1, members=1, mach=0.63, alpha=2.0),
        dict(name="fp64-2500k", kind="solve", points=2_500_000, precision="fp64", steps=1, inner=2,
             conditions=1, members=1, mach=0.63, alpha=2.0),
        # several free streams on one cloud in FP64
        dict(name="fp64-batch16-20k", kind="solve", points=20_000, precision="fp64", steps=2,
             inner=2, conditions=16, members=1, mach=0.0, alpha=0.0),
        # one residual and its derivatives, for checks and for callers with
        # their own time stepping; the transonic condition
        dict(name="fp64-eval-150k", kind="eval", points=150_000, precision="fp64", inner=2,
             mach=0.85, alpha=1.0),
        # mixed precision: the small cloud, the ordinary one
        dict(name="mixed-5k", kind="solve", points=5120, precision="mixed", steps=20, inner=2,
             conditions=1, members=1, mach=0.63, alpha=2.0),
        dict(name="mixed-600k", kind="solve", points=600_000, precision="mixed", steps=10, inner=2,
             conditions=1, members=1, mach=0.85, alpha=1.0),
        # 64 conditions on the small cloud: how the network's training data is made
        dict(name="mixed-batch64-5k", kind="solve", points=5120, precision="mixed", steps=10,
             inner=2, conditions=64, members=1, mach=0.0, alpha=0.0),
        # clouds of uneven size packed into one context
        dict(name="mixed-ragged6", kind="solve", points=600_000, precision="mixed", steps=5,
             inner=2, conditions=1, members=6, mach=0.63, alpha=2.0),
        # the network: a prediction for every point of a cloud
        dict(name="predict-46k", kind="predict", points=46080, capacity=16384, mach=0.63, alpha=2.0),
        # loss and gradients of one training batch of the study's size
        dict(name="gradients-8192", kind="gradients", batch=8192),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "mixed", "mixed", "batch", "ragged", "eval", "predict",
                       "gradients"])
    mach, alpha = round(rng.uniform(0.3, 0.8), 3), round(rng.uniform(-4.0, 6.0), 2)
    if kind == "predict":
        return dict(kind="predict", points=_log_uniform(rng, 600, 150_000),
                    capacity=rng.choice([4096, 16384, 65536]), mach=mach, alpha=alpha)
    if kind == "gradients":
        return dict(kind="gradients", batch=_log_uniform(rng, 100, 16384))
    if kind == "eval":
        return dict(kind="eval", points=_log_uniform(rng, 600, 300_000),
                    precision=rng.choice(["fp64", "fp64", "mixed"]), inner=rng.choice([0, 2, 3]),
                    mach=mach, alpha=alpha)
    case = dict(kind="solve", points=_log_uniform(rng, 600, 600_000), precision=kind, steps=1,
                inner=rng.choice([2, 2, 3]), conditions=1, members=1, mach=mach, alpha=alpha)
    if kind == "batch":
        case["precision"] = rng.choice(["fp64", "mixed"])
        case["conditions"] = rng.choice([2, 4, 8, 16, 32, 64])
        case["points"] = _log_uniform(rng, 600, 400_000 / case["conditions"])
        case["mach"] = case["alpha"] = 0.0
    if kind == "ragged":
        case["precision"] = rng.choice(["fp64", "mixed"])
        case["members"] = rng.randint(2, 8)
        case["points"] = _log_uniform(rng, 10_000, 400_000)
    pairs = case["points"] * case["conditions"]
    most = max(1.0, (600_000 if case["precision"] == "fp64" else 3_000_000) / pairs)
    case["steps"] = rng.randint(1, int(min(20, most)))
    return case


# ------------------------------------------------------------------ inputs

def _sizes(points, members):
    """Uneven member sizes that add up to about `points`."""
    share = [1.0 + 1.5 * k for k in range(members)]
    return [max(600, int(points * s / sum(share))) for s in share]


@functools.lru_cache(maxsize=8)
def _cloud(points, members=1):
    if members > 1:
        return Cl.pack([Cl.cloud_for_points(n, seed=100 + k)
                        for k, n in enumerate(_sizes(points, members))])[0]
    return Cl.cloud_for_points(points)


def _conditions(case, seed):
    if case["conditions"] > 1:
        return Cl.conditions(case["conditions"], seed=seed)
    return np.array([case["mach"]]), np.array([case["alpha"]])


def _states(cloud, mach, alpha, seed):
    return np.stack([Cl.perturbed_state(cloud, m, a, seed=seed + k)
                     for k, (m, a) in enumerate(zip(mach, alpha))])


def _solver(cloud, case, conditions=1):
    return L.Solver.from_cloud(cloud, precision=L.FP64 if case["precision"] == "fp64" else L.MIXED,
                               inner_iters=case["inner"], cfl=CFL, n_conditions=conditions)


@functools.lru_cache(maxsize=4)
def _wall_distance(points):
    return S.wall_distance(_cloud(points))


def _raw(case):
    cloud = _cloud(case["points"])
    return S.raw_inputs(cloud, _wall_distance(case["points"]), [case["mach"]], [case["alpha"]])[0]


def _params(seed):
    p = S.init_params(seed)
    p[-4:] = np.random.Generator(np.random.PCG64(seed)).normal(0.0, 0.2, 4)
    return p


def _training_batch(case, seed):
    """Rows of several conditions on the 5,120-point cloud, as shuffled
    mini-batches take them: raw inputs and targets."""
    cloud, rng = _cloud(5120), np.random.Generator(np.random.PCG64(seed))
    mach, alpha = Cl.conditions(8, seed=seed)
    raw = S.raw_inputs(cloud, _wall_distance(5120), mach, alpha).reshape(-1, 5)
    W = _states(cloud, mach, alpha, seed)
    T = np.concatenate([S.targets(W[k], mach[k], alpha[k]) for k in range(8)])
    rows = rng.permutation(raw.shape[0])[:case["batch"]]
    return np.ascontiguousarray(raw[rows]), np.ascontiguousarray(T[rows])


def prepare(case, seed):
    if case["kind"] == "predict":
        net = S.MLP(capacity=case["capacity"], seed=seed)
        net.set_params(_params(seed))
        return dict(case=case, net=net, raw=torch.from_numpy(_raw(case)).cuda())
    if case["kind"] == "gradients":
        net = S.MLP(capacity=case["batch"], seed=seed)
        net.set_params(_params(seed))
        raw, T = _training_batch(case, seed)
        feat = net.features(torch.from_numpy(raw).cuda())
        return dict(case=case, net=net, feat=feat, target=torch.from_numpy(T).cuda())
    if case["kind"] == "eval":
        cloud = _cloud(case["points"])
        solver = _solver(cloud, case)
        solver.set_freestream(case["mach"], case["alpha"])
        solver.set_state(Cl.perturbed_state(cloud, case["mach"], case["alpha"], seed=seed))
        return dict(case=case, solver=solver)
    cloud = _cloud(case["points"], case["members"])
    mach, alpha = _conditions(case, seed)
    solver = _solver(cloud, case, case["conditions"])
    solver.set_conditions(mach, alpha)
    W = torch.from_numpy(_states(cloud, mach, alpha, seed)).pin_memory()
    return dict(case=case, solver=solver, start=W, out=torch.empty_like(W).pin_memory())


# ------------------------------------------------------------------ one pass

def run(state):
    case = state["case"]
    if case["kind"] == "predict":
        return state["net"].predict(state["net"].features(state["raw"]))
    if case["kind"] == "gradients":
        loss, grads = state["net"].gradients(state["feat"], state["target"])
        return {"loss": loss, "gradients": grads}
    solver = state["solver"]
    if case["kind"] == "eval":
        R = solver.eval_residual()
        qx, qy = solver.eval_q_derivatives()
        return _typed(case, {"residual": R, "qx": qx, "qy": qy})
    solver.set_state_ptr(state["start"].data_ptr())
    solver.step(case["steps"])
    residue = solver.residual_norm()
    cl, cd = solver.forces()
    solver.get_state_ptr(state["out"].data_ptr())
    return _typed(case, {"state": state["out"], "residue": residue, "cl": cl, "cd": cd})


def _typed(case, out):
    """The mixed path computes in FP32: its results are handed on in FP32, as
    the network's training targets take them."""
    if case["precision"] == "fp64":
        return out
    return {k: v if isinstance(v, float) else
            (v.float() if isinstance(v, torch.Tensor) else v.astype(np.float32))
            for k, v in out.items()}


# ------------------------------------------------------------------ work

def work(case):
    if case["kind"] in ("predict", "gradients"):
        n = case["points"] if case["kind"] == "predict" else case["batch"]
        weights = 32 * 256 + 4 * 256 * 256 + 256 * 4
        if case["kind"] == "predict":
            return {"bytes": n * 4.0 * (5 + 4) + 4 * weights, "flops": 2.0 * n * weights}
        return {"bytes": n * 4.0 * (32 + 4) + 8 * weights, "flops": 6.0 * n * weights}
    n = case["points"]
    entries = ENTRIES * n
    # the cloud once: coordinates, normals, lists; the state in and out
    cloud_bytes = n * 33.0 + 4.0 * entries
    pairs = n * (case["conditions"] if case["kind"] == "solve" else 1)
    if case["kind"] == "eval":
        return {"bytes": cloud_bytes + n * 32.0 * 4,
                "flops": entries * (375.0 + 32 * case["inner"]) + entries * (20.0 + 32 * case["inner"])}
    per_stage = entries / n * (375.0 + 32 * case["inner"]) + 60
    return {"bytes": cloud_bytes + pairs * 64.0, "flops": 4.0 * case["steps"] * pairs * per_stage}


# ------------------------------------------------------------------ 64 bits

class _Plain:
    """The method in 64 bits, written out with torch: every neighbour list
    padded to the longest one, all points of one condition at a time."""

    def __init__(self, cloud):
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        counts = np.diff(cloud.nbr_offsets.astype(np.int64))
        K = int(counts.max())
        idx = np.zeros((cloud.n, K), dtype=np.int64)
        mask = np.arange(K)[None, :] < counts[:, None]
        idx[mask] = cloud.nbr_idx
        idx[~mask] = np.broadcast_to(np.arange(cloud.n)[:, None], idx.shape)[~mask]
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
        self.nbr = t(idx.T)  # K x n
        self.mask = t(mask.T)
        self.n, self.K, self.n_c = cloud.n, K, cloud.n_c
        xy, nrm, flag = t(cloud.xy), t(cloud.normals), t(cloud.flags.astype(np.int64))
        self.interior, self.wall, self.outer = flag == 0, flag == 1, flag == 2
        one, zero = torch.ones_like(nrm[:, 0]), torch.zeros_like(nrm[:, 0])
        self.nx = torch.where(self.interior, zero, nrm[:, 0])
        self.ny = torch.where(self.interior, one, nrm[:, 1])
        self.tx, self.ty = self.ny, -self.nx
        self.normal = nrm
        d = xy[self.nbr] - xy[None]
        dx, dy = d[..., 0], d[..., 1]
        self.hx, self.hy = 0.5 * dx, 0.5 * dy
        inf = torch.full_like(dx, math.inf)
        self.dmin = torch.where(self.mask, torch.sqrt(dx * dx + dy * dy), inf).min(0).values
        live = self.mask.double()
        sxx, sxy, syy = (live * dx * dx).sum(0), (live * dx * dy).sum(0), (live * dy * dy).sum(0)
        det = sxx * syy - sxy * sxy
        self.wx, self.wy = live * (dx * syy - dy * sxy) / det, live * (dy * sxx - dx * sxy) / det
        ds, dn = dx * self.tx + dy * self.ty, dx * self.nx + dy * self.ny
        self.split = []  # (axis, sign, weights) of the four split stencils
        for axis, a in ((0, ds), (1, dn)):
            for sign in (1, -1):
                member = self.mask & ((a < 0) if sign > 0 else (a > 0))
                if axis == 1:
                    member = member & ~(self.wall if sign > 0 else self.outer)[None]
                m = member.double()
                ss, sn, nn = (m * ds * ds).sum(0), (m * ds * dn).sum(0), (m * dn * dn).sum(0)
                D = ss * nn - sn * sn
                w = m * ((ds * nn - dn * sn) if axis == 0 else (dn * ss - ds * sn)) / D
                w = torch.where(member, w, torch.zeros_like(w))
                if axis == 1 and sign < 0:
                    w = torch.where(self.wall[None], 2.0 * w, w)
                self.split.append((axis, sign, w))
        loop = xy[:cloud.n_c]
        ahead = (torch.roll(loop, -1, 0) - loop).square().sum(1).sqrt()
        self.ds = 0.5 * (ahead + torch.roll(ahead, 1, 0))

    @staticmethod
    def q_of(W):
        rho, u, v, p = W.unbind(1)
        beta = rho / (2.0 * p)
        q1 = torch.log(rho) + torch.log(beta) / (GAMMA - 1) - beta * (u * u + v * v)
        return torch.stack([q1, 2 * beta * u, 2 * beta * v, -2 * beta], 1)

    def derivatives(self, q, inner):
        wx, wy = self.wx[..., None], self.wy[..., None]
        dq = q[self.nbr] - q[None]
        qx, qy = (wx * dq).sum(0), (wy * dq).sum(0)
        for _ in range(inner):
            c = dq - (self.hx[..., None] * (qx[self.nbr] - qx[None])
                      + self.hy[..., None] * (qy[self.nbr] - qy[None]))
            qx, qy = (wx * c).sum(0), (wy * c).sum(0)
        return qx, qy

    def _flux(self, q, axis, sign):
        """Split flux (rho, s-momentum, n-momentum, energy) along `axis` of the
        local frame for the modified states q (n x 4)."""
        beta = -0.5 * q[:, 3]
        u, v = q[:, 1] / (2 * beta), q[:, 2] / (2 * beta)
        uu = u * u + v * v
        rho = torch.exp(q[:, 0] - torch.log(beta) / (GAMMA - 1) + beta * uu)
        p = rho / (2 * beta)
        us, un = u * self.tx + v * self.ty, u * self.nx + v * self.ny
        a, b = (us, un) if axis == 0 else (un, us)
        E = p / (GAMMA - 1) + 0.5 * rho * uu
        s = a * torch.sqrt(beta)
        A = 0.5 * torch.special.erfc(-sign * s)
        B = sign * torch.exp(-s * s) / (2.0 * torch.sqrt(math.pi * beta))
        mass = rho * (a * A + B)
        ma = (p + rho * a * a) * A + rho * a * B
        mb = b * mass
        en = (p + E) * a * A + (E + 0.5 * p) * B
        return torch.stack([mass, ma, mb, en] if axis == 0 else [mass, mb, ma, en], 1)

    def residual(self, q, qx, qy):
        R = torch.zeros_like(q)
        for k in range(self.K):
            j, hx, hy = self.nbr[k], self.hx[k][:, None], self.hy[k][:, None]
            qj = q[j] - (hx * qx[j] + hy * qy[j])
            q0 = q - (hx * qx + hy * qy)
            for axis, sign, w in self.split:
                R += w[k][:, None] * (self._flux(qj, axis, sign) - self._flux(q0, axis, sign))
        ms, mn = R[:, 1].clone(), R[:, 2].clone()
        R[:, 1], R[:, 2] = ms * self.tx + mn * self.nx, ms * self.ty + mn * self.ny
        R[self.outer] = 0.0
        return R

    def steps(self, W, count, inner):
        W = W.clone()
        residue = 0.0
        for _ in range(count):
            rho, u, v, p = W.unbind(1)
            dt = CFL * self.dmin / (torch.sqrt(u * u + v * v) + torch.sqrt(GAMMA * p / rho))
            U0 = torch.stack([rho, rho * u, rho * v,
                              p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)], 1)
            U = U0.clone()
            for stage in range(4):
                q = self.q_of(W)
                R = self.residual(q, *self.derivatives(q, inner))
                if stage == 0:
                    residue = math.sqrt(float((R[:, 0] ** 2).sum())) / self.n
                step = U - 0.5 * dt[:, None] * R
                if stage == 2:
                    step = (2.0 / 3.0) * U0 + (1.0 / 3.0) * step
                tx, ty = self.normal[:, 1], -self.normal[:, 0]
                ms = step[:, 1] * tx + step[:, 2] * ty
                step[:, 1] = torch.where(self.wall, ms * tx, step[:, 1])
                step[:, 2] = torch.where(self.wall, ms * ty, step[:, 2])
                U = torch.where(self.outer[:, None], U, step)
                rho, u, v = U[:, 0], U[:, 1] / U[:, 0], U[:, 2] / U[:, 0]
                p = (GAMMA - 1) * (U[:, 3] - 0.5 * rho * (u * u + v * v))
                W = torch.where(self.outer[:, None], W, torch.stack([rho, u, v, p], 1))
        return W, residue

    def forces(self, W, mach, alpha):
        dp = W[:self.n_c, 3] - 1.0 / GAMMA
        f = -(dp * self.ds)[:, None] * self.normal[:self.n_c]
        fx, fy = float(f[:, 0].sum()), float(f[:, 1].sum())
        a, qinf = math.radians(alpha), 0.5 * mach * mach
        return (-fx * math.sin(a) + fy * math.cos(a)) / qinf, (fx * math.cos(a) + fy * math.sin(a)) / qinf


def _plain_features(raw, proj):
    x, y, d, m, a = torch.from_numpy(raw.astype(np.float64)).unbind(1)
    t = torch.stack([x, y], 1) @ torch.from_numpy(proj.astype(np.float64)).T
    f = torch.zeros(raw.shape[0], 32, dtype=torch.float64)
    f[:, :5] = torch.stack([x / 10, y / 10, torch.log(d + 1e-3) / 5, (m - 0.55) * 4, (a - 1) / 5], 1)
    f[:, 5:13], f[:, 13:21] = torch.sin(t), torch.cos(t)
    return f


def _plain_network(feat, p):
    x, at = feat, 0
    for layer in range(6):
        k, n = (32 if layer == 0 else 256), (4 if layer == 5 else 256)
        x = x @ p[at:at + n * k].reshape(n, k).T + p[at + n * k:at + n * k + n]
        at += n * k + n
        if layer < 5:
            x = torch.tanh(x)
    return x


def exact(case, seed):
    if case["kind"] == "predict":
        feat = _plain_features(_raw(case), S.projection())
        return _plain_network(feat, torch.from_numpy(_params(seed).astype(np.float64)))
    if case["kind"] == "gradients":
        raw, T = _training_batch(case, seed)
        p = torch.from_numpy(_params(seed).astype(np.float64)).requires_grad_()
        out = _plain_network(_plain_features(raw, S.projection()), p)
        loss = ((out - torch.from_numpy(T.astype(np.float64))) ** 2).mean()
        loss.backward()
        return {"loss": float(loss.detach()), "gradients": p.grad}
    if case["kind"] == "eval":
        cloud = _cloud(case["points"])
        plain = _Plain(cloud)
        W = torch.from_numpy(Cl.perturbed_state(cloud, case["mach"], case["alpha"], seed=seed))
        q = plain.q_of(W.to(plain.nbr.device))
        qx, qy = plain.derivatives(q, case["inner"])
        return {"residual": plain.residual(q, qx, qy).cpu(), "qx": qx.cpu(), "qy": qy.cpu()}
    cloud = _cloud(case["points"], case["members"])
    mach, alpha = _conditions(case, seed)
    plain = _Plain(cloud)
    W = torch.from_numpy(_states(cloud, mach, alpha, seed)).to(plain.nbr.device)
    got = [plain.steps(w, case["steps"], case["inner"]) for w in W]
    state = torch.stack([w for w, _ in got]).cpu()
    if case["conditions"] > 1:
        # the forces of a batch come as arrays, one value per condition
        f = np.array([plain.forces(w, m, a) for (w, _), m, a in zip(got, mach, alpha)])
        return {"state": state, "residue": np.array([r for _, r in got]), "cl": f[:, 0], "cd": f[:, 1]}
    if case["members"] > 1:  # several wall loops
        return {"state": state, "residue": got[0][1], "cl": None, "cd": None}
    cl, cd = plain.forces(got[0][0], float(mach[0]), float(alpha[0]))
    return {"state": state, "residue": got[0][1], "cl": cl, "cd": cd}
