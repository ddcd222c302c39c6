"""The workloads this library is measured on: batched inverse dynamics, its adjoint and forward
dynamics of serial chains in FP32 and FP64, and mixed batches of many robots, each through the
public entry points of the package.

The sizes are those of the repository's configurations and tests (7-joint arms, chains of 16 to
100 links, batches of 1024 to 262144 states, mixed requests of 6 to 100 links) and odd ones
between them. Chains and states are drawn from a seed: rotations uniform on SO(3), joint axes
uniform on the sphere, masses of 0.5 to 5 kg, q ~ U[-pi, pi], qd ~ N(0, 1), qdd ~ N(0, 2),
tau ~ N(0, 10), adjoint weights ~ N(0, 1).

A case has an ``op``:

* ``rnea``      tau = ID(q, qd, qdd) of B states of one n-link chain;
* ``vjp``       the gradients of w . tau with respect to q, qd and qdd;
* ``autograd``  tau through the differentiable call, then its backward pass;
* ``aba``       qdd = FD(q, qd, tau);
* ``fleet``     ``requests`` mixed requests (one in five forward dynamics) spread over
                ``robots`` chains of ``n_lo`` to ``n_hi`` links.
"""
import math

import numpy as np
import torch

import paper_1609_04493_gb300 as rd

TORCH = {"float32": torch.float32, "float64": torch.float64}

# Arithmetic per link that no formulation in use here goes below (FMA = 2): the recursion in
# common-normal frames, its adjoint with nothing re-derived, and the articulated-body algorithm
# (the bias recursion plus the structured inertia update and the two solves).
FLOP = {"rnea": 257, "vjp": 621, "autograd": 257 + 621, "aba": 657}
# Elements read and written per joint.
ELEMS = {"rnea": 4, "vjp": 7, "autograd": 3 + 1 + 4 + 3, "aba": 4}


def listed():
    return [
        # The smallest call: one control step of a sampling controller on a 7-joint arm.
        {"name": "rnea_arm_f32", "op": "rnea", "dtype": "float32", "n": 7, "B": 1024},
        # The same arm in FP64, as a simulator or an identification run calls it.
        {"name": "rnea_arm_f64", "op": "rnea", "dtype": "float64", "n": 7, "B": 1024},
        # The headline workload: many states of a 32-link chain.
        {"name": "rnea_chain_f32", "op": "rnea", "dtype": "float32", "n": 32, "B": 65536},
        # A link count that fills no 16-byte chunk and a batch that fills no block.
        {"name": "rnea_odd_f32", "op": "rnea", "dtype": "float32", "n": 29, "B": 49999},
        # Long chains (snake and tendon robots, chains of discretised rods).
        {"name": "rnea_long_f32", "op": "rnea", "dtype": "float32", "n": 100, "B": 65536},
        # The headline workload in FP64.
        {"name": "rnea_chain_f64", "op": "rnea", "dtype": "float64", "n": 32, "B": 65536},
        # One gradient evaluation of a trajectory optimiser: every knot of a batch of plans.
        {"name": "vjp_chain_f32", "op": "vjp", "dtype": "float32", "n": 32, "B": 8192},
        # A training step through inverse dynamics: tau and its backward pass, large batch.
        {"name": "train_chain_f32", "op": "autograd", "dtype": "float32", "n": 32, "B": 262144},
        # Forward dynamics of an arm: one step of a batch of rollouts.
        {"name": "aba_arm_f32", "op": "aba", "dtype": "float32", "n": 7, "B": 1024},
        # Forward dynamics of long chains, the simulation of a large batch.
        {"name": "aba_chain_f32", "op": "aba", "dtype": "float32", "n": 64, "B": 16384},
        # Forward dynamics in FP64, a simulator's usual precision.
        {"name": "aba_chain_f64", "op": "aba", "dtype": "float64", "n": 16, "B": 16384},
        # Mixed requests of many robots of all lengths in one call.
        {"name": "fleet_mixed_f32", "op": "fleet", "dtype": "float32", "requests": 20000,
         "robots": 1000, "n_lo": 6, "n_hi": 100},
    ]


# Per op and type: links, states, and the most joints (n * B) of a drawn case, which keeps it
# cheaper than the largest listed ones.
RANGES = {
    ("rnea", "float32"): ((6, 100), (512, 262144), 6553600),
    ("rnea", "float64"): ((6, 64), (512, 65536), 2097152),
    ("vjp", "float32"): ((6, 64), (1024, 262144), 4194304),
    ("vjp", "float64"): ((6, 32), (1024, 16384), 262144),
    ("autograd", "float32"): ((6, 64), (4096, 262144), 8388608),
    ("aba", "float32"): ((6, 64), (512, 65536), 1048576),
    ("aba", "float64"): ((6, 64), (512, 16384), 262144),
}


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(list(RANGES) + [("fleet", "float32")])
    if kind[0] == "fleet":
        n_hi = rng.randint(20, 100)
        requests = _log_int(rng, 1000, 20000)
        return {"op": "fleet", "dtype": "float32", "requests": requests,
                "robots": max(1, requests // rng.randint(5, 50)), "n_lo": rng.randint(6, 10),
                "n_hi": n_hi}
    (n_lo, n_hi), (b_lo, b_hi), joints = RANGES[kind]
    n = _log_int(rng, n_lo, n_hi)
    return {"op": kind[0], "dtype": kind[1], "n": n,
            "B": _log_int(rng, b_lo, min(b_hi, max(b_lo, joints // n)))}


# ---------------------------------------------------------------------------
# Inputs, from the seed alone
# ---------------------------------------------------------------------------

def _rotations(rng, count):
    q = rng.standard_normal((count, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)],
                    axis=1).reshape(count, 3, 3)


def _links(rng, count):
    """Model arrays of ``count`` links: home transforms, joint twists, inertias."""
    M = np.concatenate([_rotations(rng, count).reshape(count, 9),
                        rng.uniform(0.1, 0.5, size=(count, 3))], axis=1)
    w = rng.standard_normal((count, 3))
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    S = np.concatenate([-np.cross(w, rng.uniform(-0.1, 0.1, size=(count, 3))), w], axis=1)
    m = rng.uniform(0.5, 5.0, size=count)
    c = rng.uniform(-0.1, 0.1, size=(count, 3))
    d = rng.uniform(0.001, 0.05, size=(count, 3)) * m[:, None]
    R = _rotations(rng, count)
    moments = np.stack([d[:, 1] + d[:, 2], d[:, 0] + d[:, 2], d[:, 0] + d[:, 1]], axis=1)
    I = np.einsum("nij,nj,nkj->nik", R, moments, R)
    inertia = np.concatenate([m[:, None], c, I[:, [0, 1, 2], [0, 1, 2]],
                              I[:, [0, 0, 1], [1, 2, 2]]], axis=1)
    return M, S, inertia


class _Chain:
    def __init__(self, M, S, inertia):
        self.M, self.S, self.inertia, self.n = M, S, inertia, M.shape[0]


def _robots(case, seed):
    """The case's chains. Their lengths are the case's, their links the seed's."""
    rng = np.random.default_rng([1609, seed])
    if case["op"] != "fleet":
        return [_Chain(*_links(rng, case["n"]))]
    ns = np.random.default_rng([case["robots"], case["n_hi"]]).integers(
        case["n_lo"], case["n_hi"] + 1, size=case["robots"])
    at = np.concatenate([[0], np.cumsum(ns)])
    M, S, J = _links(rng, int(at[-1]))
    return [_Chain(M[a:b], S[a:b], J[a:b]) for a, b in zip(at[:-1], at[1:])]


def _requests(case):
    """(robot, kind) of each mixed request: the same for every seed, as the plan is kept while
    the states change."""
    rng = np.random.default_rng([7919, case["requests"]])
    robot = rng.integers(0, case["robots"], size=case["requests"])
    kind = np.where(rng.random(case["requests"]) < 0.2, rd.RD_REQ_FD, rd.RD_REQ_ID)
    return robot, kind


def _states(case, seed, shape):
    """q, qd, qdd, tau and w on the GPU, in the case's type."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    dt = TORCH[case["dtype"]]

    def normal(s):
        return torch.randn(shape, generator=g, device="cuda", dtype=dt) * s

    q = (torch.rand(shape, generator=g, device="cuda", dtype=dt) * 2 - 1) * math.pi
    return {"q": q, "qd": normal(1.0), "qdd": normal(2.0), "tau": normal(10.0), "w": normal(1.0)}


def _fleet_inputs(case, seed):
    """Ragged joint data of the requests: the states and the third input (qdd or tau)."""
    chains, (robot, kind) = _robots(case, seed), _requests(case)
    length = np.array([c.n for c in chains])[robot]
    x = _states(case, seed, (int(length.sum()),))
    fd = torch.from_numpy(np.repeat(kind == rd.RD_REQ_FD, length)).to("cuda")
    return chains, robot, kind, length, x["q"], x["qd"], torch.where(fd, x["tau"], x["qdd"])


def prepare(case, seed):
    if case["op"] == "fleet":
        chains, robot, kind, _, q, qd, in2 = _fleet_inputs(case, seed)
        fleet = rd.Fleet(chains)
        plan = rd.Plan(fleet, robot, kind, dtype=case["dtype"])
        return {"op": "fleet", "plan": plan, "fleet": fleet, "q": q, "qd": qd, "in2": in2}
    x = _states(case, seed, (case["B"], case["n"]))
    state = {"op": case["op"], "model": rd.Model(_robots(case, seed)[0]), **x}
    if case["op"] == "autograd":
        for k in ("q", "qd", "qdd"):
            state[k].requires_grad_(True)
    return state


def run(state):
    op = state["op"]
    if op == "fleet":
        return rd.fleet_batch(state["plan"], state["q"], state["qd"], state["in2"])
    model, q, qd = state["model"], state["q"], state["qd"]
    if op == "rnea":
        return rd.rnea(model, q, qd, state["qdd"])
    if op == "vjp":
        return rd.rnea_vjp(model, q, qd, state["qdd"], state["w"])
    if op == "aba":
        return rd.forward_dynamics(model, q, qd, state["tau"])
    tau = rd.rnea_autograd(model, q, qd, state["qdd"])
    grads = torch.autograd.grad(tau, (q, qd, state["qdd"]), state["w"])
    return (tau.detach(), *grads)


def work(case):
    size = 4 if case["dtype"] == "float32" else 8
    if case["op"] == "fleet":
        joints = case["requests"] * (case["n_lo"] + case["n_hi"]) / 2
        # constants of every robot once, then four elements per joint of the requests
        links = case["robots"] * (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": size * (4 * joints + 16 * links),
                "flops": joints * (0.8 * FLOP["rnea"] + 0.2 * FLOP["aba"])}
    joints = case["n"] * case["B"]
    return {"bytes": size * ELEMS[case["op"]] * joints, "flops": FLOP[case["op"]] * joints}


# ---------------------------------------------------------------------------
# The same results in 64 bits: recursive Newton-Euler and the articulated-body algorithm on
# whole batches of 3-vectors and 6x6 matrices, in the chain's own link frames
# ---------------------------------------------------------------------------

def _f64(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.float64)


def _cross(a, b):
    return torch.linalg.cross(*torch.broadcast_tensors(a, b))


def _apply(R, v):
    return (R * v.unsqueeze(-2)).sum(-1)


def _skew(v):
    z = torch.zeros_like(v[..., 0])
    return torch.stack([z, -v[..., 2], v[..., 1], v[..., 2], z, -v[..., 0], -v[..., 1], v[..., 0],
                        z], dim=-1).reshape(v.shape[:-1] + (3, 3))


class _Exact:
    """One link count, a batch of states, constants shared by the batch or one set per state."""

    def __init__(self, M, S, inertia):  # [n, .] or [R, n, .]
        if M.dim() == 2:
            M, S, inertia = M[None], S[None], inertia[None]
        self.n = M.shape[1]
        self.MR, self.Mp = M[..., :9].reshape(M.shape[:2] + (3, 3)), M[..., 9:]
        self.v, self.w = S[..., :3], S[..., 3:]
        self.m, self.c = inertia[..., 0:1], inertia[..., 1:4]
        xx, yy, zz, xy, xz, yz = (inertia[..., k] for k in range(4, 10))
        self.I = torch.stack([xx, xy, xz, xy, yy, yz, xz, yz, zz], -1).reshape(
            M.shape[:2] + (3, 3))

    def pose(self, i, q):
        """Rotation and origin of frame i in frame i-1: M_i exp([S_i] q_i)."""
        W = _skew(self.w[:, i])
        W2 = W @ W
        s, c, q1 = torch.sin(q)[:, None, None], torch.cos(q)[:, None, None], q[:, None, None]
        E = torch.eye(3, dtype=q.dtype, device=q.device)
        R = self.MR[:, i] @ (E + s * W + (1 - c) * W2)
        p = _apply(self.MR[:, i], _apply(q1 * E + (1 - c) * W + (q1 - s) * W2, self.v[:, i]))
        return R, p + self.Mp[:, i]

    def forward(self, q, qd, qdd):
        """Per link: pose, twist and bias wrench (f, n)."""
        B = q.shape[0]
        z = torch.zeros(B, 3, dtype=q.dtype, device=q.device)
        v = w = al = z
        a = z + torch.tensor([0.0, 0.0, 9.81], dtype=q.dtype, device=q.device)
        out = []
        for i in range(self.n):
            R, p = self.pose(i, q[:, i])
            Rt = R.transpose(-1, -2)
            sv, sw = self.v[:, i], self.w[:, i]
            jd, jdd = qd[:, i:i + 1], qdd[:, i:i + 1]
            a, al = _apply(Rt, a + _cross(al, p)), _apply(Rt, al)
            v, w = _apply(Rt, v + _cross(w, p)) + sv * jd, _apply(Rt, w) + sw * jd
            a = a + (_cross(w, sv) + _cross(v, sw)) * jd + sv * jdd
            al = al + _cross(w, sw) * jd + sw * jdd
            m, c, I = self.m[:, i], self.c[:, i], self.I[:, i]
            f = m * (a + _cross(w, v) + _cross(al, c) + _cross(w, _cross(w, c)))
            t = _cross(c, f) + _apply(I, al) + _cross(w, _apply(I, w))
            out.append((R, p, v, w, f, t))
        return out

    def rnea(self, q, qd, qdd):
        links = self.forward(q, qd, qdd)
        f = t = torch.zeros_like(links[0][2])
        tau = [None] * self.n
        for i in reversed(range(self.n)):
            f, t = f + links[i][4], t + links[i][5]
            tau[i] = (self.v[:, i] * f + self.w[:, i] * t).sum(-1)
            R, p = links[i][0], links[i][1]
            f = _apply(R, f)
            t = _apply(R, t) + _cross(p, f)
        return torch.stack(tau, 1)

    def aba(self, q, qd, tau):
        bias = tau - self.rnea(q, qd, torch.zeros_like(q))
        B, dt, dev = q.shape[0], q.dtype, q.device
        X, U, D, u = [None] * self.n, [None] * self.n, [None] * self.n, [None] * self.n
        IA, pA = None, None
        for i in reversed(range(self.n)):
            R, p = self.pose(i, q[:, i])
            Rt = R.transpose(-1, -2)
            X[i] = torch.zeros(B, 6, 6, dtype=dt, device=dev)  # twists of i-1 into frame i
            X[i][:, :3, :3] = Rt
            X[i][:, 3:, 3:] = Rt
            X[i][:, :3, 3:] = -Rt @ _skew(p)
            m, C = self.m[:, i], _skew(self.c[:, i])
            J = torch.zeros(C.shape[0], 6, 6, dtype=dt, device=dev)
            J[:, :3, :3] = m[..., None] * torch.eye(3, dtype=dt, device=dev)
            J[:, :3, 3:] = -m[..., None] * C
            J[:, 3:, :3] = m[..., None] * C
            J[:, 3:, 3:] = self.I[:, i] - m[..., None] * (C @ C)
            IA = J.expand(B, 6, 6) if IA is None else J + IA
            S = torch.cat([self.v[:, i], self.w[:, i]], -1)
            U[i] = _apply(IA, S)
            d = (S * U[i]).sum(-1)
            D[i] = torch.where(d == 0, torch.ones_like(d), d)  # a padding link
            u[i] = bias[:, i] - (0 if pA is None else (S * pA).sum(-1))
            low = IA - U[i][:, :, None] * U[i][:, None, :] / D[i][:, None, None]
            Xt = X[i].transpose(-1, -2)
            pA = _apply(Xt, U[i] * (u[i] / D[i])[:, None] + (0 if pA is None else pA))
            IA = Xt @ low @ X[i]
        a = torch.zeros(B, 6, dtype=dt, device=dev)
        qdd = []
        for i in range(self.n):
            a = _apply(X[i], a)
            qdd.append((u[i] - (U[i] * a).sum(-1)) / D[i])
            a = a + torch.cat([self.v[:, i], self.w[:, i]], -1) * qdd[i][:, None]
        return torch.stack(qdd, 1)


def _exact_fleet(case, seed):
    chains, robot, kind, length, q, qd, in2 = _fleet_inputs(case, seed)
    # every chain padded at its tip to the longest with massless links that do not move
    n = max(c.n for c in chains)
    eye = np.eye(3).reshape(9)
    M, S, J = np.zeros((len(chains), n, 12)), np.zeros((len(chains), n, 6)), np.zeros(
        (len(chains), n, 10))
    M[:, :, :9] = eye
    for k, c in enumerate(chains):
        M[k, :c.n], S[k, :c.n], J[k, :c.n] = c.M, c.S, c.inertia
    M, S, J = _f64(M), _f64(S), _f64(J)
    start = np.concatenate([[0], np.cumsum(length)[:-1]])
    col = torch.arange(n, device="cuda")
    out = torch.zeros(int(length.sum()), dtype=torch.float64, device="cuda")
    for k in (rd.RD_REQ_ID, rd.RD_REQ_FD):
        for rows in np.array_split(np.flatnonzero(kind == k), 8):
            if not len(rows):
                continue
            at = torch.from_numpy(start[rows]).to("cuda")[:, None] + col
            real = col < torch.from_numpy(length[rows]).to("cuda")[:, None]
            at = torch.where(real, at, 0)
            x = [torch.where(real, v.double()[at], 0.0) for v in (q, qd, in2)]
            rb = torch.from_numpy(robot[rows]).to("cuda")
            e = _Exact(M[rb], S[rb], J[rb])
            y = e.rnea(*x) if k == rd.RD_REQ_ID else e.aba(*x)
            out[at[real]] = y[real]
    return out


def exact(case, seed):
    if case["op"] == "fleet":
        return _exact_fleet(case, seed)
    chain, x = _robots(case, seed)[0], _states(case, seed, (case["B"], case["n"]))
    x = {k: v.double() for k, v in x.items()}
    e = _Exact(_f64(chain.M), _f64(chain.S), _f64(chain.inertia))
    parts = []
    for lo in range(0, case["B"], 32768):
        p = {k: v[lo:lo + 32768] for k, v in x.items()}
        if case["op"] == "rnea":
            parts.append((e.rnea(p["q"], p["qd"], p["qdd"]),))
        elif case["op"] == "aba":
            parts.append((e.aba(p["q"], p["qd"], p["tau"]),))
        else:
            args = [p[k].requires_grad_(True) for k in ("q", "qd", "qdd")]
            tau = e.rnea(*args)
            g = torch.autograd.grad(tau, args, p["w"])
            parts.append(g if case["op"] == "vjp" else (tau.detach(), *g))
    whole = tuple(torch.cat(c) for c in zip(*parts))
    return whole[0] if case["op"] in ("rnea", "aba") else whole
