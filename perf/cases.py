"""Performance cases: what a user of the solver, of its batched form and of the learned closure has it do.

Every case goes through the public Python entry points (`Solver`, `Batch`, `Closure` and the `ql_*` calls on caller
buffers).  The sizes are those of the repository's own workloads: the Sod tube of the benchmark and its launch-size
sweep, the paper's timed shock tubes (chi_RET-FM; Q = 200 on the generic path), the standing shock, the uneven
batch, the closure's training shape, and domains of no round size in between.
"""
import math

import numpy as np
import torch

from paper_2211_16933_gb300 import qlbm as q

DEV = "cuda" if torch.cuda.is_available() else "cpu"
TABLE_EL, TABLE_L, TABLE_DT = 0.4825, 80.0, 1e-3  # the paper's timed tubes: denseness of the left state, length, dt
NET_IN, NET_OUT, NET_LAYERS, NET_WIDTH = 7, 5, 5, 64
COARSE = 64  # coarse cells per instance of the batch cases; every domain is a multiple of it


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the benchmark's Sod tube: the largest domain, a plain FP32 run of a few steps
        dict(name="tube_fp32_4m", kind="solver", problem="tube", prec="fp32", Q=32, nx=1 << 22, chi="set", steps=4),
        # the same tube where a stage is about one wave of tiles (one launch covers the whole call)
        dict(name="tube_fp32_131k", kind="solver", problem="tube", prec="fp32", Q=32, nx=131072, chi="set", steps=20),
        # a few thousand cells: fewer tiles than the GPU has SMs
        dict(name="tube_fp32_8k", kind="solver", problem="tube", prec="fp32", Q=32, nx=8192, chi="set", steps=20),
        # the paper's smallest velocity set in FP32: latency and launches
        dict(name="table_fp32_1600", kind="solver", problem="table", prec="fp32", Q=8, nx=1600, chi="ret", steps=20),
        # the paper's sigma = 0.1 tube in its own precision, chi_RET-FM
        dict(name="table_fp64_640", kind="solver", problem="table", prec="fp64", Q=20, nx=640, chi="ret", steps=20),
        # the standing Mach 1.4 shock, run for hundreds of thousands of FP64 steps
        dict(name="shock_fp64_4096", kind="solver", problem="shock", prec="fp64", Q=32, nx=4096, chi="set", steps=10),
        # the Sod tube in FP64 on a domain that fills the GPU
        dict(name="tube_fp64_262k", kind="solver", problem="tube", prec="fp64", Q=32, nx=262144, chi="set", steps=1),
        # the paper's near-ballistic tube (generic path, any even Q)
        dict(name="table_fp64_q200", kind="solver", problem="table", prec="fp64", Q=200, nx=160, chi="ret", steps=5),
        # from host fields on, with the conservation totals read after each step (in the solver's precision: FP32
        # sums differ in their last bits); odd size, periodic, constant Prandtl number
        dict(name="wave_fp32_fields", kind="fields", problem="wave", prec="fp32", Q=24, nx=1000003, chi="set", steps=3),
        # data generation: many uneven instances advanced together, then their block-averaged fields
        dict(name="batch_fp32_256", kind="batch", prec="fp32", n=256, nmax=128, steps=2),
        # closure training: mini-batches gathered on the device, Adam; losses and updated weights
        dict(name="net_train_256", kind="train", B=256, X=512, n=1024, steps=8),
        # closure inference on one mini-batch
        dict(name="net_forward_256", kind="forward", B=256, X=512),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_problem(rng, Q):
    return rng.choice(["tube", "wave", "shock"] if Q >= 16 else ["tube", "wave"])  # 8 velocities are too few for a shock


def draw(rng):
    kind = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp64", "large_q", "fields", "batch", "train", "forward"])
    if kind == "fp32":
        Q, nx = rng.choice([8, 16, 20, 24, 32, 40]), _log_uniform(rng, 300, 3_000_000)
        steps = max(1, min(rng.randint(1, 24), int(4e8 / (Q * nx))))
        return dict(kind="solver", problem=_draw_problem(rng, Q), prec="fp32", Q=Q, nx=nx,
                    chi="set" if rng.random() < 0.75 or nx > 400_000 else "ret", steps=steps)
    if kind == "fp64":
        Q, nx = rng.choice([8, 16, 20, 24, 32, 40]), _log_uniform(rng, 150, 250_000)
        steps = max(1, min(rng.randint(1, 20), int(8e6 / (Q * nx))))
        return dict(kind="solver", problem=_draw_problem(rng, Q), prec="fp64", Q=Q, nx=nx,
                    chi=rng.choice(["set", "ret"]) if nx < 20_000 else "set", steps=steps)
    if kind == "large_q":
        return dict(kind="solver", problem="table", prec="fp64", Q=2 * rng.randint(22, 100), nx=rng.randint(100, 800),
                    chi=rng.choice(["set", "ret"]), steps=rng.randint(1, 5))
    if kind == "fields":
        return dict(kind="fields", problem="wave", prec=rng.choice(["fp32", "fp32", "fp64"]),
                    Q=rng.choice([8, 16, 24, 32]), nx=_log_uniform(rng, 1000, 100_000) | 1, chi="set",
                    steps=rng.randint(1, 3))
    if kind == "batch":
        return dict(kind="batch", prec="fp32", n=rng.randint(16, 200), nmax=rng.randint(16, 128), steps=rng.randint(1, 4))
    if kind == "train":
        return dict(kind="train", B=rng.randint(16, 256), X=rng.choice([128, 500, 512]), n=rng.randint(600, 1000),
                    steps=rng.randint(1, 4))
    return dict(kind="forward", B=rng.randint(1, 256), X=rng.choice([64, 300, 512]))


# ---------------------------------------------------------------- physical inputs (host, FP64)
def _nodes(Q):
    """Gauss-Hermite nodes and weights for exp(-p^2/2)/sqrt(2 pi) (eigenvalues of the Jacobi matrix, then Newton)."""
    p = np.linalg.eigvalsh(np.diag(np.sqrt(np.arange(1.0, Q)), 1) + np.diag(np.sqrt(np.arange(1.0, Q)), -1))
    for _ in range(3):
        h = _hermite(p, Q + 1)
        p = p - h[Q] / (math.sqrt(Q) * h[Q - 1])
    p = 0.5 * (p - p[::-1])
    return p, 1.0 / np.sum(_hermite(p, Q) ** 2, axis=0)


def _hermite(p, n):
    """He_l(p) / sqrt(l!) for l = 0 .. n - 1."""
    h = np.zeros((n, len(p)))
    h[0], h[1] = 1.0, p
    for m in range(1, n - 1):
        h[m + 1] = (p * h[m] - math.sqrt(m) * h[m - 1]) / math.sqrt(m + 1)
    return h


def _chi(eta):
    return 0.5 * (2.0 - eta) / (1.0 - eta) ** 3


def _eta0(El):
    lo, hi = 0.0, 0.49
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 6.0 * math.sqrt(2.0) * mid * _chi(mid) < El else (lo, mid)
    return 0.5 * (lo + hi)


def _z(eta):
    return 1.0 + 4.0 * eta * _chi(eta)


def _downstream(eta0, T1, mach):
    """Upstream speed and (rho, u, T) behind a standing shock of the dense gas, upstream density 1."""
    d = 1e-6
    zp = (_z(eta0 + d) - _z(eta0 - d)) / (2 * d)
    u1 = mach * math.sqrt(T1 * (_z(eta0) + eta0 * zp) + 2.0 / 3.0 * T1 * _z(eta0) ** 2)
    P1 = T1 * _z(eta0)

    def state(r):
        u2 = u1 / r
        P2 = P1 + u1 * (u1 - u2)
        T2 = P2 / (r * _z(eta0 * r))
        return (1.5 * T1 + 0.5 * u1 * u1 + P1) - (1.5 * T2 + 0.5 * u2 * u2 + P2 / r), u2, T2

    lo, hi = 1.0 + 1e-6, min(4.0, 0.49 / eta0)
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if (state(mid)[0] < 0) == (state(1.0 + 1e-6)[0] < 0) else (lo, mid)
    _, u2, T2 = state(lo)
    return u1, lo, u2, T2


def _disturbance(rng, nx, amp):
    """A smooth disturbance of a few modes, zero at both ends."""
    x = (np.arange(nx) + 0.5) / nx
    return sum(amp / m * rng.uniform(-1, 1) * np.sin(math.pi * m * x) for m in range(1, 4))


def _wave(rng, nx, amp):
    x = (np.arange(nx) + 0.5) / nx
    return sum(amp / m * rng.uniform(-1, 1) * np.cos(2 * math.pi * m * x + rng.uniform(0, 2 * math.pi))
               for m in range(1, 4))


def _problem(problem, Q, nx, chi, seed):
    """One domain: its parameters, initial (rho, u, T) and the ghost states."""
    rng = np.random.default_rng(seed)
    P = dict(Q=Q, nx=nx, length=1.0, El=0.1, kn=0.05, periodic=False, pr_dense=True, ret=chi == "ret", ghost=None)
    pmax = float(_nodes(Q)[0][-1])
    if problem == "wave":
        # smooth periodic fields around (1, 0, 1)
        P.update(kn=0.1, periodic=True, pr_dense=False)
        f = [1.0 + _wave(rng, nx, 0.05), _wave(rng, nx, 0.1), 1.0 + _wave(rng, nx, 0.05)]
    elif problem == "shock":
        # a tanh profile between the two states of a standing shock
        P.update(length=128.0, kn=1.0 / 128.0, El=float(rng.uniform(0.05, 0.2)))
        T1 = 0.45 if Q < 24 else 0.7
        u1, r2, u2, T2 = _downstream(_eta0(P["El"]), T1, float(rng.uniform(1.3, 1.5)))
        s = 0.5 * (1.0 + np.tanh(((np.arange(nx) + 0.5) / nx - 0.5) * 128.0 / 4.0))
        f = [1.0 + (r2 - 1.0) * s, u1 + (u2 - u1) * s, T1 + (T2 - T1) * s]
        P["ghost"] = np.array([[1.0, u1, T1]] * 3 + [[r2, u2, T2]] * 3)
    else:
        # a Sod tube (densities 1 and 1/8, gas at rest), each half with a smooth disturbance on it
        left = np.arange(nx) < nx // 2
        f = [np.where(left, 1.0, 0.125) * (1.0 + _disturbance(rng, nx, 0.02)), _disturbance(rng, nx, 0.02),
             1.0 + _disturbance(rng, nx, 0.02)]
        P["ghost"] = np.array([[1.0, 0.0, 1.0]] * 3 + [[0.125, 0.0, 1.0]] * 3)
        if problem == "table":
            # the mean free path of each velocity set's row of the paper's table: sigma over E_l
            sigma = {8: 0.01, 20: 0.1}.get(Q, 1.0 if Q > 40 else 0.05)
            P.update(length=TABLE_L, El=TABLE_EL, kn=sigma / (TABLE_EL * TABLE_L))
    P["dt"] = TABLE_DT if problem == "table" else 0.4 * P["length"] / nx / pmax
    if P["ret"] and P["El"] * P["kn"] * nx > 250:  # the ball of chi_RET-FM reaches at most 256 cells
        P["kn"] = 250 / (P["El"] * nx)
    P["fields"] = f
    return P


def _batch_problems(case, seed):
    """Half sound waves, half standing shocks, of uneven sizes and velocity sets."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["n"]):
        nx = COARSE * int(rng.integers(4, case["nmax"] + 1))
        Q = int(rng.choice([16, 24, 32]))
        out.append(_problem("shock" if i % 2 else "wave", Q, nx, "set", int(rng.integers(1 << 30))))
    return out


def _net_inputs(case, seed, n):
    rng = np.random.default_rng(seed)
    X = case["X"]
    x = np.empty((n, X, NET_IN), dtype=np.float32)
    t = np.arange(X) / X
    for c in range(NET_IN):
        a = rng.standard_normal((n, 3, 1)) * np.array([1.0, 0.5, 0.3])[None, :, None]
        ph = rng.uniform(0, 2 * np.pi, (n, 3, 1))
        x[:, :, c] = (a * np.sin(2 * np.pi * (np.arange(3) + 1)[None, :, None] * t + ph)).sum(1)
    y = np.empty((n, X, NET_OUT), dtype=np.float32)
    for c in range(NET_OUT):
        y[:, :, c] = np.tanh(x[:, :, c] * x[:, :, (c + 1) % NET_IN]) * 0.5
    per = (np.arange(n) % 2).astype(np.int32)
    return x, y, per, rng.permutation(n)


def _net_params(seed):
    """He-uniform weights W[cout][5][cin] and small biases per layer, channels padded to 16 with zeros."""
    rng = np.random.default_rng(seed + 7)
    out = []
    for m in range(NET_LAYERS):
        ci = NET_IN if m == 0 else NET_WIDTH
        co = NET_OUT if m == NET_LAYERS - 1 else NET_WIDTH
        W = np.zeros((16 if m == NET_LAYERS - 1 else co, 5, 16 if m == 0 else ci))
        a = math.sqrt(6.0 / (5 * ci))
        W[:co, :, :ci] = rng.uniform(-a, a, (co, 5, ci))
        b = np.zeros(W.shape[0])
        b[:co] = rng.uniform(-0.1, 0.1, co)
        out += [W.ravel(), b]
    return np.concatenate(out).astype(np.float32)


# ---------------------------------------------------------------- prepare and run
class _View:
    """The device state of a solver as an array, [Q][nx] pairs in place (the solver is kept alive with it)."""

    def __init__(self, solver, ptr, stride):
        self.solver = solver
        b = 4 if solver.precision == q.QL_FP32 else 8
        self.__cuda_array_interface__ = dict(shape=(solver.Q, solver.nx, 2), typestr="<f%d" % b, data=(ptr, False),
                                             strides=(2 * b * stride, 2 * b, b), version=2)


def _psi(s):
    ptr, stride = q.ql_state_device(s.ctx)
    return torch.as_tensor(_View(s, ptr, stride), device=DEV)


def _solver(P, prec):
    return q.Solver(P["Q"], P["nx"], P["length"], P["dt"], P["El"], P["kn"],
                    bc=q.QL_BC_PERIODIC if P["periodic"] else q.QL_BC_FIXED, init_kind=q.QL_INIT_FIELDS,
                    rho=P["fields"][0], u=P["fields"][1], T=P["fields"][2], ghost=P["ghost"],
                    precision=q.QL_FP32 if prec == "fp32" else q.QL_FP64,
                    pr_mode=q.QL_PR_DENSE if P["pr_dense"] else q.QL_PR_CONST,
                    chi_mode=q.QL_CHI_RET_FM if P["ret"] else q.QL_CHI_SET)


def _pinned(a):
    t = torch.empty(a.shape, dtype=torch.float64, pin_memory=True)
    t.numpy()[...] = a
    return t.numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solver", "fields"):
        P = _problem(case["problem"], case["Q"], case["nx"], case["chi"], seed)
        st = dict(kind=kind, steps=case["steps"], solver=_solver(P, case["prec"]))
        if kind == "fields":
            st["fields"] = [_pinned(a) for a in P["fields"]]
        return st
    if kind == "batch":
        keep, insts = [], []
        for P in _batch_problems(case, seed):
            insts.append(q.make_instance(
                P["Q"], P["nx"], P["length"], P["dt"], P["El"], P["kn"],
                bc=q.QL_BC_PERIODIC if P["periodic"] else q.QL_BC_FIXED, init_kind=q.QL_INIT_FIELDS,
                rho=P["fields"][0], u=P["fields"][1], T=P["fields"][2], ghost=P["ghost"],
                pr_mode=q.QL_PR_DENSE if P["pr_dense"] else q.QL_PR_CONST, keep=keep))
        b = q.Batch(insts, precision=q.QL_FP32 if case["prec"] == "fp32" else q.QL_FP64)
        out = torch.empty(case["n"], 5, COARSE, dtype=torch.float64, device=DEV)
        return dict(kind=kind, steps=case["steps"], batch=b, out=out)
    n = case["n"] if kind == "train" else case["B"]
    x, y, per, perm = _net_inputs(case, seed, n)
    net = q.Closure(NET_IN, NET_OUT, case["X"], case["B"], seed=seed)
    net.set_params(_net_params(seed))
    st = dict(kind=kind, net=net, x=torch.from_numpy(x).to(DEV), per=torch.from_numpy(per).to(DEV))
    if kind == "train":
        st["y"] = torch.from_numpy(y).to(DEV)
        st["perm"] = torch.from_numpy(np.resize(perm, case["steps"] * case["B"]).astype(np.int32)).to(DEV)
        st["lr"] = np.full(case["steps"], 1e-3, dtype=np.float32)
        st["losses"] = torch.empty(case["steps"], dtype=torch.float32, device=DEV)
    else:
        st["pred"] = torch.empty(case["B"], case["X"], NET_OUT, dtype=torch.float32, device=DEV)
    return st


def run(state):
    kind = state["kind"]
    if kind == "solver":
        s = state["solver"]
        s.step(state["steps"])
        return _psi(s)
    if kind == "fields":
        s = state["solver"]
        q.ql_load_fields(s.ctx, *state["fields"])
        totals = np.zeros((state["steps"], 3), dtype=np.float32 if s.precision == q.QL_FP32 else np.float64)
        for j in range(state["steps"]):
            s.step(1)
            totals[j] = s.totals()
        return dict(totals=totals, psi=_psi(s))
    if kind == "batch":
        b, out = state["batch"], state["out"]
        b._stream.wait_stream(torch.cuda.current_stream())
        b.run(state["steps"])
        b.fields(COARSE, out)
        torch.cuda.current_stream().wait_stream(b._stream)
        return out.float()  # as training data are kept
    net = state["net"]
    if kind == "train":
        net.train_steps(state["x"], state["y"], state["per"], state["perm"], state["lr"], state["losses"])
        return dict(losses=state["losses"], params=net.get_params())
    net.forward(state["x"], state["per"], state["pred"])
    return state["pred"]


# ---------------------------------------------------------------- work
def _updates(case):
    if case["kind"] == "batch":
        # the expected sum over the instances (their sizes depend on the seed): 24 velocities, mean size
        return case["n"] * 24 * COARSE * 0.5 * (4 + case["nmax"]) * case["steps"]
    return case["nx"] * case["Q"] * case["steps"]


def work(case):
    """A Runge-Kutta step reads and writes 16 words per (cell, velocity) when each stage is one pass over the state
    (stage 1: a pair in, a pair out; stages 2 and 3: two pairs in, one out); flops per stage: a WENO-5 face value of
    two components, the Q-term equilibrium sum shared by +p and -p, moments, targets and the update."""
    kind = case["kind"]
    if kind in ("solver", "fields", "batch"):
        Q = case.get("Q", 24)
        word = 4 if case["prec"] == "fp32" else 8
        n = _updates(case)
        w = dict(bytes=16.0 * word * n, flops=3.0 * n * (110 + Q + 30))
        if kind == "fields":  # fields in, the first state out, totals after each step (a pass over the state)
            w["bytes"] += 3 * 8.0 * case["nx"] + 2.0 * word * case["nx"] * Q * (case["steps"] + 1)
        if kind == "batch":
            w["bytes"] += 2.0 * word * n / case["steps"]
        return w
    macs = 5 * (NET_IN * 64 + 3 * 64 * 64 + 64 * NET_OUT)
    pos = float(case["B"] * case["X"])
    if kind == "train":
        # forward, input gradient (not of the first layer) and weight gradient; activations written and read
        return dict(bytes=case["steps"] * pos * (4 * NET_IN + 4 * NET_OUT + 4 * 64 * 2 * 3),
                    flops=case["steps"] * pos * 2.0 * (3 * macs - 5 * NET_IN * 64))
    return dict(bytes=pos * 4 * (NET_IN + NET_OUT), flops=pos * 2.0 * macs)


# ---------------------------------------------------------------- the same in 64 bits, plain torch
def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


class _Ref:
    """The finite-difference lattice Boltzmann scheme of the paper on one domain, in FP64."""

    def __init__(self, P):
        self.P, self.nx = P, P["nx"]
        p, w = _nodes(P["Q"])
        self.p, self.G = _t(p), _t(w[:, None] * _hermite(p, P["Q"]).T)
        self.dx, self.dt = P["length"] / P["nx"], P["dt"]
        self.eta0 = _eta0(P["El"])
        self.tau0 = 5.0 * math.sqrt(2.0 * math.pi) / 16.0 * P["kn"] * P["length"] * _chi(self.eta0)
        if not P["periodic"]:
            g = _t(P["ghost"]).T
            self.ghost = self.equilibrium(g[0], g[1], g[2])
        if P["ret"]:
            sigma = P["El"] * P["kn"] * P["length"]
            W = 0
            while (W + 0.5) * self.dx < sigma:
                W += 1

            def below(x):
                h = np.clip(sigma + x, 0.0, 2.0 * sigma)
                return h * h * (3.0 * sigma - h) / (4.0 * sigma ** 3)

            d = np.arange(-W, W + 1)
            self.W, self.K = W, below((d + 0.5) * self.dx) - below((d - 0.5) * self.dx)
        self.psi = self.equilibrium(*[_t(a) for a in P["fields"]])

    def g(self, u, T):
        Q = self.P["Q"]
        c = torch.empty(Q, u.numel(), dtype=torch.float64, device=u.device)
        c[0], c[1] = 1.0, u
        for m in range(2, Q):
            c[m] = u * c[m - 1] / math.sqrt(m) + math.sqrt((m - 1) / m) * (T - 1.0) * c[m - 2]
        return self.G @ c

    def equilibrium(self, rho, u, T):
        g = self.g(u, T) * rho
        return torch.stack([g, 2.0 * T * g], dim=2)

    def pad(self, psi):
        if self.P["periodic"]:
            return torch.cat([psi[:, -3:], psi, psi[:, :3]], dim=1)
        return torch.cat([self.ghost[:, :3], psi, self.ghost[:, 3:]], dim=1)

    def moments(self, a):
        phi, th, p = a[:, :, 0], a[:, :, 1], self.p
        S0, S1, S2, S3 = phi.sum(0), p @ phi, (p * p) @ phi, (p * p * p) @ phi
        R0, R1 = th.sum(0), p @ th
        u = S1 / S0
        c2 = S2 - u * S1
        T = (c2 + R0) / (3.0 * S0)
        qx = 0.5 * (S3 - 3 * u * S2 + 2 * u * u * S1 + R1 - u * R0)
        return S0, u, T, qx, c2, (S0, S1, S2 + R0)

    def grad(self, v):
        n = self.nx
        return ((v[6:] - v[:n]) / 60.0 - 0.15 * (v[5:5 + n] - v[1:1 + n]) + 0.75 * (v[4:4 + n] - v[2:2 + n])) / self.dx

    def face(self, f):
        a, b, b2, c = f[0] - f[1], f[2] - f[1], f[3] - f[2], f[4] - f[3]
        s = [a * (a + 2.75 * b) + 2.5 * b * b, b * (b - 1.25 * b2) + b2 * b2, c * (c - 2.75 * b2) + 2.5 * b2 * b2]
        m = torch.maximum(torch.maximum(s[0], s[1]), s[2])
        m = torch.where(m > 0, m, torch.ones_like(m))
        s = [(x / m) ** 2 for x in s]
        w = [s[1] * s[2], 6.0 * s[0] * s[2], 3.0 * s[0] * s[1]]
        num = w[0] * (a / 3.0 + b * (5.0 / 6.0)) + w[1] * (b / 6.0 + b2 / 3.0) + w[2] * (b2 * (2.0 / 3.0) - c / 6.0)
        return f[2] + num / torch.clamp(w[0] + w[1] + w[2], min=1e-300)

    def rhs(self, psi):
        P, n = self.P, self.nx
        a = self.pad(psi)
        rho, u, T, qx, _, _ = self.moments(a)
        inner = slice(3, 3 + n)
        dlnn, du, dlnT = self.grad(torch.log(rho)), self.grad(u), self.grad(torch.log(T))
        if P["ret"]:
            W, r = self.W, rho[inner]
            if P["periodic"]:
                at = torch.arange(-3 - W, n + 3 + W, device=r.device) % n
                ext = r[at]
            else:
                ext = torch.cat([rho[:1].expand(W), rho, rho[-1:].expand(W)])
            nbar = sum(float(self.K[d]) * ext[d:d + n + 6] for d in range(2 * W + 1))
            chi_all = _chi(self.eta0 * nbar)
            chi, dlnchi = chi_all[inner], self.grad(torch.log(chi_all))
        rho, u, T, qx = rho[inner], u[inner], T[inner], qx[inner]
        eta = self.eta0 * rho
        if not P["ret"]:
            chi, dlnchi = _chi(eta), eta * (3.0 / (1.0 - eta) - 1.0 / (2.0 - eta)) * dlnn
        Y = 4.0 * eta * chi
        muf = 1.0 + 0.8 * Y + 0.16 * (1.0 + 12.0 / math.pi) * Y * Y
        itau = rho * chi * torch.sqrt(T) / (self.tau0 * muf)
        laf = 1.0 + 1.2 * Y + 0.36 * (1.0 + 32.0 / (9.0 * math.pi)) * Y * Y
        Pr = 2.0 / 3.0 * muf / laf if P["pr_dense"] else torch.full_like(Y, 2.0 / 3.0)
        A = (1.0 - Pr) * qx / (5.0 * rho * T * T)
        Gx = dlnchi + 2.0 * dlnn
        ng = self.g(u, T) * rho
        L = torch.empty_like(psi)
        rows = max(1, int(1 << 23) // n)
        for k0 in range(0, P["Q"], rows):
            k = slice(k0, min(P["Q"], k0 + rows))
            p = self.p[k, None]
            xi = p - u
            x2 = xi * xi / T
            tp = itau * (1.0 + A * xi * (x2 - 3.0)) - Y * (xi * Gx + 0.6 * (x2 - 1.0) * du + 0.3 * xi * (x2 + 1.0 / 3.0) * dlnT)
            tt = itau * (1.0 + A * xi * (x2 - 1.0)) - Y * (xi * Gx + 0.6 * (x2 - 1.0 / 3.0) * du
                                                           + 0.3 * xi * (x2 + 7.0 / 3.0) * dlnT)
            target = torch.stack([ng[k] * tp, 2.0 * T * ng[k] * tt], dim=2)
            h = torch.empty(p.shape[0], n + 1, 2, dtype=torch.float64, device=psi.device)
            for up in (True, False):
                r = torch.nonzero((self.p[k] > 0) == up).flatten()
                if r.numel():
                    b = a[k][r]
                    h[r] = self.face([b[:, m:m + n + 1] for m in (range(5) if up else range(5, 0, -1))])
            L[k] = target - psi[k] * itau[None, :, None] - (p / self.dx)[:, :, None] * (h[:, 1:] - h[:, :-1])
        return L

    def step(self):
        a = self.psi
        b = a + self.dt * self.rhs(a)
        b = 0.75 * a + 0.25 * (b + self.dt * self.rhs(b))
        self.psi = a / 3.0 + 2.0 / 3.0 * (b + self.dt * self.rhs(b))


def _net64(params, x, per):
    """The network of `params` (FP64, flat) on x [B][X][NET_IN]; layers of 5 taps, ReLU between them."""
    a, off = x.permute(0, 2, 1), 0
    for m in range(NET_LAYERS):
        ci, co = (16 if m == 0 else 64), (16 if m == NET_LAYERS - 1 else 64)
        W = params[off:off + co * 5 * ci].view(co, 5, ci).permute(0, 2, 1)
        b = params[off + co * 5 * ci:off + co * 5 * ci + co]
        off += co * 5 * ci + co
        if m == 0:
            W = W[:, :NET_IN]
        wrap = torch.cat([a[:, :, -2:], a, a[:, :, :2]], dim=2)
        ends = torch.cat([a[:, :, :1], a[:, :, :1], a, a[:, :, -1:], a[:, :, -1:]], dim=2)
        w = torch.where((per != 0)[:, None, None], wrap, ends)
        X = a.shape[2]
        z = b[None, :, None] + sum(torch.matmul(W[:, :, j], w[:, :, j:j + X]) for j in range(5))
        a = torch.relu(z) if m < NET_LAYERS - 1 else z
    return a[:, :NET_OUT].permute(0, 2, 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solver":
        r = _Ref(_problem(case["problem"], case["Q"], case["nx"], case["chi"], seed))
        for _ in range(case["steps"]):
            r.step()
        return r.psi
    if kind == "fields":
        r = _Ref(_problem(case["problem"], case["Q"], case["nx"], case["chi"], seed))
        totals = np.zeros((case["steps"], 3))
        for j in range(case["steps"]):
            r.step()
            S = r.moments(r.psi)[5]
            totals[j] = [float(S[0].sum()) * r.dx, float(S[1].sum()) * r.dx, 0.5 * float(S[2].sum()) * r.dx]
        return dict(totals=totals, psi=r.psi)
    if kind == "batch":
        out = torch.empty(case["n"], 5, COARSE, dtype=torch.float64, device=DEV)
        for i, P in enumerate(_batch_problems(case, seed)):
            r = _Ref(P)
            for _ in range(case["steps"]):
                r.step()
            rho, u, T, qx, pxx, _ = r.moments(r.psi)
            for f, v in enumerate((rho, u, T, qx, pxx)):
                out[i, f] = v.view(COARSE, -1).mean(1)
        return out
    n = case["n"] if kind == "train" else case["B"]
    x, y, per, perm = _net_inputs(case, seed, n)
    x, y, per = _t(x), _t(y), torch.from_numpy(per).to(DEV)
    w = _t(_net_params(seed))
    if kind == "forward":
        with torch.no_grad():
            return _net64(w, x, per)
    w.requires_grad_(True)
    m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []
    at = np.resize(perm, case["steps"] * case["B"]).reshape(case["steps"], case["B"])
    for s in range(case["steps"]):
        i = torch.from_numpy(at[s]).to(DEV)
        loss = ((_net64(w, x[i], per[i]) - y[i]) ** 2).mean()
        (g,) = torch.autograd.grad(loss, w)
        losses.append(loss.detach())
        with torch.no_grad():
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            w -= 1e-3 * (m / (1 - 0.9 ** (s + 1))) / (torch.sqrt(v / (1 - 0.999 ** (s + 1))) + 1e-8)
    return dict(losses=torch.stack(losses), params=w.detach())
