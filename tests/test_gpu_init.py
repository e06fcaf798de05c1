"""Initial FP32 states (double-FP32 sums) against the FP64 sums of the same fields, over the range the double-FP32
form takes and on fields outside it (which take the FP64 sums), for every compiled velocity set.

A value is n g = n (e + o) with e and o sums of Q / 2 terms held to about 2^-46 of their largest term; rounding to FP32
adds 2^-24 of the value.  The bound below allows 2^-44 of the sum of the terms' magnitudes, and one and a half FP32
roundings (the FP32 theta multiplies a value that is itself held to 2^-46)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _terms(q, Q, u, T):
    """Sum over l of |G[k][l] c_l| per (velocity, cell), FP64."""
    p, w = (np.asarray(a) for a in q.ql_velocity_set(Q))
    h, c = np.zeros((Q, Q)), np.zeros((Q, len(u)))
    h[:, 0], h[:, 1], c[0], c[1] = 1.0, p, 1.0, u
    for l in range(2, Q):
        h[:, l] = (p * h[:, l - 1] - np.sqrt(l - 1) * h[:, l - 2]) / np.sqrt(l)
        c[l] = u * c[l - 1] / np.sqrt(l) + np.sqrt((l - 1) / l) * (T - 1) * c[l - 2]
    return np.abs(w[:, None] * h) @ np.abs(c)


@pytest.mark.parametrize("Q", [8, 16, 20, 24, 32, 40])
@pytest.mark.parametrize("kind", ["rest", "ordinary", "tiny", "edge", "outside"])
def test_fp32_state_is_the_rounded_fp64_state(gpu, Q, kind):
    q, nx = gpu, 301
    rng = np.random.default_rng(Q)
    rho, u, T = rng.uniform(0.1, 2.0, nx), rng.uniform(-1.0, 1.0, nx), rng.uniform(0.4, 1.7, nx)
    if kind == "rest":
        u[:], T[:] = 0.0, 1.0
    elif kind == "tiny":
        rho, u, T = rho * 1e-12, u * 10.0 ** rng.uniform(-40, -3, nx), 1.0 + u * 10.0 ** rng.uniform(-16, -3, nx)
    elif kind == "edge":  # the last arguments of the double-FP32 form, and the first beyond it
        u, T = np.where(rng.random(nx) < 0.5, 1.99, -2.01), rng.uniform(0.05, 3.0, nx)
    elif kind == "outside":  # |u| >= 8 in every other cell
        u[::2] = 8.5
    if Q == 40 and kind == "outside":
        u[::2] = 8.01
    args = (Q, nx, 1.0, 1e-5, 0.1, 0.05)
    kw = dict(bc=q.QL_BC_PERIODIC, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T)
    a, b = q.Solver(*args, precision=q.QL_FP32, **kw), q.Solver(*args, precision=q.QL_FP64, **kw)
    size = rho * _terms(q, Q, u, T)
    for x, y, f in zip(a.state(), b.state(), (1.0, 2.0 * T)):
        x, y = x.T, y.T  # [velocity][cell]
        assert (np.abs(x - y) <= 1.5 * 2.0 ** -24 * np.abs(y) + 2.0 ** -44 * np.abs(f) * size + 1e-44).all()
    a.close()
    b.close()
