"""WENO-5 face values of the FP64 kernels (App. A.2) value by value, where the right-hand-side tests, which compare
with the largest value of a row, cannot see an error.

At a Knudsen number of 1e200 with the Enskog term off the right-hand side is the advection alone, L = -p (h_R - h_L) / dx,
so the rows of a state can be any positive numbers; every velocity gets the same ones in another scale.  The reference
evaluates the faces in extended precision from the same FP64 values.  Tolerance per value: 2e-14 of (s_R + s_L) |p| / dx,
where s = |f0| + sum_q w_q C_q with C_q the sum of the magnitudes in a candidate (F^q - f0).  An FP64 face has about 25
roundings of 1.1e-16 on weights and candidates, and an indicator (a quadratic form with condition number at most 35)
passes a relative error of its differences on at most 4 times: 25 x 4 x 1.1e-16 = 1.1e-14.  Domains: a few blocks of
the small-domain kernels, and one that the tile kernels take (the rows repeat, and so does the reference)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _faces(f):
    """(h, s) of the right face of every cell of periodic rows f for a positive velocity."""
    m2, m1, p1, p2 = (np.roll(f, k) for k in (2, 1, -1, -2))
    a, b, g, c = m2 - m1, f - m1, p1 - f, p2 - p1
    beta = [a * a + LD(2.75) * a * b + LD(2.5) * b * b, b * b - LD(1.25) * b * g + g * g,
            c * c - LD(2.75) * c * g + LD(2.5) * g * g]
    s = [x * x for x in beta]
    w = [s[1] * s[2], 6 * s[0] * s[2], 3 * s[0] * s[1]]
    d = w[0] + w[1] + w[2]
    flat = d == 0  # the stencils that carry weight are constant
    d = np.where(flat, LD(1), d)
    cand = [(2 * a + 5 * b) / 6, (b + 2 * g) / 6, (4 * g - c) / 6]
    size = [(2 * abs(a) + 5 * abs(b)) / 6, (abs(b) + 2 * abs(g)) / 6, (4 * abs(g) + abs(c)) / 6]
    h = f + sum(x * y for x, y in zip(w, cand)) / d
    return h, abs(f) + sum(x * y for x, y in zip(w, size)) / d


def _check_advection(q, block, Q, repeat):
    """block: positive values of one period of a row."""
    block = np.asarray(block, dtype=np.float64)
    nx = len(block) * repeat
    s = q.Solver(Q, nx, 1.0, 1e-9, 1e-3, 1e200, bc=q.QL_BC_PERIODIC, init_kind=q.QL_INIT_FIELDS, rho=np.ones(nx),
                 u=np.zeros(nx), T=np.ones(nx), precision=q.QL_FP64, pr_mode=q.QL_PR_CONST, enskog=0)
    scale = 2.0 ** (np.arange(Q) % 3)  # exact
    rows = np.tile(block, repeat)[:, None] * scale
    s.set_state(rows, rows)
    got = s.rhs()
    f = block.astype(LD)
    hp, sp = _faces(f)
    hm, sm = (x[::-1] for x in _faces(f[::-1]))  # value at the left face of each cell for a negative velocity
    want = {1: -(hp - np.roll(hp, 1)), -1: np.roll(hm, -1) - hm}
    size = {1: sp + np.roll(sp, 1), -1: np.roll(sm, -1) + sm}
    for L in got:
        for k in range(Q):
            sgn, r = (1, LD(s.p[k])) if s.p[k] > 0 else (-1, LD(-s.p[k]))
            # a negative velocity: L = -p (h_R - h_L) / dx = |p| (h_R - h_L) / dx
            x = (L[:, k].reshape(repeat, -1) / (r * LD(scale[k]) / LD(s.dx))).astype(LD)
            err = abs(x - want[sgn]) / size[sgn]
            assert err.max() <= 2e-14, (k, float(err.max()), int(err.max(0).argmax()))
    s.close()


def _power_of_two_rows():
    """Five-cell patterns f0 + (2^-k, 0, 0, 1, 3) g and their mirror images between random cells: the first stencil's indicator
    vanishes against the other two, and all three are powers of two."""
    rng = np.random.default_rng(3)
    out = []
    for g in (0.25, 0.5, 1.0, 2.0):
        for k in range(12, 25):
            pat = 8.0 + g * np.array([2.0 ** -k, 0.0, 0.0, 1.0, 3.0])
            for f in (pat, pat[::-1]):
                out += list(f) + list(rng.uniform(7.0, 9.0, 3))
    return out


@pytest.mark.parametrize("repeat", [1, 160])
def test_weights_of_powers_of_two(gpu, repeat):
    _check_advection(gpu, _power_of_two_rows(), 8, repeat)


def _steep_rows():
    """Positive rows whose neighbouring values differ by large factors: tails that fall and rise by e^5 and e^12 per cell, a flat
    tail beside a jump of 22 and 25 decades, a Gaussian population across a temperature jump, random factors, and (values of
    ordinary size) random data and jumps by 1.5, 2, 3 and 8."""
    rng = np.random.default_rng(17)
    u = lambda n, amp: 1.0 + amp * rng.uniform(0, 1, n)
    out = [np.exp(-5.0 * np.arange(12)) * u(12, 0.1), np.exp(-60.0 + 5.0 * np.arange(12)) * u(12, 0.1),
           np.exp(-12.0 * np.arange(6)) * u(6, 0.1), np.exp(-72.0 + 12.0 * np.arange(7)) * u(7, 0.1)]
    for tail, high in ((1e-25, 1.0), (1e-25, 1e-3), (1e-22, 1.0)):
        out += [tail * u(8, 0.3), high * u(8, 0.3)]
    T = np.concatenate([np.full(6, 0.4), np.linspace(0.4, 1.3, 7), np.full(6, 1.3)])
    for p in (3.0, 5.0, 7.0):
        f = np.exp(-p * p / (2 * T)) * u(len(T), 1e-3)
        out += [f, f[::-1]]
    out += [np.exp(rng.uniform(-12, 12, 200)), rng.uniform(0, 1, 200)]
    for r in (1.5, 2.0, 3.0, 8.0):
        out += [u(5, 0.01), u(7, 0.01) / r]
    return np.concatenate(out)


@pytest.mark.parametrize("repeat", [1, 250])
def test_steep_rows_keep_the_relative_precision_of_small_values(gpu, repeat):
    _check_advection(gpu, _steep_rows(), 8, repeat)


@pytest.mark.parametrize("repeat", [1, 300])
def test_differences_near_the_smallest_normal_number(gpu, repeat):
    """Tails of 1e-300 and 1e-305, alone and beside a value of 1: their differences' unit of 2^-59 is below the normal range."""
    rng = np.random.default_rng(29)
    u = lambda n: 1.0 + rng.uniform(0, 1, n)
    _check_advection(gpu, np.concatenate([1e-300 * u(200), u(20), 1e-305 * u(200), u(20)]), 8, repeat)
