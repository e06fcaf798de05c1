"""The tile stage kernels of the solver, at the smallest domains that take them (a few cells more than the small-domain
kernels do: 131072 in FP64, 16384 in FP32), for every compiled velocity set, both chi modes and both precisions.

A periodic domain of four equal periods must give, period by period, the bits of one period alone, which is small
enough for the small-domain kernels (same arithmetic in the same order).  Lengths and Knudsen numbers differ by factors
of four, so that cell size, ball and relaxation time are the same numbers in both, whatever the order in which they are
rounded.  Fixed boundaries are compared with the oracle's right-hand side, to 1e-11 (FP64) and 2e-5 (FP32) of its
largest value, the tolerances of the other right-hand-side tests."""
import numpy as np
import pytest

import oracle as O
from paper_2211_16933_gb300 import inputs

pytestmark = pytest.mark.gpu
PERIOD = {0: 32769, 1: 4097}  # four of them: 131076 and 16388 cells, with ragged last tiles


def _solver(q, precision, Q, nx, periods, ball):
    """`periods` periods of nx cells each; ball: cells that the chi_RET-FM ball reaches on each side (None: chi_SET)."""
    length, El = nx * 2.0 ** -16, 0.25
    kn = 2.0 ** -6 if ball is None else (ball - 0.25) * 2.0 ** -16 / (El * length)  # sigma = El kn length
    rho, u, T = inputs.smooth_periodic_fields(nx, seed=Q)
    s = q.Solver(Q, periods * nx, periods * length, 2e-7, El, kn / periods, bc=q.QL_BC_PERIODIC,
                 init_kind=q.QL_INIT_FIELDS, rho=np.tile(rho, periods), u=np.tile(u, periods), T=np.tile(T, periods),
                 precision=precision, chi_mode=q.QL_CHI_SET if ball is None else q.QL_CHI_RET_FM)
    ph, th = s.state()
    noise = inputs.state_noise((nx, Q), 11)
    s.set_state(ph * np.tile(noise, (periods, 1)), th * np.tile(noise, (periods, 1)))
    return s


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ball", [None, 3])
@pytest.mark.parametrize("Q", [8, 16, 20, 24, 32, 40])
def test_tile_kernels_give_the_bits_of_the_small_domain_kernels(gpu, Q, ball, precision):
    nx = PERIOD[precision]
    one, four = (_solver(gpu, precision, Q, nx, n, ball) for n in (1, 4))
    assert one.sigma == four.sigma and one.dx == four.dx
    for a, b in zip(one.rhs(), four.rhs()):
        np.testing.assert_array_equal(b, np.tile(a, (4, 1)))
    for s in (one, four):
        s.step(1)
        s.step(2)
    for a, b in zip(one.state(), four.state()):
        np.testing.assert_array_equal(b, np.tile(a, (4, 1)))
    one.close()
    four.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("Q", [20, 40])
@pytest.mark.parametrize("ball", [None, 3])
def test_tile_kernels_at_fixed_boundaries_match_oracle(gpu, Q, ball, precision):
    q, nx, El, length = gpu, 4 * PERIOD[precision], 0.3, 1.0
    rho, u, T = inputs.smooth_periodic_fields(nx, seed=3)
    ghost = np.array([[rho[0], u[0], T[0]]] * 3 + [[rho[-1], u[-1], T[-1]]] * 3) * [1.01, 1.0, 0.99]
    kn = 0.05 if ball is None else (ball - 0.3) / (El * nx)
    dt = inputs.cfl_dt(length / nx, float(np.abs(q.ql_velocity_set(Q)[0]).max()), 0.2)
    s = q.Solver(Q, nx, length, dt, El, kn, bc=q.QL_BC_FIXED, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T, ghost=ghost,
                 precision=precision, chi_mode=q.QL_CHI_SET if ball is None else q.QL_CHI_RET_FM)
    m = O.make_model(Q, nx, length, dt, El, kn, bc=O.BC_FIXED, chi_mode=O.CHI_SET if ball is None else O.CHI_RET_FM)
    O.set_ghosts(m, ghost[:3], ghost[3:])
    ph, th = O.equilibrium_state(m, rho, u, T)
    noise = inputs.state_noise(ph.shape, 11)
    s.set_state(ph * noise, th * noise)
    want, got = O.rhs(m, ph * noise, th * noise), s.rhs()
    for x, y in zip(got, want):
        assert np.abs(x - y).max() <= (1e-11, 2e-5)[precision] * np.abs(y).max()
    s.close()
