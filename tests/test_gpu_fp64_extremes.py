"""FP64 kernels where a reciprocal, root or logarithm meets an argument outside the normal range: an infinite Knudsen
number (no collisions: the relaxation rate is the reciprocal of an infinite time) gives what 1e200 gives, bit for bit, on
the small-domain kernels, on the tile kernels and on a velocity set without tiles.  A gas whose density is below the smallest
normal number (but has a finite reciprocal) can be stepped."""
import numpy as np
import pytest

from paper_2211_16933_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,Q,nx", [(0, 16, 200), (0, 32, 1000), (0, 12, 90), (0, 8, 131080), (1, 16, 200), (1, 8, 16400)])
def test_an_infinite_knudsen_number_means_no_collisions(gpu, precision, Q, nx):
    q = gpu
    rho, u, T = inputs.smooth_periodic_fields(nx, seed=nx)
    dt = inputs.cfl_dt(1.0 / nx, float(np.abs(q.ql_velocity_set(Q)[0]).max()), 0.2)
    out = []
    for kn in (np.inf, 1e200 if precision == 0 else 1e30):
        s = q.Solver(Q, nx, 1.0, dt, 0.1, kn, bc=q.QL_BC_PERIODIC, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T,
                     precision=precision)
        s.step(3)
        out.append(s.state())
        s.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all()
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("Q,nx", [(8, 64), (12, 64), (8, 131080)])
def test_a_density_below_the_normal_range(gpu, Q, nx):
    q = gpu
    rho, u, T = np.full(nx, 1.5e-308), np.zeros(nx), np.ones(nx)
    s = q.Solver(Q, nx, 1.0, 1e-4 / nx, 0.1, 0.05, bc=q.QL_BC_PERIODIC, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T,
                 precision=q.QL_FP64)
    s.step(3)
    m = s.moments()
    # uniform: nothing changes but for the rounding of subnormal populations (spacing 5e-324, 40 of them and 9 stages)
    assert np.abs(m["rho"] / rho - 1.0).max() <= 400 * 5e-324 / 1.5e-308 + 1e-13
    s.close()
