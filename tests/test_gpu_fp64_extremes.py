"""FP64 kernels where a reciprocal, root or logarithm meets an argument outside the normal range: an infinite Knudsen
number (no collisions: the relaxation rate is the reciprocal of an infinite time) gives what 1e200 gives, bit for bit, on
the small-domain kernels, on the tile kernels and on a velocity set without tiles."""
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
