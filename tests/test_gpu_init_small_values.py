"""Initial FP32 states value by value, where populations of fast velocities are small sums of large terms: each value is the
FP64 state's, rounded once.  Bound: half a unit in the last place is at most 2^-24 of the value; pairs that the kernel
leaves to the FP64 sums are those sums rounded, and the double-FP32 sums (2^-46 of the terms' magnitudes) are kept only where
the value is at least 2^-12 of these, so they add 2^-34 of the value, 2^-10 of the bound, twice for theta: (1 + 2^-9) 2^-24."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q", [8, 16, 20, 24, 32, 40])
@pytest.mark.parametrize("u0,du,T0,dT", [(0.0, 0.1, 1.0, 0.05), (0.0, 1.0, 0.9, 0.5), (1.2, 0.2, 0.5, 0.1),
                                         (-1.0, 0.4, 0.85, 0.15), (0.0, 0.02, 1.0, 0.02), (0.0, 7.9, 4.0, 3.9)])
def test_fp32_values_are_fp64_values_rounded(gpu, Q, u0, du, T0, dT):
    q, nx = gpu, 500
    rng = np.random.default_rng(Q)
    rho, u, T = rng.uniform(0.1, 2.0, nx), rng.uniform(u0 - du, u0 + du, nx), rng.uniform(T0 - dT, T0 + dT, nx)
    args = (Q, nx, 1.0, 1e-5, 0.1, 0.05)
    kw = dict(bc=q.QL_BC_PERIODIC, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T)
    a, b = q.Solver(*args, precision=q.QL_FP32, **kw), q.Solver(*args, precision=q.QL_FP64, **kw)
    for x, y in zip(a.state(), b.state()):
        assert (np.abs(x - y) <= (1.0 + 2.0 ** -9) * 2.0 ** -24 * np.abs(y) + 1e-44).all()
    a.close()
    b.close()
