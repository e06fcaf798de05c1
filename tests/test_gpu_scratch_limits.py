"""ql_create where the memory does not suffice for the buffers that only the small-domain kernels need (per-cell
coefficients in FP64, the second density array of chi_RET-FM in FP32): the solver is created, and its steps give the
same bits.  The allocator hook refuses what goes beyond a limit just below the unlimited solver's total."""
import numpy as np
import pytest

from paper_2211_16933_gb300 import inputs

pytestmark = pytest.mark.gpu


def _solver(q, limit, precision, Q, nx, ball):
    class Limited(q.Solver):
        total = 0

        def _attach_torch(self, o, device, use_torch):
            super()._attach_torch(o, device, use_torch)
            inner = self._alloc_cb

            def alloc(nbytes, user):
                if limit is not None and self.total + nbytes > limit:
                    return None
                self.total += nbytes
                return inner(nbytes, user)

            self._limited_cb = q.ALLOC_FN(alloc)
            o.alloc = self._limited_cb

    rho, u, T = inputs.smooth_periodic_fields(nx, seed=nx)
    dt = inputs.cfl_dt(1.0 / nx, float(np.abs(q.ql_velocity_set(Q)[0]).max()), 0.2)
    kn = 0.05 if ball is None else (ball - 0.3) / (0.3 * nx)
    return Limited(Q, nx, 1.0, dt, 0.3, kn, bc=q.QL_BC_PERIODIC, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T,
                   precision=precision, chi_mode=q.QL_CHI_SET if ball is None else q.QL_CHI_RET_FM)


@pytest.mark.parametrize("precision,Q,nx,ball", [(0, 16, 1000, None), (0, 40, 300, 3), (0, 24, 2000, 9), (1, 20, 1000, 2),
                                                 (0, 12, 3000, None), (0, 50, 700, 7)])
def test_solvers_without_room_for_the_small_domain_buffers(gpu, precision, Q, nx, ball):
    free = _solver(gpu, None, precision, Q, nx, ball)
    tight = _solver(gpu, free.total - 1, precision, Q, nx, ball)
    assert tight.total < free.total
    for s in (free, tight):
        s.step(1)
        s.step(2)
    for a, b in zip(free.state() + free.rhs(), tight.state() + tight.rhs()):
        np.testing.assert_array_equal(a, b)
    tight.close()
    free.close()


def test_no_room_for_the_state_is_still_refused(gpu):
    free = _solver(gpu, None, 0, 16, 500, None)
    with pytest.raises(gpu.QLError) as e:
        _solver(gpu, free.total // 4, 0, 16, 500, None)
    assert e.value.status == gpu.QL_ENOMEM
    free.close()
