"""ql_step_noalloc gives the bits of ql_step on FP64 domains whose per-cell buffers fit behind the stage buffers in the scratch
array (two launches per stage), on ones where only the stage buffers fit, and beyond the two-launch stages' range."""
import numpy as np
import pytest

from paper_2211_16933_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q,nx,periodic", [(8, 8, True), (16, 31, False), (40, 1000, True), (32, 49000, False), (32, 60000, True),
                                           (8, 131072, False), (8, 131073, True)])
def test_noalloc_gives_the_bits_of_ql_step(gpu, Q, nx, periodic):
    import torch
    q = gpu
    rho, u, T = inputs.smooth_periodic_fields(nx, seed=nx)
    dt = inputs.cfl_dt(1.0 / nx, float(np.abs(q.ql_velocity_set(Q)[0]).max()), 0.2)
    bc = q.QL_BC_PERIODIC if periodic else q.QL_BC_FIXED
    kw = dict(bc=bc, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T, precision=q.QL_FP64, pr_mode=q.QL_PR_DENSE)
    if not periodic:
        kw["ghost"] = np.array([[rho[0], u[0], T[0]]] * 3 + [[rho[-1], u[-1], T[-1]]] * 3) * [1.01, 1.0, 0.99]
    ref, own = (q.Solver(Q, nx, 1.0, dt, 0.1, 0.05, **kw) for _ in range(2))
    psi, stride = q.ql_state_device(own.ctx)
    o = q.ql_opts()
    o.precision, o.pr_mode, o.enskog, o.device, o.pr_const, o.rho_ref = q.QL_FP64, q.QL_PR_DENSE, 1, 0, 2.0 / 3.0, 1.0
    o.stream = torch.cuda.current_stream().cuda_stream
    for steps in (1, 2):
        q.ql_step_noalloc(q.ql_velset(Q, 0), q.ql_grid(nx, 1.0, dt), 0.1, 0.05, q.ql_bc(bc, 0), o, psi, stride, steps)
        ref.step(steps)
        for a, b in zip(own.state(), ref.state()):
            np.testing.assert_array_equal(a, b)
    own.close()
    ref.close()
