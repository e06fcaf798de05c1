"""The stage kernels of small domains (FP32), and FP64 stages as two launches (small domains, and velocity sets
without compiled tiles), at the sizes where they can go
wrong: domains below one block of cells or one warp's strip, one cell more, several of each; balls of chi_RET-FM
that the cell kernel averages itself (up to 5 cells) and wider ones; a domain of more cells than the per-cell
buffers hold.  Tiled velocity sets must give the bits of the tile kernels, which the batched form always runs; the
other sets are compared with the oracle's right-hand side to 1e-11 of its largest value, the tolerance of the other
right-hand-side tests."""
import numpy as np
import pytest

import oracle as O
from paper_2211_16933_gb300 import inputs

pytestmark = pytest.mark.gpu


def _setup(q, Q, nx, periodic, ball, seed):
    """Smooth fields on nx cells; ball: cells that the chi_RET-FM ball reaches on each side (None: chi_SET)."""
    rho, u, T = inputs.smooth_periodic_fields(nx, seed)
    El, length = 0.3, 1.0
    kn = 0.05 if ball is None else max(ball - 0.3, 0.2) / (El * nx)
    dt = inputs.cfl_dt(length / nx, float(np.abs(q.ql_velocity_set(Q)[0]).max()), 0.2)
    kw = dict(bc=q.QL_BC_PERIODIC if periodic else q.QL_BC_FIXED, init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T,
              chi_mode=q.QL_CHI_SET if ball is None else q.QL_CHI_RET_FM)
    if not periodic:
        kw["ghost"] = np.array([[rho[0], u[0], T[0]]] * 3 + [[rho[-1], u[-1], T[-1]]] * 3) * [1.01, 1.0, 0.99]
    return (Q, nx, length, dt, El, kn), kw


def _same_as_batch(q, precision, Q, nx, periodic, ball):
    args, kw = _setup(q, Q, nx, periodic, ball, seed=nx + Q)
    s = q.Solver(*args, precision=precision, **kw)
    keep = []
    plain, pkw = _setup(q, 8, 40, True, None, seed=1)  # a batch needs a chi_SET instance
    b = q.Batch([q.make_instance(*args, keep=keep, **kw), q.make_instance(*plain, keep=keep, **pkw)],
                precision=precision)
    s.step(2)
    s.step(1)
    b.run(3)
    assert not b.sync().any()
    for x, y in zip(s.state(), b.state(0)):
        np.testing.assert_array_equal(x, y)
    s.close()
    b.close()


@pytest.mark.parametrize("Q,nx,periodic,ball", [
    (8, 8, True, None), (8, 26, False, None), (16, 27, True, None), (32, 31, False, None), (24, 32, True, None),
    (32, 1000, False, None), (16, 8, True, 2), (8, 22, False, 2), (24, 23, True, 5), (32, 63, False, 5),
    (16, 64, True, 6), (32, 500, False, 9)])
def test_two_launch_stages_give_the_bits_of_the_tile_kernels(gpu, Q, nx, periodic, ball):
    _same_as_batch(gpu, gpu.QL_FP64, Q, nx, periodic, ball)


@pytest.mark.parametrize("Q,nx,periodic,ball", [
    (8, 8, True, None), (16, 29, False, None), (24, 30, True, None), (32, 31, False, None), (8, 61, False, None),
    (32, 1000, True, None), (16, 8, True, 1), (8, 30, False, 1), (24, 61, True, 3), (32, 90, False, 16),
    (16, 91, True, 16), (16, 200, True, 17)])
def test_fp32_stages_of_small_domains_give_the_bits_of_the_tile_kernels(gpu, Q, nx, periodic, ball):
    """30 cells per CTA, the velocity pairs dealt to its warps, balls of up to 16 cells averaged in the stage."""
    _same_as_batch(gpu, gpu.QL_FP32, Q, nx, periodic, ball)


@pytest.mark.parametrize("Q,nx,periodic,ball", [(6, 131072 + 37, True, None), (4, 131072 + 1, False, None),
                                                (50, 45, True, 7), (12, 40, False, 3)])
def test_other_velocity_sets_against_the_oracle(gpu, Q, nx, periodic, ball):
    q = gpu
    (_, _, length, dt, El, kn), kw = args = _setup(q, Q, nx, periodic, ball, seed=5)
    s = q.Solver(*args[0], precision=q.QL_FP64, **kw)
    m = O.make_model(Q, nx, length, dt, El, kn, bc=O.BC_PERIODIC if periodic else O.BC_FIXED,
                     chi_mode=O.CHI_SET if ball is None else O.CHI_RET_FM)
    if not periodic:
        O.set_ghosts(m, kw["ghost"][:3], kw["ghost"][3:])
    ph, th = O.equilibrium_state(m, kw["rho"], kw["u"], kw["T"])
    noise = inputs.state_noise(ph.shape, 11)
    s.set_state(ph * noise, th * noise)
    want, got = O.rhs(m, ph * noise, th * noise), s.rhs()
    for x, y in zip(got, want):
        assert np.abs(x - y).max() <= 1e-11 * np.abs(y).max()
    s.close()
