"""Block-averaged fields of a batch (ql_batch_fields) against the per-cell fields of ql_batch_moments averaged here:
one fine cell per coarse cell, a few, a block's worth, and more than the 256 that one block takes in one turn,
on uneven instances, in both precisions.  Tolerance: the sums of at most 32 velocities and 700 cells round to a few
times 1e-14 of the largest term (about 4 for the heat flux), the double-FP32 sums of FP32 moments to 2^-46 of it."""
import numpy as np
import pytest

from paper_2211_16933_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncoarse,mult", [(700, (1, 2)), (35, (1, 9)), (16, (16, 31)), (3, (86, 700)), (1, (257, 513))])
def test_batch_fields_are_block_averages(gpu, precision, ncoarse, mult):
    import torch
    q = gpu
    keep, insts = [], []
    for i, m in enumerate(mult):
        nx, Q = ncoarse * m, (8, 16, 24, 32)[(i + ncoarse) % 4]
        p, _ = q.ql_velocity_set(Q)
        rho, u, T = inputs.smooth_periodic_fields(nx, seed=3 + i)
        insts.append(q.make_instance(Q, nx, 1.0, inputs.cfl_dt(1.0 / nx, abs(p).max()), 0.1, 0.05,
                                     init_kind=q.QL_INIT_FIELDS, rho=rho, u=u, T=T, keep=keep))
    b = q.Batch(insts, precision=precision)
    b.run(2)
    out = torch.full((len(insts), 5, ncoarse), float("nan"), dtype=torch.float64, device="cuda")
    b._stream.wait_stream(torch.cuda.current_stream())
    b.fields(ncoarse, out)
    assert not b.sync().any()
    got = out.cpu().numpy()
    for i in range(len(insts)):
        m = b.moments(i)
        for f, k in enumerate(("rho", "u", "T", "q", "Pxx")):
            want = m[k].reshape(ncoarse, -1).mean(1)
            assert np.abs(got[i, f] - want).max() <= 1e-12, (i, k)
    b.close()
