"""The closure's device error word: an index out of range in one ql_closure_train_steps call is reported by that call
and not again by later calls of other entry points, and a new closure starts without flags whatever its memory held."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(B=4, X=64):
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(B, X, 7, device="cuda", generator=g)
    return x, 0.5 * torch.randn(B, X, 5, device="cuda", generator=g), (torch.arange(B, device="cuda") % 2).int()


def test_a_bad_index_is_reported_once(gpu):
    import torch
    net, (x, y, per) = gpu.Closure(7, 5, 64, 4, seed=3), _batch()
    before = net.gradients(x, y, per)
    bad = torch.tensor([0, 1, 2, 9], dtype=torch.int32, device="cuda")
    with pytest.raises(gpu.QLError) as e:
        net.train_steps(x, y, per, bad, np.zeros(1, dtype=np.float32))
    assert e.value.status == gpu.QL_EINVAL
    after = net.gradients(x, y, per)  # learning rate 0: the same network
    assert after[0] == before[0]
    np.testing.assert_array_equal(after[1], before[1])
    assert net.train_step(x, y, per, 0.0, want_loss=True) == before[0]
    net.train_steps(x, y, per, bad.clamp(max=3), np.zeros(1, dtype=np.float32))
    net.close()


def test_a_new_closure_has_no_flags(gpu):
    """Its memory comes from an allocator that hands out blocks full of ones."""
    import ctypes as C

    import torch
    q, blocks = gpu, {}

    def alloc(nbytes, user):
        t = torch.full((max(int(nbytes), 1),), 255, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        blocks[t.data_ptr()] = t
        return t.data_ptr()

    def free(p, user):
        blocks.pop(p, None)

    hooks = q.ALLOC_FN(alloc), q.FREE_FN(free)
    d, o, c = q.ql_closure_desc(), q.ql_opts(), C.c_void_p()
    d.in_channels, d.out_channels, d.width, d.layers, d.ksize, d.positions, d.max_batch = 7, 5, 64, 5, 5, 64, 4
    for i in range(8):
        d.in_scale[i] = d.out_scale[i] = 1.0
    o.stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    o.alloc, o.free = hooks
    assert q.lib().ql_closure_create(C.byref(d), C.byref(o), C.byref(c)) == q.QL_OK
    x, y, per = _batch()
    loss = C.c_float()
    st = q.lib().ql_closure_gradients(c, C.c_void_p(x.data_ptr()), C.c_void_p(y.data_ptr()), C.c_void_p(per.data_ptr()), 4,
                                      C.byref(loss), None)
    assert st == q.QL_OK, q.lib().ql_closure_last_error(c)
    assert np.isfinite(loss.value)
    q.lib().ql_closure_destroy(c)
