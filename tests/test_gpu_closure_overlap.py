"""ql_closure_forward with an output that overlaps its inputs gives what separate arrays give, bit for bit: y shifted
against x by less than its length in either direction, y in the place of x, and y over the padding kinds.  More samples
than the GPU holds blocks of the whole-network kernel at once, so that some are read after others are written."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,shift", [(7, 5, 0), (7, 5, 64 * 7 * 37), (5, 7, 64 * 5 * 37), (6, 6, 0), (6, 6, 4), (7, 5, None)])
def test_forward_over_its_own_inputs(gpu, cin, cout, shift):
    import torch
    B, X = 700, 64
    net = gpu.Closure(cin, cout, X, B, seed=5)
    g = torch.Generator(device="cuda").manual_seed(2)
    x = torch.randn(B, X, cin, device="cuda", generator=g)
    per = (torch.arange(B, device="cuda") % 2).int()
    want = torch.empty(B, X, cout, device="cuda")
    net.forward(x, per, want)
    n, m = x.numel(), want.numel()
    for forward in (True, False):
        if shift is None:  # y over periodic
            y = torch.empty(m, device="cuda")
            p = y[m // 2:m // 2 + B].view(torch.int32)
            p.copy_(per)
            net.forward(x, p, y)
        else:  # y starts `shift` floats after x, or before it
            buf = torch.empty(n + m + 2 * shift, device="cuda")
            at = (0, shift) if forward else (shift, 0)
            xs, y = buf[at[0]:at[0] + n].view(B, X, cin), buf[at[1]:at[1] + m]
            xs.copy_(x)
            net.forward(xs, per, y)
        assert torch.equal(y.view(B, X, cout), want)
    net.close()
