"""Bias and head gradients, sums over all pixels, against 64-bit sums of the device's
own activation gradients (BF16, exactly known) and head gradient (FP32).

Blocks add their partial sums into 16 slots in single precision, c additions a
slot, and the slots are added in double precision and rounded once.  An
addition errs by at most 2^-24 of the running total, at random by a third of
it; totals grow evenly, so c of them err by 2^-24 sqrt(c) / 5, and 16
independent slots by a quarter of that.  The final rounding is at most 2^-24.
The bound on the norm, 2^-24 (1 + sqrt(c) / 4), leaves a factor of five on the
additions; with one chain for all blocks the errors were 1.5e-7 to 3.4e-7.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1701_03549_gb300 import fire, surrogate      # noqa: E402

LAYERS = 8


@pytest.mark.parametrize("S,n", [(8, 20), (16, 1), (16, 64), (32, 8),
                                 (32, 32), (64, 8), (128, 1)])
def test_sums(S, n):
    torch.manual_seed(S + n)
    ctx = fire.Context(0, torch.cuda.current_stream())
    theta = surrogate.init_params(2 * S + n)
    net = fire.Net(ctx, S, n)
    net.set_params(theta)
    x = torch.rand((n, S, S, 16), device="cuda").to(torch.bfloat16)
    t = torch.rand((n, S, S), device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    net.backward(x, t, loss, sync=True)
    grad = torch.tensor(net.get(fire.NET_GRAD), device="cuda").double()
    prob = torch.empty((n, S, S), device="cuda")
    net.forward(x, prob, sync=True)
    P = n * S * S

    def err(got, want):
        return float((got - want).norm() / want.norm())

    def bound(c):
        return 2.0 ** -24 * (1 + max(1.0, c) ** 0.5 / 4)

    def buf(which, l):
        o = torch.empty((n, S, S, 128), dtype=torch.bfloat16, device="cuda")
        return net.buffer(which, l, n, o).double().reshape(-1, 128)

    # head: blocks of 64 pixels at these sizes
    g = ((prob - t) * np.float32(1 / np.float32(P))).double().reshape(-1, 1)
    assert err(grad[-129:-1], (g * buf(fire.BUF_ACT, 7)).sum(0)) < bound(P / 1024)
    assert abs(float(grad[-1] - g.sum())) < bound(P / 1024) * float(g.abs().sum())
    # biases: blocks of 64 pixels (S = 8), at most 152 blocks otherwise
    c = P / 1024 if S < 16 else min(P / 1024, 152 / 16)
    off = 0
    for l in range(LAYERS):
        off += 128 * 9 * (128 if l else 16)
        dz = buf(fire.BUF_DZ, l)
        assert err(grad[off:off + 128], dz.sum(0)) < bound(c), l
        off += 128
    # the loss that comes back with them
    y, tt = prob.double(), t.double()
    want = -(tt * y.log() + (1 - tt) * (1 - y).log()).mean()
    assert abs(float(loss) - float(want)) < 1e-5 * float(want)
    net.free()
    ctx.close()


def test_loss_into_any_address():
    """A loss pointer that is not 8-byte aligned is taken as before."""
    ctx = fire.Context(0, torch.cuda.current_stream())
    net = fire.Net(ctx, 16, 1)
    net.set_params(surrogate.init_params(1))
    x = torch.rand((1, 16, 16, 16), device="cuda").to(torch.bfloat16)
    t = torch.rand((1, 16, 16), device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    net.backward(x, t, loss, sync=True)
    raw = torch.zeros(16, dtype=torch.uint8, device="cuda")
    ctx.check(ctx.lib.fire_net_backward(
        ctx.h, net.h, 1, x.data_ptr(), t.data_ptr(),
        fire.FIRE_DEVICE_PTRS | fire.FIRE_SYNC, raw.data_ptr() + 3))
    got = raw.cpu().numpy()[3:11].copy().view(np.float64)[0]
    assert got == pytest.approx(float(loss), rel=1e-12)
    net.free()
    ctx.close()
