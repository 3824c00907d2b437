"""Every convolution of the surrogate on its own, forward and backward, at the
sizes where its kernels change path: tiles of several rows (S < 128), one row
(S = 128), half a row (S = 256) and a quarter (S = 512), every dilation, odd
sample counts.

Each layer is computed in 64 bits from the device's own input of that layer
(BF16, so exactly known), which leaves one layer's rounding in the comparison:

An output z is an FP32 sum of K = 9 C_in products, so it is within
K 2^-24 sum|w x| of the exact one (the products are exact in FP32), and its
BF16 rounding adds at most 2^-8 |z|.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1701_03549_gb300 import fire, surrogate  # noqa

DIL = (1, 1, 2, 4, 8, 16, 32, 64)


def _conv64(x, w, d, sign):
    """sum_t x[p + sign off(t)] w[:, t, :]^T in float64, and its absolute sum."""
    S = x.shape[1]
    xp = torch.nn.functional.pad(x, (0, 0, d, d, d, d))
    z = torch.zeros(x.shape[:3] + (w.shape[0],), dtype=torch.float64,
                    device=x.device)
    za = torch.zeros_like(z)
    for t in range(9):
        r, c = d + sign * (t // 3 - 1) * d, d + sign * (t % 3 - 1) * d
        xs = xp[:, r:r + S, c:c + S, :]
        z += xs @ w[:, t, :].T
        za += xs.abs() @ w[:, t, :].abs().T
    return z, za


@pytest.mark.parametrize("S,n", [(8, 3), (16, 1), (16, 3), (32, 2), (64, 1),
                                 (128, 1), (256, 1), (512, 1)])
def test_layers(S, n):
    torch.manual_seed(S + n)
    ctx = fire.Context(0, torch.cuda.current_stream())
    theta = surrogate.init_params(S + n, head_bias=-1.0)
    theta += np.float32(0.01) * np.random.default_rng(S).standard_normal(
        theta.size).astype(np.float32)   # nonzero biases
    net = fire.Net(ctx, S, n)
    net.set_params(theta)
    x = torch.rand((n, S, S, 16), device="cuda").to(torch.bfloat16)
    t = torch.rand((n, S, S), device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    net.backward(x, t, loss, sync=True)
    th = torch.tensor(theta, device="cuda")

    def buf(which, l):
        o = torch.empty((n, S, S, 128), dtype=torch.bfloat16, device="cuda")
        return net.buffer(which, l, n, o).double()

    off, hin = 0, x.double()
    for l, d in enumerate(DIL):
        ci = hin.shape[-1]
        nw = 128 * 9 * ci
        w = th[off:off + nw].view(128, 9, ci).to(torch.bfloat16).double()
        b = th[off + nw:off + nw + 128].double()
        h, dz = buf(fire.BUF_ACT, l), buf(fire.BUF_DZ, l)
        # forward
        z, za = _conv64(hin, w, d, 1)
        z = torch.relu(z + b)
        tol = 2.0 ** -8 * z.abs() + (9 * ci + 1) * 2.0 ** -24 * (za + b.abs())
        assert bool(((h - z).abs() <= tol).all()), (l, "forward")
        # input gradient, masked by the layer below
        if l > 0:
            wt = w.permute(2, 1, 0).contiguous()
            g, ga = _conv64(dz, wt, d, -1)
            g = torch.where(hin > 0, g, torch.zeros_like(g))
            tol = 2.0 ** -8 * g.abs() + 9 * 128 * 2.0 ** -24 * ga
            got = buf(fire.BUF_DZ, l - 1)
            assert bool(((got - g).abs() <= tol).all()), (l, "input gradient")
        off += nw + 128
        hin = h
    net.free()
    ctx.close()


@pytest.mark.parametrize("S,n", [(8, 3), (16, 1), (16, 3), (32, 2), (64, 1),
                                 (64, 3), (128, 1), (256, 1), (512, 1)])
def test_weight_gradients(S, n):
    """dW and db of every layer from the device's own dz and layer input.

    The pixels (P) are split over at least 50 blocks per tap, each a chain of
    FP32 additions of 16-pixel products (at most P / 800 + 8 of them), and the
    blocks' sums (at most 152) are added with atomics; an addition errs by at
    most 2^-23 of what it adds up to (the tensor core truncates), which the sum
    of absolute products bounds.
    """
    torch.manual_seed(S + n)
    ctx = fire.Context(0, torch.cuda.current_stream())
    theta = surrogate.init_params(2 * S + n, head_bias=-1.0)
    net = fire.Net(ctx, S, n)
    net.set_params(theta)
    x = torch.rand((n, S, S, 16), device="cuda").to(torch.bfloat16)
    t = torch.rand((n, S, S), device="cuda")
    net.backward(x, t, None, sync=True)
    grad = torch.tensor(net.get(fire.NET_GRAD), device="cuda").double()
    eps = (n * S * S / 800 + 160) * 2.0 ** -23

    def buf(which, l):
        o = torch.empty((n, S, S, 128), dtype=torch.bfloat16, device="cuda")
        return net.buffer(which, l, n, o).double()

    off, hin = 0, x.double()
    for l, d in enumerate(DIL):
        ci = hin.shape[-1]
        nw = 128 * 9 * ci
        dz = buf(fire.BUF_DZ, l).reshape(-1, 128)
        hp = torch.nn.functional.pad(hin, (0, 0, d, d, d, d))
        gw = grad[off:off + nw].view(128, 9, ci)
        for tap in range(9):
            r, c = (tap // 3) * d, (tap % 3) * d
            xs = hp[:, r:r + S, c:c + S, :].reshape(-1, ci)
            want, mag = dz.T @ xs, dz.abs().T @ xs.abs()
            assert bool(((gw[:, tap] - want).abs() <= eps * mag).all()), (l, tap)
        gb = grad[off + nw:off + nw + 128]
        assert bool(((gb - dz.sum(0)).abs() <= eps * dz.abs().sum(0)).all()), l
        off += nw + 128
        hin = buf(fire.BUF_ACT, l)
    net.free()
    ctx.close()
