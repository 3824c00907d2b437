"""The surrogate's convolutions at S = 1024, whose layer of dilation 32 streams
strips of 192 pixels in three stages (its teeth would be below 8 pixels), and with
several samples where a tile is a row or less of one: forward, input gradient,
weight and bias gradients against 64-bit sums, with the tolerances of
test_gpu_conv_layers.py.  From S = 512 on the rows at both ends, around a
dilation's distance from them and in the middle stand for the others.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1701_03549_gb300 import fire, surrogate      # noqa: E402

DIL = (1, 1, 2, 4, 8, 16, 32, 64)


def _conv64(x, w, d, sign, r0, r1):
    """Rows r0 to r1 of sum_t x[p + sign off(t)] w[:, t, :]^T in float64, and of
    its absolute sum."""
    S = x.shape[1]
    a, b = max(0, r0 - d), min(S, r1 + d)
    xp = torch.nn.functional.pad(x[:, a:b].double(),
                                 (0, 0, d, d, d - r0 + a, r1 + d - b))
    z = torch.zeros((x.shape[0], r1 - r0, S, w.shape[0]), dtype=torch.float64,
                    device=x.device)
    za = torch.zeros_like(z)
    for t in range(9):
        r, c = d + sign * (t // 3 - 1) * d, d + sign * (t % 3 - 1) * d
        xs = xp[:, r:r + r1 - r0, c:c + S, :]
        z += xs @ w[:, t, :].T
        za += xs.abs() @ w[:, t, :].abs().T
    return z, za


def _rows(S, d):
    if S < 512:
        return [(0, S)]
    return [(0, 6), (max(0, d - 2), d + 2), (S // 2 - 3, S // 2 + 3),
            (S - d - 2, min(S, S - d + 2)), (S - 6, S)]


@pytest.mark.parametrize("S,n", [(128, 3), (256, 2), (512, 2), (1024, 1)])
def test_layers_and_gradients(S, n):
    torch.manual_seed(S + n)
    ctx = fire.Context(0, torch.cuda.current_stream())
    theta = surrogate.init_params(S + n, head_bias=-1.0)
    theta += np.float32(0.01) * np.random.default_rng(S).standard_normal(
        theta.size).astype(np.float32)   # nonzero biases
    net = fire.Net(ctx, S, n)
    net.set_params(theta)
    x = torch.rand((n, S, S, 16), device="cuda").to(torch.bfloat16)
    t = torch.rand((n, S, S), device="cuda")
    net.backward(x, t, None, sync=True)
    th = torch.tensor(theta, device="cuda")
    grad = torch.tensor(net.get(fire.NET_GRAD), device="cuda").double()
    eps = (n * S * S / 800 + 160) * 2.0 ** -23

    def buf(which, l):
        o = torch.empty((n, S, S, 128), dtype=torch.bfloat16, device="cuda")
        return net.buffer(which, l, n, o)

    off, hin = 0, x
    for l, d in enumerate(DIL):
        ci = hin.shape[-1]
        nw = 128 * 9 * ci
        w = th[off:off + nw].view(128, 9, ci).to(torch.bfloat16).double()
        b = th[off + nw:off + nw + 128].double()
        h, dz = buf(fire.BUF_ACT, l), buf(fire.BUF_DZ, l)
        below = buf(fire.BUF_DZ, l - 1) if l else None
        for r0, r1 in _rows(S, d):
            z, za = _conv64(hin, w, d, 1, r0, r1)
            z = torch.relu(z + b)
            tol = 2.0 ** -8 * z.abs() + (9 * ci + 1) * 2.0 ** -24 * (za + b.abs())
            got = h[:, r0:r1].double()
            assert bool(((got - z).abs() <= tol).all()), (l, r0, "forward")
            if l:
                g, ga = _conv64(dz, w.permute(2, 1, 0).contiguous(), d, -1, r0, r1)
                g = torch.where(hin[:, r0:r1] > 0, g, torch.zeros_like(g))
                tol = 2.0 ** -8 * g.abs() + 9 * 128 * 2.0 ** -24 * ga
                got = below[:, r0:r1].double()
                assert bool(((got - g).abs() <= tol).all()), (l, r0, "input gradient")
        # weight and bias gradients over all pixels, sample by sample
        gw = grad[off:off + nw].view(128, 9, ci)
        want = torch.zeros((9, 128, ci), dtype=torch.float64, device="cuda")
        mag, db, dba = torch.zeros_like(want), 0.0, 0.0
        for i in range(n):
            zi = dz[i].double().reshape(-1, 128)
            db, dba = db + zi.sum(0), dba + zi.abs().sum(0)
            hp = torch.nn.functional.pad(hin[i].double(), (0, 0, d, d, d, d))
            for tap in range(9):
                r, c = (tap // 3) * d, (tap % 3) * d
                xs = hp[r:r + S, c:c + S, :].reshape(-1, ci)
                want[tap] += zi.T @ xs
                mag[tap] += zi.abs().T @ xs.abs()
        assert bool(((gw.transpose(0, 1) - want).abs() <= eps * mag).all()), l
        assert bool(((grad[off + nw:off + nw + 128] - db).abs() <= eps * dba).all()), l
        off += nw + 128
        hin = h
    net.free()
    ctx.close()
