"""fire_simulate_batch inside a stream capture that the caller began, with no call
of that shape before: a map whose state fits in shared memory needs nothing from
the library's buffers there, so the capture holds, and the graph stays valid when
the context later moves those buffers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1701_03549_gb300 import fire, synth          # noqa: E402


# fires per SM on both sides of the rules that prefer state in global memory
@pytest.mark.parametrize("H,W,n,steps", [
    (70, 90, 8, False), (70, 90, 8, True), (512, 512, 100, True),
    (512, 512, 1300, False), (512, 512, 4096, False), (640, 640, 400, False),
    (640, 640, 400, True)])
def test_captured_batch(H, W, n, steps):
    land = synth.landscape(H, W, seed=7)
    ign = np.tile(np.asarray(synth.centre_ignition(land.veg), np.int32), (n, 1))
    rng = np.random.default_rng(n)
    p = np.tile(np.asarray(synth.TRUTH_BETA), (n, 1)) + rng.normal(0, 2, (n, 5))
    dev = dict(device="cuda")
    args = (torch.tensor(p, **dev), torch.tensor(ign, **dev),
            torch.arange(5, 5 + n, dtype=torch.int64, **dev))
    out = torch.zeros((n, 6), dtype=torch.int32, **dev)
    bs = torch.zeros((n, H, W), dtype=torch.int32, **dev) if steps else None
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ctx = fire.Context(0, st)
        m = ctx.landscape_upload(land)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st,
                              capture_error_mode="thread_local"):
            m.simulate_batch(*args, want_steps=steps, device=True, out=out,
                             burn_step=bs)
        g.replay()
        torch.cuda.synchronize()
        first = out.clone()
        # the same call outside the capture, which may take another shape
        out.zero_()
        m.simulate_batch(*args, want_steps=steps, device=True, out=out,
                         burn_step=bs, sync=True)
        assert torch.equal(first, out) and int(first[:, 0].sum()) > n
        # a larger map moves the context's buffers; the graph runs as before
        big = ctx.landscape_upload(synth.uniform_landscape(1400, 1400))
        q = torch.full((64, 5), -1.0, dtype=torch.float64, **dev)
        o2 = torch.zeros((64, 6), dtype=torch.int32, **dev)
        big.simulate_batch(q, torch.full((64, 2), 9, dtype=torch.int32, **dev),
                           args[2][:1].repeat(64), device=True, out=o2,
                           sync=True)
        out.zero_()
        if steps:
            want = bs.clone()
            bs.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(first, out)
        if steps:
            assert torch.equal(want, bs)
        m.free()
        big.free()
        ctx.close()
