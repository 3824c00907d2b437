"""Predicted fitness of candidates on coarse grids large enough for a cluster of
blocks per candidate (S >= 128 and fewer than eight candidates per SM), and on
both sides of that rule, against the oracle: a NaN candidate among them.

Every sum adds at most 65536 terms of one sign in double precision: on the
device in chains of at most 64 per thread, five of the shuffles and 64 of the
warps, in numpy pairwise.  So each side is within 2^-53 x 256 = 3e-14 of the
exact sums, and the ratio, whose numerator cancels less than tenfold on these
inputs, within 1e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import surrogate as sg                      # noqa: E402
from paper_1701_03549_gb300 import fire                 # noqa: E402


@pytest.mark.parametrize("S,n", [(64, 16), (128, 1), (128, 16), (256, 1),
                                 (256, 16), (128, "below"), (128, "at")])
def test_predicted_fitness(S, n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = {"below": 8 * sms - 1, "at": 8 * sms}.get(n, n)
    rng = np.random.default_rng([S, n])
    prob = rng.random((n, S, S), dtype=np.float32)
    if n > 7:
        prob[7] = np.nan
    tf = (rng.uniform(size=(S, S)) * (rng.uniform(size=(S, S)) < 0.4)
          ).astype(np.float32)
    ctx = fire.Context(0, torch.cuda.current_stream())
    pd, td = torch.tensor(prob, device="cuda"), torch.tensor(tf, device="cuda")
    keep = torch.full((max(1, n // 4),), -1, dtype=torch.int32, device="cuda")
    for kind in (0, 1):
        pred = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
        fire.fire_net_screen(ctx, S, pd, td, 16.0, kind, keep.numel(), pred,
                             keep, sync=True)
        want = sg.predicted_fitness(prob, tf, kind, 16)
        got = pred.cpu().numpy()
        ok = ~np.isnan(want)
        assert np.array_equal(np.isnan(got), ~ok)
        assert np.allclose(got[ok], want[ok], rtol=1e-12, atol=0)
        order = np.argsort(np.where(np.isnan(got), np.inf, got), kind="stable")
        assert np.array_equal(keep.cpu().numpy(), order[:keep.numel()])
    ctx.close()
