"""The nearest burnable target cell of a point (fire_snap_ignitions) on maps of
every outline: against a search over all target cells, ties to the lower index;
and its cost, which goes by the map's tiles and not by the square around them.
"""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1701_03549_gb300 import fire, synth          # noqa: E402


def _snap(ctx, m, rows, cols):
    genes = np.zeros((len(rows), 2))
    genes[:, 0], genes[:, 1] = cols, rows
    return np.asarray(fire.fire_snap_ignitions(ctx, m, genes, 0, 1, 1))


@pytest.mark.parametrize("cells", [1, 3, 40, 2000])
@pytest.mark.parametrize("H,W", [(1, 1), (31, 33), (1, 5000), (4000, 3),
                                 (33, 3000), (2999, 70), (97, 260),
                                 (512, 512)])
def test_against_all_target_cells(H, W, cells):
    rng = np.random.default_rng([H, W, cells])
    land = synth.uniform_landscape(H, W)
    water = rng.random((H, W)) < 0.2
    target = np.zeros(H * W, bool)
    # a cluster in one corner and cells anywhere: near and far points
    target[rng.integers(0, H * W, cells)] = True
    if cells > 1:
        target[rng.integers(0, H * W, cells)] &= rng.random(cells) < 0.5
    keep = rng.integers(0, H * W)
    target[keep] = True
    water.ravel()[keep] = False
    target = target.reshape(H, W)
    land.veg[water] = 0
    ctx = fire.Context(0, torch.cuda.current_stream())
    m = ctx.landscape_upload(land)
    m.target_upload(target)
    n = 64
    rows, cols = rng.integers(0, H, n), rng.integers(0, W, n)
    rows[:4], cols[:4] = [0, 0, H - 1, H - 1], [0, W - 1, 0, W - 1]
    got = _snap(ctx, m, rows, cols)
    rr, cc = np.nonzero(target & (land.veg != 0))   # row-major order
    d = (rr[None] - rows[:, None]) ** 2 + (cc[None] - cols[:, None]) ** 2
    k = d.argmin(1)                                 # the first of equal ones
    assert np.array_equal(got.reshape(-1, 2), np.stack([rr[k], cc[k]], 1))
    m.free()
    ctx.close()


def test_long_maps_cost_no_more_than_square_ones():
    """4096 tiles in one row, one column and a square, the target in the far
    corner: the same words to search.  (Whole rings took a second here.)"""
    ctx = fire.Context(0, torch.cuda.current_stream())
    best = {}
    for H, W in ((2048, 2048), (32, 131072), (131072, 32), (64, 65536)):
        m = ctx.landscape_upload(synth.uniform_landscape(H, W))
        target = np.zeros((H, W), bool)
        target[H - 1, W - 1] = True
        m.target_upload(target)
        z = np.zeros(16)
        for _ in range(4):
            t = time.perf_counter()
            got = _snap(ctx, m, z, z)
            dt = time.perf_counter() - t
            best[H, W] = min(dt, best.get((H, W), dt))
        assert (got.reshape(-1, 2) == [H - 1, W - 1]).all()
        m.free()
    ctx.close()
    # the point in the corner of the square sees all directions but two, as
    # the ends of a line do: 4 leaves room for the batches' waits
    assert max(best.values()) < 4 * best[2048, 2048], best
