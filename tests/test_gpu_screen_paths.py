"""The two single-precision screens of the trial decision against the oracle:
fixed point where map and coefficients fit its range, float pairs elsewhere.
Coefficients on both sides of each limit (fx_scale in fire_device.cuh), maps
with uniform and varying wind, and a map with one slope out of range.  Every
trajectory is compared cell by cell: decisions near a threshold fall back to
double precision in either screen, so they are all exact.
"""
import numpy as np
import pytest

from paper_1701_03549_gb300 import synth

pytestmark = pytest.mark.gpu


def _coefficients():
    """Rows around the limits: |b_j| 63.9 and 127.9, |b0| + |b1| + |b2| +
    1.4143 |b3| + 2 |b4| 255 and 511.  The rest of a row keeps z moderate, so
    that fires neither die at once nor decide without a draw."""
    rows = [list(synth.TRUTH_BETA), [0.3, -0.4, 0.5, 1.0, -0.5], [0.0] * 5]
    for lim in (63.9, 127.9):
        for v in (np.nextafter(lim, 0), np.nextafter(lim, 200), lim + 1):
            for j in (2, 3, 4):
                b = [-0.2, 0.1, 0.4, 0.6, 0.2]
                b[j] = v if j != 3 else -v
                rows.append(b)
    for lim in (255.0, 511.0):
        for v in (lim / 2 - 1.2, lim / 2 - 0.4, lim / 2 + 1.0):
            rows.append([-v, v + 0.4, 0.1, 0.2, 0.1])
    rows += [[1e4, -1e4, 1.0, 1.0, 1.0], [1e300, -1e300, 0.0, 1.0, 0.0]]
    return np.array(rows, np.float64)


@pytest.mark.parametrize("cell", [False, True])
@pytest.mark.parametrize("wind", [None, 7])
@pytest.mark.parametrize("steep", [False, True])
def test_paths_match_the_oracle(cell, wind, steep):
    pytest.importorskip("torch")
    import oracle
    from paper_1701_03549_gb300 import fire

    oracle.build()
    land = synth.landscape(45, 70, seed=11, wind_seed=wind)
    if steep:   # sig = slope / 100 beyond the fixed-point range in one cell
        land.slope[20, 30] = 250.0
    p = _coefficients()
    n = len(p)
    ign = np.tile(np.asarray(synth.centre_ignition(land.veg), np.int32), (n, 1))
    seeds = np.arange(5, 5 + n, dtype=np.uint64)
    target = np.random.default_rng(3).random(land.shape) < 0.4
    ctx = fire.Context(0)
    m = ctx.landscape_upload(land)
    m.target_upload(target)
    F = oracle.Features(land)
    res, bs = m.simulate_batch(p, ign, seeds, want_steps=True,
                               cell_uniform=cell)
    for i in range(n):
        o, obs = F.simulate(p[i], tuple(ign[i]), int(seeds[i]), target=target,
                            mode=1 if cell else 0)
        assert np.array_equal(bs[i], obs), (i, p[i])
        for k in ("burnt", "inter", "target", "steps", "status", "trials"):
            assert int(res[k][i]) == o[k], (i, k)
    assert np.unique(res["burnt"]).size > 5   # the rows are not all trivial
    m.free()
    ctx.close()
