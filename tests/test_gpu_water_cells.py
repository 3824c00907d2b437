"""Covariates of cells that cannot burn have no say in how a map is simulated: with
NaN, -9999 and winds of their own in them a map runs as fast as without, and its
fires are the oracle's, cell by cell.  Maps that open with such cells, maps of
them alone and maps with one burnable cell out of the fixed-point range too.
"""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1701_03549_gb300 import fire, synth          # noqa: E402


def _spoil(land, rng):
    """No-data values of every kind in the water cells, the first row's cells
    among them."""
    land.veg[0, :7] = 0
    bad = np.array([np.nan, -9999.0, np.inf, 1e30, 777.0], np.float32)
    water = np.nonzero(land.veg == 0)
    for raster in (land.slope, land.aspect, land.wind):
        raster[water] = rng.choice(bad, water[0].size)
    return land


@pytest.mark.parametrize("cell", [False, True])
@pytest.mark.parametrize("wind", [None, 7])
@pytest.mark.parametrize("steep", [False, True])
def test_fires_match_the_oracle(wind, cell, steep):
    import oracle

    oracle.build()
    rng = np.random.default_rng(3)
    land = _spoil(synth.landscape(45, 70, seed=11, wind_seed=wind), rng)
    ign = synth.centre_ignition(land.veg)
    if steep:
        land.slope[tuple(np.argwhere(land.veg != 0)[700])] = 250.0
    p = np.array([synth.TRUTH_BETA, [0.3, -0.4, 0.5, 1.0, -0.5], [0.0] * 5,
                  [-0.2, 0.1, 64.0, -64.5, 130.0]])
    p = np.concatenate([p, rng.normal(0, 3, (12, 5))])
    n = len(p)
    seeds = np.arange(9, 9 + n, dtype=np.uint64)
    # the oracle reads the same map with plain values in the water
    clean = synth.Landscape(land.veg, land.elev, land.slope.copy(),
                            land.aspect.copy(), land.wind.copy())
    for raster in (clean.slope, clean.aspect, clean.wind):
        raster[land.veg == 0] = 0.0
    F = oracle.Features(clean)
    ctx = fire.Context(0)
    m = ctx.landscape_upload(land)
    res, bs = m.simulate_batch(p, np.tile(np.asarray(ign, np.int32), (n, 1)),
                               seeds, want_steps=True, cell_uniform=cell)
    for i in range(n):
        o, obs = F.simulate(p[i], ign, int(seeds[i]), mode=1 if cell else 0)
        assert np.array_equal(bs[i], obs), i
        for k in ("burnt", "steps", "status", "trials"):
            assert int(res[k][i]) == o[k], (i, k)
    assert np.unique(res["burnt"]).size > 5
    m.free()
    ctx.close()


def test_a_map_without_burnable_cells():
    ctx = fire.Context(0)
    land = synth.uniform_landscape(70, 300, veg_code=0)
    land.slope[:] = np.nan
    m = ctx.landscape_upload(land)
    args = [torch.tensor(a, device="cuda") for a in (
        np.zeros((2, 5)), np.array([[3, 4], [60, 299]], np.int32),
        np.array([1, 2], np.int64))]
    out = torch.zeros((2, 6), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    m.simulate_batch(*args, device=True, out=out, sync=True)
    # FIRE_STATUS_BAD_IGNITION, reported per simulation
    assert (fire.results_view(out)["status"] & 4 == 4).all()
    m.free()
    ctx.close()


@pytest.mark.parametrize("wind", [None, 7])
def test_speed_of_a_map_with_nodata_water(wind):
    """Runs alternate; the float-pair screen for the whole map, which one such
    water cell chose before, takes 1.3 times as long on this chain of steps."""
    ctx = fire.Context(0, torch.cuda.current_stream())
    lands = [synth.landscape(70, 90, seed=107, wind_seed=wind),
             _spoil(synth.landscape(70, 90, seed=107, wind_seed=wind),
                    np.random.default_rng(3))]
    lands[0].veg[0, :7] = 0
    maps = [ctx.landscape_upload(l) for l in lands]
    n = 8
    p = torch.tensor(synth.gauss_population(n, 3), device="cuda")
    g = torch.tensor(np.tile(np.asarray(
        synth.centre_ignition(lands[0].veg), np.int32), (n, 1)), device="cuda")
    s = torch.arange(5, 5 + n, device="cuda")
    out = [torch.zeros((n, 6), dtype=torch.int32, device="cuda")
           for _ in maps]
    best = [1e9, 1e9]
    for _ in range(40):
        for i, m in enumerate(maps):
            torch.cuda.synchronize()
            t = time.perf_counter()
            m.simulate_batch(p, g, s, device=True, out=out[i])
            torch.cuda.synchronize()
            best[i] = min(best[i], time.perf_counter() - t)
    assert torch.equal(out[0], out[1]) and int(out[0][:, 0].max()) > 1000
    assert best[1] < 1.12 * best[0], best
    for m in maps:
        m.free()
    ctx.close()
