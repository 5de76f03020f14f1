"""GPU: the column histogram of the FP32 form (csrc/col_hist.cuh) against the
oracle, at the sizes where its lane mapping, hand-over and folds can go wrong:
every points-per-step count (d = 1..32), exact and run-time dimensions, bin
counts up to the largest the columns hold, point counts below one hand-over,
and columns folded several times."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1010_2107_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gv():
    from paper_1010_2107_gb300 import gvegas
    gvegas.lib()
    return gvegas


def _check(gv, orc, ctx, cfg, fn, d, N, ncall):
    """Bins and estimate of one evaluation pass within 1e-5 of sum |w| (the FP32
    form's bar: a weight's rounding is below 1e-5 of itself)."""
    I, _ = gv.vegas_eval(ctx, 2)
    _, bins = gv.vegas_get_grid(ctx, bin_sums=True)
    o = orc.iteration(cfg, fn, orc.uniform_grid(d, N), 2)
    p = orc.sample_batch(cfg, orc.uniform_grid(d, N), 2, np.arange(ncall))
    w = np.abs(orc.integrand(fn, p["x"]) * p["jac"])
    assert np.all(np.abs(bins[0] - o["S1"]) <= 1e-5 * w.sum())
    assert np.all(np.abs(bins[1] - o["S2"]) <= 1e-5 * (w ** 2).sum())
    # every axis holds every point once: its sums are the totals
    np.testing.assert_allclose(bins[0].sum(1), bins[0].sum(1)[0], rtol=1e-6)
    assert abs(I - o["I"]) <= 1e-5 * w.mean()


@pytest.mark.parametrize("ncall", [2, 65, 20011])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 13, 16, 17, 20, 24, 31, 32])
def test_columns_every_points_per_step(gv, orc, d, ncall):
    params = np.concatenate([np.linspace(0.5, 1.5, d), np.linspace(0.3, 0.7, d)])
    N = {1: 2, 2: 100, 5: 37}.get(d, 50)
    with gv.vegas_create(wl.GENZ_CONTINUOUS, d, params, nbins=N, ncall=ncall, precision="fp32") as ctx:
        assert gv.vegas_get_tile(ctx)["cap"] == 0  # columns, not buckets
        cfg = orc.make_cfg(d, nbins=N, ncall=ncall, ybits=24)
        _check(gv, orc, ctx, cfg, orc.Integrand(wl.GENZ_CONTINUOUS, d, params), d, N, ncall)


@pytest.mark.parametrize("d,nstrat,nc", [(3, 2, 500), (4, 4, 3), (7, 2, 33), (8, 4, 8)])
def test_columns_stratified(gv, orc, d, nstrat, nc):
    params = np.concatenate([np.linspace(0.5, 1.5, d), np.linspace(0.3, 0.7, d)])
    ncall = nstrat ** d * nc
    with gv.vegas_create(wl.GENZ_CONTINUOUS, d, params, ncall=ncall, nstrat=nstrat, precision="fp32") as ctx:
        assert gv.vegas_get_tile(ctx)["cap"] == 0
        cfg = orc.make_cfg(d, ncall=ncall, nstrat=nstrat, ybits=24)
        _check(gv, orc, ctx, cfg, orc.Integrand(wl.GENZ_CONTINUOUS, d, params), d, 50, ncall)


@pytest.mark.parametrize("d", [7, 16])
def test_columns_folded_many_times(gv, orc, d):
    """64-thread CTAs, one per SM: each lane's column takes several times the
    additions it may hold between folds."""
    params = np.concatenate([np.linspace(0.5, 1.5, d), np.linspace(0.3, 0.7, d)])
    ncall = 1_500_001
    with gv.vegas_create(wl.GENZ_CONTINUOUS, d, params, ncall=ncall, precision="fp32") as ctx:
        gv.vegas_set_launch(ctx, 64, 1)
        assert gv.vegas_get_tile(ctx)["cap"] == 0
        cfg = orc.make_cfg(d, ncall=ncall, ybits=24)
        _check(gv, orc, ctx, cfg, orc.Integrand(wl.GENZ_CONTINUOUS, d, params), d, 50, ncall)
