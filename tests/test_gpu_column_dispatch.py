"""GPU: which per-bin sums a shape gets (csrc/abi.cu: columns or bucketed tiles),
on both sides of every line of the rule, and that either gives the oracle's sums:
the columns' memory (eight warps per SM), the least work beyond 50 bins for
kernels that know the dimension and for the others, and CTAs asked for by hand."""
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


def _check(gv, orc, d, N, ncall, columns, threads=None):
    params = np.concatenate([np.linspace(0.5, 1.5, d), np.linspace(0.3, 0.7, d)])
    with gv.vegas_create(wl.GENZ_CONTINUOUS, d, params, nbins=N, ncall=ncall, precision="fp32") as ctx:
        if threads:
            gv.vegas_set_launch(ctx, threads)
        assert (gv.vegas_get_tile(ctx)["cap"] == 0) == columns
        I, _ = gv.vegas_eval(ctx, 2)
        _, bins = gv.vegas_get_grid(ctx, bin_sums=True)
    cfg = orc.make_cfg(d, nbins=N, ncall=ncall, ybits=24)
    o = orc.iteration(cfg, orc.Integrand(wl.GENZ_CONTINUOUS, d, params), orc.uniform_grid(d, N), 2)
    # (positive weights: their sums are the scale of the FP32 form's bar, 1e-5)
    assert np.all(np.abs(bins[0] - o["S1"]) <= 1e-5 * o["S1"][0].sum())
    assert np.all(np.abs(bins[1] - o["S2"]) <= 1e-5 * o["S2"][0].sum())
    assert I == pytest.approx(o["I"], rel=1e-5)


@pytest.mark.parametrize("d,fits", [(1, 107), (2, 109), (8, 105), (16, 103), (20, 99), (32, 95)])
def test_memory_of_eight_warps(gv, orc, d, fits):
    ncall = 6_000_000 // 20 if d > 2 else 5000  # enough work for columns at each of these
    _check(gv, orc, d, fits, ncall, True)
    if d < 32:
        _check(gv, orc, d, fits + 1, ncall, False)
    else:  # buckets end at 2751 cells
        with pytest.raises(gv.VegasError) as e:
            _check(gv, orc, d, fits + 1, ncall, False)
        assert e.value.status == gv.EINVAL


@pytest.mark.parametrize("ncall,threads", [(1000, None), (1000, 64), (200_001, 64)])
def test_where_no_bucket_fits_columns_take_any_work(gv, orc, ncall, threads):
    _check(gv, orc, 32, 90, ncall, True, threads)


@pytest.mark.parametrize("d,N,least", [(4, 51, 500_000), (8, 64, 250_000), (16, 100, 125_000), (32, 51, 62_500),
                                       (7, 51, 857_143), (9, 80, 666_667), (20, 64, 100_000)])
def test_least_work_beyond_50_bins(gv, orc, d, N, least):
    _check(gv, orc, d, N, least, True)
    _check(gv, orc, d, N, least - 1, False)
    _check(gv, orc, d, 50, 1003, True)


@pytest.mark.parametrize("d,N,threads,columns", [(6, 51, None, False), (3, 100, None, False), (2, 100, None, True),
                                                 (8, 72, 64, True), (8, 128, 64, True), (8, 128, 128, True), (7, 200, 64, True),
                                                 (8, 50, 64, True), (8, 50, 512, True), (8, 72, 512, False)])
def test_dimensions_and_widths(gv, orc, d, N, threads, columns):
    _check(gv, orc, d, N, 70_001, columns, threads)
