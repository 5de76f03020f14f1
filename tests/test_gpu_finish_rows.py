"""GPU: the finishing kernel's reduction of the partial rows (csrc/finalize.cu)
around its thread counts, slices and loads in flight: bins on both sides of 64
and 128, row counts from one to several per thread."""
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


@pytest.mark.parametrize("precision,rel", [("fp64", 1e-12), ("fp32_acc64", 1e-5), ("fp32", 1e-5)])
@pytest.mark.parametrize("N", [64, 65, 85, 86, 128, 129, 160, 256])
@pytest.mark.parametrize("ncall", [200, 40_001, 300_007])
def test_bin_sums_over_all_rows(gv, orc, N, ncall, precision, rel):
    """S1, S2 of every bin of one pass against the oracle's (bars of the parity
    tests: 1e-12 of the weights' sum in FP64, 1e-5 with FP32 weights), in narrow
    CTAs too, which leave several times the rows."""
    d = 2
    params = np.concatenate([np.linspace(0.5, 1.5, d), np.linspace(0.3, 0.7, d)])
    o = orc.iteration(orc.make_cfg(d, nbins=N, ncall=ncall, ybits=24), orc.Integrand(wl.GENZ_CONTINUOUS, d, params),
                      orc.uniform_grid(d, N), 0)
    with gv.vegas_create(wl.GENZ_CONTINUOUS, d, params, nbins=N, ncall=ncall, precision=precision, ybits=24) as ctx:
        for threads in (None, 64, 256):
            if threads:
                gv.vegas_set_launch(ctx, threads)
            I, _ = gv.vegas_eval(ctx, 0)
            _, bins = gv.vegas_get_grid(ctx, bin_sums=True)
            assert np.all(np.abs(bins[0] - o["S1"]) <= rel * o["S1"][0].sum())
            assert np.all(np.abs(bins[1] - o["S2"]) <= rel * o["S2"][0].sum())
            assert I == pytest.approx(o["I"], rel=rel)
