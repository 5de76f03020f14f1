"""GPU: the batch's automatic rounds per item and its autotuner (csrc/batch.cu)."""
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


def _ms(gv, b):
    gv.vegas_batch_profile(b, 2)
    return min(sum(gv.vegas_batch_profile(b, 4).values()) for _ in range(6))


CASES = [(64, 4, 14, 19, 50), (64, 4, 14, 19, 100), (64, 16, 14, 18, 100), (16, 16, 10, 13, 50)]


@pytest.mark.parametrize("count,dmax,lo,hi,nbins", CASES)
def test_automatic_rounds_beat_buckets(gv, count, dmax, lo, hi, nbins):
    """The automatic shape against bucketed tiles of 32 rounds (which these
    batches had before columns), low dimensions above all, whose items are short
    for their folds; measured 0.55 to 0.97 of them."""
    ins = wl.genz_batch(count, seed=5, dmax=dmax, log2n_min=lo, log2n_max=hi)
    with gv.vegas_batch_create(ins, nbins=nbins, seed=1, precision="fp32", ybits=24) as b:
        assert gv.vegas_batch_get_tile(b)["cap"] == 0
        r0 = gv.vegas_batch_iterate(b, 1, refine=False)
        auto = _ms(gv, b)
        gv.vegas_batch_set_tile(b, 2)
        gv.vegas_batch_set_launch(b, 256, 32)
        assert auto <= 1.02 * _ms(gv, b)
        gv.vegas_batch_reset(b)
        r1 = gv.vegas_batch_iterate(b, 1, refine=False)
        np.testing.assert_allclose([r["I"] for r in r0], [r["I"] for r in r1], rtol=2e-5, atol=1e-7)


@pytest.mark.parametrize("count,dmax,lo,hi,nbins", CASES)
@pytest.mark.parametrize("threads", [None, 128])
def test_tuning_does_not_slow_a_batch(gv, count, dmax, lo, hi, nbins, threads):
    """Whatever shape was set before: at 100 bins with 128 threads columns do not
    fit, with 256 they do, and both are tried."""
    ins = wl.genz_batch(count, seed=5, dmax=dmax, log2n_min=lo, log2n_max=hi)
    with gv.vegas_batch_create(ins, nbins=nbins, seed=1, precision="fp32", ybits=24) as b:
        auto = _ms(gv, b)
        if threads:
            gv.vegas_batch_set_launch(b, threads, 32)
        tuned = gv.vegas_batch_autotune(b)
        shape = gv.vegas_batch_get_launch(b)
        assert (tuned["threads"], tuned["rounds"]) == (shape["threads"], shape["rounds"])
        assert _ms(gv, b) <= 1.03 * auto
