"""GPU: the batch's column-histogram kernels (csrc/batch_dim.cuh) against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gv():
    from paper_1010_2107_gb300 import gvegas
    gvegas.lib()
    return gvegas


@pytest.mark.parametrize("nbins,threads,rounds", [(50, 256, 128), (64, 256, 8), (100, 256, 3), (100, 128, 3), (2, 64, 40)])
def test_column_histogram_kernels_of_every_dimension(gv, orc, nbins, threads, rounds):
    """The batch's automatic kernels (lane-owned columns) of all sixteen
    dimensions: one CTA and two per SM, items of many hand-overs (folds within
    an item) and of a few, ragged point counts, every family.  Bars as for the
    bucketed kernels: 1e-5 of the sums of |w| and w^2."""
    kinds = [0, 1, 2, 3, 4, 6, 7]
    ins = []
    for d in range(1, 17):
        k = kinds[d % 7]
        a, u = np.linspace(0.5, 1.5, d), np.linspace(0.3, 0.7, d)
        p = {2: a, 3: np.r_[a, 0.2], 4: np.array([1 / 3, 2 / 3, 0.3]), 7: np.r_[a, u[:2]]}.get(k, np.r_[a, u])
        ins.append(dict(kind=k, ndim=d, ncall=40_009 + 100 * d, params=p))
    with gv.vegas_batch_create(ins, nbins=nbins) as b:
        gv.vegas_batch_set_launch(b, threads, rounds)
        # (at 100 bins CTAs of four warps leave fewer than eight per SM: buckets)
        assert (gv.vegas_batch_get_tile(b)["cap"] == 0) == ((nbins, threads) != (100, 128))
        r = gv.vegas_batch_iterate(b, 1)
        got = [gv.vegas_batch_get_grid(b, i, bin_sums=True)[1] for i in range(len(ins))]
    for i, q in enumerate(ins):
        d = q["ndim"]
        cfg = orc.make_cfg(d, nbins=nbins, ncall=q["ncall"], ybits=24, instance=i)
        fn = orc.Integrand(q["kind"], d, q["params"])
        o = orc.iteration(cfg, fn, orc.uniform_grid(d, nbins), 0)
        pts = orc.sample_batch(cfg, orc.uniform_grid(d, nbins), 0, np.arange(q["ncall"]))
        w = np.abs(orc.integrand(fn, pts["x"]) * pts["jac"])
        assert abs(r[i]["I"] - o["I"]) <= 1e-5 * w.mean(), i
        assert np.all(np.abs(got[i][0] - o["S1"]) <= 1e-5 * w.sum()), i
        assert np.all(np.abs(got[i][1] - o["S2"]) <= 1e-5 * (w ** 2).sum()), i
