"""GPU: a change of launch shape whose buffers cannot be allocated.  The
allocation is failed on the host (vegas_fail_alloc_after); the context must go
on in its previous shape, with the graphs and buffers it had."""
from __future__ import annotations

import pytest

from paper_1010_2107_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gv():
    from paper_1010_2107_gb300 import gvegas
    gvegas.lib()
    return gvegas


@pytest.mark.parametrize("change", ["launch", "tile"])
def test_failed_shape_change_keeps_the_context(gv, change):
    """Few hypercubes, so that partial rows, totals and the cubes' parts all grow
    with narrower CTAs: each growth fails in turn, before anything was given up
    (no further allocation in that call), and the cached graphs, frozen passes
    included, then give what an untouched context gives."""
    d = 2
    kw = dict(ncall=16 * 16384, nstrat=4, precision="fp32", seed=9)
    mk = lambda: gv.vegas_create(wl.DOUBLE_GAUSSIAN, d, wl.double_gaussian_params(w=0.2), **kw)

    def calls(ctx):
        out = [gv.bases_integrate(ctx, 2, 0.0, 3, 0.0), gv.vegas_eval(ctx, 1), gv.vegas_get_grid(ctx).tolist()]
        gv.vegas_reset_grid(ctx)
        gv.vegas_set_iteration(ctx, 0)
        return out

    with mk() as ref, mk() as ctx:
        want = calls(ref)
        assert calls(ctx) == want  # and captures the graphs
        shape = gv.vegas_get_launch(ctx), gv.vegas_get_tile(ctx)
        failed = 0
        for j in range(8):
            n0 = gv.vegas_alloc_count()
            gv.vegas_fail_alloc_after(j)
            try:
                gv.vegas_set_launch(ctx, 128) if change == "launch" else gv.vegas_set_tile(ctx, 1)
                break
            except gv.VegasError as e:
                assert e.status == gv.ENOMEM
            finally:
                gv.vegas_fail_alloc_after(-1)
            failed += 1
            assert gv.vegas_alloc_count() - n0 == j + 1
            assert (gv.vegas_get_launch(ctx), gv.vegas_get_tile(ctx)) == shape
            assert calls(ctx) == want
        assert failed == (3 if change == "launch" else failed) and failed >= 1
        assert (gv.vegas_get_launch(ctx), gv.vegas_get_tile(ctx)) != shape
        r, w = gv.bases_integrate(ctx, 2, 0.0, 3, 0.0)[0], want[0][0]
        assert r["I"] == pytest.approx(w["I"], rel=1e-5)


@pytest.mark.parametrize("change", ["launch", "tile"])
@pytest.mark.parametrize("precision,ybits", [("fp32", 24), ("fp64", 53)])
def test_failed_shape_change_keeps_the_batch(gv, precision, ybits, change):
    """As above for a batch: items and partial rows grow with fewer rounds per
    item (or, where a tile brings buckets with fewer rounds, with the tile);
    shape, graphs, frozen passes and results stay."""
    insts = wl.genz_batch(6, seed=5, log2n_min=17, log2n_max=18)
    if change == "tile":  # work enough for 128 rounds with columns
        insts = wl.genz_batch(40, seed=5, log2n_min=22, log2n_max=22) if precision == "fp32" else insts
    mk = lambda: gv.vegas_batch_create(insts, nbins=50, seed=1, precision=precision, ybits=ybits)

    def calls(b):
        gv.vegas_batch_reset(b)
        return [r["I"] for r in gv.vegas_batch_iterate(b, 2, refine=False)]

    with mk() as b:
        want = calls(b)
        shape = gv.vegas_batch_get_launch(b), gv.vegas_batch_get_tile(b)
        failed = 0
        for j in range(4):
            n0 = gv.vegas_alloc_count()
            gv.vegas_fail_alloc_after(j)
            try:
                gv.vegas_batch_set_launch(b, 64, 4) if change == "launch" else gv.vegas_batch_set_tile(b, 2)
                break
            except gv.VegasError as e:
                assert e.status == gv.ENOMEM
            finally:
                gv.vegas_fail_alloc_after(-1)
            failed += 1
            assert gv.vegas_alloc_count() - n0 == j + 1
            assert (gv.vegas_batch_get_launch(b), gv.vegas_batch_get_tile(b)) == shape
            assert calls(b) == want
        if change == "launch":
            assert failed == 2 and gv.vegas_batch_get_launch(b)["threads"] == 64
        assert calls(b) == pytest.approx(want, rel=1e-5)
