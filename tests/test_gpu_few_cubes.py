"""GPU: hypercubes shared by several groups of lanes (few cubes with many
points) and frozen-grid iterations that share one launch, against the oracle
and against the same iterations run one by one."""
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


def _params(d):
    return np.concatenate([np.linspace(2.0, 4.0, d), np.linspace(0.3, 0.7, d)])


# few cubes, cubes of a ragged number of points, a count that is no power of two, one of many cubes
SHAPES = [(1, 2, 40_001), (2, 2, 5003), (2, 3, 1001), (3, 6, 500), (4, 5, 7), (4, 8, 33)]


@pytest.mark.parametrize("d,g,nc", SHAPES)
@pytest.mark.parametrize("precision", ["fp64", "fp32_acc64", "fp32"])
def test_cubes_in_parts_match_the_oracle(gv, orc, d, g, nc, precision):
    """Estimate, variance, bins and cube sums of an evaluation pass (with the
    histogram) and of a frozen-grid iteration (without).  Bars: FP64 1e-12 of
    the sums; FP32 1e-5, its weights' rounding (the variance, a difference of
    sums, twice as much of the mean square)."""
    ncall, tol = g ** d * nc, 1e-12 if precision == "fp64" else 1e-5
    with gv.vegas_create(wl.GENZ_GAUSSIAN, d, _params(d), ncall=ncall, nstrat=g, precision=precision, ybits=24) as ctx:
        cfg = orc.make_cfg(d, ncall=ncall, nstrat=g, ybits=24)
        fn = orc.Integrand(wl.GENZ_GAUSSIAN, d, _params(d))
        o = orc.iteration(cfg, fn, orc.uniform_grid(d, 50), 0)
        p = orc.sample_batch(cfg, orc.uniform_grid(d, 50), 0, np.arange(ncall))
        w = np.abs(orc.integrand(fn, p["x"]) * p["jac"])
        I, var = gv.vegas_eval(ctx, 0)
        _, bins = gv.vegas_get_grid(ctx, bin_sums=True)
        cubes = gv.vegas_get_cube_sums(ctx)
        gv.vegas_iterate(ctx, 1, refine=False)
        hist, frozen_cubes = gv.vegas_get_history(ctx), gv.vegas_get_cube_sums(ctx)
        gv.vegas_set_iteration(ctx, 0)
        gv.bases_integrate(ctx, 0, 0.0, 1, 0.0)
        cmax = gv.vegas_get_cube_max(ctx)
    ref = w.reshape(-1, nc)
    for got in (cubes, frozen_cubes):
        np.testing.assert_allclose(got[:, 0], ref.sum(1), rtol=tol, atol=tol * ref.sum(1).max())
        np.testing.assert_allclose(got[:, 1], (ref ** 2).sum(1), rtol=2 * tol, atol=tol * (ref ** 2).sum(1).max())
    np.testing.assert_allclose(cmax, ref.max(1), rtol=tol, atol=tol * ref.max())
    vtol = 2 * tol * (w ** 2).mean() / ncall + 2 * tol * o["var"]
    for got_I, got_var in ((I, var), hist[0]):
        assert abs(got_I - o["I"]) <= tol * w.mean()
        assert abs(got_var - o["var"]) <= vtol
    assert np.all(np.abs(bins[0] - o["S1"]) <= tol * w.sum())
    assert np.all(np.abs(bins[1] - o["S2"]) <= tol * (w ** 2).sum())


@pytest.mark.parametrize("nstrat,ncall", [(0, 50_003), (0, 3_000_017), (2, 8 * 4001), (16, 4096 * 200)])
@pytest.mark.parametrize("precision", ["fp64", "fp32_acc64", "fp32"])
def test_frozen_iterations_in_one_launch_equal_single_ones(gv, precision, nstrat, ncall):
    """Eleven frozen-grid iterations in one call (launches of eight and three)
    and one by one: the same estimates bit for bit, the last one's cube sums,
    and the same maxima as BASES's integration phase records."""
    d, n = 3, 11
    with gv.vegas_create(wl.GENZ_GAUSSIAN, d, _params(d), ncall=ncall, nstrat=nstrat, precision=precision) as ctx:
        gv.vegas_iterate(ctx, n, refine=False)
        together = gv.vegas_get_history(ctx)
        r = gv.vegas_iterate(ctx, 0)
        cubes = gv.vegas_get_cube_sums(ctx) if nstrat else None
        gv.vegas_reset_results(ctx)
        gv.vegas_set_iteration(ctx, 0)
        for _ in range(n):
            gv.vegas_iterate(ctx, 1, refine=False, result=False)
        single = gv.vegas_get_history(ctx)
        s = gv.vegas_iterate(ctx, 0)
        assert np.array_equal(together, single)
        assert r == s and r["iters_done"] == n and r["samples"] == n * ncall
        if nstrat:
            assert np.array_equal(cubes, gv.vegas_get_cube_sums(ctx))
        gv.vegas_set_iteration(ctx, 0)
        gv.bases_integrate(ctx, 0, 0.0, n, 0.0)
        assert np.array_equal(gv.vegas_get_history(ctx), single)
        cmax = gv.vegas_get_cube_max(ctx)
        gv.vegas_set_iteration(ctx, 0)  # an ACC target: one iteration per launch
        out, _ = gv.bases_integrate(ctx, 0, 0.0, n, 1e-30)
        assert out["iters_done"] == n and np.array_equal(gv.vegas_get_history(ctx), single)
        assert np.array_equal(gv.vegas_get_cube_max(ctx), cmax)
