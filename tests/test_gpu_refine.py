"""GPU: the grid optimisation with 64-bit integer sums (csrc/refine.cuh)
against the oracle's, over bin counts, damping exponents and sums of squares
of very different sizes."""
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


@pytest.mark.parametrize("alpha", [0.0, 0.4, 1.5, 6.0, 20.0])
@pytest.mark.parametrize("N", [2, 3, 31, 32, 33, 64, 65, 129, 256])
@pytest.mark.parametrize("a", [1e-8, 3.0, 60.0])
def test_refined_edges_match_the_oracle(gv, orc, N, alpha, a):
    """One iteration's edges from the GPU's own bin sums; the bar is that of
    the loop's parity tests (edges within 1e-13 of the unit axis), for weights
    that are flat (a = 1e-8), peaked, and spread over 1e-300 .. 1 (a = 60)."""
    d = 2
    params = np.concatenate([np.full(d, a), np.full(d, 0.37)])
    with gv.vegas_create(wl.GENZ_GAUSSIAN, d, params, nbins=N, ncall=5003, alpha=alpha) as ctx:
        e0 = gv.vegas_get_grid(ctx)
        gv.vegas_iterate(ctx, 1)
        edges, bins = gv.vegas_get_grid(ctx, bin_sums=True)
    ref = orc.refine(bins[1], e0, alpha)
    assert np.max(np.abs(edges - ref)) <= 1e-13
    assert np.all(np.diff(edges, axis=1) >= 0) and np.all(edges[:, 0] == 0) and np.all(edges[:, -1] == 1)


def test_batched_refinement_of_many_bins(gv, orc):
    """More bins than 128: the batch's finalisation gives one thread to each."""
    d, N = 3, 200
    ins = [dict(kind=wl.GENZ_GAUSSIAN, ndim=d, ncall=20000, params=wl.genz_gaussian_params(d, a=4.0))]
    with gv.vegas_batch_create(ins, nbins=N, precision="fp64") as b:
        e0 = gv.vegas_batch_get_grid(b, 0)
        gv.vegas_batch_iterate(b, 1)
        edges, bins = gv.vegas_batch_get_grid(b, 0, bin_sums=True)
    assert np.max(np.abs(edges - orc.refine(bins[1], e0))) <= 1e-13


@pytest.mark.parametrize("scale,moves", [(1e152, True), (1e153, False)])
def test_sums_that_overflow_together_leave_the_grid(gv, orc, scale, moves):
    """Every bin's sum of squares finite, their total past the largest double:
    the axis is left as it is, as the oracle does; a tenth of it still refines."""
    src = """
template <typename T>
__device__ T vegas_user_f(const T* x, int d, const T* p) { return x[0] < T(0.5) ? p[0] : T(0.1) * p[0]; }
"""
    with gv.vegas_create_user(src, 1, [scale], nbins=50, ncall=2000) as ctx:
        e0 = gv.vegas_get_grid(ctx)
        gv.vegas_iterate(ctx, 1)
        edges, bins = gv.vegas_get_grid(ctx, bin_sums=True)
    assert np.all(np.isfinite(bins[1]))
    ref = orc.refine(bins[1], e0)
    assert np.array_equal(ref, e0) == (not moves)
    assert np.max(np.abs(edges - ref)) <= (1e-13 if moves else 0.0)
