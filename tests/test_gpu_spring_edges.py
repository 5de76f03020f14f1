"""GPU: SPRING calls off the common path (csrc/abi.cu, csrc/sample_kernel.cuh)."""
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


@pytest.mark.parametrize("nstrat", [0, 2])
@pytest.mark.parametrize("precision,ybits", [("fp64", 53), ("fp64", 24), ("fp32", 24)])
def test_no_positive_maximum_is_an_error_and_draws_nothing(gv, precision, ybits, nstrat):
    """Every weight zero (a transverse-momentum cut above the beam energy): no
    cube can be drawn.  The call answers ESTATE, also when it is the first to
    allocate the tables, and the context goes on with other parameters."""
    d = 8
    ncall = 20 * max(1, nstrat) ** d
    with gv.vegas_create(wl.RAMBO_BW, d, wl.rambo_params(2, ptmin=900.0), ncall=ncall, nstrat=nstrat,
                         precision=precision, ybits=ybits) as ctx:
        gv.bases_integrate(ctx, 1, 0.0, 1, 0.0)
        assert np.all(gv.vegas_get_cube_max(ctx) == 0.0)
        for n in (1, 5000):
            with pytest.raises(gv.VegasError) as e:
                gv.spring_generate(ctx, 0, n)
            assert e.value.status == gv.ESTATE
        gv.vegas_set_params(ctx, wl.rambo_params(2, ptmin=1.0, drmin=0.01))
        gv.bases_integrate(ctx, 1, 0.0, 1, 0.0)
        r = gv.spring_generate(ctx, 0, 5000)
        assert r["n_events"] > 0 and np.all((r["x"] >= 0) & (r["x"] <= 1)) and np.all(np.diff(r["trial"].astype(int)) > 0)
        gv.vegas_set_params(ctx, wl.rambo_params(2, ptmin=900.0))
        gv.bases_integrate(ctx, 1, 0.0, 1, 0.0)
        with pytest.raises(gv.VegasError) as e:
            gv.spring_generate(ctx, 0, 5000)
        assert e.value.status == gv.ESTATE
