"""GPU: frozen passes of the smallest tables.  Their shared memory, one table and
the groups' sums, exceeds what the refining pass of the same integrator asks for
(few bins, few points per tile), so each kernel's launch limit has to cover the
frozen shape as well as the refining one (csrc/abi.cu configure_launch)."""
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


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("ybits", [24, 53])
@pytest.mark.parametrize("nbins,nstrat,ncall", [(2, 6, 423_672), (2, 0, 100_003), (3, 5, 40_000), (2, 0, 64)])
def test_frozen_passes(gv, precision, ybits, nbins, nstrat, ncall):
    with gv.vegas_create(wl.GENZ_PRODUCT_PEAK, 1, np.array([1.0, 0.5]), nbins=nbins, nstrat=nstrat, ncall=ncall,
                         precision=precision, ybits=ybits) as ctx:
        r = gv.vegas_iterate(ctx, 3, refine=False)
    # 1 / (1 + (x - 1/2)^2) over [0, 1] is 2 atan(1/2)
    exact = 2.0 * np.arctan(0.5)
    assert abs(r["I"] - exact) <= 6.0 * r["sigma"] + 1e-6
