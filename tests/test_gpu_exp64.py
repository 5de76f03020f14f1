"""GPU: exp64 (csrc/common.cuh), the FP64 integrands' exponential, against
30-digit values: over its range, around the multiples of ln 2 / 64 where the
reduction turns, on both sides of 708 where the library takes over, and at zeros,
underflow, infinities and NaN.  Reached through a user integrand, whose source is
compiled with the kernels' headers."""
from __future__ import annotations

import decimal
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = """
template <typename T>
__device__ T vegas_user_f(const T* x, int d, const T* p) { return T(gv::exp64(p[1] == 0.0 ? p[0] : fma(p[1], x[0], p[0]))); }
"""


@pytest.fixture(scope="module")
def gv():
    from paper_1010_2107_gb300 import gvegas
    gvegas.lib()
    return gvegas


@pytest.fixture(scope="module")
def ctx(gv):
    with gv.vegas_create_user(SRC, 1, [0.0, 1.0], nbins=2, ncall=4096) as c:
        yield c


def _ulps(args, got):
    """Errors in units in the last place of the exact values."""
    with decimal.localcontext(decimal.Context(prec=40)):
        out = []
        for a, g in zip(args, got):
            e = decimal.Decimal(float(a)).exp()
            u = decimal.Decimal(math.ulp(float(e)))
            out.append(abs(float((decimal.Decimal(float(g)) - e) / u)))
    return np.array(out)


@pytest.mark.parametrize("lo,hi", [(-707.9, 707.9), (-30.0, 0.0), (-1e-3, 1e-3), (-1e-300, 1e-300)])
def test_over_the_range(gv, ctx, lo, hi):
    """Below 0.84 ulp: 0.5 from the last rounding, at most 0.31 from the
    polynomial's end, the rest from its roundings."""
    gv.vegas_set_params(ctx, [lo, hi - lo])
    s = gv.vegas_sample_dump(ctx, 0, np.arange(4096))
    # the argument as the kernel forms it: rounded once
    x = s["x"][:, 0]
    with decimal.localcontext(decimal.Context(prec=60)):
        args = np.array([float(decimal.Decimal(lo) + decimal.Decimal(hi - lo) * decimal.Decimal(float(v))) for v in x])
    assert np.max(_ulps(args, s["f"])) <= 0.84


def _at(gv, ctx, a):
    gv.vegas_set_params(ctx, [a, 0.0])
    return float(gv.vegas_sample_dump(ctx, 0, np.arange(1))["f"][0])


def test_where_the_reduction_turns(gv, ctx):
    step = math.log(2.0) / 64
    args = []
    for n in (-65000, -4097, -64, -1, 0, 1, 31, 32, 63, 64, 65, 4096, 65000):
        for c in (n * step, (n + 0.5) * step):
            args += [c, np.nextafter(c, -np.inf), np.nextafter(c, np.inf)]
    assert np.max(_ulps(args, [_at(gv, ctx, float(a)) for a in args])) <= 0.84


def test_edges(gv, ctx):
    assert _at(gv, ctx, 0.0) == 1.0 and _at(gv, ctx, -0.0) == 1.0
    assert _at(gv, ctx, math.inf) == math.inf and _at(gv, ctx, -math.inf) == 0.0
    assert math.isnan(_at(gv, ctx, math.nan))
    assert _at(gv, ctx, 710.0) == math.inf and _at(gv, ctx, -746.0) == 0.0
    # both sides of the hand-over; the library's own bound is 1 ulp
    for c in (708.0, -708.0):
        args = [np.nextafter(c, 0.0), c, np.nextafter(c, 2 * c), 1.001 * c]
        assert np.max(_ulps(args, [_at(gv, ctx, float(a)) for a in args])) <= 1.0
    # subnormal results: an absolute error of one smallest number
    for a in (-708.5, -720.0, -740.0, -745.0):
        with decimal.localcontext(decimal.Context(prec=40)):
            e = decimal.Decimal(a).exp()
            assert abs(decimal.Decimal(_at(gv, ctx, a)) - e) <= decimal.Decimal(5e-324) * 2 + e * decimal.Decimal(2.3e-16)
