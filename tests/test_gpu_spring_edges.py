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


def _spring_into(gv, ctx, n, x_ptr, t_ptr):
    """spring_generate through the C ABI with raw addresses (None: not asked for)."""
    import ctypes
    k, ov, npos = ctypes.c_uint32(), ctypes.c_uint32(), ctypes.c_uint32()
    st = gv.lib().spring_generate(
        ctx.handle, 0, n, None if x_ptr is None else ctypes.cast(x_ptr, ctypes.POINTER(ctypes.c_double)),
        None if t_ptr is None else ctypes.cast(t_ptr, ctypes.POINTER(ctypes.c_uint64)),
        ctypes.byref(k), ctypes.byref(ov), ctypes.byref(npos))
    assert st == gv.OK
    return k.value, ov.value, npos.value


def _buffer(nbytes, kind):
    """A host byte buffer filled with 0xA5 and the offset to use in it."""
    import torch
    off = {"pageable": 16, "pinned": 16, "pinned-odd": 20, "pageable-odd": 3}[kind]
    b = torch.empty(nbytes + off + 64, dtype=torch.uint8, pin_memory=kind.startswith("pinned"))
    b.fill_(0xA5)
    return b, off


@pytest.mark.parametrize("kx,kt", [("pinned", "pinned"), ("pageable", "pinned"), ("pinned", "pageable"),
                                   ("pinned-odd", "pinned"), ("pinned", "pinned-odd"),
                                   ("pageable-odd", "pageable-odd"), ("pinned", None), (None, "pinned"),
                                   ("pageable", None), (None, "pageable")])
def test_events_do_not_depend_on_the_callers_buffers(gv, kx, kt):
    """Pinned buffers (written by the GPU), pageable ones (copied), one of each,
    one alone, and addresses off the elements' alignment (copied): the same
    events and counts byte for byte, and nothing past them, for one trial, sizes
    around a chunk of 4096, and a larger call after smaller ones."""
    d = 4
    with gv.vegas_create(wl.DOUBLE_GAUSSIAN, d, wl.double_gaussian_params(w=0.15), ncall=4 ** d * 32, nstrat=4,
                         precision="fp32") as ctx:
        gv.bases_integrate(ctx, 2, 0.0, 2, 0.0)
        for n in (1, 4095, 4097, 30011):
            ref = gv.spring_generate(ctx, 0, n)
            m = ref["n_events"]
            assert n == 1 or 0 < m < n
            bx, ox = _buffer(8 * d * n, kx) if kx else (None, 0)
            bt, ot = _buffer(8 * n, kt) if kt else (None, 0)
            got = _spring_into(gv, ctx, n, bx.data_ptr() + ox if kx else None, bt.data_ptr() + ot if kt else None)
            assert got == (m, ref["overflow"], ref["nonpos"])
            for b, o, want in ((bx, ox, ref["x"]), (bt, ot, ref["trial"])):
                if b is not None:
                    raw = np.ascontiguousarray(want).tobytes()
                    assert b.numpy()[o:o + len(raw)].tobytes() == raw
                    assert np.all(b.numpy()[:o] == 0xA5) and np.all(b.numpy()[o + len(raw):] == 0xA5)


def test_every_failed_allocation_of_the_first_call(gv):
    """Each allocation of a context's first SPRING call fails in turn (on the
    host), on one context: every call answers ENOMEM, none leaves tables half
    there, and the first that gets all of them draws the events of an untouched
    context; so does a larger call after its own failures."""
    d = 3
    kw = dict(ncall=4 ** d * 50, nstrat=4, precision="fp64", ybits=24, seed=3)
    mk = lambda: gv.vegas_create(wl.GENZ_GAUSSIAN, d, wl.genz_gaussian_params(d, a=4.0), **kw)
    with mk() as ref, mk() as ctx:
        for c in (ref, ctx):  # no refining iteration: the same grid and maxima bit for bit in both
            gv.bases_integrate(c, 0, 0.0, 2, 0.0)
        for n, least in ((4096, 10), (9000, 3)):
            want, failed = gv.spring_generate(ref, 0, n), 0
            for j in range(32):
                gv.vegas_fail_alloc_after(j)
                try:
                    got = gv.spring_generate(ctx, 0, n)
                    break
                except gv.VegasError as e:
                    assert e.status == gv.ENOMEM
                    failed += 1
                finally:
                    gv.vegas_fail_alloc_after(-1)
            assert failed >= least
            assert got["n_events"] == want["n_events"] > 0
            np.testing.assert_array_equal(got["trial"], want["trial"])
            np.testing.assert_array_equal(got["x"], want["x"])
