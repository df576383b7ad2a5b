"""Lengths that the kernels cannot compute with are refused by ct_geom_create on
the host: infinite ones and ones past single precision, and a pixel pitch so
small that the back-projector's row margin passes what an int holds.  An
infinite pitch once reached the projector as a NaN row coordinate.  No GPU is
needed: the checks come before any CUDA call.
"""
import ctypes

import pytest


@pytest.fixture(scope="module")
def libct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct
    return ct


def create(libct, **kw):
    base = dict(kind=1, nx=16, ny=16, nz=16, voxel_mm=1.0, n_views=8, angle_start_rad=0.0,
                angle_span_rad=6.283185307179586, nu=25, nv=16, du_mm=1.5, dv_mm=1.5, sod_mm=500.0,
                sdd_mm=1000.0, vol_dtype=0, sino_dtype=0)
    base.update(kw)
    h = ctypes.c_void_p()
    d = libct.ct_geom_desc(**base)
    st = libct.lib().ct_geom_create(ctypes.byref(d), ctypes.byref(h))
    if h.value:
        libct.lib().ct_geom_destroy(h)
    return st


FLAT = dict(kind=0, nz=1, nv=1)


@pytest.mark.parametrize("value", [float("inf"), float("nan"), 1e39])
@pytest.mark.parametrize("bad", [("du_mm", {}), ("dv_mm", {}), ("sdd_mm", {}), ("sod_mm", {}), ("voxel_mm", {}),
                                 ("du_mm", FLAT), ("voxel_mm", FLAT)], ids=lambda b: b[0] + ("_2d" if b[1] else ""))
def test_lengths_outside_single_precision_are_refused(libct, bad, value):
    assert create(libct, **{bad[0]: value}, **bad[1]) == libct.CT_EINVAL
    assert libct.lib().ct_last_error()


@pytest.mark.parametrize("dv", [1e-9, 1e-12, 1e-30])
def test_row_margin_past_an_int_is_refused(libct, dv):
    assert create(libct, dv_mm=dv) == libct.CT_EINVAL
    assert b"too large" in libct.lib().ct_last_error()


def test_lengths_that_a_2d_scan_does_not_use_are_not_looked_at(libct):
    for kw in (dict(sod_mm=float("inf")), dict(sdd_mm=float("nan")), dict(dv_mm=float("inf"))):
        assert create(libct, **FLAT, **kw) != libct.CT_EINVAL
