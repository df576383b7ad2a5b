"""The ramp filter's longest rows: the last lengths of each transform against the
FP64 oracle on single rows (relative L2 <= 1e-5, as for every operator), and one
column more than it takes, which is refused with a message by every call that
filters, while the calls that do not filter run.
"""
import math

import numpy as np
import pytest
import torch

import ct_inputs as ci
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct as _ct
    return _ct


def par2d(nu, views=3):
    return ci.Geometry(name="par2d_%d" % nu, kind=ci.PARALLEL_2D, nx=20, ny=21, nz=1, vox=1.0, n_views=views, ang0=0.1,
                       span=math.pi, nu=nu, nv=1, du=1.0, dv=1.0)


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("nu", [1024, 1025, 1536, 1537, 2048])
def test_long_rows(ct, nu, transpose):
    spec = par2d(nu)
    y = ci.random_vector(spec.m, seed=87).astype(np.float32).reshape(spec.sino_shape)
    f = ct.ramp_F(ct.Geometry.from_spec(spec), torch.from_numpy(y).cuda(), transpose=transpose).double().cpu().numpy()
    ref = (oracle.ramp_Ft if transpose else oracle.ramp_F)(spec, y.astype(np.float64)).reshape(f.shape)
    assert np.linalg.norm(f - ref) <= 1e-5 * np.linalg.norm(ref)


def test_longer_rows_are_refused_where_they_would_be_filtered(ct):
    spec = par2d(2049)
    g = ct.Geometry.from_spec(spec)
    x, y = torch.rand(spec.vol_shape, device="cuda"), torch.rand(spec.sino_shape, device="cuda")
    xo, yo, opts = torch.empty_like(x), torch.empty_like(y), ct.make_opts(b_kind="fbp")
    state = ct.GmresState(g, 2, "device", opts)
    for call in (lambda: ct.ct_ramp_F(g, y, yo), lambda: ct.ct_backproject_B(g, y, xo, "fbp"),
                 lambda: ct.ct_adjoint_Bt(g, x, yo, "fbp"), lambda: ct.ct_bagmres_solve(g, y, 2, xo, opts),
                 lambda: ct.ct_abgmres_solve(g, y, 2, xo, opts), lambda: ct.ct_bagmres_vjp(g, x, 2, yo, opts),
                 lambda: state.start(y)):
        with pytest.raises(ct.CTError) as ei:
            call()
        assert ei.value.status == ct.CT_EINVAL and "2048" in str(ei.value)
    state.close()
    ct.ct_project_A(g, x, yo)
    ct.ct_backproject_B(g, y, xo, "un")
    ct.ct_adjoint_Bt(g, x, yo, "un")
    assert ct.ct_bagmres_solve(g, y, 2, xo, ct.make_opts(b_kind="un")).iters == 2
