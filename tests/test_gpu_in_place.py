"""2D images that are projected without copies: on both sides of the rule that
chooses them (the launches recorded say which way a call went), the values are
bit for bit those of ct_project_A_noalloc, which always makes the copies.
"""
import math

import numpy as np
import pytest
import torch

import ct_inputs as ci

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct as _ct
    yield _ct
    _ct.profile_enable(False)


def par2d(nx, ny, views, nu, ang0=0.15):
    return ci.Geometry(name="par2d_%dx%d_%d_%d" % (nx, ny, views, nu), kind=ci.PARALLEL_2D, nx=nx, ny=ny, nz=1,
                       vox=1.0, n_views=views, ang0=ang0, span=math.pi, nu=nu, nv=1, du=1.0, dv=1.0)


IN_PLACE = [par2d(1, 1, 1, 1), par2d(9, 7, 5, 33), par2d(64, 64, 90, 95), par2d(96, 96, 90, 140), par2d(48, 49, 600, 70),
            par2d(30, 300, 200, 306), par2d(24, 22, 10, 160, ang0=0.0), par2d(95, 96, 400, 139)]
COPIED = [par2d(96, 96, 1500, 140), par2d(64, 64, 700, 95), par2d(97, 96, 9, 30), par2d(9, 1000, 60, 1005),
          par2d(80, 80, 500, 118)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", IN_PLACE + COPIED, ids=lambda s: s.name)
def test_in_place_reads(ct, spec, dtype):
    g = ct.Geometry.from_spec(spec, vol_dtype=dtype)
    x = torch.from_numpy(ci.random_vector(spec.n, seed=93).astype(np.float32).reshape(spec.vol_shape)).cuda()
    y, ref = torch.empty(spec.sino_shape, device="cuda"), torch.empty(spec.sino_shape, device="cuda")
    ct.ct_project_A_noalloc(g, x, ref)
    ct.profile_enable(True)
    ct.profile_reset()
    ct.ct_project_A(g, x, y)
    torch.cuda.synchronize()
    launches = ct.profile_read()
    ct.profile_enable(False)
    assert launches["plane_copies"][1] == (0 if spec in IN_PLACE else 1)
    assert torch.equal(y, ref)
