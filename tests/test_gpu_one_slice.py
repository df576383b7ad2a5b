"""One-row projections where the batches of planes end, against the FP64 oracle (relative L2 <= 1e-5, as for every
operator): plane counts one below, at and above a batch (4 or 8) times
the warps that share them, elongated images, cone beams of one row.
"""
import math

import numpy as np
import pytest
import torch

import ct_inputs as ci
import oracle

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5


@pytest.fixture(scope="module")
def ct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct as _ct
    return _ct


def par2d(nx, ny, views, nu, ang0=0.15):
    return ci.Geometry(name="par2d_%dx%d_%d_%d" % (nx, ny, views, nu), kind=ci.PARALLEL_2D, nx=nx, ny=ny, nz=1,
                       vox=1.0, n_views=views, ang0=ang0, span=math.pi, nu=nu, nv=1, du=1.0, dv=1.0)


ROWS = [par2d(3, 4, 7, 9), par2d(5, 31, 9, 40), par2d(32, 33, 8, 50), par2d(63, 65, 9, 30), par2d(64, 127, 7, 150),
        par2d(300, 11, 31, 310), par2d(140, 130, 63, 200), par2d(260, 30, 600, 270),
        ci._cone("row_17", 0, 2.0, 9, 40, 1, 1.0, nxyz=(17, 63, 3), dv=3.0),
        ci._cone("row_128", 0, 2.0, 64, 150, 1, 1.0, nxyz=(128, 65, 4), dv=3.0)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", ROWS, ids=lambda s: s.name)
def test_one_row_projection(ct, spec, dtype):
    g = ct.Geometry.from_spec(spec, vol_dtype=dtype)
    x = torch.from_numpy(ci.random_vector(spec.n, seed=91).astype(np.float32).reshape(spec.vol_shape))
    y = ct.project_A(g, x.cuda()).double().cpu().numpy()
    if dtype == "bf16":
        x = x.to(torch.bfloat16)
    ref = oracle.project_A(spec, x.double().numpy()).reshape(y.shape)
    assert np.linalg.norm(y - ref) <= OP_TOL * np.linalg.norm(ref)
