"""The projector's kernels at the sizes where the launch changes from one to
another, against the FP64 oracle (relative L2 <= 1e-5, as for every operator).

The paired walk: its window, its clamped window (a detector that reaches far
beyond the slices), and without a window (a detector coarser than the
slices); ray counts off the 16 rays of a thread and plane counts off the
loop's unroll.  The one-row walk: 1, 2, 4 and 8 warps a ray.
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


SCANS = [
    ci._cone("window_33x37_17", 0, 3.0, 9, 35, 17, 4.0, nxyz=(33, 37, 15), ang0=0.3),
    ci._cone("window_5x6_64", 0, 3.0, 7, 32, 64, 3.9, nxyz=(5, 6, 90), ang0=0.8),
    ci._cone("clamped_tall", 0, 2.0, 11, 48, 41, 3.0, nxyz=(32, 30, 8)),
    ci._cone("no_window_coarse", 0, 1.0, 13, 21, 18, 4.0, nxyz=(40, 38, 33), ang0=0.2),
    ci._cone("one_row_cone", 0, 2.0, 40, 200, 1, 1.0, nxyz=(50, 46, 5), dv=3.0),
    par2d(9, 7, 5, 33),       # 8 warps a ray
    par2d(61, 70, 80, 450),   # 4
    par2d(40, 48, 150, 500),  # 2
    par2d(130, 97, 500, 400),  # 1
    # the largest image that is read without copies, and the next
    par2d(96, 96, 500, 400),
    par2d(97, 96, 60, 150),
    # whole warps of rays beside the image, parallel to its sides but for a slope of 1e-17
    par2d(24, 22, 10, 160, ang0=0.0),
    par2d(181, 181, 270, 257, ang0=0.0),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", SCANS, ids=lambda s: s.name)
def test_projector_kernels_match_oracle(ct, spec, dtype):
    g = ct.Geometry.from_spec(spec, vol_dtype=dtype)
    x = ci.random_vector(spec.n, seed=81).astype(np.float32).reshape(spec.vol_shape)
    xd = torch.from_numpy(x)
    y = ct.project_A(g, xd.cuda()).double().cpu().numpy()
    if dtype == "bf16":
        xd = xd.to(torch.bfloat16)
    ref = oracle.project_A(spec, xd.double().numpy()).reshape(y.shape)
    assert np.linalg.norm(y - ref) <= OP_TOL * np.linalg.norm(ref)



@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", [s for s in SCANS if s.kind == ci.PARALLEL_2D], ids=lambda s: s.name)
def test_images_read_in_place_match_the_copies(ct, spec, dtype):
    # ct_project_A_noalloc always makes copies; the operations are the same
    g = ct.Geometry.from_spec(spec, vol_dtype=dtype)
    x = torch.from_numpy(ci.random_vector(spec.n, seed=82).astype(np.float32).reshape(spec.vol_shape)).cuda()
    y = torch.empty(spec.sino_shape, device="cuda")
    ct.ct_project_A_noalloc(g, x, y)
    assert torch.equal(ct.project_A(g, x), y)
