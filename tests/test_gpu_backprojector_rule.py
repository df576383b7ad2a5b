"""Back-projections on both sides of the rules that choose between runs of 4
slices a thread and slabs of 12 and 16, in FP32 and bf16 storage, against the
FP64 oracle (relative L2 <= 1e-5, as for every operator), at sizes that are
ragged in every axis; and a scan of more views than the slab kernel's shared
memory holds, which had no kernel in a volume that it serves.
"""
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


def cone(nx, ny, nz, views, nu=60, nv=30):
    return ci._cone("cone_%dx%dx%d_%d" % (nx, ny, nz, views), 0, 128.0 / max(nx, ny), views, nu, nv, 5.0,
                    nxyz=(nx, ny, nz))


# blocks of runs of 4 slices: 896 and 960 (6 an SM are 912), 600 and 612 (4 an SM are 608); slabs of 12 and 16
# either way around for FP32 and bf16
SCANS = [cone(111, 109, 63, 5), cone(127, 113, 63, 5), cone(79, 77, 78, 5), cone(95, 135, 47, 5), cone(159, 157, 47, 4),
         cone(81, 117, 136, 4), cone(100, 98, 99, 4), cone(200, 200, 20, 4), cone(250, 255, 15, 4)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", SCANS, ids=lambda s: s.name)
def test_back_projection(ct, spec, dtype):
    g = ct.Geometry.from_spec(spec, sino_dtype=dtype)
    y = torch.from_numpy(ci.random_vector(spec.m, seed=94).astype(np.float32).reshape(spec.sino_shape))
    x = ct.backproject_B(g, y.cuda(), "un").double().cpu().numpy()
    if dtype == "bf16":
        y = y.to(torch.bfloat16)
    ref = oracle.backproject_B(spec, y.double().numpy()).reshape(x.shape)
    assert np.linalg.norm(x - ref) <= OP_TOL * np.linalg.norm(ref)


def test_more_views_than_shared_memory_holds(ct):
    spec = cone(150, 60, 120, 7000, nu=6, nv=5)
    g = ct.Geometry.from_spec(spec)
    y = torch.from_numpy(ci.random_vector(spec.m, seed=95).astype(np.float32).reshape(spec.sino_shape)).cuda()
    x = ct.backproject_B(g, y, "un")
    # the same views as two scans of half the angles each: a sum of two (FP32 sums of 3500 terms, 1e-5)
    half = torch.zeros_like(x)
    for i in range(2):
        part = ci.Geometry(**dict(vars(spec), name="half", n_views=3500, ang0=spec.ang0 + i * spec.span / 2,
                                  span=spec.span / 2))
        half += ct.backproject_B(ct.Geometry.from_spec(part), y[i * 3500:(i + 1) * 3500].contiguous(), "un")
    assert float((x - half).norm()) <= OP_TOL * float(half.norm())
