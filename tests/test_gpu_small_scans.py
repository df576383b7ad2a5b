"""The paired walk on BF16 copies, with its clamp (a detector taller than the
slices, whose plane loop is unrolled by 3) and without, at plane counts off the
unroll, against the FP64 oracle on the rounded volume (relative L2 <= 1e-5, as for
every operator).
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


def cone(nx, ny, nz, views, nu, nv, du, ang0=0.3, **kw):
    return ci._cone("cone_%dx%dx%d_%d_%dx%d_%g" % (nx, ny, nz, views, nu, nv, ang0), 0, 128.0 / max(nx, ny), views, nu,
                    nv, du, nxyz=(nx, ny, nz), ang0=ang0, **kw)


@pytest.mark.parametrize("spec", [cone(36, 50, 7, 6, 69, 15, 3.5), cone(31, 29, 30, 5, 49, 33, 6.0),
                                  cone(17, 18, 40, 5, 31, 31, 9.0), cone(40, 35, 6, 4, 60, 41, 4.0)], ids=lambda s: s.name)
def test_bf16_projection(ct, spec):
    g = ct.Geometry.from_spec(spec, vol_dtype="bf16")
    x = torch.from_numpy(ci.random_vector(spec.n, seed=89).astype(np.float32).reshape(spec.vol_shape))
    y = ct.project_A(g, x.cuda()).double().cpu().numpy()
    ref = oracle.project_A(spec, x.to(torch.bfloat16).double().numpy()).reshape(y.shape)
    assert np.linalg.norm(y - ref) <= OP_TOL * np.linalg.norm(ref)
