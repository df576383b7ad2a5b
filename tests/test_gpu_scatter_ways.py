"""The transposes on both sides of the rules that choose how they scatter
(straight into the output, into accumulators, into accumulators kept twice),
against the FP64 oracle (relative L2 <= 1e-5, as for every operator; FP32 sums
in any order): few rays a voxel, detector rows finer than slices, one-row and
one-view scans, oversampled detectors, thin slabs, odd sizes in every axis.  And
with no scratch memory to be had: B_un^T still runs, A^T is refused.
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
    yield _ct
    _ct.fault_set(None)


def par2d(nx, ny, views, nu):
    return ci.Geometry(name="par2d_%dx%d_%d_%d" % (nx, ny, views, nu), kind=ci.PARALLEL_2D, nx=nx, ny=ny, nz=1, vox=1.0,
                       n_views=views, ang0=0.15, span=math.pi, nu=nu, nv=1, du=1.0, dv=1.0)


def cone(nx, ny, nz, views, nu, nv, du, **kw):
    return ci._cone("cone_%dx%dx%d_%d_%dx%d" % (nx, ny, nz, views, nu, nv), 0, 128.0 / max(nx, ny), views, nu, nv, du,
                    nxyz=(nx, ny, nz), ang0=0.3, **kw)


AT = [par2d(90, 101, 4, 150), cone(31, 33, 35, 5, 47, 41, 6.0), cone(131, 129, 67, 2, 61, 33, 4.5), cone(33, 31, 12, 6, 47, 40, 5.0),
      cone(130, 60, 201, 3, 41, 23, 7.0), cone(70, 71, 9, 12, 90, 1, 3.0)]
BT = [par2d(40, 41, 90, 60), par2d(60, 61, 1, 90), par2d(60, 61, 40, 90), cone(33, 35, 5, 3, 47, 9, 6.0),
      cone(65, 63, 5, 40, 67, 9, 4.5), cone(17, 19, 21, 9, 31, 27, 9.0), cone(49, 47, 41, 19, 55, 31, 6.0),
      cone(49, 47, 41, 1, 55, 31, 6.0)]
AT_SIDDON = [cone(13, 15, 11, 4, 21, 12, 12.0), cone(60, 57, 44, 20, 81, 51, 3.5), cone(9, 7, 8, 30, 121, 103, 2.0),
             cone(70, 60, 150, 3, 180, 71, 1.7)]


def check(a, ref):
    a = a.double().cpu().numpy()
    ref = ref.reshape(a.shape)
    assert np.linalg.norm(a - ref) <= OP_TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("spec", AT, ids=lambda s: s.name)
def test_projector_transpose(ct, spec):
    y = ci.random_vector(spec.m, seed=96).astype(np.float32).reshape(spec.sino_shape)
    at = ct.adjoint_At(ct.Geometry.from_spec(spec), torch.from_numpy(y).cuda())
    check(at, oracle.adjoint_At(spec, y.astype(np.float64)))


@pytest.mark.parametrize("memory", ["plenty", "none"])
@pytest.mark.parametrize("spec", BT, ids=lambda s: s.name)
def test_back_projector_transpose(ct, spec, memory):
    x = ci.random_vector(spec.n, seed=97).astype(np.float32).reshape(spec.vol_shape)
    g, xd, y = ct.Geometry.from_spec(spec), torch.from_numpy(x).cuda(), torch.empty(spec.sino_shape, device="cuda")
    ct.fault_set("oom" if memory == "none" else None)
    try:
        ct.ct_adjoint_Bt(g, xd, y, "un")
    finally:
        ct.fault_set(None)
    check(y, oracle.adjoint_Bt(spec, x.astype(np.float64), filtered=False))


@pytest.mark.parametrize("projector,spec", [("siddon", s) for s in AT_SIDDON] + [("joseph", par2d(811, 797, 3, 301))],
                         ids=lambda s: getattr(s, "name", s))
def test_transpose_of_the_projector(ct, projector, spec):
    """<A x, y> = <x, A^T y>, where the oracle has other coordinates: rays in voxel boundary planes (a matter of
    convention), and images so large that FP32 coordinates part from FP64 ones by more than the tolerance."""
    y = ci.random_vector(spec.m, seed=98, positive=True).astype(np.float32).reshape(spec.sino_shape)
    x = ci.random_vector(spec.n, seed=99, positive=True).astype(np.float32).reshape(spec.vol_shape)
    g = ct.Geometry.from_spec(spec, projector=projector)
    ax = ct.project_A(g, torch.from_numpy(x).cuda()).double().cpu().numpy()
    at = ct.adjoint_At(g, torch.from_numpy(y).cuda()).double().cpu().numpy()
    lhs, rhs = float((ax * y).sum()), float((x * at).sum())
    assert abs(lhs - rhs) <= OP_TOL * abs(lhs)


def test_no_scratch_memory(ct):
    spec = AT[2]
    g = ct.Geometry.from_spec(spec)
    x, y = torch.empty(spec.vol_shape, device="cuda"), torch.ones(spec.sino_shape, device="cuda")
    ct.fault_set("oom")
    try:
        with pytest.raises(ct.CTError) as ei:
            ct.ct_adjoint_At(g, y, x)
        assert ei.value.status == ct.CT_ENOMEM
        with pytest.raises(ct.CTError) as ei:   # the filter needs a sinogram to write to
            ct.ct_adjoint_Bt(g, x, y, "fbp")
        assert ei.value.status == ct.CT_ENOMEM
    finally:
        ct.fault_set(None)
    ct.ct_adjoint_At(g, y, x)
