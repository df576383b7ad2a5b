"""One-row projections and single-slice back-projections where the batches of
planes and views end, against the FP64 oracle (relative L2 <= 1e-5, as for every
operator): plane and view counts one below, at and above a batch (4 or 8) times
the warps that share them, elongated images, cone beams of one row and of one
slice, detectors that miss part of the image.
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
SLICES = [par2d(9, 8, v, 12) for v in (1, 7, 8, 9, 63, 64, 65)] + \
         [par2d(150, 41, 33, 170), par2d(90, 300, 31, 60), par2d(230, 210, 17, 330)] + \
         [ci._cone("slice_%d" % v, 0, 2.0, v, 60, 9, 1.5, nxyz=(40, 37, 1)) for v in (7, 16, 65)]


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


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", SLICES, ids=lambda s: s.name)
def test_one_slice_back_projection(ct, spec, dtype):
    g = ct.Geometry.from_spec(spec, sino_dtype=dtype)
    y = torch.from_numpy(ci.random_vector(spec.m, seed=92).astype(np.float32).reshape(spec.sino_shape))
    x = ct.backproject_B(g, y.cuda(), "un").double().cpu().numpy()
    if dtype == "bf16":
        y = y.to(torch.bfloat16)
    ref = oracle.backproject_B(spec, y.double().numpy()).reshape(x.shape)
    assert np.linalg.norm(x - ref) <= OP_TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("spec", [SLICES[5], SLICES[9], SLICES[12]], ids=lambda s: s.name)
def test_one_slice_in_a_solve(ct, spec):
    """Inside BA-GMRES the projector writes the entries' four values, not row differences."""
    from oracle import krylov
    g = ct.Geometry.from_spec(spec)
    b = oracle.project_A(spec, ci.phantom(spec)[0].astype(np.float64)).astype(np.float32)
    x, _ = ct.bagmres(g, torch.from_numpy(b.reshape(spec.sino_shape)).cuda(), 3, b_kind="un")
    ops = oracle.Operators(spec, "un")
    ref = krylov.ba_gmres(ops.A, ops.B, b.astype(np.float64).reshape(-1), 3, keep_basis=False)["x_final"]
    assert np.linalg.norm(x.double().cpu().numpy().reshape(-1) - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("views", [1, 9])
def test_readings_of_skipped_views_are_not_touched(ct, views):
    """A view that a voxel misses adds exactly nothing, whatever the detector's last readings are."""
    spec = par2d(41, 43, views, 15)
    g = ct.Geometry.from_spec(spec)
    y = np.zeros(spec.m, dtype=np.float32)
    y.reshape(views, 15)[:, 7] = 1.0
    seen = ct.backproject_B(g, torch.from_numpy(y.reshape(spec.sino_shape)).cuda(), "un").cpu().numpy() != 0
    y.reshape(views, 15)[0, 7] = np.inf
    bad = ~np.isfinite(ct.backproject_B(g, torch.from_numpy(y.reshape(spec.sino_shape)).cuda(), "un").cpu().numpy())
    assert bad.any() and np.count_nonzero(bad & ~seen) <= np.count_nonzero(seen)
    assert np.count_nonzero(~bad) > 0.5 * spec.n
