"""The transposes' kernels at the sizes where their launches change, against
the FP64 oracle (relative L2 <= 1e-5, as for every operator): 1 to 16 warps a
tile of A^T, 1 to 32 blocks a run of B_un^T, odd row lengths (a pair of cells is
aligned in one accumulator on one row and in the other on the next), and the
detector's and the grid's first and last columns.  Non-finite data stays on
the cells that its rays touch.
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
    return ci.Geometry(name="par2d_%dx%d" % (nx, ny), kind=ci.PARALLEL_2D, nx=nx, ny=ny, nz=1, vox=1.0,
                       n_views=views, ang0=ang0, span=math.pi, nu=nu, nv=1, du=1.0, dv=1.0)


def cone(name, nx, ny, nz, views, nu, nv, du, **kw):
    return ci._cone(name, 0, 1.0, views, nu, nv, du, nxyz=(nx, ny, nz), ang0=0.3, **kw)


SCANS = [par2d(9, 7, 3, 33), par2d(100, 81, 60, 150),
         par2d(24, 22, 10, 160, ang0=0.0),   # warps of rays beside the image, parallel to its sides
         cone("thin", 31, 33, 5, 9, 41, 9, 1.7),
         cone("odd_rows", 33, 31, 17, 11, 47, 21, 1.5),
         cone("mid", 65, 60, 40, 40, 97, 47, 1.6),
         cone("wide", 90, 87, 33, 64, 130, 50, 1.5),
         cone("tall_detector", 32, 30, 8, 20, 47, 60, 1.4),
         cone("coarse", 40, 38, 33, 13, 21, 18, 4.0)]


@pytest.mark.parametrize("spec", SCANS, ids=lambda s: s.name)
def test_transposes_match_oracle(ct, spec):
    g = ct.Geometry.from_spec(spec)
    x = ci.random_vector(spec.n, seed=85).astype(np.float32).reshape(spec.vol_shape)
    y = ci.random_vector(spec.m, seed=86).astype(np.float32).reshape(spec.sino_shape)
    at = ct.adjoint_At(g, torch.from_numpy(y).cuda()).double().cpu().numpy()
    ref = oracle.adjoint_At(spec, y.astype(np.float64)).reshape(at.shape)
    assert np.linalg.norm(at - ref) <= OP_TOL * np.linalg.norm(ref)
    for kind in ("un", "fbp"):
        bt = ct.adjoint_Bt(g, torch.from_numpy(x).cuda(), kind).double().cpu().numpy()
        ref = oracle.adjoint_Bt(spec, x.astype(np.float64), filtered=kind == "fbp").reshape(bt.shape)
        assert np.linalg.norm(bt - ref) <= OP_TOL * np.linalg.norm(ref), kind


def test_matched_solve_uses_the_transpose(ct):
    """CGLS and BA-GMRES with B = A^T, whose workspaces hold the accumulators."""
    from oracle import krylov
    spec = SCANS[4]
    g = ct.Geometry.from_spec(spec)
    b = oracle.project_A(spec, ci.phantom(spec)[0].astype(np.float64)).astype(np.float32)
    bd = torch.from_numpy(b.reshape(spec.sino_shape)).cuda()
    ops = oracle.Operators(spec, "at")
    x, _ = ct.cgls(g, bd, 4, b_kind="at")
    ref = krylov.cgls(ops.A, ops.B, b.astype(np.float64).reshape(-1), 4)
    xr = ref["x_final"] if "x_final" in ref else ref["x"]
    assert np.linalg.norm(x.double().cpu().numpy().reshape(-1) - xr) <= 1e-4 * np.linalg.norm(xr)
    x, res = ct.bagmres(g, bd, 4, b_kind="at")
    ref = krylov.ba_gmres(ops.A, ops.B, b.astype(np.float64).reshape(-1), 4, keep_basis=False)
    assert np.linalg.norm(x.double().cpu().numpy().reshape(-1) - ref["x_final"]) <= 1e-4 * np.linalg.norm(ref["x_final"])


def test_nonfinite_reading_touches_its_own_cells_only(ct):
    spec = SCANS[4]
    g = ct.Geometry.from_spec(spec)
    r = (spec.n_views // 2 * spec.nv + 9) * spec.nu + 20
    y = np.zeros(spec.m, dtype=np.float32)
    y[r] = 1.0
    touched = ct.adjoint_At(g, torch.from_numpy(y.reshape(spec.sino_shape)).cuda()).cpu().numpy() != 0
    y[r] = np.inf
    bad = ~np.isfinite(ct.adjoint_At(g, torch.from_numpy(y.reshape(spec.sino_shape)).cuda()).cpu().numpy())
    assert touched.any() and np.array_equal(bad & touched, touched)
    # a weight of exactly zero times Inf is NaN in a sample's four cells, no further
    assert np.count_nonzero(bad) <= np.count_nonzero(touched) * 2
