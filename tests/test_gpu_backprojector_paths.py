"""The back-projector's kernels at the sizes where the launch changes from one
to another, against the FP64 oracle (relative L2 <= 1e-5 for an operator, 1e-4
for a solve, as everywhere).

Small volumes: 1, 2 and 8 warps a run, runs past nz, tiles past nx and ny.
Slabs of 12 and of 16 slices (ragged in every axis), whose entries hold row
differences (operator calls) or four values (the projector writes them inside
a BA-GMRES solve with B_un).
"""
import math

import numpy as np
import pytest
import torch

import ct_inputs as ci
import oracle
from oracle import krylov

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct as _ct
    return _ct


def par2d(nx, ny, views, nu):
    return ci.Geometry(name="par2d_%dx%d" % (nx, ny), kind=ci.PARALLEL_2D, nx=nx, ny=ny, nz=1, vox=1.0,
                       n_views=views, ang0=0.15, span=math.pi, nu=nu, nv=1, du=1.0, dv=1.0)


def cone(name, nx, ny, nz, views, nu, nv, du, vox=1.0):
    return ci._cone(name, 0, vox, views, nu, nv, du, nxyz=(nx, ny, nz), ang0=0.3)


SLAB12 = cone("slab12", 163, 157, 59, 10, 190, 70, 1.6)
SLAB16 = cone("slab16", 170, 150, 61, 7, 200, 66, 1.7)
SCANS = [
    par2d(31, 9, 11, 40),      # 8 warps a run
    par2d(200, 333, 13, 300),  # 2
    cone("slice", 33, 30, 1, 17, 60, 9, 1.2),
    cone("run_past_nz", 65, 33, 5, 19, 70, 12, 1.9),
    cone("small_split1", 100, 97, 40, 6, 120, 45, 2.0),
    SLAB12,
    SLAB16,
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("spec", SCANS, ids=lambda s: s.name)
def test_backprojector_kernels_match_oracle(ct, spec, dtype):
    g = ct.Geometry.from_spec(spec, sino_dtype=dtype)
    y = torch.from_numpy(ci.random_vector(spec.m, seed=83).astype(np.float32).reshape(spec.sino_shape))
    x = ct.backproject_B(g, y.cuda(), "un").double().cpu().numpy()
    if dtype == "bf16":
        y = y.to(torch.bfloat16)
    ref = oracle.backproject_B(spec, y.double().numpy()).reshape(x.shape)
    assert np.linalg.norm(x - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("spec", [SCANS[0], SCANS[4], SLAB12], ids=lambda s: s.name)
def test_projector_written_entries(ct, spec):
    g = ct.Geometry.from_spec(spec)
    b = oracle.project_A(spec, ci.phantom(spec)[0].astype(np.float64)).astype(np.float32)
    x, res = ct.bagmres(g, torch.from_numpy(b.reshape(spec.sino_shape)).cuda(), 2, b_kind="un")
    ops = oracle.Operators(spec, "un")
    ref = krylov.ba_gmres(ops.A, ops.B, b.astype(np.float64).reshape(-1), 2, keep_basis=False)
    xg = x.double().cpu().numpy().reshape(-1)
    assert np.linalg.norm(xg - ref["x_final"]) <= 1e-4 * np.linalg.norm(ref["x_final"])
    assert np.max(np.abs(res.resid - ref["resid"])) <= 1e-4 * ref["resid"][0]


# transform lengths 8, 2^a, 3 2^a with and without a radix-2 stage, and the first row length past each
@pytest.mark.parametrize("nu", [1, 3, 47, 48, 49, 64, 65, 96, 97, 128, 129, 192, 193, 384, 385, 768, 769])
@pytest.mark.parametrize("transpose", [False, True])
def test_ramp_lengths(ct, nu, transpose):
    spec = par2d(40, 40, 7, nu)   # an odd row count: the last row has no partner
    g = ct.Geometry.from_spec(spec)
    y = ci.random_vector(spec.m, seed=87).astype(np.float32).reshape(spec.sino_shape)
    out = ct.ramp_F(g, torch.from_numpy(y).cuda(), transpose).double().cpu().numpy()
    ref = (oracle.ramp_Ft if transpose else oracle.ramp_F)(spec, y.astype(np.float64)).reshape(out.shape)
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)
