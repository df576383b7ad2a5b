"""Orthogonalisation of vectors whose length is not a multiple of a 16-byte group
or whose start is not aligned: the coefficients of a sweep of single passes
against FP64 (numpy) on the same vectors, in groups with a remainder and one
element at a time, around the lengths where the launch changes.  Tolerances: a
compensated dot product of unit vectors with q carries about one FP32 rounding
of a rounding, 2^-48, and the norm's square root halves it, 1e-14 of ||q||; plain
FP32 chains of up to 30 products with random signs, 30 x 2^-24 / sqrt(number of
chains), 1e-7 (chains are longest for one element at a time: at most 27 products
here).  And whole solves on ragged grids against the oracle (1e-4, as everywhere).
"""
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


@pytest.mark.parametrize("mode,tol", [(0, 1e-14), (1, 1e-7)])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", [1, 3, 5, 1023, 4097, 8195, 100003, 1245189, 2490371, 2490373])
def test_sweep_coefficients(ct, n, offset, mode, tol):
    rng = np.random.default_rng(n + offset)
    j, ldv = 3, (n + 63) // 64 * 64
    V = np.zeros((j, ldv), dtype=np.float32)
    V[:, :n] = rng.standard_normal((j, n))
    V[:, :n] /= np.linalg.norm(V[:, :n].astype(np.float64), axis=1, keepdims=True)
    V[:, n:] = np.nan   # past the vectors: never read into a sum
    q = rng.standard_normal(n).astype(np.float32)
    buf = torch.full((n + 8,), float("nan"), device="cuda")
    qd = buf[offset:offset + n]
    qd.copy_(torch.from_numpy(q))
    h = torch.zeros(j + 1, dtype=torch.float64, device="cuda")
    ct.ct_mgs_sweep(torch.from_numpy(V).cuda(), ldv, j, n, qd, h, mode)
    h = h.cpu().numpy()
    norm = np.linalg.norm(q.astype(np.float64))
    for i in range(j):   # the same update, q -= fl(h_i) v_i with one rounding
        v = V[i, :n].astype(np.float64)
        assert abs(h[i] - q.astype(np.float64) @ v) <= tol * norm
        q = (q.astype(np.float64) - np.float64(np.float32(h[i])) * v).astype(np.float32)
    assert abs(h[j] - np.linalg.norm(q.astype(np.float64))) <= tol * norm
    assert np.array_equal(qd.cpu().numpy(), q)
    rest = np.concatenate([buf[:offset].cpu().numpy(), buf[offset + n:].cpu().numpy()])
    assert np.isnan(rest).all()   # nothing written past q


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("vol", ["f32", "bf16"])
def test_long_vectors_on_a_device_and_a_host_basis(ct, vol, mode):
    """Vectors past the one-launch sweep, ragged: both bases take the same passes, bit for bit."""
    spec = ci._cone("cone_143x139x131", 0, 0.9, 3, 40, 20, 7.0, nxyz=(143, 139, 131))
    g = ct.Geometry.from_spec(spec, vol_dtype=vol)
    b = torch.from_numpy(ci.random_vector(spec.m, seed=84).astype(np.float32)).cuda()
    out = []
    for basis in ("device", "host"):
        st = ct.GmresState(g, 3, basis, ct.make_opts(b_kind="un", dot_mode=mode))
        st.start(b)
        x = torch.empty(spec.vol_shape, device="cuda")
        out.append((st.extend(3, x).resid.copy(), x))
        st.close()
    assert np.array_equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert np.all(np.diff(out[0][0]) <= 1e-12 * out[0][0][0])


@pytest.mark.parametrize("vol", ["f32", "bf16"])
@pytest.mark.parametrize("nxyz", [(15, 13, 11), (23, 18, 7), (14, 15, 9)], ids=str)
def test_ragged_solve(ct, nxyz, vol):
    spec = ci._cone("cone_%dx%dx%d" % nxyz, 0, 8.0, 24, 33, 21, 9.0, nxyz=nxyz)   # 1, 2 and 2 past a multiple of 4
    b = oracle.project_A(spec, ci.phantom(spec)[0].astype(np.float64)).astype(np.float32)
    ops = oracle.Operators(spec, "un")
    ref = krylov.ba_gmres(ops.A, ops.B, b.astype(np.float64).reshape(-1), 4, keep_basis=False)["x_final"]
    g = ct.Geometry.from_spec(spec, vol_dtype=vol)
    x, _ = ct.bagmres(g, torch.from_numpy(b.reshape(spec.sino_shape)).cuda(), 4, b_kind="un")
    err = np.linalg.norm(x.double().cpu().numpy().reshape(-1) - ref) / np.linalg.norm(ref)
    # bf16 copies and basis: 2^-9 a voxel, a solve of 4 iterations a few times that
    assert err <= (1e-4 if vol == "f32" else 2e-2)
