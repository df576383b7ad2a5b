"""The orthogonalisation's kernels at the sizes where the launch changes from
one to another.

Coefficients of a sweep of single passes against FP64 (numpy) on the same
vectors: one block, several, more elements than a register-resident sweep
takes, lengths that are not a multiple of a 16-byte group, and values whose
squares leave FP32's range.  Tolerances: a compensated dot product of unit
vectors with q carries about one FP32 rounding of a rounding, 2^-48, and the
norm's square root halves it: 1e-14 of ||q||; plain FP32 chains of up to 30
products with random signs, 30 x 2^-24 / sqrt(number of chains): 1e-7.

The one-launch sweep against single passes: a BA-GMRES state with its basis on
the device uses the first, one with its basis in host memory the second, and
both must return the same bits.
"""

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
    return _ct


@pytest.mark.parametrize("mode,tol", [(0, 1e-14), (1, 1e-7)])
@pytest.mark.parametrize("n,scale", [(1, 1.0), (7, 1.0), (8192, 1.0), (8196, 1.0), (100003, 1.0), (1245188, 1.0),
                                     (2490372, 1.0), (4096, 3e18)])
def test_sweep_coefficients(ct, n, scale, mode, tol):
    rng = np.random.default_rng(n)
    j = 3
    V = rng.standard_normal((j, n)).astype(np.float32)
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    q = (rng.standard_normal(n) * scale).astype(np.float32)
    qd, Vd = torch.from_numpy(q).cuda(), torch.from_numpy(V).cuda()
    h = torch.zeros(j + 1, dtype=torch.float64, device="cuda")
    ct.ct_mgs_sweep(Vd, n, j, n, qd, h, mode)
    h = h.cpu().numpy()
    norm = np.linalg.norm(q.astype(np.float64))
    for i in range(j):   # the same update, q -= fl(h_i) v_i with one rounding
        assert abs(h[i] - q.astype(np.float64) @ V[i].astype(np.float64)) <= tol * norm
        q = (q.astype(np.float64) - np.float64(np.float32(h[i])) * V[i].astype(np.float64)).astype(np.float32)
    assert abs(h[j] - np.linalg.norm(q.astype(np.float64))) <= tol * norm
    assert np.array_equal(qd.cpu().numpy(), q)


def cone(nx, ny, nz, views=5):
    return ci._cone("cone_%dx%dx%d" % (nx, ny, nz), 0, 128.0 / max(nx, ny), views, 40, 20, 7.0, nxyz=(nx, ny, nz))


SCANS = [ci.PAR2D_64,          # one block
         cone(21, 19, 11),     # not a multiple of 4
         cone(44, 36, 29),     # a few blocks
         cone(128, 120, 82),   # every SM, 16 elements a thread and a few of 32
         cone(140, 136, 130)]  # 32 elements a thread, nearly all of them


@pytest.mark.parametrize("vol", ["f32", "bf16"])
@pytest.mark.parametrize("mode,reorth", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("spec", SCANS, ids=lambda s: s.name)
def test_one_launch_sweep_equals_single_passes(ct, spec, mode, reorth, vol):
    g = ct.Geometry.from_spec(spec, vol_dtype=vol)
    b = torch.from_numpy(ci.random_vector(spec.m, seed=84).astype(np.float32)).cuda()
    out = []
    for basis in ("device", "host"):
        st = ct.GmresState(g, 5, basis, ct.make_opts(b_kind="un", dot_mode=mode, reorth=reorth))
        st.start(b)
        x = torch.empty(spec.vol_shape, device="cuda")
        res = st.extend(5, x)
        out.append((x.cpu().numpy(), res.resid.copy()))
        st.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])
