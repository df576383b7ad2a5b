"""Scratch memory: every call takes it from the library's own pool, the pool keeps
at most 1/32 of the device's memory while a geometry lives and gives it back with
the last one, and geometries created, used and destroyed by several threads at
once give what they give alone.
"""
import ctypes
import gc
import json
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

import ct_inputs as ci

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
USED_MEM_HIGH = 8   # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.fixture(scope="module")
def ct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct as _ct
    return _ct


@pytest.fixture()
def default_pool_high():
    """high() is the most that was ever taken from the device's default pool since the fixture began."""
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    pool, value = ctypes.c_void_p(), ctypes.c_ulonglong(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(value)) == 0

    def high():
        v = ctypes.c_ulonglong(0)
        assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
        return v.value
    return high


def test_calls_leave_the_default_pool_alone(ct, default_pool_high):
    spec = ci.CONE_ANISO
    g = ct.Geometry.from_spec(spec)
    x = torch.from_numpy(ci.phantom(spec)[0]).cuda()
    y = ct.project_A(g, x)
    xo, gb = torch.empty_like(x), torch.empty_like(y)
    calls = {
        "A": lambda: ct.project_A(g, x), "B": lambda: ct.backproject_B(g, y, "fbp"), "At": lambda: ct.adjoint_At(g, y),
        "Bt": lambda: ct.adjoint_Bt(g, x, "fbp"),
        "ba": lambda: ct.ct_bagmres_solve(g, y, 3, xo, workspace=None),
        "host": lambda: ct.ct_bagmres_solve_host(g, y.cpu().pin_memory(), 3, torch.empty(spec.vol_shape).pin_memory(),
                                                 workspace=None),
        "restarted": lambda: ct.ct_bagmres_restarted(g, y, 2, 2, xo, workspace=None),
        "ab": lambda: ct.ct_abgmres_solve(g, y, 3, xo, workspace=None),
        "cgls": lambda: ct.ct_cgls_solve(g, y, 3, xo, workspace=None),
        "vjp": lambda: ct.ct_bagmres_vjp(g, x, 3, gb, workspace=None),
    }
    for name, call in calls.items():
        call()
        torch.cuda.synchronize()
        assert default_pool_high() == 0, name


SCRIPT = r"""
import json, sys
sys.path.insert(0, %r)
import torch, ct_inputs as ci
from paper_2201_07408_gb300 import ct
torch.zeros(1, device="cuda")
small = ct.Geometry.from_spec(ci.PAR2D_64)
y = torch.rand(small.sino_shape, device="cuda"); ct.backproject_B(small, y, "un")
small.close(); torch.cuda.synchronize()
free0, total = torch.cuda.mem_get_info()
out = []
for _ in range(2):
    g, h = ct.Geometry.from_spec(ci.CONE_256), ct.Geometry.from_spec(ci.CONE_SMALL)
    y = torch.rand(g.sino_shape, device="cuda"); x = torch.empty(g.vol_shape, device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ct.ct_backproject_B(g, y, x, "un"); torch.cuda.synchronize()
    kept = before - torch.cuda.mem_get_info()[0]
    g.close()
    still = before - torch.cuda.mem_get_info()[0]
    h.close(); del x, y; torch.cuda.empty_cache(); torch.cuda.synchronize()
    out.append([kept, still, free0 - torch.cuda.mem_get_info()[0]])
print(json.dumps([total, out]))
"""


def test_the_pool_is_bounded_and_given_back(ct):
    r = subprocess.run([sys.executable, "-c", SCRIPT % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    total, rounds = json.loads(r.stdout.strip().splitlines()[-1])
    for kept, still, lost in rounds:
        assert 0 < kept <= total // 32 + (64 << 20)   # (the driver maps in blocks of some MiB)
        assert still > 0                                # another geometry lives
        assert lost <= 64 << 20                         # the last one is gone


def test_geometries_come_and_go_on_several_threads(ct):
    specs = [ci.CONE_SMALL, ci.CONE_ANISO, ci.CONE_THIN, ci.PAR2D_64]
    ref = []
    for i, s in enumerate(specs):
        g = ct.Geometry.from_spec(s)
        b = ct.project_A(g, torch.from_numpy(ci.phantom(s, seed=i)[0]).cuda())
        x = torch.empty(s.vol_shape, device="cuda")
        r = ct.ct_bagmres_solve(g, b, 4, x, ct.make_opts(b_kind="fbp"), workspace=None)
        ref.append((b, x.cpu().numpy(), r.resid.copy()))
        g.close()
    gc.collect()
    errors = []

    def work(i):
        try:
            st = torch.cuda.Stream()
            for _ in range(12):
                g = ct.Geometry.from_spec(specs[i])
                x = torch.empty(specs[i].vol_shape, device="cuda")
                st.wait_stream(torch.cuda.default_stream())
                r = ct.ct_bagmres_solve(g, ref[i][0], 4, x, ct.make_opts(b_kind="fbp"), stream=st, workspace=None)
                y = torch.empty(specs[i].sino_shape, device="cuda")
                ct.ct_project_A(g, x, y, stream=st)
                st.synchronize()
                g.close()   # others' calls in flight, and now and then the last geometry
                assert np.array_equal(x.cpu().numpy(), ref[i][1]) and np.array_equal(r.resid, ref[i][2])
        except Exception as e:   # reported below
            errors.append((i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(specs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert not any(t.is_alive() for t in threads) and not errors, errors
