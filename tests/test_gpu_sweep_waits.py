"""The one-launch Gram-Schmidt sweep where its waits run out, and where it cannot
be launched, both made on the host (ct_fault_set): a block that publishes nothing
ends the solve with CT_ETIMEOUT, the iterations before it intact, and the next
start on the same state solves as if nothing had been; a refused cooperative
launch gives way to single passes with the same bits, also in the middle of a
solve.
"""
import numpy as np
import pytest
import torch

import ct_inputs as ci


@pytest.fixture(scope="module")
def ct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2201_07408_gb300 import ct as _ct
    yield _ct
    _ct.fault_set(None)


@pytest.mark.parametrize("spec,canon", [("sweep_stall:3", "sweep_stall:3"), ("sweep_refused", "sweep_refused"),
                                        ("sweep_refused,sweep_stall:2,oom,nan_at_iter:9",
                                         "nan_at_iter:9,oom,sweep_stall:2,sweep_refused")])
def test_fault_specs(ct, spec, canon):
    ct.fault_set(spec)
    assert ct.fault_get() == canon
    ct.fault_set(None)


@pytest.mark.parametrize("bad", ["sweep_stall", "sweep_stall:0", "sweep_stall:x", "sweep_refused:1", "sweep_stalls:1"])
def test_malformed_fault_specs(ct, bad):
    with pytest.raises(ct.CTError):
        ct.fault_set(bad)
    assert ct.fault_get() == ""


# 11 blocks (16 elements a thread), and every SM with 32 elements a thread
SCANS = [ci.CONE_SMALL, ci._cone("cone_128x120x82", 0, 1.0, 5, 40, 20, 7.0, nxyz=(128, 120, 82))]


@pytest.fixture(params=SCANS, ids=lambda s: s.name)
def scan(request, ct):
    spec = request.param
    g = ct.Geometry.from_spec(spec)
    b = ct.project_A(g, torch.from_numpy(ci.phantom(spec)[0]).cuda())
    return spec, g, b


@pytest.mark.gpu
@pytest.mark.parametrize("reorth", [0, 1])
def test_a_silent_block_ends_the_solve(ct, scan, reorth):
    spec, g, b = scan
    opts = lambda: ct.make_opts(b_kind="un", reorth=reorth)
    x, y = torch.empty(spec.vol_shape, device="cuda"), torch.empty(spec.vol_shape, device="cuda")
    clean = ct.ct_bagmres_solve(g, b, 6, x, opts())
    for stall in (1, 4):
        ct.fault_set("sweep_stall:%d" % stall)
        try:
            with pytest.raises(ct.CTError) as ei:
                ct.ct_bagmres_solve(g, b, 6, y, opts())
        finally:
            ct.fault_set(None)
        assert ei.value.status == ct.CT_ETIMEOUT
        r = ei.value.result
        assert r.iters == stall - 1
        np.testing.assert_array_equal(r.resid[:stall], clean.resid[:stall])
        assert np.all(r.resid[stall:] == -1.0)
    again = ct.ct_bagmres_solve(g, b, 6, y, opts())
    assert torch.equal(x, y) and np.array_equal(again.resid, clean.resid)


@pytest.mark.gpu
def test_a_state_starts_again_after_a_stall(ct, scan):
    spec, g, b = scan
    x, y = torch.empty(spec.vol_shape, device="cuda"), torch.empty(spec.vol_shape, device="cuda")
    st = ct.GmresState(g, 6, "device", ct.make_opts(b_kind="un"))
    st.start(b)
    clean = st.extend(6, x)
    st.start(b)
    st.extend(2, y)
    ct.fault_set("sweep_stall:3")
    try:
        with pytest.raises(ct.CTError) as ei:
            st.extend(6, y)
    finally:
        ct.fault_set(None)
    assert ei.value.status == ct.CT_ETIMEOUT and st.iters == 2
    st.start(b)   # finds the slots as the stall left them
    res = st.extend(6, y)
    assert torch.equal(x, y) and np.array_equal(res.resid, clean.resid)
    st.close()


@pytest.mark.gpu
@pytest.mark.parametrize("reorth", [0, 1])
@pytest.mark.parametrize("refused", [(0, 6), (2, 3), (1, 4)], ids=str)
def test_refused_launches_give_way_to_passes(ct, scan, refused, reorth):
    spec, g, b = scan
    x, y = torch.empty(spec.vol_shape, device="cuda"), torch.empty(spec.vol_shape, device="cuda")
    clean = ct.ct_bagmres_solve(g, b, 6, x, ct.make_opts(b_kind="un", reorth=reorth))
    st = ct.GmresState(g, 6, "device", ct.make_opts(b_kind="un", reorth=reorth))
    st.start(b)
    for k in range(1, 7):
        ct.fault_set("sweep_refused" if refused[0] < k <= refused[1] else None)
        try:
            res = st.extend(k, y)
        finally:
            ct.fault_set(None)
    assert torch.equal(x, y) and np.array_equal(res.resid, clean.resid)
    st.close()
