"""The work that is timed: single operators, training steps and whole solves on
scans from a 64 x 64 slice to a 512^3 cone-beam volume.

A case names an operation (``op``) and the scan it runs on.  The scans are
the framework's workloads (the 128 mm field of view at 64^2, 128^3, 256^3 and
512^3) and grids of the same kind with odd sizes.  Inputs are what the
operation meets in use: volumes are reconstructed images (ellipsoid phantoms
with noise), sinograms are noisy measured data (analytic line integrals of
the phantom, photon noise), image gradients are dense.

``exact`` evaluates the same operators from their definitions in 64 bits with
torch: Joseph's bilinear samples, the voxel-driven bilinear back-projection,
the linear ramp convolution, ray lengths from sorted plane crossings, and
GMRES / CGLS over those.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_07408_gb300 import autograd as ct_autograd
from paper_2201_07408_gb300 import ct

PARALLEL, CONE = 0, 1


# --- cases ------------------------------------------------------------------------
def _scan(op, nx, ny, nz, views, nu, nv, du, dv=None, vox=None, kind=CONE, ang0=0.0, span=2 * math.pi,
          sod=500.0, sdd=1000.0, b_kind="un", k=0, vol="f32", sino="f32", projector="joseph", **more):
    return dict(op=op, kind=kind, nx=nx, ny=ny, nz=nz, vox=128.0 / max(nx, ny) if vox is None else vox,
                views=views, ang0=ang0, span=span, nu=nu, nv=nv, du=du, dv=du if dv is None else dv, sod=sod,
                sdd=sdd, b_kind=b_kind, k=k, vol=vol, sino=sino, projector=projector, **more)


def _par2d(op, n, views, nu, **more):
    return _scan(op, n, n, 1, views, nu, 1, 1.0, dv=1.0, vox=1.0, kind=PARALLEL, span=math.pi, **more)


def listed():
    return [
        # one forward projection of a 2D slice: the smallest call, in loops of users' own iterations
        _par2d("A", 64, 90, 95, name="project_2d_64"),
        # a whole small solve: ten BA-GMRES iterations on the noisy 2D scan, bound by its launches
        _par2d("ba", 64, 90, 95, k=10, name="bagmres_2d_64"),
        # one step of a data-fidelity loss on a small odd volume: projection and its exact transpose
        _scan("step", 40, 36, 28, 45, 70, 30, 4.0, dv=4.5, vox=3.0, ang0=0.3, name="train_step_40x36x28"),
        # projection with BF16 copies of a ragged volume (short scan)
        _scan("A", 150, 131, 97, 211, 233, 151, 1.25, ang0=0.2, span=3.6, vol="bf16", name="project_bf16_150x131x97"),
        # the projection of the 256^3 scan: half of every iteration there
        _scan("A", 256, 256, 256, 360, 384, 256, 0.75, name="project_256"),
        # FDK reconstruction of a ragged mid-size scan
        _scan("B", 181, 175, 90, 271, 301, 157, 0.95, b_kind="fbp", ang0=0.1, name="fbp_181x175x90"),
        # unfiltered back-projection of the 256^3 scan from BF16 storage
        _scan("B", 256, 256, 256, 360, 384, 256, 0.75, sino="bf16", name="backproject_bf16_256"),
        # the matched transpose on the 256^3 scan (gradient of a data term, matched CGLS)
        _scan("At", 256, 256, 256, 360, 384, 256, 0.75, name="adjoint_256"),
        # the gradient through a converged solve: GMRES on the transposes
        _scan("vjp", 128, 128, 128, 128, 192, 128, 1.5, b_kind="fbp", k=6, name="solve_vjp_128"),
        # a training step with the line-intersection projector
        _scan("step", 128, 128, 128, 128, 192, 128, 1.5, ang0=0.1, projector="siddon", name="train_step_siddon_128"),
        # a whole solve at 128^3: BA-GMRES with the filtered back-projector
        _scan("ba", 128, 128, 128, 128, 192, 128, 1.5, b_kind="fbp", k=20, name="bagmres_128"),
        # FDK reconstruction of the 512^3 scan: the largest single call
        _scan("B", 512, 512, 512, 720, 768, 512, 0.375, b_kind="fbp", name="fbp_512"),
    ]


def draw(rng):
    op = rng.choice(["A", "A", "B", "B", "At", "Bt", "step", "ba", "ab", "cgls", "vjp"])
    solve = op in ("ba", "ab", "cgls", "vjp")
    b_kind = rng.choice(["un", "fbp"]) if op in ("B", "Bt", "ba") else "fbp" if op in ("vjp", "ab") else "un"
    k = rng.randint(3, 8) if solve else 0
    if rng.random() < 0.15:   # a 2D slice
        n = int(round(math.exp(rng.uniform(math.log(48), math.log(512)))))
        nu = int(n * rng.uniform(1.2, 1.6))
        return _scan(op, n, max(8, int(n * rng.uniform(0.7, 1.0))), 1, max(8, int(n * rng.uniform(0.5, 1.4))), nu, 1,
                     1.0, dv=1.0, vox=1.0, kind=PARALLEL, ang0=rng.uniform(0, 6.28), span=math.pi, b_kind=b_kind, k=k)
    n = int(round(math.exp(rng.uniform(math.log(32), math.log(112 if solve else 240)))))
    m = max(8, int(n * rng.uniform(0.75, 1.0)))
    nx, ny = (n, m) if rng.random() < 0.5 else (m, n)
    nz = max(6, int(n * rng.uniform(0.3, 1.0)))
    vox = 128.0 / n
    sod = rng.uniform(400.0, 700.0)
    sdd = sod * rng.uniform(1.5, 2.2)
    nu = int(n * rng.uniform(1.2, 1.6))
    nv = max(5, int(nz * rng.uniform(0.9, 1.3)))
    du = 144.0 * (sdd / sod) * rng.uniform(0.85, 1.1) / nu
    dv = du * rng.uniform(0.9, 1.2)
    projector = "siddon" if op in ("A", "step") and rng.random() < 0.3 else "joseph"
    vol = "bf16" if op == "A" and projector == "joseph" and rng.random() < 0.4 else "f32"
    sino = "bf16" if op == "B" and b_kind == "un" and rng.random() < 0.4 else "f32"
    if projector == "siddon":   # no detector row in a voxel boundary plane, where a ray's lengths are a convention
        nv += (nv ^ nz) & 1
    return _scan(op, nx, ny, nz, max(12, int(n * rng.uniform(0.7, 1.4))), nu, nv, du, dv=dv, vox=vox,
                 ang0=rng.uniform(0, 6.28), span=rng.choice([2 * math.pi, 2 * math.pi, 3.6]), sod=sod, sdd=sdd,
                 b_kind=b_kind, k=k, vol=vol, sino=sino, projector=projector)


# --- inputs -----------------------------------------------------------------------
def _axes(c, dtype, dev):
    return [(torch.arange(n, dtype=dtype, device=dev) - (n - 1) / 2.0) * c["vox"] for n in (c["nx"], c["ny"], c["nz"])]


def _ellipsoids(c, seed):
    """Twelve ellipsoids (ellipses in 2D) inside the field of view: centre, semi-axes, rotation, density."""
    rng = np.random.default_rng([seed, 77])
    r = 0.5 * min(c["nx"], c["ny"]) * c["vox"]
    zh = 0.45 * c["nz"] * c["vox"]
    out = []
    for _ in range(12):
        q = rng.standard_normal(4)
        q /= np.linalg.norm(q)
        if c["kind"] == PARALLEL:
            q[1] = q[2] = 0.0
            q /= np.linalg.norm(q)
        w, x, y, z = q
        rot = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                        [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                        [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])
        semi = rng.uniform(0.08, 0.47, 3) * r
        rad, ph = 0.5 * r * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        cz = 0.0
        if c["kind"] == PARALLEL:
            semi[2] = 1e6
        else:
            semi = np.minimum(semi, rng.uniform(0.3, 0.8) * zh)
            cz = rng.uniform(-1, 1) * (zh - semi.max())
        out.append((np.array([rad * math.cos(ph), rad * math.sin(ph), cz]), semi, rot, rng.uniform(0.002, 0.02)))
    return out


def _image(c, seed, dev):
    """A reconstructed image: the phantom plus noise of 3 % of its range in every voxel."""
    x, y, z = _axes(c, torch.float32, dev)
    vol = torch.zeros(c["nz"], c["ny"], c["nx"], device=dev)
    for cen, semi, rot, dens in _ellipsoids(c, seed):
        q = torch.zeros_like(vol)
        for a in range(3):
            f = rot[:, a] / semi[a]
            q += ((z - cen[2]) * f[2])[:, None, None].add((y - cen[1])[:, None] * f[1] + (x - cen[0]) * f[0]).square_()
        vol += (q <= 1.0) * dens
    gen = torch.Generator(device=dev).manual_seed(int(seed) * 2 + 1)
    vol += torch.randn(vol.shape, device=dev, generator=gen) * 0.0006
    return vol


def _data(c, seed, dev):
    """Measured data -log(counts / I0): the phantom's line integrals with photon noise (I0 = 1e5)."""
    ells = _ellipsoids(c, seed)
    b = torch.empty(c["views"], c["nv"], c["nu"], device=dev)
    for s in range(c["views"]):
        S, d = _rays(c, s, dev, torch.float32)
        dn = torch.sqrt(sum(t * t for t in d))
        p = 0.0
        for cen, semi, rot, dens in ells:
            a1 = a2 = bb = 0.0
            for a in range(3):
                f = rot[:, a] / semi[a]
                o = (S[0] - cen[0]) * f[0] + (S[1] - cen[1]) * f[1] + (S[2] - cen[2]) * f[2]
                e = d[0] * f[0] + d[1] * f[1] + d[2] * f[2]
                a1, a2, bb = a1 + e * e, a2 + o * o, bb + o * e
            p = p + torch.sqrt(torch.clamp(bb * bb - a1 * (a2 - 1.0), min=0.0)) / a1 * (2.0 * dens)
        b[s] = p * dn
    gen = torch.Generator(device=dev).manual_seed(int(seed) * 2)
    if c["kind"] == PARALLEL:
        return b + torch.randn(b.shape, device=dev, generator=gen) * (0.01 * b.max())
    counts = 1e5 * torch.exp(-b)   # mean counts are in the thousands and more: the Gaussian limit of the photon noise
    counts += torch.sqrt(counts) * torch.randn(b.shape, device=dev, generator=gen)
    return -torch.log(torch.clamp(counts, min=1.0) / 1e5)


def prepare(case, seed):
    c, dev = case, torch.device("cuda", torch.cuda.current_device())
    geom = ct.Geometry(c["kind"], c["nx"], c["ny"], c["nz"], c["vox"], c["views"], c["ang0"], c["span"], c["nu"],
                       c["nv"], c["du"], c["dv"], c["sod"], c["sdd"], device=dev, vol_dtype=c["vol"],
                       sino_dtype=c["sino"], projector=c["projector"])
    st = {"case": c, "geom": geom}
    if c["op"] in ("A", "Bt", "step", "vjp"):
        st["x"] = _image(c, seed, dev)
    if c["op"] in ("B", "At", "step", "ba", "ab", "cgls"):
        st["b"] = _data(c, seed, dev)
    return st


# --- one pass ---------------------------------------------------------------------
def run(state):
    c, g, op = state["case"], state["geom"], state["case"]["op"]
    if op == "A":
        return ct.project_A(g, state["x"])
    if op == "B":
        return ct.backproject_B(g, state["b"], c["b_kind"])
    if op == "At":
        return ct.adjoint_At(g, state["b"])
    if op == "Bt":
        return ct.adjoint_Bt(g, state["x"], c["b_kind"])
    if op == "step":
        x = state["x"].detach().requires_grad_(True)
        y = ct_autograd.project_A(g, x)
        (0.5 * (y - state["b"]).square().sum()).backward()
        return [y.detach(), x.grad]
    if op == "vjp":
        gb = torch.empty(g.sino_shape, dtype=torch.float32, device=g.device)
        res = ct.ct_bagmres_vjp(g, state["x"], c["k"], gb, ct.make_opts(b_kind=c["b_kind"]))
        return [gb, res.resid.astype(np.float32)]
    solve = {"ba": ct.bagmres, "ab": ct.abgmres, "cgls": ct.cgls}[op]
    x, res = solve(g, state["b"], c["k"], b_kind=c["b_kind"])
    # the residual history comes from single-precision operators: as such numbers it is compared
    return [x, res.resid.astype(np.float32)]


def work(case):
    """Bytes: inputs and outputs once (and the basis of a solve: each new vector is orthogonalised against all
    before it, so each is read once and written once an iteration).  Flops: one bilinear sample (4 products, 4
    sums) for each ray and plane of a projection or its transpose and for each voxel and view of a
    back-projection or its transpose, the crossed voxels for the line-intersection projector, 5 N log2 N for
    each transform of a filtered row, 4 a basis element and vector."""
    c = case
    n, m = c["nx"] * c["ny"] * c["nz"], c["views"] * c["nv"] * c["nu"]
    rows = c["views"] * c["nv"]
    nf = 2 ** math.ceil(math.log2(2 * c["nu"] - 1))
    steps = max(c["nx"], c["ny"])
    fa = m * (2.0 * (steps + c["nx"] // 2) if c["projector"] == "siddon" else 8.0 * steps)
    fb = 8.0 * n * c["views"] + (rows * 5.0 * nf * math.log2(nf) if c["b_kind"] == "fbp" else 0.0)
    io, op, k = 4.0 * (n + m), c["op"], c["k"]
    if op in ("A", "At"):
        return {"bytes": io, "flops": fa}
    if op in ("B", "Bt"):
        return {"bytes": io, "flops": fb}
    if op == "step":
        return {"bytes": 2 * io + 4.0 * m, "flops": 2 * fa}
    length = m if op == "ab" else n
    sweeps = 0 if op == "cgls" else k * (k + 1) / 2
    return {"bytes": io + 4.0 * length * (sweeps + k), "flops": (k + 1) * fb + k * fa + 4.0 * length * sweeps}


# --- the same in 64 bits ------------------------------------------------------------
def _rays(c, s, dev, dtype=torch.float64):
    """A point and the direction (three tensors that broadcast to nv x nu) of the rays of view s."""
    th = c["ang0"] + s * c["span"] / c["views"]
    co, si = math.cos(th), math.sin(th)
    u = ((torch.arange(c["nu"], dtype=dtype, device=dev) - (c["nu"] - 1) / 2.0) * c["du"])[None, :]
    v = ((torch.arange(c["nv"], dtype=dtype, device=dev) - (c["nv"] - 1) / 2.0) * c["dv"])[:, None]
    zero = torch.zeros_like(u)
    if c["kind"] == PARALLEL:
        return (u * co, u * si, zero), (zero - si, zero + co, zero)
    return ((zero + c["sod"] * co, zero + c["sod"] * si, zero),
            (-c["sdd"] * co - u * si, -c["sdd"] * si + u * co, v.expand(-1, c["nu"])))


def _planes(c, s, dev):
    """For each dominant axis of view s: (x-dominant?, columns, sample grid, step lengths)."""
    S, d = _rays(c, s, dev)
    xdom = (d[0].abs() >= d[1].abs() * (1 - 1e-9)).reshape(-1)
    x, y, _ = _axes(c, torch.float64, dev)
    for is_x in (True, False):
        cols = torch.nonzero(xdom if is_x else ~xdom).reshape(-1)
        if not cols.numel():
            continue
        (Sa, Sb, Sz), (da, db, dz) = [[t[..., cols] for t in (q if is_x else (q[1], q[0], q[2]))] for q in (S, d)]
        a = (x if is_x else y)[:, None, None]
        nb = c["ny"] if is_x else c["nx"]
        t = (a - Sa) / da
        fb = (Sb + t * db) / c["vox"] + (nb - 1) / 2.0
        fz = (Sz + t * dz) / c["vox"] + (c["nz"] - 1) / 2.0
        shape = (a.shape[0], c["nv"], cols.numel())
        grid = torch.stack([((2 * fb + 1) / nb - 1).expand(shape), ((2 * fz + 1) / c["nz"] - 1).expand(shape)], -1)
        yield is_x, cols, grid, c["vox"] * torch.sqrt(da * da + db * db + dz * dz) / da.abs()


def _sample(img, grid):
    return torch.nn.functional.grid_sample(img, grid, mode="bilinear", padding_mode="zeros", align_corners=False)


def _spread(out, img, grid):
    """The transpose of _sample."""
    return torch.ops.aten.grid_sampler_2d_backward(out, img, grid, 0, 0, False, [True, False])[0]


def _A64(c, vol):
    if c["projector"] == "siddon":
        return _siddon64(c, vol, None)
    y = torch.zeros(c["views"], c["nv"], c["nu"], dtype=torch.float64, device=vol.device)
    xs, ys = vol.permute(2, 0, 1)[:, None].contiguous(), vol.permute(1, 0, 2)[:, None].contiguous()
    for s in range(c["views"]):
        for is_x, cols, grid, step in _planes(c, s, vol.device):
            y[s][:, cols] = _sample(xs if is_x else ys, grid).sum((0, 1)) * step
    return y


def _At64(c, y):
    if c["projector"] == "siddon":
        return _siddon64(c, None, y)
    xs = torch.zeros(c["nx"], 1, c["nz"], c["ny"], dtype=torch.float64, device=y.device)
    ys = torch.zeros(c["ny"], 1, c["nz"], c["nx"], dtype=torch.float64, device=y.device)
    for s in range(c["views"]):
        for is_x, cols, grid, step in _planes(c, s, y.device):
            acc = xs if is_x else ys
            acc += _spread((y[s][:, cols] * step).expand(grid.shape[0], 1, -1, -1).contiguous(), acc, grid)
    return xs[:, 0].permute(1, 2, 0) + ys[:, 0].permute(1, 0, 2)


def _siddon64(c, vol, y):
    """Line-intersection projection of vol, or its transpose on y, from sorted plane crossings."""
    dev = (vol if y is None else y).device
    n = (c["nx"], c["ny"], c["nz"])
    out = torch.zeros(c["views"], c["nv"], c["nu"], dtype=torch.float64, device=dev) if y is None else \
        torch.zeros(n[0] * n[1] * n[2], dtype=torch.float64, device=dev)
    for s in range(c["views"]):
        S, d = [[t.expand(c["nv"], c["nu"]).reshape(-1, 1) / c["vox"] for t in q] for q in _rays(c, s, dev)]
        ts, lo, hi = [], -math.inf, math.inf
        for a in range(3):
            t = (torch.arange(n[a] + 1, dtype=torch.float64, device=dev) - n[a] / 2.0 - S[a]) / d[a]
            par = d[a].abs() < 1e-12
            inside = (S[a] > -n[a] / 2.0) & (S[a] < n[a] / 2.0)
            t = torch.where(par, torch.where(inside, -math.inf, math.inf), t)
            first, last = torch.minimum(t[:, :1], t[:, -1:]), torch.maximum(t[:, :1], t[:, -1:])
            lo = torch.clamp(first, min=lo) if a == 0 else torch.maximum(lo, first)
            hi = torch.where(par & inside, math.inf, last) if a == 0 else \
                torch.minimum(hi, torch.where(par & inside, math.inf, last))
            ts.append(t)
        hi = torch.maximum(lo, hi)
        t = torch.sort(torch.minimum(torch.maximum(torch.cat(ts, 1), lo), hi), 1)[0]
        t = torch.nan_to_num(t, nan=0.0, posinf=0.0, neginf=0.0)
        length = (t[:, 1:] - t[:, :-1]) * torch.sqrt(sum(q * q for q in d))
        mid = 0.5 * (t[:, 1:] + t[:, :-1])
        idx, ok = 0, length > 0
        for a in (2, 1, 0):
            i = torch.floor(S[a] + mid * d[a] + n[a] / 2.0).long()
            ok = ok & (i >= 0) & (i < n[a])
            idx = idx * n[a] + i
        idx, length = torch.where(ok, idx, 0), torch.where(ok, length, 0.0) * c["vox"]
        if y is None:
            out[s] = (vol.reshape(-1)[idx] * length).sum(1).reshape(c["nv"], c["nu"])
        else:
            out.index_add_(0, idx.reshape(-1), (length * y[s].reshape(-1, 1)).reshape(-1))
    return out if y is None else out.reshape(n[::-1])


def _voxel_grid(c, s, dev):
    """Detector position of every voxel in view s as a sample grid, and the weights of its columns."""
    x, y, z = _axes(c, torch.float64, dev)
    th = c["ang0"] + s * c["span"] / c["views"]
    co, si = math.cos(th), math.sin(th)
    if c["kind"] == PARALLEL:
        u = (x * co)[None, :] + (y * si)[:, None]
        mag, kb = torch.ones_like(u), c["vox"] ** 2 / c["du"]
    else:
        mag = c["sdd"] / (c["sod"] - (x * co)[None, :] - (y * si)[:, None])
        u = mag * ((y * co)[:, None] - (x * si)[None, :])
        kb = c["vox"] ** 3 / (c["du"] * c["dv"])
    shape = (1, c["nz"], c["ny"] * c["nx"])
    gu = (2 * (u / c["du"] + (c["nu"] - 1) / 2.0) + 1) / c["nu"] - 1
    gv = (2 * (z[:, None] * mag.reshape(1, -1) / c["dv"] + (c["nv"] - 1) / 2.0) + 1) / c["nv"] - 1
    return torch.stack([gu.reshape(1, 1, -1).expand(shape), gv[None].expand(shape)], -1), (kb * mag * mag).reshape(-1)


def _F64(c, y, transpose=False):
    u = (torch.arange(c["nu"], dtype=torch.float64, device=y.device) - (c["nu"] - 1) / 2.0) * c["du"]
    v = (torch.arange(c["nv"], dtype=torch.float64, device=y.device) - (c["nv"] - 1) / 2.0) * c["dv"]
    if c["kind"] == PARALLEL:
        cosw, tau = 1.0, c["du"]
        scale = math.pi / c["views"] * c["du"] / c["vox"] ** 2 * tau
    else:
        r = c["sod"] / c["sdd"]
        cosw, tau = c["sdd"] / torch.sqrt(c["sdd"] ** 2 + u[None, :] ** 2 + v[:, None] ** 2), c["du"] * r
        scale = math.pi / c["views"] * r * r * c["du"] * c["dv"] / c["vox"] ** 3 * tau
    q = torch.arange(c["nu"], dtype=torch.float64, device=y.device)
    h = torch.where(q % 2 == 1, -1.0 / (math.pi * q.clamp(min=1.0) * tau) ** 2, 0.0)
    h[0] = 1.0 / (4.0 * tau * tau)
    ln = 2 * c["nu"]
    kern = torch.zeros(ln, dtype=torch.float64, device=y.device)
    kern[:c["nu"]] = h
    kern[ln - c["nu"] + 1:] = h[1:].flip(0)
    spec = torch.fft.rfft(kern * scale)
    y = y if transpose else y * cosw
    y = torch.fft.irfft(torch.fft.rfft(y, ln) * spec, ln)[..., :c["nu"]]
    return y * cosw if transpose else y


def _B64(c, y):
    if c["b_kind"] == "fbp":
        y = _F64(c, y)
    if c["sino"] == "bf16":
        y = y.to(torch.bfloat16).double()
    x = torch.zeros(c["nz"], c["ny"] * c["nx"], dtype=torch.float64, device=y.device)
    for s in range(c["views"]):
        grid, w = _voxel_grid(c, s, y.device)
        x += _sample(y[s][None, None], grid)[0, 0] * w
    return x.reshape(c["nz"], c["ny"], c["nx"])


def _Bt64(c, x):
    y = torch.zeros(c["views"], c["nv"], c["nu"], dtype=torch.float64, device=x.device)
    x = x.reshape(c["nz"], -1)
    for s in range(c["views"]):
        grid, w = _voxel_grid(c, s, x.device)
        y[s] = _spread((x * w)[None, None].contiguous(), y[s][None, None], grid)[0, 0]
    return _F64(c, y, True) if c["b_kind"] == "fbp" else y


def _gmres64(op, r0, k):
    """(basis, coefficients of x_k, residual history) of k GMRES iterations on op z = r0."""
    beta = r0.norm()
    V, H = [r0 / beta], np.zeros((k + 1, k))
    hist, y = [float(beta)], None
    for j in range(k):
        q = op(V[j])
        for i in range(j + 1):
            H[i, j] = float((q * V[i]).sum())
            q = q - H[i, j] * V[i]
        H[j + 1, j] = float(q.norm())
        V.append(q / H[j + 1, j])
        e = np.zeros(j + 2)
        e[0] = hist[0]
        y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
        hist.append(float(np.linalg.norm(H[:j + 2, :j + 1] @ y - e)))
    return sum(float(a) * v for a, v in zip(y, V)), np.array(hist)


def exact(case, seed):
    c, op = case, case["op"]
    n, m = c["nx"] * c["ny"] * c["nz"], c["views"] * c["nv"] * c["nu"]
    a, b = float(m) * max(c["nx"], c["ny"]), float(n) * c["views"]
    # seconds that these evaluations take, from the samples of each kind
    k = max(1, c["k"])
    if {"A": a, "B": b, "At": 2 * a, "Bt": 2 * b, "step": 3 * a, "vjp": 2 * k * (a + b)}.get(op, k * (a + b)) > 2.2e10:
        return None
    st = prepare(c, seed)
    x, y = (st[t].double() if t in st else None for t in ("x", "b"))
    if op == "A":
        return _A64(c, x.to(torch.bfloat16).double() if c["vol"] == "bf16" else x)
    if op == "B":
        return _B64(c, y)
    if op == "At":
        return _At64(c, y)
    if op == "Bt":
        return _Bt64(c, x)
    if op == "step":
        p = _A64(c, x)
        return [p, _At64(c, p - y)]
    if op == "ba":
        z, hist = _gmres64(lambda v: _B64(c, _A64(c, v)), _B64(c, y), k)
        return [z, hist]
    if op == "ab":
        z, hist = _gmres64(lambda v: _A64(c, _B64(c, v)), y, k)
        return [_B64(c, z), hist]
    if op == "vjp":
        z, hist = _gmres64(lambda v: _At64(c, _Bt64(c, v)), x, k)
        return [_Bt64(c, z), hist]
    z, r, hist = torch.zeros(c["nz"], c["ny"], c["nx"], dtype=torch.float64, device=y.device), y, [float(y.norm())]
    s = _B64(c, r)
    p, gamma = s, float(s.square().sum())
    for _ in range(k):
        q = _A64(c, p)
        alpha = gamma / float(q.square().sum())
        z, r = z + alpha * p, r - alpha * q
        s = _B64(c, r)
        new = float(s.square().sum())
        p, gamma = s + (new / gamma) * p, new
        hist.append(float(r.norm()))
    return [z, np.array(hist)]
