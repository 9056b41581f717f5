"""The work that a user of the library has it do, as timed cases.

Each case is one call (or one forward and backward call) of the Python binding on
device-resident fields, with the plan and the output buffers kept between calls, as a
time-stepping program keeps them.  Sizes are this repository's own: its test and benchmark
grids, and grids of the same ranges."""
import math

import numpy as np
import torch

from paper_2609_19130_gb300 import FP64, MIXED, Grid, Plan, Projection
from paper_2609_19130_gb300 import _native as N

FFT_SIZES = (1, 2, 3, 4, 6, 8, 12, 16, 24, 32)
# every supported number of cells along x and y from 16 on
XY_SIZES = sorted({a * b for a in FFT_SIZES for b in FFT_SIZES if a * b >= 16})
BATCH_XY, BATCH_Z = (64, 96, 128, 192), (64, 128, 256)
# no drawn case is larger than the largest listed one; fp64 and one-sweep cases stay smaller
MOST_CELLS, MOST_CELLS_FP64, MOST_CELLS_ONE_SWEEP = 1024 * 1024 * 512, 1 << 25, 1 << 25


def _case(kind, nx, ny, nz, beta, precision="mixed", refine=1, **more):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "beta": beta, "precision": precision,
         "refine": refine if precision == "mixed" else 0, "dt": 1e-3}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one fp64 projection of a test-sized uniform grid (latency)
        dict(_case("project", 32, 32, 32, 0.0, "fp64"), name="fp64_32"),
        # a small, ragged grid of a coarse run or of a development loop, default precision
        dict(_case("project", 96, 72, 45, 2.0), name="mixed_96x72x45"),
        # the mid-size channel in both precisions, z clustered at the walls
        dict(_case("project", 256, 256, 256, 2.0, "fp64"), name="fp64_256"),
        dict(_case("project", 256, 256, 256, 2.0), name="mixed_256"),
        # the DNS channel with its implicit pressure update, two refinement sweeps
        dict(_case("pressure", 384, 384, 192, 2.0, refine=2), name="channel_384x384x192"),
        # the benchmark's DNS-scale grid and input, two refinement sweeps
        dict(_case("project", 1024, 1024, 512, 2.5, refine=2), name="dns_1024x1024x512"),
        # a jet domain: an open top (phi = 0 there), long in x, an odd number of levels
        dict(_case("outlet", 512, 192, 301, 1.5, refine=2), name="outlet_512x192x301"),
        # a closed box: walls in x and y as well (cosine transforms)
        dict(_case("walls", 256, 192, 129, 2.0), name="walls_256x192x129"),
        # a batch of independent uneven grids, each with its own stretching
        dict(_case("batch", 0, 0, 0, 0.0, refine=2, grids=64, sizes=1), name="batch_64"),
        # a training step through the differentiable projection: forward and gradients
        dict(_case("grad", 256, 256, 256, 2.0, grids=8), name="grad_8x256"),
        # the implicit viscous solve of the velocity that precedes each projection
        dict(_case("viscous", 384, 384, 192, 2.0, diffusion=1e-4), name="viscous_384x384x192"),
        dict(_case("viscous", 192, 144, 101, 1.5, "fp64", diffusion=1e-3), name="viscous_fp64_192x144x101"),
    ]


def draw(rng):
    kind = rng.choice(("project", "project", "project", "pressure", "outlet", "walls", "batch", "grad", "viscous"))
    precision = "fp64" if rng.random() < 0.3 else "mixed"
    refine = rng.choice((1, 2))
    beta = 0.0 if rng.random() < 0.2 else round(rng.uniform(1.0, 2.5), 3)
    if kind == "batch":
        return _case(kind, 0, 0, 0, 0.0, precision, refine,
                     grids=rng.randint(2, 24 if precision == "fp64" else 64), sizes=rng.randint(2, 1 << 20))
    grids = rng.randint(1, 8) if kind == "grad" else 1
    most = MOST_CELLS_FP64 if precision == "fp64" else MOST_CELLS_ONE_SWEEP if refine == 1 else MOST_CELLS
    if kind in ("grad", "viscous"):
        most = MOST_CELLS_FP64 // grids
    while True:
        nx, ny = (min(XY_SIZES, key=lambda s, t=math.exp(rng.uniform(math.log(16), math.log(1024))): abs(s - t))
                  for _ in range(2))
        nz = round(math.exp(rng.uniform(math.log(9), math.log(512))))
        if 4096 <= nx * ny * nz <= most:
            break
    more = {}
    if kind == "grad":
        more["grids"] = grids
    if kind == "viscous":
        more["diffusion"] = round(10 ** rng.uniform(-5, -2), 7)
    return _case(kind, nx, ny, nz, beta, precision, refine, **more)


# ------------------------------------------------------------------ grids and fields
def _z_faces(nz, beta, lz):
    s = np.arange(nz + 1) / nz
    return lz * s if beta == 0.0 else 0.5 * lz * (1.0 + np.tanh(beta * (2.0 * s - 1.0)) / math.tanh(beta))


def _grids(case):
    """(nx, ny, nz, lx, ly, lz, z faces, walls, outlet) of each grid of the case."""
    if case["kind"] == "batch":
        r = np.random.RandomState(case["sizes"])
        got = []
        for _ in range(case["grids"]):
            nx, ny, nz = int(r.choice(BATCH_XY)), int(r.choice(BATCH_XY)), int(r.choice(BATCH_Z))
            got.append((nx, ny, nz, 2 * math.pi, 2 * math.pi, 2.0, _z_faces(nz, float(r.uniform(1.0, 3.0)), 2.0),
                        False, False))
        return got
    nx, ny, nz, beta = case["nx"], case["ny"], case["nz"], case["beta"]
    box = (1.0, 1.0, 1.0) if nx == ny == nz and beta == 0.0 else (2 * math.pi, 2 * math.pi, 2.0)
    one = (nx, ny, nz) + box + (_z_faces(nz, beta, box[2]), case["kind"] == "walls", case["kind"] == "outlet")
    return [one] * (case["grids"] if case["kind"] == "grad" else 1)


def _shapes(grid):
    nx, ny, nz, wall = grid[0], grid[1], grid[2], int(grid[7])
    return (nz, ny, nx + wall), (nz, ny + wall, nx), (nz + 1, ny, nx)


def _seal(u, v, w, grid):
    """No flow through the walls."""
    w[0].zero_()
    if not grid[8]:
        w[-1].zero_()
    if grid[7]:
        for f in (u[:, :, 0], u[:, :, -1], v[:, 0], v[:, -1]):
            f.zero_()


def _velocity(case, grid, gen):
    """u*, v*, w*: smooth Fourier modes with an energy spectrum of k^-5/3 and a little noise where
    a resolved flow is meant (periodic x and y, 256 cells and more), else uniform in [-1, 1]."""
    nx, ny, nz = grid[:3]
    out = []
    for c, shape in enumerate(_shapes(grid)):
        f = torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen).mul_(2.0).sub_(1.0)
        if not grid[7] and min(nx, ny) >= 256 and case["kind"] != "grad":
            f.mul_(0.01)
            kx = torch.arange(nx // 2 + 1, device="cuda", dtype=torch.float64)
            ky = torch.fft.fftfreq(ny, 1.0 / ny, device="cuda", dtype=torch.float64)
            k2 = ky[:, None] ** 2 + kx[None, :] ** 2
            z = torch.arange(shape[0], device="cuda", dtype=torch.float64)
            z = z / nz if c == 2 else (z + 0.5) / nz
            for q in range(1 if c == 2 else 0, 33, 4):
                k = torch.sqrt(k2 + q * q)
                amp = torch.where((k > 0) & (k <= 32), k.clamp(min=1.0) ** (-11.0 / 6.0), torch.zeros_like(k))
                phase = torch.randn(amp.shape + (2,), dtype=torch.float64, device="cuda", generator=gen)
                plane = torch.fft.irfft2(torch.view_as_complex(phase) * amp, s=(ny, nx)) * (0.2 * nx * ny)
                prof = torch.sin(math.pi * q * z) if c == 2 else torch.cos(math.pi * q * z)
                f.addcmul_(prof[:, None, None], plane[None])
        out.append(f)
    _seal(*out, grid)
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _inputs(case, seed):
    """Per grid the fields that the call reads: velocity, and p_n or the gradients of a loss."""
    gen, got = _generator(seed), []
    for grid in _grids(case):
        f = _velocity(case, grid, gen)
        cells = (grid[2], grid[1], grid[0])
        if case["kind"] == "pressure":
            f.append(torch.rand(cells, dtype=torch.float64, device="cuda", generator=gen))
        if case["kind"] == "grad":  # d loss / d (u, v, w, phi): weights drawn from N(0, 1)
            f += [torch.randn(s, dtype=torch.float64, device="cuda", generator=gen) for s in _shapes(grid) + (cells,)]
        got.append(f)
    return got


def _flat(fields):
    """The fields of a batch in one buffer, and the view of each: a batch's outputs as its owner keeps them."""
    buf = torch.empty(sum(f.numel() for f in fields), dtype=torch.float64, device="cuda")
    views, at = [], 0
    for f in fields:
        views.append(buf[at:at + f.numel()].view(f.shape))
        at += f.numel()
    return buf, views


def prepare(case, seed):
    grids, fields = _grids(case), _inputs(case, seed)
    wall = N.IBF_BC_NEUMANN
    plan = Plan([Grid(g[0], g[1], g[2], g[3], g[4], g[5], zf=g[6], bc_x=wall if g[7] else N.IBF_BC_PERIODIC,
                      bc_y=wall if g[7] else N.IBF_BC_PERIODIC, bc_zhi=N.IBF_BC_DIRICHLET if g[8] else wall)
                 for g in grids],
                precision=FP64 if case["precision"] == "fp64" else MIXED, refine_steps=case["refine"],
                pressure=N.IBF_P_IMPLICIT if case["kind"] == "pressure" else N.IBF_P_PHI,
                inv_re=1e-3 if case["kind"] == "pressure" else 0.0)
    state = {"case": case, "plan": plan}
    if case["kind"] == "grad":  # one tensor per field with the grids as its leading dimension
        state["in"] = [torch.stack([f[i] for f in fields]).requires_grad_() for i in range(3)]
        state["grad"] = [torch.stack([f[i] for f in fields]) for i in range(3, 7)]
        return state
    cells = [torch.empty((g[2], g[1], g[0]), dtype=torch.float64, device="cuda") for g in grids]
    like = [[f[0], f[1], f[2], c] for f, c in zip(fields, cells)]
    if case["kind"] == "batch":
        cols = [_flat([row[i] for row in like]) for i in range(4)]
        state["whole"] = [buf for buf, _ in cols]
        state["out"] = [tuple(views[i] for _, views in cols) for i in range(len(grids))]
    else:
        state["out"] = [tuple(torch.empty_like(f) for f in row[:3 if case["kind"] == "viscous" else 4]) for row in like]
    state["in"] = [tuple(f) for f in fields]
    return state


def run(state):
    case, plan = state["case"], state["plan"]
    if case["kind"] == "viscous":
        return plan.viscous_solve(state["in"], case["diffusion"], out=state["out"])[0]
    if case["kind"] == "grad":
        out = Projection.apply(plan, case["dt"], 1.0, *state["in"])
        grads = torch.autograd.grad(out, state["in"], state["grad"])
        return {"out": [o.detach() for o in out], "grad": list(grads)}
    if case["kind"] == "batch":
        plan.project_batch(state["in"], case["dt"], out=state["out"])
        return state["whole"]
    f = state["in"][0]
    return plan.project(f[0], f[1], f[2], case["dt"], out=state["out"][0], p=f[3] if len(f) > 3 else None)


def work(case):
    nbytes = flops = 0.0
    for g in _grids(case):
        n = float(g[0]) * g[1] * g[2]
        fields = {"viscous": 6, "pressure": 8, "grad": 14}.get(case["kind"], 7)  # fp64 fields read or written
        nbytes += 8.0 * fields * n
        # transforms there and back (5/2 n log2 per real direction), sweeps, stencils; again for each sweep
        solve = 2 * 2.5 * (math.log2(g[0]) + math.log2(g[1])) + 14
        times = {"viscous": 3.0, "grad": 2.0 * (1 + case["refine"])}.get(case["kind"], 1.0 + case["refine"])
        flops += n * (times * solve + 30)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit values
def _transform(f, grid, back=False):
    """x and y transforms of the fields [nz, ny, nx]: Fourier where periodic, cosine at walls."""
    nx, ny = grid[:2]
    if not grid[7]:
        return torch.fft.irfft2(f, s=(ny, nx)) if back else torch.fft.rfft2(f)
    for axis, n in ((2, nx), (1, ny)):
        i = torch.arange(n, dtype=torch.float64, device="cuda")
        c = torch.cos(math.pi / (2 * n) * torch.remainder(i[:, None] * (2 * i[None, :] + 1), 4 * n))  # [mode, cell]
        if back:
            c = c * (2.0 / n)
            c[0] *= 0.5
        f = torch.tensordot(f, c, dims=([axis], [0 if back else 1])).movedim(-1, axis)
    return f


def _modes(grid):
    """Eigenvalues of the second differences along x and y, [ny, modes of x]."""
    nx, ny, wall = grid[0], grid[1], grid[7]
    m = torch.arange(nx if wall else nx // 2 + 1, dtype=torch.float64, device="cuda")
    n = torch.arange(ny, dtype=torch.float64, device="cuda")
    per = 2 if wall else 1
    lx = -4.0 * (nx / grid[3]) ** 2 * torch.sin(math.pi * m / (per * nx)) ** 2
    ly = -4.0 * (ny / grid[4]) ** 2 * torch.sin(math.pi * n / (per * ny)) ** 2
    return lx, ly


def _thomas(lo, up, diag, rhs):
    """Solves rows k of x[k-1] lo[k] + x[k] diag(k) + x[k+1] up[k] = rhs[k]; diag(k): per mode."""
    nz, cp = rhs.shape[0], []
    x = torch.empty_like(rhs)
    for k in range(nz):
        d = diag(k) - (lo[k] * cp[-1] if k else 0.0)
        cp.append(up[k] / d)
        x[k] = (rhs[k] - (lo[k] * x[k - 1] if k else 0.0)) / d
    for k in range(nz - 2, -1, -1):
        x[k] -= cp[k] * x[k + 1]
    return x


def _metrics(grid):
    zf = np.asarray(grid[6], dtype=np.float64)
    hz = np.diff(zf)
    gz = np.full(len(zf), np.inf)  # distances across the faces; no coupling at walls
    gz[1:-1] = 0.5 * (zf[2:] - zf[:-2])
    if grid[8]:
        gz[-1] = zf[-1] - 0.5 * (zf[-2] + zf[-1])
    return hz, gz


def _col(a):
    return torch.as_tensor(a, dtype=torch.float64, device="cuda")[:, None, None]


def _poisson(b, grid):
    """phi with the discrete Laplacian b (less b's weighted mean at a closed top), of zero weighted mean."""
    hz, gz = _metrics(grid)
    closed = not grid[8]
    if closed:
        b = b - (b.mean(dim=(1, 2)) * torch.as_tensor(hz, device="cuda")).sum() / hz.sum()
    nz = grid[2]
    lo, up = 1.0 / (hz * gz[:-1]), 1.0 / (hz * gz[1:])
    lx, ly = _modes(grid)
    lam = ly[:, None] + lx[None, :]
    lam[0, 0] = -1.0  # the mean of each plane is solved apart
    bh = _transform(b, grid)
    del b
    mean = bh[:, 0, 0].real.clone()
    bh[:, 0, 0] = 0.0
    inner = up.copy()
    inner[-1] = 0.0
    diag = lambda k: lam - (lo[k] + up[k])  # noqa: E731
    x = _thomas(lo, inner, diag, bh)
    for k in range(nz):  # one step of refinement
        bh[k] -= diag(k) * x[k]
        if k:
            bh[k] -= lo[k] * x[k - 1]
        if k + 1 < nz:
            bh[k] -= inner[k] * x[k + 1]
    x += _thomas(lo, inner, diag, bh)
    del bh
    # plane means: fluxes from the bottom up, then values
    flux = np.cumsum(hz * mean.cpu().numpy().astype(np.longdouble))
    phi = np.zeros(nz, dtype=np.longdouble)
    phi[-1] = 0.0 if closed else -flux[-1] * gz[-1]
    phi[:-1] = phi[-1] - np.cumsum((flux[:-1] * gz[1:-1])[::-1])[::-1]
    if closed:
        phi -= (phi * hz).sum() / hz.sum()
    x[:, 0, 0] = torch.as_tensor(phi.astype(np.float64), device="cuda").to(x.dtype)
    return _transform(x, grid, back=True)


def _divergence(u, v, w, grid):
    hz, _ = _metrics(grid)
    rdx, rdy = grid[0] / grid[3], grid[1] / grid[4]
    if grid[7]:
        d = (u[:, :, 1:] - u[:, :, :-1]).mul_(rdx).add_((v[:, 1:] - v[:, :-1]).mul_(rdy))
    else:
        d = (u.roll(-1, 2) - u).mul_(rdx).add_((v.roll(-1, 1) - v).mul_(rdy))
    return d.add_((w[1:] - w[:-1]).div_(_col(hz)))


def _project64(u, v, w, grid, dt):
    rdx, rdy = grid[0] / grid[3], grid[1] / grid[4]
    _, gz = _metrics(grid)
    b = _divergence(u, v, w, grid).div_(dt)
    phi = _poisson(b, grid)
    u, v, w = u.clone(), v.clone(), w.clone()
    if grid[7]:
        u[:, :, 1:-1] -= (phi[:, :, 1:] - phi[:, :, :-1]) * (dt * rdx)
        v[:, 1:-1] -= (phi[:, 1:] - phi[:, :-1]) * (dt * rdy)
    else:
        u -= (phi - phi.roll(1, 2)) * (dt * rdx)
        v -= (phi - phi.roll(1, 1)) * (dt * rdy)
    w[1:-1] -= (phi[1:] - phi[:-1]) * (dt / _col(gz[1:-1]))
    if grid[8]:
        w[-1] += phi[-1] * (dt / gz[-1])
    return u, v, w, phi, b


def _gradient64(gu, gv, gw, gp, grid, dt):
    """g + D^T S^T (g_phi / dt - G^T g), S the Poisson solve, S^T = V S V^-1 with the cells' volumes V."""
    rdx, rdy = grid[0] / grid[3], grid[1] / grid[4]
    hz, gz = _metrics(grid)
    src = gp / dt - (gu - gu.roll(-1, 2)) * rdx - (gv - gv.roll(-1, 1)) * rdy
    face = gw / _col(gz)
    src -= face[:-1] - face[1:]
    psi = _poisson(src / _col(hz), grid) * _col(hz)
    gw = gw.clone()
    gw[:-1] -= psi / _col(hz)
    gw[1:] += psi / _col(hz)
    return gu + (psi.roll(1, 2) - psi) * rdx, gv + (psi.roll(1, 1) - psi) * rdy, gw


def _viscous64(f, grid, beta, on_faces):
    hz, gz = _metrics(grid)
    if on_faces:  # w: the interior faces, zero on the walls
        lo, up = 1.0 / (gz[1:-1] * hz[:-1]), 1.0 / (gz[1:-1] * hz[1:])
        mid = lo + up
        inner = f[1:-1]
    else:  # u, v: the mirror value at a no-slip wall lies one cell height away
        lo, up = 1.0 / (hz * gz[:-1]), 1.0 / (hz * gz[1:])
        mid = lo + up
        mid[0] += 2.0 / hz[0] ** 2
        mid[-1] += 2.0 / hz[-1] ** 2
        inner = f
    lx, ly = _modes(grid)
    h = torch.fft.rfft2(inner) / ((1.0 - beta * lx)[None, :] * (1.0 - beta * ly)[:, None])
    x = _thomas(-beta * lo, -beta * up, lambda k: 1.0 + beta * mid[k], torch.fft.irfft2(h, s=inner.shape[1:]))
    if not on_faces:
        return x
    return torch.cat([torch.zeros_like(f[:1]), x, torch.zeros_like(f[:1])])


def exact(case, seed):
    grids, dt = _grids(case), case["dt"]
    got = []
    for grid, f in zip(grids, _inputs(case, seed)):
        if case["kind"] == "viscous":
            return tuple(_viscous64(f[c], grid, case["diffusion"], c == 2) for c in range(3))
        u, v, w, phi, b = _project64(f[0], f[1], f[2], grid, dt)
        if case["kind"] == "pressure":  # p_n + phi - dt / (2 Re) lap phi
            mean = (b.mean(dim=(1, 2)) * torch.as_tensor(np.diff(grid[6]), device="cuda")).sum() / grid[5]
            phi = f[3] + phi - 0.5 * dt * 1e-3 * (b - mean)
        got.append([u, v, w, phi])
        if case["kind"] == "grad":
            got[-1] += _gradient64(*f[3:7], grid, dt)
    if case["kind"] == "grad":
        cols = [torch.stack([g[i] for g in got]) for i in range(7)]
        return {"out": cols[:4], "grad": cols[4:]}
    if case["kind"] == "batch":
        return [torch.cat([g[i].reshape(-1) for g in got]) for i in range(4)]
    return tuple(got[0])
