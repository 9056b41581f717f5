"""The mixed path's two-cell kernels (even nx, rows divisible by 4) against the one-cell ones.

The reference arm is a plan of two rows per CTA, which turns the half-block and two-cell
right-hand sides off, called with a u* off a 16-byte boundary, which turns the two-cell
correction off.  The tested arm has 4 to 16 rows; its fields lie on 16-byte boundaries or all
off them (8-byte loads), x and y are periodic or wall-bounded, with and without a mass source.

Both arms solve the same systems from the same right-hand sides, so without a sweep they agree
to the error of the fp32 solve, about 100 x 2^-24 at most on these grids, and every sweep
multiplies that by as much again: bounds 1e-5, 1e-9 and 1e-11 of the largest value (the adjoint,
whose source is 1/dt larger than its result, ten times that).  A cell left out or taken twice,
a wrong neighbour or a wrong row is of the order of the values or, in a sweep's residual, of the
correction before it; a low word lost or misplaced is 2^-24.

The order of the plane sums differs too.  Whole-number fields, spacings and a time step of
powers of two make the right-hand sides whole multiples of a power of two far below 2^48 of
them, whose float-float sums are exact in any order.  Random fields on a stretched z give every
coefficient and value its low word; a plane mean is then known to about 2^-48 of max|b| (a
random walk of roundings), 2^-45 allowed, of which the (0,0) solve makes lz^2 in phi and dt lz
in w: added to the bounds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_19130_gb300 import MIXED, Grid, Plan  # noqa: E402
from paper_2609_19130_gb300 import _native as N  # noqa: E402

pytestmark = pytest.mark.gpu
NEU, PER, DIR = N.IBF_BC_NEUMANN, N.IBF_BC_PERIODIC, N.IBF_BC_DIRICHLET
DT = 2.0 ** -10


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


def shifted(t):
    """A copy of t that starts 8 bytes past a 16-byte boundary."""
    buf = torch.empty(t.numel() + 3, dtype=t.dtype, device=t.device)
    off = 1 if buf.data_ptr() % 16 == 0 else 2
    out = buf[off:off + t.numel()].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == 8
    return out


def call(grid, rows, refine, pressure, f, p, q, grads):
    plan = Plan([grid], precision=MIXED, refine_steps=refine, pressure=pressure, inv_re=2.0 ** -6,
                tuning=[dict(rows=rows)])
    assert plan.tuning()["rows"] == rows
    # fields written before, so that every cell of the output is seen to be written
    out = [torch.full(s, float("nan"), dtype=torch.float64, device="cuda") for s in grid.shapes + (p.shape,)]
    plan.project(*f, DT, out=out, p=p if pressure else None, q=q)
    back = [torch.full(s, float("nan"), dtype=torch.float64, device="cuda") for s in grid.shapes]
    plan.backward_into([tuple(grads)], [tuple(back)], DT)
    torch.cuda.synchronize()
    assert plan.sync_status() in (N.IBF_OK, N.IBF_WARN_INCOMPATIBLE_RHS)
    plan.close()
    return out, back


def make(grid, gen, whole):
    """u*, v*, w*, p, q and the gradients of u, v, w, phi."""
    cells = (grid.nz, grid.ny, grid.nx)
    got = []
    for s in grid.shapes + (cells, cells) + grid.shapes + (cells,):
        if whole:
            got.append(torch.randint(-8, 9, s, device="cuda", generator=gen).to(torch.float64))
        else:
            got.append(torch.randn(s, dtype=torch.float64, device="cuda", generator=gen))
    return got


def arms(grid, rows, refine, pressure, source, aligned, whole):
    assert rows % 4 == 0 and rows <= grid.ny + grid.ny % 2 and grid.nx % 2 == 0
    gen = torch.Generator(device="cuda").manual_seed(11)
    f = make(grid, gen, whole)
    move = (lambda t: t) if aligned else shifted
    q = f[4] if source else None
    ref = call(grid, 2, refine, pressure, [shifted(f[0])] + f[1:3], f[3], q, [shifted(f[5])] + f[6:])
    got = call(grid, rows, refine, pressure, [move(t) for t in f[:3]], move(f[3]), move(q) if source else None,
               [move(t) for t in f[5:]])
    return f, got, ref


def agree(got, ref, refine, slack):
    tol = (1e-5, 1e-9, 1e-11, 1e-11)[refine]
    for i, (a, b, s) in enumerate(zip(got[0] + got[1], ref[0] + ref[1], slack)):
        assert float((a - b).abs().max()) <= (tol if i < 4 else 10.0 * tol) * float(b.abs().max()) + s


# nx below, at and past a warp's 64 cells and a CTA's; odd row counts, single and odd last rows
PERIODIC = [(2, 3, 4, 4), (6, 4, 5, 4), (64, 9, 3, 4), (64, 9, 3, 8), (72, 18, 7, 8), (96, 72, 9, 12), (144, 16, 4, 16),
            (512, 6, 3, 4), (1024, 8, 2, 8), (128, 128, 3, 12), (32, 12, 1, 12)]
WALLS = [(2, 3, 4, 4), (64, 9, 3, 8), (72, 18, 7, 8), (192, 32, 5, 12)]
CASES = ([s + (PER, PER) for s in PERIODIC] +
         [s + bc for s in WALLS for bc in ((NEU, PER), (PER, NEU), (NEU, NEU))])
ids = lambda c: "%dx%dx%d_rows%d%s%s" % (c[:4] + ("_wx" if c[4] == NEU else "", "_wy" if c[5] == NEU else ""))  # noqa: E731


@pytest.mark.parametrize("case", CASES, ids=ids)
@pytest.mark.parametrize("refine,pressure,source,top", [(0, N.IBF_P_PHI, True, DIR), (1, N.IBF_P_PHI, False, NEU),
                                                        (2, N.IBF_P_PHI, True, DIR), (3, N.IBF_P_IMPLICIT, False, NEU)])
@pytest.mark.parametrize("aligned", [True, False])
def test_exact_sums(case, refine, pressure, source, top, aligned):
    nx, ny, nz, rows, bx, by = case
    grid = Grid(nx, ny, nz, nx / 4.0, ny / 8.0, nz / 4.0, bc_x=bx, bc_y=by, bc_zhi=top)
    _, got, ref = arms(grid, rows, refine, pressure, source, aligned, True)
    agree(got, ref, refine, [0.0] * 7)


@pytest.mark.parametrize("case", CASES, ids=ids)
@pytest.mark.parametrize("refine,pressure,source,top", [(1, N.IBF_P_PHI, True, NEU), (2, N.IBF_P_EXPLICIT, False, DIR)])
@pytest.mark.parametrize("aligned", [True, False])
def test_low_words(case, refine, pressure, source, top, aligned):
    nx, ny, nz, rows, bx, by = case
    grid = Grid(nx, ny, nz, 2.0, 1.7, 1.0, beta=1.5, bc_x=bx, bc_y=by, bc_zhi=top)
    f, got, ref = arms(grid, rows, refine, pressure, source, aligned, False)
    hz = np.diff(0.5 * (1.0 + np.tanh(1.5 * (2.0 * np.arange(nz + 1) / nz - 1.0)) / np.tanh(1.5)))
    # max|b| and the adjoint's source (g_phi / dt and differences of g, per cell height)
    over = nx / grid.lx + ny / grid.ly + 1.0 / hz.min()
    bmax = max(float(t.abs().max()) for t in f[:5]) * (2.0 * over + 1.0) / DT
    smax = max(float(t.abs().max()) for t in f[5:]) * (2.0 * over + 1.0 / DT) / hz.min()
    mean = 2.0 ** -45
    agree(got, ref, refine, [mean * bmax * DT * grid.lz] * 3 + [mean * bmax * grid.lz ** 2] + [mean * smax * grid.lz ** 2] * 3)
