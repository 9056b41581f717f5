"""The two-cell kernels of the mixed path (even nx, periodic x and y, 16-byte aligned fields)
against the one-cell kernels, which every other call takes.

Shifting one field by 8 bytes sends the correction of the same call to the one-cell kernel and
the right-hand sides to 8-byte accesses.  Both do the
same packed float-float operations lane for lane; only the order of the plane sums' float-
float additions may differ, a change of 2^-48 of those sums.  That can flip the fp32 rounding
of the (0,0) mode's phi (6e-8 of it), which each refinement sweep corrects to its own fp32
rounding: bounds of 1e-6 without a sweep and 1e-12 with."""
import pytest

torch = pytest.importorskip("torch")

from paper_2609_19130_gb300 import MIXED, Grid, Plan  # noqa: E402
from paper_2609_19130_gb300 import _native as N  # noqa: E402

pytestmark = pytest.mark.gpu


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


# widths below, at and past a warp's 64 cells and a CTA's; odd and single rows and planes
SHAPES = [(2, 3, 4), (6, 1, 5), (32, 12, 1), (64, 9, 3), (72, 18, 7), (96, 72, 9), (144, 16, 4), (512, 6, 3),
          (1024, 8, 2), (128, 128, 3)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("refine,pressure,outlet", [(0, N.IBF_P_PHI, False), (1, N.IBF_P_PHI, False),
                                                    (2, N.IBF_P_PHI, True), (3, N.IBF_P_IMPLICIT, False),
                                                    (1, N.IBF_P_EXPLICIT, True)])
def test_same_as_one_cell(shape, refine, pressure, outlet):
    nx, ny, nz = shape
    grid = Grid(nx, ny, nz, 2.0, 1.7, 1.0, beta=1.5, bc_zhi=N.IBF_BC_DIRICHLET if outlet else N.IBF_BC_NEUMANN)
    plan = Plan([grid], precision=MIXED, refine_steps=refine, pressure=pressure, inv_re=0.01)
    gen = torch.Generator(device="cuda").manual_seed(7)
    f = [torch.randn(s, dtype=torch.float64, device="cuda", generator=gen) for s in grid.shapes + ((nz, ny, nx),)]
    p = f[3] if pressure else None
    ref = plan.project(shifted(f[0]), f[1], f[2], 1e-3, p=p)
    got = plan.project(f[0], f[1], f[2], 1e-3, p=p)
    tol = 1e-12 if refine else 1e-6
    for a, b in zip(got, ref):
        assert float((a - b).abs().max()) <= tol * float(b.abs().max())
    grads = [[torch.empty_like(x) for x in f[:3]] for _ in range(2)]
    plan.backward_into([(f[0], shifted(f[1]), f[2], f[3])], [grads[0]], 1e-3)
    plan.backward_into([tuple(f)], [grads[1]], 1e-3)
    torch.cuda.synchronize()
    for a, b in zip(*grads):
        assert float((a - b).abs().max()) <= tol * float(b.abs().max())
    plan.close()
