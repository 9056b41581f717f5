"""The rounding of the wall-bounded y transforms: the plane-parallel path against the streaming
one on domains much longer in y than high, where the low y-modes of the z systems magnify an
fp32 rounding to 1e-8 of phi after one sweep.

Both run the same transforms, twiddles, pivots and Thomas recurrences with the same roundings,
so only the (0,0) mode's fp64 sums differ in their order: a few fp64 roundings (1e-13) in fp64;
on the mixed path an fp32 rounding of the (0,0) mode may flip, which the sweep corrects to fp32
rounding of its fp32 correction (6e-8 squared): 1e-12 of the largest value."""
import math

import pytest

torch = pytest.importorskip("torch")

from paper_2609_19130_gb300 import FP64, MIXED, Grid, Plan  # noqa: E402
from paper_2609_19130_gb300 import _native as N  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


@pytest.mark.parametrize("nx,ny", [(4, 72), (4, 192), (6, 256), (3, 512), (2, 768), (4, 1024)])
@pytest.mark.parametrize("prec,tol", [(FP64, 1e-13), (MIXED, 1e-12)])
def test_wall_transforms_round_alike(nx, ny, prec, tol):
    g = Grid(nx, ny, 5, 2 * math.pi, 2 * math.pi * ny / 64.0, 2.0, beta=1.0, bc_y=N.IBF_BC_NEUMANN)
    gen = torch.Generator(device="cuda").manual_seed(2)
    u, v, w = (torch.rand(s, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1 for s in g.shapes)
    for f in (v[:, 0], v[:, -1], w[0], w[-1]):
        f.zero_()
    out = []
    for tri in (2, 1):
        plan = Plan([g], precision=prec, refine_steps=1, tuning=[dict(yz_kernel=1, tri=tri)])
        out.append(plan.project(u, v, w, 1e-3))
        torch.cuda.synchronize()
        plan.close()
    for a, b in zip(*out):
        assert float((a - b).abs().max()) <= tol * float(b.abs().max())
