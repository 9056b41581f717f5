"""The plane-parallel y/z path (all planes' y transforms at once, then whole z systems)
against the streaming kernels on the same grid.

Both run the same transforms, pivots and Thomas recurrences in the same order, so only the
(0,0) mode's fp64 sums differ in their order: the fields agree to a few fp64 roundings of
those sums (1e-13) in fp64; on the mixed path an fp32 rounding of the (0,0) mode may flip,
which the sweep corrects to fp32 rounding of its fp32 correction (6e-8 squared): 1e-12."""
import pytest

torch = pytest.importorskip("torch")

from paper_2609_19130_gb300 import FP64, MIXED, Grid, Plan  # noqa: E402
from paper_2609_19130_gb300 import _native as N  # noqa: E402

pytestmark = pytest.mark.gpu
NEU, PER, DIR = N.IBF_BC_NEUMANN, N.IBF_BC_PERIODIC, N.IBF_BC_DIRICHLET


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


def run(grids, prec, tunings, seed=3):
    plan = Plan(grids, precision=prec, refine_steps=1, tuning=tunings)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ins = []
    for g in grids:
        f = [torch.rand(s, dtype=torch.float64, device="cuda", generator=gen) - 0.5 for s in g.shapes]
        f[2][0].zero_()
        f[2][-1].zero_()
        if g.bc_x == NEU:
            f[0][:, :, 0] = f[0][:, :, -1] = 0.0
        if g.bc_y == NEU:
            f[1][:, 0] = f[1][:, -1] = 0.0
        ins.append(tuple(f))
    outs = plan.project_batch(ins, 1e-3)
    torch.cuda.synchronize()
    assert plan.sync_status() in (N.IBF_OK, N.IBF_WARN_INCOMPATIBLE_RHS)
    plan.close()
    return outs


def close(a, b, tol):
    for x, y in zip(a, b):
        assert torch.isfinite(x).all()
        assert float((x - y).abs().max()) <= tol * float(y.abs().max())


# sizes at the edges of the z batches (8 levels), of a warp's and a CTA's modes, of the y
# transforms' groups (one and several column blocks, radix 3, ny = 1, 32-point DFTs), and one
# with more levels than the fused (0,0) solve takes
SHAPES = [(16, 12, 2), (24, 9, 7), (32, 1, 8), (18, 16, 9), (64, 48, 17), (96, 72, 33), (12, 512, 3),
          (16, 768, 5), (1024, 8, 16), (6, 6, 1100), (256, 64, 24)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec,tol", [(FP64, 1e-13), (MIXED, 1e-12)])
def test_same_as_streaming(shape, prec, tol):
    grid = Grid(*shape, 2.0, 1.7, 1.0, beta=1.5)
    ref = run([grid], prec, [dict(yz_kernel=1, tri=1)])[0]
    for tuning in (dict(yz_kernel=1, tri=2), dict(yz_kernel=3, mb=3)):
        close(run([grid], prec, [tuning])[0], ref, tol)


@pytest.mark.parametrize("bc", [(NEU, PER, NEU), (PER, NEU, NEU), (NEU, NEU, DIR), (PER, PER, DIR)])
@pytest.mark.parametrize("prec,tol", [(FP64, 1e-13), (MIXED, 1e-12)])
def test_walls_and_outlet(bc, prec, tol):
    grid = Grid(36, 32, 13, 2.0, 1.7, 1.0, beta=1.5, bc_x=bc[0], bc_y=bc[1], bc_zhi=bc[2])
    close(run([grid], prec, [dict(yz_kernel=1, tri=2)])[0], run([grid], prec, [dict(yz_kernel=1, tri=1)])[0], tol)


@pytest.mark.parametrize("prec,tol", [(FP64, 1e-13), (MIXED, 1e-12)])
def test_batch_with_other_kernels(prec, tol):
    """Plane-parallel grids beside a streaming and a slab one (the (0,0) modes then have their own launch)."""
    grids = [Grid(32, 24, 9, beta=1.0), Grid(64, 12, 16), Grid(24, 32, 5, beta=2.0), Grid(48, 16, 21)]
    tun = [dict(yz_kernel=1, tri=2), dict(yz_kernel=1, tri=1), dict(yz_kernel=3), dict(yz_kernel=2, mb=1)]
    got = run(grids, prec, tun)
    alone = run(grids, prec, [dict(yz_kernel=1, tri=1)] * 4)
    planes = run(grids, prec, [dict(yz_kernel=1, tri=2)] * 4)
    for a, b, c in zip(got, alone, planes):
        close(a, b, tol)
        close(c, b, tol)
