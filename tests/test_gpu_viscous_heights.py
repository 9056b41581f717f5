"""The viscous solve at the heights, planes and widths where its kernels change form, against
the oracle.

z: the tile kernel copies a column in four groups of levels and sweeps it in turns of two
batches of eight, so columns from 25 levels on fill several groups and from 33 on whole
turns; w has one level less than u and v.  Planes of a multiple of four cells (two in fp64)
take 16-byte copies.  Above 816 levels (fp64: 408) the streaming z kernel takes over.
y and x: 512, 768 and 288 cells factor into 24- and 32-point transforms.

Bounds (max error of max|oracle|): fp64 1e-12, as for the small grids.  Mixed: 2e-6, the
bound of the small grids (fp32 transforms and sweep), with beta = 4 hz^2 at the closest faces:
the off-diagonals are four times the identity's entry, so values decay over about
sqrt(beta)/hz = 2 levels, and the sweeps' roundings (2^-24 each) accumulate over those only.
In fp64 also beta = 0.02, which couples tens of levels: 60 x 2^-53 for the tallest.  The wide
grids have few levels, far apart: the betas of the small grids."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from oracle import viscous as V  # noqa: E402
from paper_2609_19130_gb300 import FP64, MIXED, Grid, Plan, synth  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {FP64: 1e-12, MIXED: 2e-6}


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


def check(nx, ny, nz, prec, stretch, betas=None):
    g = Grid(nx, ny, nz, 2 * math.pi, 1.3, 2.0, beta=stretch)
    zf = O.zfaces_tanh(nz, g.lz, g.beta)
    f = synth.uniform_velocity_np(83, nx, ny, nz)
    plan = Plan([g], precision=prec, refine_steps=0)
    dev = [tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in f)]
    for beta in betas or [4.0 * float(np.diff(zf).min()) ** 2] + ([0.02] if prec == FP64 else []):
        ref = V.viscous_solve(nx, ny, nz, g.lx, g.ly, zf, *f, beta)
        got = plan.viscous_solve(dev, beta)[0]
        torch.cuda.synchronize()
        for a, b, nm in zip(got, ref, "uvw"):
            e = float(np.abs(a.cpu().numpy() - b).max() / np.abs(b).max())
            assert e <= TOL[prec], (nm, beta, e)
    plan.close()


PLANES = [(12, 16), (6, 3), (3, 3)]  # 192, 18 and 9 columns: whole and partial tiles; copies of 16, 8 and 4 bytes


@pytest.mark.parametrize("plane", PLANES, ids=lambda p: "%dx%d" % p)
@pytest.mark.parametrize("nz", [25, 33, 34, 65, 101, 192])
@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_tile_heights(plane, nz, prec):
    check(*plane, nz, prec, 0.5)


@pytest.mark.parametrize("plane,nz,prec", [((6, 4), 408, FP64), ((6, 4), 409, FP64), ((3, 3), 420, FP64),
                                           ((6, 4), 816, MIXED), ((6, 4), 817, MIXED), ((3, 3), 830, MIXED)],
                         ids=lambda v: str(v))
def test_tall_columns(plane, nz, prec):
    """The last height of the tile kernel and the streaming kernel above it."""
    check(*plane, nz, prec, 0.0)


@pytest.mark.parametrize("shape", [(6, 512, 9), (4, 768, 5), (12, 288, 4), (512, 4, 9), (288, 6, 4)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_wide_transforms(shape, prec):
    check(*shape, prec, 0.5, (1e-4, 0.02))
