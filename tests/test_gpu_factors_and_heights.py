"""Transforms with factors of 16 and more along a wall-bounded y, and z systems of the heights
at which their kernels change form, against the FP64 oracle.

Wall-bounded y: 192 and 256 cells factor into 16 x 12 and 16 x 16, 288 into 24 x 12, 512 to 1024
into 32 x 16 to 32 x 32.  z: the tile kernel's four groups of levels hold more than one turn of
its sweeps from 65 levels on; grids of few modes keep it up to 560 levels.  Mode counts per
plane: multiples of four, even and odd (copies of 16, 8 and 4 bytes).

Bounds of the parity tests: relative L2 of phi 1e-12 in fp64, 1e-9 on the mixed path, here after
two sweeps (one leaves the square of 2^-24 times the number of cells along the longest
direction, which at 1024 cells is at that bound); velocities 1e-11 and 1e-9 of max|u*|.  The
oracle's plain sums of n terms are off by 2^-52 sqrt(n) / 5 of a mode of white input, and a solve
multiplies the error of the lowest of n modes by up to 2 n / pi of the input's size there: on
512 cells and more that is above 1e-12, and fp64's bound four times it, 2^-52 n^1.5 / 2."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2609_19130_gb300 import FP64, MIXED, Grid, Plan, synth  # noqa: E402
from paper_2609_19130_gb300 import _native as N  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {FP64: (1e-12, 1e-11), MIXED: (1e-9, 1e-9)}


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


def check(nx, ny, nz, wx, wy, prec, ly, stretch):
    neu = N.IBF_BC_NEUMANN
    g = Grid(nx, ny, nz, 2 * math.pi, ly, 2.0, beta=stretch, bc_x=neu if wx else 0, bc_y=neu if wy else 0)
    og = O.Grid(nx, ny, nz, lx=g.lx, ly=ly, lz=2.0, beta=stretch, wall_x=wx, wall_y=wy)
    f = synth.uniform_velocity_np(29, nx, ny, nz, wall_x=wx, wall_y=wy)
    phi, u, v, w, _ = O.project(og, *f, dt=1e-3)
    plan = Plan([g], precision=prec, refine_steps=2)
    got = plan.project(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in f), 1e-3)
    torch.cuda.synchronize()
    got = [t.cpu().numpy() for t in got]
    plan.close()
    tp, tu = TOL[prec]
    if prec == FP64:
        tp = max(tp, 2.0 ** -53 * max(nx, ny) ** 1.5)
    e = np.linalg.norm(got[3] - phi) / np.linalg.norm(phi)
    assert e <= tp, e
    umax = max(np.abs(a).max() for a in f)
    for a, b in zip(got, (u, v, w)):
        assert np.abs(a - b).max() <= tu * umax


@pytest.mark.parametrize("nx,ny", [(4, 192), (6, 256), (4, 288), (3, 512), (2, 768), (4, 1024)])
@pytest.mark.parametrize("wx", [False, True])
@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_wall_bounded_y(nx, ny, wx, prec):
    check(nx, ny, 5, wx, True, prec, 2 * math.pi * ny / 64.0, 1.0)


@pytest.mark.parametrize("nx,ny", [(8, 6), (6, 4), (4, 3)])
@pytest.mark.parametrize("nz", [65, 101, 192, 401, 560, 561])
def test_z_systems(nx, ny, nz):
    check(nx, ny, nz, False, False, MIXED, 1.3, 0.0)
