"""ibf_project_noalloc's host time per call against ibf_project's, on a grid so small that the
host side is what a caller waits for.

Both enqueue the same streaming solve.  The entry point without allocation also builds its
tables, sends them as launch arguments and sets the shared-memory caps of the kernels it may
launch (15; 0.7 us each).  Setting those of every kernel of the library made it 3.9 times
ibf_project's time; with its own kernels only it is 1.7 times, bound 2.5 (smallest of 300 calls
each, which other work on the host can only lengthen)."""
import ctypes as C
import time

import pytest

torch = pytest.importorskip("torch")

from paper_2609_19130_gb300 import MIXED, Grid, Plan, synth  # noqa: E402
from paper_2609_19130_gb300 import _native as N  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


def test_host_time_of_a_call():
    grid = Grid(16, 16, 8, beta=1.0)
    u, v, w = synth.uniform_velocity_torch(3, grid.nx, grid.ny, grid.nz, "cuda")
    out = [torch.empty_like(t) for t in (u, v, w)]
    out.append(torch.empty((grid.nz, grid.ny, grid.nx), dtype=torch.float64, device="cuda"))
    fin = N.ibf_fields(u.data_ptr(), v.data_ptr(), w.data_ptr(), None)
    fout = N.ibf_fields(*(t.data_ptr() for t in out))
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    lib = N.lib()
    plan = Plan([grid], precision=MIXED, refine_steps=1, tuning=[dict(yz_kernel=1, tri=1)])
    cg = N.ibf_grid(grid.nx, grid.ny, grid.nz, grid.lx, grid.ly, grid.lz, None, grid.beta, grid.bc_x, grid.bc_y,
                    grid.bc_zlo, grid.bc_zhi)
    opts = N.ibf_opts(N.IBF_MIXED, 1, 0, 0)

    def with_plan():
        return lib.ibf_project(plan.handle, C.byref(fin), C.byref(fout), 1e-3, 1.0, None, stream)

    def noalloc():
        return lib.ibf_project_noalloc(C.byref(cg), C.byref(opts), C.byref(fin), C.byref(fout), 1e-3, 1.0, stream)

    def shortest(call):
        for _ in range(20):
            assert call() == N.IBF_OK
        best = 1e9
        for _ in range(300):
            torch.cuda.synchronize()
            t = time.perf_counter()
            call()
            best = min(best, time.perf_counter() - t)
        torch.cuda.synchronize()
        return best

    ratio = shortest(noalloc) / shortest(with_plan)
    plan.close()
    assert ratio <= 2.5, ratio
