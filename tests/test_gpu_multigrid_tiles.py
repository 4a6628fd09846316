"""The multigrid's tiled sweeps (32 x 32 nodes and their halo) at grids that
are one tile, one tile wide, and many, from a guess and from zero: V-cycles
must bring the residual of the 5-point equations down as whole-grid red-black
sweeps do.  The reference is a plain numpy V(2,2) cycle of the same operators,
to which FP64 cycles agree within 1e-11 of the solution (rounding through a few
hundred sweeps)."""
import numpy as np
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import rel_l2, require_gpu, to_np

pytestmark = pytest.mark.gpu


def sweeps(p, f, cx, cy, n):
    ny, nx = p.shape
    jj, ii = np.mgrid[1:ny - 1, 1:nx - 1]
    for k in range(2 * n):
        v = (cx * (p[1:-1, :-2] + p[1:-1, 2:]) + cy * (p[:-2, 1:-1] + p[2:, 1:-1]) - f[1:-1, 1:-1]) / (2 * (cx + cy))
        at = (ii + jj) % 2 == k % 2
        p[1:-1, 1:-1][at] = v[at]


def vcycle(p, f, dx, dy):
    my, mx = p.shape[0] - 1, p.shape[1] - 1
    cx, cy = 1 / dx ** 2, 1 / dy ** 2
    if min(mx, my) == 2:
        p[1:-1, 1:-1] = O.poisson_solve(f[1:-1, 1:-1], mx, my, dx, dy)
        return
    sweeps(p, f, cx, cy, 2)
    r = np.zeros_like(p)
    r[1:-1, 1:-1] = f[1:-1, 1:-1] - O.laplacian5(p, dx, dy)
    c = np.zeros((my // 2 + 1, mx // 2 + 1))
    vcycle(c, O.restrict(r), 2 * dx, 2 * dy)
    p += O.prolong(c)
    p[0] = p[-1] = 0
    p[:, 0] = p[:, -1] = 0
    sweeps(p, f, cx, cy, 2)


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-11), ("f32", 1e-5)])
@pytest.mark.parametrize("nx,ny", [(8, 16), (128, 128), (128, 256), (256, 512), (512, 256)])
def test_cycles_equal_whole_grid_sweeps(nx, ny, dtype, tol):
    require_gpu()
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=0, dt=1e-5, dtype=dtype, y0=0.0,
                 y1=float(ny) / nx)
    rhs = inputs.random_field(nx, ny, seed=nx + ny)
    for cycles in (1, 2):
        qg.qg_set_solver(b.h, qg.QG_SOLVER_MULTIGRID, cycles)
        p = np.zeros((ny + 1, nx + 1))
        for _ in range(cycles):
            vcycle(p, O.embed(rhs), 1.0 / nx, 1.0 / nx)
        assert rel_l2(to_np(b.poisson_solve(rhs)), p[1:-1, 1:-1]) <= tol
    b.close()
