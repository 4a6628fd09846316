"""FP32 V-cycles reach the rounding of FP32: a residual that loses digits
(psi's second differences formed by cancellation) leaves psi's error 50 to 100
times above it, however many cycles run, and different from one cycle count
to the next.

Tolerance: the rounding of one value of psi is up to 6e-8 of it, and the smooth
part of the field is corrected on the coarse grids to the rounding of each
update; 2e-7 leaves a factor of three for the updates' sum.  A lost digit in
the residual leaves 2e-6 or more.  (512 x 1024: the six cycles that the rate of
convergence asks for are past at 8.)"""
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import rel_l2, require_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,cycles", [(64, 128, 12), (128, 256, 12), (512, 1024, 8), (512, 1024, 12),
                                          (512, 1024, 13)])
def test_fp32_vcycles_reach_rounding(nx, ny, cycles):
    require_gpu()
    rhs = inputs.smooth_field(nx, ny, seed=nx + cycles, noise=0.1)
    ref = O.poisson_solve(rhs, nx, ny, 1.0 / nx, 2.0 / ny)
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype="f32")
    qg.qg_set_solver(b.h, qg.QG_SOLVER_MULTIGRID, cycles)
    assert rel_l2(to_np(b.poisson_solve(rhs)), ref) <= 2e-7
    b.close()
