"""Engine 50's two-layer mode-space solve and its CTAs of at least four pairs:
pair counts that leave CTAs partly filled, the longest FP32 transform with one
pair per CTA, and determinants far from one (a small Rossby number, no
coupling), against the oracle.  Tolerances: the solver's stated 1e-12 (FP64)
and 2e-6 (FP32), five times that for the coupled pair."""
import numpy as np
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import rel_l2, require_gpu, to_np

pytestmark = pytest.mark.gpu

TOL = {"f64": 5e-12, "f32": 1e-5}


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,Ro,Fr", [(256, 128, 2.49e-4, 0.087), (512, 256, 2.49e-4, 0.087),
                                         (128, 1024, 2.49e-4, 0.087), (128, 4096, 2.49e-4, 0.087),
                                         (4096, 128, 2.49e-4, 0.087), (128, 256, 1e-10, 0.087),
                                         (128, 256, 2.49e-4, 0.0), (128, 256, 1e-15, 0.0)])
def test_coupled_solve(monkeypatch, dtype, nx, ny, Ro, Fr):
    require_gpu()
    monkeypatch.setenv("QG_SOLVE_ENGINE", "50")
    b = qg.Basin(nx, ny, Re=697.16, Ro=Ro, levels=0, dt=1e-5, dtype=dtype, layers=2, Fr=Fr, delta=0.2,
                 sigma=1.43e-3, y0=-0.5, y1=0.5)
    assert qg.qg_solve_engine(b.h) == 50
    Q = [inputs.smooth_field(nx, ny, seed=k, noise=0.1) for k in (1, 2)]
    ref = O.elliptic_two_layer(Q[0], Q[1], nx, ny, 1 / nx, 1 / ny, Ro, Fr, 0.2)
    got = to_np(b.poisson_solve(np.stack(Q)))
    b.close()
    for k in (0, 1):
        assert rel_l2(got[k], ref[k]) <= TOL[dtype], rel_l2(got[k], ref[k])
