"""Engine 50's half-length sine transforms at the edges of their range: the
shortest sides (FFT length 256, one thread per row), rows of 1 to 32 threads
on either side, pairs per CTA that do not divide the pairs, two layers, and a
batch of the shortest grids, against the oracle's sine-transform solve
(Section 4.3).  Tolerances: the solver's stated 1e-12 (FP64) and 2e-6 (FP32)."""
import numpy as np
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import assert_fields_close, rel_l2, require_gpu, to_np

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 2e-6}


@pytest.fixture(autouse=True)
def _force_engine(monkeypatch):
    monkeypatch.setenv("QG_SOLVE_ENGINE", "50")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(128, 256), (256, 128), (128, 4096), (4096, 128)])
def test_short_sides(dtype, nx, ny):
    require_gpu()
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype=dtype)
    assert qg.qg_solve_engine(b.h) == 50
    rhs = inputs.random_field(nx, ny, seed=nx + ny)
    ref = O.poisson_solve(rhs, nx, ny, 1.0 / nx, 2.0 / ny)
    assert_fields_close(to_np(b.poisson_solve(rhs)), ref, TOL[dtype], 32 * TOL[dtype])
    b.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(128, 256), (256, 256)])
def test_two_layers(dtype, nx, ny):
    """Both through qg_poisson_solve and in the step's own buffers (psi)."""
    require_gpu()
    p = dict(Ro=2.49e-4, Fr=0.087, delta=0.2, sigma=1.43e-3)
    b = qg.Basin(nx, ny, Re=697.16, levels=0, dt=1e-5, dtype=dtype, layers=2, y0=-0.5, y1=0.5, **p)
    assert qg.qg_solve_engine(b.h) == 50
    Q = [inputs.smooth_field(nx, ny, seed=k, noise=0.1) for k in (1, 2)]
    ref = O.elliptic_two_layer(Q[0], Q[1], nx, ny, 1 / nx, 1 / ny, p["Ro"], p["Fr"], p["delta"])
    got = to_np(b.poisson_solve(np.stack(Q)))
    for k in (0, 1):
        b.set_state(Q[k], k)
        assert rel_l2(got[k], ref[k]) <= TOL[dtype] * 5
    for k in (0, 1):
        assert rel_l2(to_np(b.psi(k)), ref[k]) <= TOL[dtype] * 5
    b.close()


def test_batch_of_the_shortest_grids_equals_standalone_handles(monkeypatch):
    """Queue items of eight and four pairs; bitwise the stand-alone states."""
    require_gpu()
    monkeypatch.setenv("QG_FINE_ROWS", "64")
    m = [dict(nx=128, ny=256, Re=200.0, Ro=0.0016, levels=0, dt=2e-5),
         dict(nx=256, ny=512, Re=300.0, Ro=0.0016, levels=1, dt=2e-5),
         dict(nx=512, ny=1024, Re=400.0, Ro=0.0016, levels=2, dt=1e-5)]
    ens = qg.Ensemble(m, dtype="f32")
    assert ens.kernel_count() == 3 * (1 + 3)
    solo = [qg.Basin(dtype="f32", **k) for k in m]
    for i, k in enumerate(m):
        w = inputs.perturbation(k["nx"], k["ny"], seed=i) * 50.0
        ens.member(i).set_state(w)
        solo[i].set_state(w)
        solo[i].step(3)
    ens.step(3)
    ens.synchronize()
    for i, b in enumerate(solo):
        b.synchronize()
        assert np.array_equal(to_np(ens.member(i).state()), to_np(b.state())), i
        b.close()
    ens.close()
