"""Engine 42 (sine sums with one output per thread): the smallest and largest
sides it takes, tables in and out of shared memory, one and two layers, and
steps whose right-hand side comes in partial planes, against the oracle.
Tolerances: the solver's stated 1e-12 (FP64) and 2e-6 (FP32), 1e-4 after 50
FP32 steps, 1e-12 after 50 FP64 ones."""
import numpy as np
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import assert_fields_close, rel_l2, require_gpu, to_np

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 2e-6}


@pytest.fixture(autouse=True)
def _force_engine(monkeypatch):
    monkeypatch.setenv("QG_SOLVE_ENGINE", "42")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (8, 256), (256, 8), (16, 64), (64, 128), (256, 256)])
def test_solve(nx, ny, dtype):
    require_gpu()
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype=dtype)
    assert qg.qg_solve_engine(b.h) == 42
    rhs = inputs.smooth_field(nx, ny, seed=nx + ny, noise=0.3)
    ref = O.poisson_solve(rhs, nx, ny, 1.0 / nx, 2.0 / ny)
    assert rel_l2(to_np(b.poisson_solve(rhs)), ref) <= TOL[dtype]
    b.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_two_layers(dtype):
    require_gpu()
    nx, ny = 32, 64
    p = dict(Ro=2.49e-4, Fr=0.087, delta=0.2, sigma=1.43e-3)
    b = qg.Basin(nx, ny, Re=697.16, levels=0, dt=1e-5, dtype=dtype, layers=2, y0=-0.5, y1=0.5, **p)
    Q = [inputs.smooth_field(nx, ny, seed=k, noise=0.1) for k in (1, 2)]
    ref = O.elliptic_two_layer(Q[0], Q[1], nx, ny, 1 / nx, 1 / ny, p["Ro"], p["Fr"], p["delta"])
    got = to_np(b.poisson_solve(np.stack(Q)))
    for k in (0, 1):
        assert rel_l2(got[k], ref[k]) <= TOL[dtype] * 5
    b.close()


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-12), ("f32", 1e-4)])
@pytest.mark.parametrize("levels", [0, 1, 2])
def test_steps(levels, dtype, tol):
    require_gpu()
    nx, ny = 64, 128
    w0 = inputs.perturbation(nx, ny, seed=5) * 20.0
    ref = O.run(w0, O.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=levels, dt=1e-4), 50)
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=levels, dt=1e-4, dtype=dtype)
    assert qg.qg_solve_engine(b.h) == 42
    b.set_state(w0)
    b.step(50)
    assert_fields_close(to_np(b.state()), ref, tol, 8 * tol)
    b.close()


def test_unsupported_sides_and_the_fallback():
    """Past 256 intervals a side another engine solves; the choice made while an
    engine that does not take the grid is asked for stays among the
    transforms."""
    require_gpu()
    b = qg.Basin(512, 256, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype="f64")
    assert qg.qg_solve_engine(b.h) in (4, 16, 32, 33, 34, 50)
    b.close()
