"""The fine stage with one node per thread (tiles of 16 x 8 nodes, 16 x 16 at
l = 4), forced through QG_FINE_ROWS, against the oracle: every level, both
types, grids narrower than a tile and with many seams, a forcing field and
the adaptive step.  Tolerances: the stated 1e-12 per 100 FP64 steps and 1e-4
per 100 FP32 steps; tile seams are also checked on their own."""
import numpy as np
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import assert_fields_close, rel_l2, require_gpu, to_np

pytestmark = pytest.mark.gpu


def basin(nx, ny, levels, dtype, monkeypatch, dt):
    rows = 16 if levels == 4 else 8
    monkeypatch.setenv("QG_FINE_ROWS", f"{rows}x1")
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=levels, dt=dt, dtype=dtype)
    assert qg.qg_stencil_tile(b.h) == (rows, 1)
    return b


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-12), ("f32", 1e-4)])
@pytest.mark.parametrize("nx,ny,levels", [(8, 8, 0), (8, 16, 0), (16, 8, 0), (128, 256, 0), (64, 128, 1), (128, 64, 2),
                                          (128, 256, 3), (128, 256, 4)])
def test_follows_the_oracle(nx, ny, levels, dtype, tol, monkeypatch):
    require_gpu()
    w0 = inputs.perturbation(nx, ny, seed=16) * 20.0
    F = inputs.perturbed_forcing_field(nx, ny, seed=3, Ro=0.0016)
    b = basin(nx, ny, levels, dtype, monkeypatch, 5e-5)
    for forcing in (None, F):
        ref = O.run(w0, O.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=levels, dt=5e-5, forcing=forcing), 50)
        b.set_forcing(forcing)
        b.set_state(w0)
        b.step(50)
        assert_fields_close(to_np(b.state()), ref, tol, 8 * tol, xper=16, yper=8)
    b.close()


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-11), ("f32", 1e-4)])
@pytest.mark.parametrize("levels", [0, 2])
def test_adaptive_step(levels, dtype, tol, monkeypatch):
    """The bounds of the sweep's adaptive-step test."""
    require_gpu()
    nx, ny = 64, 128
    w0 = inputs.gyre_state(nx, ny, seed=4)
    ref, dts = O.run_adaptive(w0, O.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=levels, dt=5e-4), 10, 0.01)
    assert min(dts) < 5e-4      # Eq. dt, not the cap, sets the step
    b = basin(nx, ny, levels, dtype, monkeypatch, 5e-4)
    qg.qg_set_cfl(b.h, 0.01)
    b.set_state(w0)
    b.step(10)
    assert rel_l2(to_np(b.state()), ref) <= tol
    t, last = qg.qg_get_time(b.h)
    assert np.isclose(t, sum(dts), rtol=tol) and np.isclose(last, dts[-1], rtol=tol)
    b.close()
