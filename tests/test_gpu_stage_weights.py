"""The weights of a TVDRK3 stage (those of w^n and of w^(s), the Laplacian's
centre among them) add up to one: a defect, however small, multiplies the
state by the same factor in every step.

Measured as the projection of the FP32 state's error on the 64-bit state
after 23 steps.  The roundings of the nodes are independent and average out:
about five of at most 2^-24 per node and stage, 69 stages, over 8 000 nodes and
more leave 23 * 3 * 5 * 6e-8 / sqrt(8000) = 2e-7 if they all had their
greatest size, about a tenth of that at the sizes they have; the bound is
1e-7.  A centre weight rounded together with that of w^(s) gives 5.1e-7,
4.8e-7 and 7.8e-7 in these cases."""
import numpy as np
import pytest

from oracle import qg_oracle as O
from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,levels,Re,tile", [
    (256, 512, 2, 350.0, "128"), (256, 512, 2, 350.0, "32x4"), (256, 512, 2, 350.0, "8x1"),
    (256, 512, 0, 800.0, "128"), (256, 512, 0, 800.0, "8x1"), (64, 128, 1, 300.0, "128"),
    (64, 128, 1, 300.0, "8x1")])
def test_no_drift(monkeypatch, nx, ny, levels, Re, tile):
    require_gpu()
    monkeypatch.setenv("QG_FINE_ROWS", tile)
    w0 = inputs.gyre_state(nx, ny, seed=3).astype(np.float32).astype(np.float64)
    dt = 4e-3 / nx
    ref = O.run(w0, O.Basin(nx, ny, Re=Re, Ro=0.0016, levels=levels, dt=dt), 23)
    b = qg.Basin(nx, ny, Re=Re, Ro=0.0016, levels=levels, dt=dt, dtype="f32")
    assert "x".join(map(str, qg.qg_stencil_tile(b.h))) == (tile if "x" in tile else tile + "x8")
    b.set_state(w0)
    b.step(23)
    err = to_np(b.state()) - ref
    b.close()
    drift = float((err * ref).sum() / (ref * ref).sum())
    assert abs(drift) <= 1e-7, drift


def test_no_drift_of_ensemble_members():
    require_gpu()
    m = [dict(nx=64, ny=128, Re=300.0, Ro=0.0016, levels=1, dt=4e-3 / 64),
         dict(nx=64, ny=128, Re=800.0, Ro=0.0016, levels=1, dt=4e-3 / 64)]
    e = qg.Ensemble(m, dtype="f32")
    w0 = inputs.gyre_state(64, 128, seed=4).astype(np.float32).astype(np.float64)
    for i in range(2):
        e.member(i).set_state(w0)
    e.step(23)
    for i in range(2):
        ref = O.run(w0, O.Basin(64, 128, Re=m[i]["Re"], Ro=0.0016, levels=1, dt=4e-3 / 64), 23)
        err = to_np(e.member(i).state()) - ref
        drift = float((err * ref).sum() / (ref * ref).sum())
        assert abs(drift) <= 1e-7, (i, drift)
    e.close()
