"""The restriction's partial planes 1 to 3 are zero off the seams whatever the
handle stepped before: multigrid sums all four planes at every node, and engine
50 reads planes 1 and 3 between the seams on sides of 128 intervals (256 x 512,
l = 1, tiles 64 columns wide).  A handle that stepped NaN, and a member of an
ensemble that did, steps a new state bitwise as a fresh one."""
import numpy as np
import pytest

from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,levels,tile,cycles", [
    (256, 512, 1, "128", 0), (256, 512, 1, "8x1", 0), (512, 256, 1, "32", 0), (512, 512, 2, "64", 0),
    (1024, 512, 3, "128", 0), (256, 512, 1, "128", 2), (256, 512, 2, "8x1", 2)])
def test_basin(monkeypatch, nx, ny, levels, tile, cycles):
    require_gpu()
    monkeypatch.setenv("QG_FINE_ROWS", tile)
    monkeypatch.setenv("QG_SOLVE_ENGINE", "50")
    w = inputs.gyre_state(nx, ny, seed=7)
    out = []
    for stale in (False, True):
        b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=levels, dt=1e-5, dtype="f32")
        if cycles:
            qg.qg_set_solver(b.h, qg.QG_SOLVER_MULTIGRID, cycles)
        if stale:
            b.set_state(np.full((ny - 1, nx - 1), np.nan))
            b.step(2)
        b.set_state(w)
        b.step(3)
        out.append(to_np(b.state()))
        b.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


def test_ensemble_members():
    require_gpu()
    m = [dict(nx=256, ny=512, Re=200.0, Ro=0.0016, levels=1, dt=1e-5),
         dict(nx=256, ny=512, Re=300.0, Ro=0.0016, levels=1, dt=1e-5),
         dict(nx=128, ny=256, Re=300.0, Ro=0.0016, levels=2, dt=1e-5)]
    w = [inputs.gyre_state(k["nx"], k["ny"], seed=i) for i, k in enumerate(m)]
    out = []
    for stale in (False, True):
        e = qg.Ensemble(m, dtype="f32")
        if stale:
            for i, k in enumerate(m):
                e.member(i).set_state(np.full((k["ny"] - 1, k["nx"] - 1), np.nan))
            e.step(2)
        for i in range(3):
            e.member(i).set_state(w[i])
        e.step(3)
        out.append([to_np(e.member(i).state()) for i in range(3)])
        e.close()
    for i in range(3):
        assert np.isfinite(out[0][i]).all() and np.array_equal(out[0][i], out[1][i]), i
