"""The refinement of the FP32 diagnostics reads nothing that an earlier call left
in memory: after states of NaN have gone through the handle's scratch memory
(tapes, transfers), the diagnostics of a healthy state are bitwise those of a
fresh handle; and they leave the steps that follow bitwise as they are."""
import numpy as np
import pytest

from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu, to_np

pytestmark = pytest.mark.gpu

KW = dict(Re=200.0, Ro=0.0016, dt=1e-5, dtype="f32")


@pytest.mark.parametrize("bad", [float("nan"), 1e12])
@pytest.mark.parametrize("nx,ny,levels,engine", [(512, 256, 0, "50"), (512, 1024, 1, "50"),
                                                 (128, 256, 1, "34"), (64, 128, 1, "42"),
                                                 (64, 128, 1, "40"), (64, 64, 0, "4")])
def test_diagnostics_do_not_depend_on_earlier_calls(monkeypatch, nx, ny, levels, engine, bad):
    require_gpu()
    monkeypatch.setenv("QG_SOLVE_ENGINE", engine)
    w = inputs.gyre_state(nx, ny, seed=5)
    a = qg.Basin(nx, ny, levels=levels, **KW)
    a.set_state(w)
    want = a.diagnostics()
    a.close()
    b = qg.Basin(nx, ny, levels=levels, **KW)
    assert qg.qg_solve_engine(b.h) == int(engine)
    junk = np.full((ny - 1, nx - 1), bad)
    for first in (6, 1, 2, 3):
        # states of junk in a long tape's memory, then a short tape at its front
        b.set_state(junk)
        qg.qg_tape_begin(b.h, 1, 6)
        b.step(5)
        qg.qg_tape_end(b.h)
        b.restrict(junk, 1)
        qg.qg_tape_begin(b.h, 1, first)
        b.set_state(w)
        assert b.diagnostics() == want, first
        qg.qg_tape_end(b.h)
    b.close()


@pytest.mark.parametrize("nx,ny,levels", [(64, 128, 0), (128, 256, 1), (512, 1024, 1), (256, 256, 2)])
def test_diagnostics_leave_the_steps_alone(nx, ny, levels):
    require_gpu()
    w = inputs.gyre_state(nx, ny, seed=6)
    b = qg.Basin(nx, ny, levels=levels, **KW)
    out = []
    for ask in (False, True):
        b.set_state(w)
        for _ in range(3):
            b.step(2)
            if ask:
                b.diagnostics()
        out.append((to_np(b.state()), to_np(b.psi())))
    b.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
