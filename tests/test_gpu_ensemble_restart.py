"""New states for an ensemble that has stepped: the partial sums of R^l w of
all coarsened members come from one launch when every state is new, from each
member's own launch when only some are; both must equal stand-alone handles."""
import numpy as np
import pytest

from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu, to_np

pytestmark = pytest.mark.gpu

MEMBERS = [
    dict(nx=16, ny=16, Re=200.0, Ro=0.0016, levels=1, dt=1e-4, amp=1.0),
    dict(nx=32, ny=64, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, amp=1.0),
    dict(nx=64, ny=128, Re=312.5, Ro=0.0025, levels=1, dt=1e-4, amp=1.3),
    dict(nx=256, ny=128, Re=200.0, Ro=0.0016, levels=3, dt=2e-5, amp=0.9),
    dict(nx=128, ny=512, Re=200.0, Ro=0.0016, levels=2, dt=2e-5, amp=0.9),
]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_new_states_after_steps(dtype, monkeypatch):
    """The same engine and tile on both sides: bitwise equal (tolerance 0,
    the arithmetic is the same)."""
    require_gpu()
    monkeypatch.setenv("QG_SOLVE_ENGINE", "4")
    monkeypatch.setenv("QG_FINE_ROWS", "64")
    ens = qg.Ensemble(MEMBERS, dtype=dtype)
    solo = [qg.Basin(m["nx"], m["ny"], Re=m["Re"], Ro=m["Ro"], levels=m["levels"], dt=m["dt"],
                     amp=m["amp"], dtype=dtype) for m in MEMBERS]
    for k, new in enumerate([range(5), range(5), [3], [0, 1, 2, 4]]):
        for i in new:
            m = MEMBERS[i]
            w = inputs.perturbation(m["nx"], m["ny"], seed=100 * k + i) * 50.0
            ens.member(i).set_state(w)
            solo[i].set_state(w)
        ens.step(3)
        ens.synchronize()
        for i, b in enumerate(solo):
            b.step(3)
            b.synchronize()
            assert np.array_equal(to_np(ens.member(i).state()), to_np(b.state())), (k, i)
    for b in solo:
        b.close()
    ens.close()
