"""Calls that a program may capture into a CUDA graph of its own: the energy sum,
the reverse steps and the stand-alone operators, on a handle's first use and
after the handle has replayed its own graphs, several times in one capture.
The captured work gives what the calls give.  Each case in a process of its
own: a capture that fails leaves the next one's state undefined."""
import os
import subprocess
import sys

import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SCRIPT = """
import sys
import torch
from paper_1308_3290_gb300 import inputs, qg

what, before = sys.argv[1], int(sys.argv[2])
new = lambda *s: torch.zeros(*s, device="cuda")
s = torch.cuda.Stream()
with torch.cuda.stream(s):
    b = qg.Basin(64, 128, Re=200.0, Ro=0.0016, levels=1, dt=1e-4, dtype="f32")
    b.set_state(inputs.gyre_state(64, 128, seed=1))
    w = torch.as_tensor(inputs.gyre_state(64, 128, seed=2), dtype=torch.float32, device="cuda").contiguous()
    if what == "energy":
        out = [torch.zeros(1, dtype=torch.float64, device="cuda")]
        call = lambda: qg.qg_energy_accumulate(b.h, 1.0, out[0])
    elif what == "adjoint":
        qg.qg_tape_begin(b.h, 1, 12)
        b.step(12)
        out = [new(127, 63), new(127, 63)]
        call = lambda: (qg.qg_energy_gradient(b.h, 1.0, out[0]), qg.qg_adjoint_step(b.h, 1, out[0], out[1]))
    else:
        out = [new(63, 31), new(63, 31), new(127, 63), w.clone()]
        def call():
            qg.qg_restrict(b.h, w, out[0], 1)
            qg.qg_poisson_solve(b.h, out[0], out[1], 1)
            qg.qg_prolong(b.h, out[1], out[2], 1)
            qg.qg_restrict(b.h, out[3], out[3], 1)      # overlapping: through scratch
    for _ in range(before):
        call()
    s.synchronize()
    save = [o.clone() for o in out]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for _ in range(3):
            call()
    g.replay()
    s.synchronize()
    got = [o.clone() for o in out]
    # the same three calls without the capture, on a handle of the same state
    for o, k in zip(out, save):
        o.copy_(k)
    if what == "adjoint":
        b.set_state(inputs.gyre_state(64, 128, seed=1))
        qg.qg_tape_begin(b.h, 1, 12)
        b.step(12)
        for o in out:
            o.zero_()
        for _ in range(before):
            call()
    for _ in range(3):
        call()
    b.synchronize()
    for a, c in zip(got, out):
        assert torch.isfinite(a).all() and float(a.abs().max()) > 0
        assert torch.equal(a, c), float((a - c).abs().max())
print("SAME")
"""


@pytest.mark.parametrize("what", ["energy", "adjoint", "operators"])
@pytest.mark.parametrize("before", [0, 1, 4])
def test_capture(what, before):
    require_gpu()
    r = subprocess.run([sys.executable, "-c", _SCRIPT, what, str(before)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "SAME" in r.stdout, r.stdout[-500:] + r.stderr[-2500:]


def test_a_tape_is_not_begun_in_a_capture():
    """Its states have to outlive the caller's graph: refused, for a handle that
    has reversed a tape before too, and the handle goes on."""
    require_gpu()
    script = """
import torch
from paper_1308_3290_gb300 import inputs, qg
s = torch.cuda.Stream()
with torch.cuda.stream(s):
    b = qg.Basin(64, 128, Re=200.0, Ro=0.0016, levels=1, dt=1e-4, dtype="f32")
    b.set_state(inputs.gyre_state(64, 128, seed=1))
    qg.qg_tape_begin(b.h, 1, 4)
    qg.qg_tape_end(b.h)
    b.synchronize()
    g = torch.cuda.CUDAGraph()
    status = None
    try:
        with torch.cuda.graph(g, stream=s):
            try:
                qg.qg_tape_begin(b.h, 1, 4)
            except qg.QGError as e:
                status = e.status
                raise
    except Exception:
        pass
    assert status == qg.QG_ERR_OOM, status
print("REFUSED")
"""
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert "REFUSED" in r.stdout, r.stdout[-500:] + r.stderr[-2500:]
