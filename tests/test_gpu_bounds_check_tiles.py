"""The bounds-checked build (QG_BOUNDS_CHECK) over the kernels that
bounds_workload.py does not force: the sine sums (engine 42) at the ends of
their range, the one-node tiles at every level, engine 50's short sides (one
thread per row, the spare row, CTAs partly filled, two layers, a batch), the
adjoint at every level in both types, the first stage's extras, the dense
transfers, and an ensemble's new states in one launch.  In a process of its own,
as there; no check may fail.  And no two kernels' checks share a number."""
import glob
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SCRIPT = """
import os, sys
import torch
from paper_1308_3290_gb300 import adjoint, build, inputs, qg

qg.load(build.build(variant="bounds"))
bad = 0
def check(name):
    global bad
    s = qg.qg_bounds_check_result()
    print(name, s, flush=True)
    bad = bad or s

def basin(nx, ny, lv, dtype, **kw):
    return qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=lv, dt=2e-5, dtype=dtype, **kw)

def two(nx, ny, lv, dtype):
    b = qg.Basin(nx, ny, Re=697.16, Ro=2.49e-4, levels=lv, dt=1e-5, dtype=dtype, layers=2, Fr=0.087,
                 delta=0.2, sigma=1.43e-3, y0=-0.5, y1=0.5)
    for k in (0, 1):
        b.set_state(inputs.smooth_field(nx, ny, seed=k, amp=0.05), k)
    b.step(2)
    b.psi(0)
    b.synchronize()
    b.close()

def steps(b, nx, ny):
    b.set_state(inputs.perturbation(nx, ny, seed=1) * 20.0)
    b.step(2)
    b.diagnostics()
    b.psi()
    b.close()

for dtype in ("f32", "f64"):
    os.environ["QG_SOLVE_ENGINE"] = "42"
    for nx, ny, lv in ((8, 8, 0), (8, 256, 0), (256, 8, 0), (256, 256, 0), (64, 128, 1), (256, 512, 2)):
        b = basin(nx, ny, lv, dtype)
        assert qg.qg_solve_engine(b.h) == 42
        b.poisson_solve(inputs.smooth_field(nx >> lv, ny >> lv, seed=2), lv)
        steps(b, nx, ny)
    two(8, 16, 0, dtype)
    two(64, 64, 1, dtype)
    check("engine 42 " + dtype)
    os.environ["QG_SOLVE_ENGINE"] = "50"
    for nx, ny, lv in ((128, 256, 0), (256, 128, 0), (128, 1024, 0), (1024, 128, 0), (256, 512, 1), (512, 512, 1)):
        b = basin(nx, ny, lv, dtype)
        assert qg.qg_solve_engine(b.h) == 50
        b.poisson_solve(inputs.smooth_field(nx >> lv, ny >> lv, seed=2), lv)
        steps(b, nx, ny)
    two(128, 256, 0, dtype)
    two(256, 128, 0, dtype)
    two(512, 512, 1, dtype)
    check("engine 50 " + dtype)
    del os.environ["QG_SOLVE_ENGINE"]
    for lv in range(5):
        os.environ["QG_FINE_ROWS"] = "16x1" if lv == 4 else "8x1"
        b = basin(128, 256, lv, dtype)
        assert qg.qg_stencil_tile(b.h)[1] == 1
        b.set_forcing(inputs.perturbed_forcing_field(128, 256, seed=3, Ro=0.0016))
        qg.qg_set_cfl(b.h, 0.5)
        qg.qg_stats_begin(b.h)
        steps(b, 128, 256)
        del os.environ["QG_FINE_ROWS"]
        b = basin(128, 256, lv, dtype)
        T = b.tdtype
        F = torch.as_tensor(inputs.perturbed_forcing_field(128, 256, seed=5, Ro=0.0016), dtype=T,
                            device="cuda").contiguous().requires_grad_(True)
        w0 = torch.as_tensor(inputs.perturbation(128, 256, seed=5), dtype=T, device="cuda")
        adjoint.mean_kinetic_energy(F, b, w0, 6, 3, 2).backward()
        for k in (1, 2, 6):
            b.prolong(b.restrict(w0, k), k)
        b.close()
        check("level %d %s" % (lv, dtype))
    m = [dict(nx=n, ny=2 * n, Re=200.0, Ro=0.0016, levels=lv, dt=2e-5)
         for n, lv in ((128, 0), (256, 1), (64, 1), (64, 2), (32, 0), (512, 2))]
    e = qg.Ensemble(m, dtype=dtype)
    for i, k in enumerate(m):
        e.member(i).set_state(inputs.perturbation(k["nx"], k["ny"], seed=i))
    e.step(2)
    e.synchronize()
    e.close()
    for lv in (0, 1):
        b = basin(256, 512, lv, dtype)
        qg.qg_set_solver(b.h, qg.QG_SOLVER_MULTIGRID, 2)
        steps(b, 256, 512)
    check("ensemble, multigrid " + dtype)
print("FIRST_FAILED_SITE", bad)
"""


@pytest.mark.gpu
def test_no_index_leaves_its_buffer():
    from tests.gpu_util import require_gpu
    require_gpu()
    env = {k: v for k, v in os.environ.items() if not k.startswith("QG_")}
    r = subprocess.run([sys.executable, "-c", _SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0 and "FIRST_FAILED_SITE 0" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_check_numbers_name_one_place():
    """A number that stands in two files cannot name the place of a failed check
    (node_tile.cuh's are shared by the kernels that include it)."""
    where = {}
    for f in sorted(glob.glob(os.path.join(ROOT, "paper_1308_3290_gb300", "csrc", "*.cu*"))):
        if f.endswith("bounds.cuh"):
            continue
        text = open(f).read()
        for m in re.finditer(r"QG_IN\(", text):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            n = re.search(r", *(\d+|PH == 0 \? \d+ : \d+)\)$", text[m.start():i])
            assert n, (f, text[m.start():i])
            for v in re.findall(r"\d+", n.group(1).replace("PH == 0", "")):
                where.setdefault(int(v), set()).add(os.path.basename(f))
    assert len(where) > 60
    assert {k: v for k, v in where.items() if len(v) > 1} == {}
