"""What the tuner keeps: a basin's choice and an ensemble member's of the same
shape are entries of their own (a member is offered neither the sine sums nor
the one-node tile), and a choice made with the tile forced is not kept.  Each
case in a process of its own, through the QG_TUNE_CACHE file."""
import json
import os
import subprocess
import sys

import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_PROLOG = """
import json, os
from paper_1308_3290_gb300 import qg
kw = dict(nx=64, ny=128, Re=200.0, Ro=0.0016, levels=1, dt=1e-4)
def choice(h):
    return [qg.qg_solve_engine(h)] + list(qg.qg_stencil_tile(h))
"""


def run(body, cache, **env):
    e = dict(os.environ, QG_TUNE_CACHE=str(cache), **env)
    for k in ("QG_SOLVE_ENGINE", "QG_FINE_ROWS"):
        if k not in env:
            e.pop(k, None)
    r = subprocess.run([sys.executable, "-c", _PROLOG + body], env=e, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


@pytest.mark.parametrize("dtype,esz", [("f64", 8), ("f32", 4)])
def test_a_members_choice_is_not_a_basins(tmp_path, dtype, esz):
    require_gpu()
    cache = tmp_path / "tune.txt"
    # the basin's entry is there; the ensemble created first leaves it alone
    line = f"64 128 1 1 {esz} 42 8 1"
    cache.write_text(line + "\n")
    got = run(f"""
e = qg.Ensemble([kw, kw], dtype="{dtype}")
m = choice(e.member(0).h)
b = qg.Basin(dtype="{dtype}", **kw)
print(json.dumps([m, choice(b.h)]))
""", cache)
    assert got[1] == [42, 8, 1]
    assert got[0][0] != 42 and got[0][2] != 1
    lines = cache.read_text().splitlines()
    assert [x for x in lines if not x.startswith(("member ", "group "))] == [line]
    # the member's entry is taken by members only
    cache.write_text(f"member 64 128 1 1 {esz} 16 64 8\n" + line + "\n")
    got = run(f"""
b = qg.Basin(dtype="{dtype}", **kw)
e = qg.Ensemble([kw, kw], dtype="{dtype}")
print(json.dumps([choice(e.member(1).h), choice(b.h)]))
""", cache)
    assert got == [[16, 64, 8], [42, 8, 1]]


def test_a_forced_tiles_choice_is_not_kept(tmp_path):
    require_gpu()
    cache = tmp_path / "tune.txt"
    body = """
b = qg.Basin(dtype="f32", **kw)
print(json.dumps(choice(b.h)))
"""
    assert run(body, cache, QG_FINE_ROWS="64")[1:] == [64, 8]
    assert not cache.exists() or cache.read_text() == ""
    got = run(body, cache)
    assert cache.read_text().split() == ["64", "128", "1", "1", "4"] + [str(v) for v in got]


@pytest.mark.parametrize("dtype,esz", [("f64", 8), ("f32", 4)])
def test_a_forced_engine_that_does_not_take_the_grid(tmp_path, dtype, esz):
    """64 x 128, l = 1 is too short for engine 50: the choice is among the others
    but the sine sums (42), with an empty cache and with one that names 42, and
    is not kept."""
    require_gpu()
    cache = tmp_path / "tune.txt"
    body = f"""
b = qg.Basin(dtype="{dtype}", **kw)
print(json.dumps(choice(b.h)))
"""
    line = f"64 128 1 1 {esz} 42 8 1\n"
    for text in ("", line):
        cache.write_text(text)
        assert run(body, cache, QG_SOLVE_ENGINE="50")[0] not in (42, 50)
        assert cache.read_text() == text


@pytest.mark.parametrize("nx,ny,levels,dtype,never", [
    (64, 128, 1, "f32", (4, 16, 32, 33, 41)), (64, 128, 1, "f64", (16, 32)),
    (512, 1024, 0, "f32", (4, 16, 32, 33)), (512, 1024, 0, "f64", (16, 32))])
def test_engines_that_are_not_timed(tmp_path, nx, ny, levels, dtype, never):
    """Where engine 42 or 50 takes the grid, some engines are not candidates; on
    a grid that neither takes (8 x 512) another one is found."""
    require_gpu()
    body = f"""
b = qg.Basin({nx}, {ny}, Re=200.0, Ro=0.0016, levels={levels}, dt=1e-5, dtype="{dtype}")
c = qg.Basin(8, 512, Re=200.0, Ro=0.0016, levels=0, dt=1e-5, dtype="{dtype}")
print(json.dumps([qg.qg_solve_engine(b.h), qg.qg_solve_engine(c.h)]))
"""
    got = run(body, tmp_path / "tune.txt")
    assert got[0] not in never
    assert got[1] in (4, 16, 32, 33, 34)
