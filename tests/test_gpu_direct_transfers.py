"""qg_restrict and qg_prolong between device buffers (straight from one to the
other), between host buffers, and where source and destination overlap in
memory (through scratch, as the host buffers go), bit for bit the same; and
state exchange of odd row lengths from addresses off 16 bytes."""
import numpy as np
import pytest

from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("nx,ny,levels", [(16, 32, 1), (64, 8, 2), (128, 256, 3), (32, 32, 4)])
def test_every_buffer_kind(nx, ny, levels, dtype):
    torch = require_gpu()
    tdt = torch.float32 if dtype == "f32" else torch.float64
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype=dtype)
    mx, my = nx >> levels, ny >> levels
    fine = torch.as_tensor(inputs.random_field(nx, ny, seed=1), dtype=tdt)
    coarse = torch.as_tensor(inputs.random_field(mx, my, seed=2), dtype=tdt)
    for call, src, shape in ((qg.qg_restrict, fine, (my - 1, mx - 1)),
                             (qg.qg_prolong, coarse, (ny - 1, nx - 1))):
        host = torch.empty(shape, dtype=tdt)
        call(b.h, src.contiguous(), host, levels)
        b.synchronize()
        dev = torch.empty(shape, dtype=tdt, device="cuda")
        call(b.h, src.cuda(), dev, levels)
        b.synchronize()
        assert torch.equal(dev.cpu(), host)
        # one buffer holds both, the destination starting inside the source
        n, m = src.numel(), dev.numel()
        buf = torch.zeros(n + m, dtype=tdt, device="cuda")
        buf[:n] = src.cuda().flatten()
        out = buf[n // 2:n // 2 + m].view(shape)
        call(b.h, buf[:n].view(src.shape), out, levels)
        b.synchronize()
        assert torch.equal(out.cpu(), host)
    b.close()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (8, 64), (64, 8), (128, 256)])
def test_state_round_trip(nx, ny, dtype):
    torch = require_gpu()
    tdt = torch.float32 if dtype == "f32" else torch.float64
    b = qg.Basin(nx, ny, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype=dtype)
    n = (nx - 1) * (ny - 1)
    for off in (0, 1, 2, 3):
        big = torch.randn(n + 8, dtype=tdt, device="cuda")
        out = torch.full((n + 8,), 7.0, dtype=tdt, device="cuda")
        qg.qg_set_state(b.h, big[off:off + n], 0)
        qg.qg_get_state(b.h, out[off:off + n], 0)
        b.synchronize()
        assert torch.equal(out[off:off + n], big[off:off + n])
        assert bool((out[:off] == 7.0).all()) and bool((out[off + n:] == 7.0).all())
    b.close()
