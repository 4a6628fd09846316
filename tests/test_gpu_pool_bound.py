"""What a handle's scratch pool keeps: no more than 256 MiB (four fields of this
handle are less) after a synchronisation, also when a tape and other calls'
scratch were live together, and nothing once the handle is gone."""
import pytest

from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

MIB = 2**20


def test_bound():
    torch = require_gpu()
    n = 2048                       # a padded FP32 field: 2049 rows of 2080 values, 16.3 MiB
    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]
    w = torch.as_tensor(inputs.perturbation(n, n, seed=1), dtype=torch.float32, device="cuda").contiguous()
    out = torch.empty_like(w)
    start = free()
    b = qg.Basin(n, n, Re=200.0, Ro=0.0016, levels=1, dt=1e-6, dtype="f32")
    b.set_state(w)
    with pytest.raises(qg.QGError):
        qg.qg_tape_begin(b.h, 1, 10**6)     # 17 TB: only the work fields are allocated, and stay
    b.synchronize()
    base = free()
    qg.qg_tape_begin(b.h, 1, 14)            # 15 states: 244 MiB
    for _ in range(2):
        qg.qg_poisson_solve(b.h, w, out, 0)     # 33 MiB beside them
    qg.qg_tape_end(b.h)
    b.synchronize()
    # (memory is mapped in granules of 2 MiB)
    assert base - free() <= 258 * MIB
    b.close()
    assert start - free() <= 8 * MIB            # (loaded kernels)
