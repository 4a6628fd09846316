"""Tapes of more states than any memory holds: QG_ERR_OOM, also where the bytes
wrap around in 64 bits (an 8 x 8 FP32 state takes 9 * 32 * 4 = 1152 = 2^7 * 9
bytes: 2^57 of them wrap to zero), and the handle records and reverses
afterwards."""
import pytest

from paper_1308_3290_gb300 import inputs, qg
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

BIG = 2**63 - 1


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("every,steps", [(1, BIG), (1, 2**57 - 1), (1, 2**57), (1, 2**58 - 1), (2, BIG),
                                         (2**57 - 1, 2**57 - 1), (BIG, 1), (BIG, BIG), (BIG - 1, 5),
                                         (2**56, 2**62)])
def test_out_of_memory(dtype, every, steps):
    torch = require_gpu()
    b = qg.Basin(8, 8, Re=200.0, Ro=0.0016, levels=0, dt=1e-4, dtype=dtype)
    with pytest.raises(qg.QGError) as e:
        qg.qg_tape_begin(b.h, every, steps)
    assert e.value.status == qg.QG_ERR_OOM
    b.set_state(inputs.perturbation(8, 8, seed=1))
    qg.qg_tape_begin(b.h, 2, 4)
    b.step(4)
    lam = torch.zeros((7, 7), dtype=torch.float32 if dtype == "f32" else torch.float64, device="cuda")
    g = torch.zeros_like(lam)
    qg.qg_energy_gradient(b.h, 1.0, lam)
    qg.qg_adjoint_step(b.h, 4, lam, g)
    qg.qg_tape_end(b.h)
    b.synchronize()
    assert torch.isfinite(g).all() and float(g.abs().max()) > 0
    b.close()
