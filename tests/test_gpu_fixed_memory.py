"""Device memory of the fixed-point copies: operators that cannot use them do not keep them."""
import pytest

import synth
from paper_2302_02863_gb300 import vfd

pytestmark = pytest.mark.gpu


def _assembled(mesh, log_kappa):
    """(operator, bytes of device memory that it took)."""
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    op = vfd.vfd_assemble(mesh, synth.config2_s_field(), synth.const_field(log_kappa), 0.9)
    torch.cuda.synchronize()
    return op, before - torch.cuda.mem_get_info()[0]


def test_copies_that_do_not_fit_are_released():
    import torch
    m = synth.disk_mesh(45, R=1.1, jitter=0.2, seed=9)
    mesh = vfd.vfd_mesh(2, m.coords, m.cells, m.cell_is_interior, leaf_m=64, cheb_p=8)
    i = mesh.info
    _assembled(mesh, 0.0)   # modules and streams
    op, size = _assembled(mesh, 0.0)
    # e^-620: entries below 2^-830, which FP64 holds and the copies do not
    small, ssize = _assembled(mesh, -620.0)
    copies = 8 * (i["near_entries"] + i["far_blocks"] * i["rank"] ** 2)
    assert copies > 100 << 20
    assert size - ssize > 0.8 * copies, (size, ssize, copies)
    x = torch.randn(mesh.n_dof, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    y, z = (vfd.vfd_apply(o, x, torch.empty_like(x)) for o in (op, small))
    import math
    z = z * math.exp(310.0) * math.exp(310.0)
    # the FP64 assembly rounds an exponent of about 900 at every operation: 2^-53 x 900 a few times
    assert float((y - z).abs().max() / y.abs().max()) < 2e-12
    # and the many-column call runs without them
    X = x.repeat(64, 1)
    Z = vfd.vfd_apply(small, X, torch.empty_like(X))
    assert vfd.vfd_op_apply_stats(small)["tensor_columns"] == 0
    assert float((Z * math.exp(310.0) * math.exp(310.0) - y).abs().max() / y.abs().max()) < 2e-12
