"""CG and PCG where the apply leaves so many partial sums of p.Ap (more than 4096: leaves of a few
DoFs) that they are summed in two stages."""
import pytest

import synth
from paper_2302_02863_gb300 import vfd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf", [(9000, 2), (8300, 2), (3000, 2), (6000, 5)])
@pytest.mark.parametrize("kind", ["none", "two_level", "jacobi"])
def test_solve_with_many_leaves(n, leaf, kind):
    import torch
    m = synth.interval_mesh(n)
    mesh = vfd.vfd_mesh(1, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=6)
    op = vfd.vfd_assemble(mesh, synth.const_field(0.4), synth.random_fourier_field(5, 0.3, d=1), 0.9)
    if kind != "none":
        vfd.vfd_precondition(op, vfd.VFD_PREC_TWO_LEVEL if kind == "two_level" else vfd.VFD_PREC_BLOCK_JACOBI)
    F = torch.randn(mesh.n_dof, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    U = torch.zeros_like(F)
    st, its, rel = vfd.vfd_solve(op, F, U, rtol=1e-9, max_it=5000)
    assert st == vfd.VFD_OK and rel[0] <= 1e-9, (its, rel)
    r = F - vfd.vfd_apply(op, U, torch.empty_like(U))
    # the recursive residual of a few hundred iterations drifts by less than the tolerance
    assert float(r.norm() / F.norm()) <= 2e-9
    again = torch.zeros_like(F)
    st, its2, _ = vfd.vfd_solve(op, F, again, rtol=1e-9, max_it=5000)
    assert its2 == its and torch.equal(again, U)   # sums in a fixed order
