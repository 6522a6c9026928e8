"""Errors of the fixed-point and digit arithmetic against extended precision."""
import numpy as np
import pytest

import synth
from paper_2302_02863_gb300 import vfd

pytestmark = pytest.mark.gpu
LD = np.longdouble   # 64 bits of mantissa or more


def _near_entry(x, cells, i, j, s):
    """Entry (i, j) of the near part on an interval: 3-point Gauss rules, cells that touch left out."""
    g = LD(0.5) * np.sqrt(LD(3) / LD(5))
    t, w = np.array([LD(0.5) - g, LD(0.5), LD(0.5) + g]), np.array([LD(5), LD(8), LD(5)]) / LD(18)
    out = LD(0)
    for a in np.nonzero((cells == i).any(1))[0]:
        for b in np.nonzero((cells == j).any(1))[0]:
            if set(cells[a]) & set(cells[b]):
                continue
            (a0, a1), (b0, b1) = x[cells[a]].astype(LD), x[cells[b]].astype(LD)
            p, q = a0 + (a1 - a0) * t, b0 + (b1 - b0) * t
            fa, fb = (t if cells[a][1] == i else 1 - t), (t if cells[b][1] == j else 1 - t)
            gamma = np.exp(-(1 + 2 * LD(s)) * np.log(np.abs(p[:, None] - q[None])))
            out -= 2 * abs(a1 - a0) * abs(b1 - b0) * ((w * fa)[:, None] * (w * fb)[None] * gamma).sum()
    return out


@pytest.mark.parametrize("s", [0.05, 0.5, 0.9])
def test_near_entries_of_an_interval(s):
    """An evaluation errs by at most 4.8e-15 (exponents to 40, tables and products of 64 bits); an entry
    is a sum of positive terms, the quadrature points add 2^-53 of a coordinate over a distance, below
    1e-15 on a mesh of 24 cells."""
    import torch
    m = synth.interval_mesh(24)
    x, cells = np.asarray(m.coords).reshape(-1), np.asarray(m.cells).reshape(-1, 2)
    mesh = vfd.vfd_mesh(1, m.coords, m.cells, m.cell_is_interior, leaf_m=64, lam=0.0)
    op = vfd.vfd_assemble(mesh, synth.const_field(s), synth.const_field(0.0), 0.95)
    dof, n = vfd.vfd_mesh_dofs(mesh)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    K = vfd.vfd_apply_parts(op, vfd.VFD_PART_KNEAR, eye, torch.empty_like(eye)).cpu().numpy()   # row j: K e_j
    vert = np.nonzero(dof >= 0)[0]
    worst = 0.0
    for i in vert[::3]:
        for j in vert:
            ref = _near_entry(x, cells, i, j, s)
            got = K[dof[j], dof[i]]
            worst = max(worst, float(abs(got - ref) / abs(ref)) if ref else abs(got))
    assert worst <= 6e-15


@pytest.mark.parametrize("leaf,p,lam", [(64, 4, 0.0), (32, 6, 0.75), (20, 8, 0.75)])
@pytest.mark.parametrize("nrhs", [1, 8, 64])
def test_apply_of_normal_columns(leaf, p, lam, nrhs):
    """Root mean square of a row's error in units of |A||x|: below 2^-53, one rounding."""
    import torch
    m = synth.disk_mesh(16, seed=3)
    mesh = vfd.vfd_mesh(2, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=p, lam=lam)
    s = synth.sigmoid_field(synth.random_fourier_field(21, 1.0), 0.1, 0.9)
    op = vfd.vfd_assemble(mesh, s, synth.random_fourier_field(22, 0.5), 0.95)
    n = mesh.n_dof
    eye, A = torch.eye(n, dtype=torch.float64, device="cuda"), torch.empty(n, n, dtype=torch.float64, device="cuda")
    for i in range(0, n, 4):
        vfd.vfd_apply_noalloc(op, eye[i:i + 4], A[i:i + 4])
    A = A.T.cpu().numpy().astype(LD)
    vfd.vfd_op_set_tensor_columns(op, 64)
    X = torch.randn(nrhs, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    Y = vfd.vfd_apply(op, X, torch.empty_like(X)).cpu().numpy()
    assert vfd.vfd_op_apply_stats(op)["tensor_columns"] == (64 if nrhs == 64 else 0)
    few = slice(0, 8)
    x = X.cpu().numpy()[few].astype(LD).T
    err = (Y[few].T - A @ x) / (np.abs(A) @ np.abs(x))
    assert float(np.sqrt((err ** 2).mean())) <= 2.0 ** -53
