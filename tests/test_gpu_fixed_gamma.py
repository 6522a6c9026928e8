"""The fixed-point kernel evaluations of the assembly against the FP64 ones.

A constant c added to log kappa scales every part of the operator by e^c; with
c = 120 the fields leave the fixed-point formats and the assembly takes its FP64
path, so the two operators, the second scaled back, have to agree part by part.
"""
import math
from types import SimpleNamespace

import numpy as np
import pytest

import synth
from paper_2302_02863_gb300 import vfd

pytestmark = pytest.mark.gpu
SHIFT = 120.0

# the FP64 path rounds an exponent of up to SHIFT + 60 at every operation (2^-53
# of it, a few times: below 1e-13); the fixed path's error is below 1e-14.  Near
# blocks and the density are sums of positive terms; the far field's bases and the
# singular rules' basis differences change sign, which costs another factor of 10
TOL = {"rho": 1e-13, vfd.VFD_PART_M: 1e-13, vfd.VFD_PART_KNEAR: 1e-13, vfd.VFD_PART_KFAR: 1e-12,
       vfd.VFD_PART_B: 1e-12}

MESHES = {
    "interval": lambda: synth.interval_mesh(150),
    "interval_wide": lambda: synth.interval_mesh(37, R=9.0),
    "disk": lambda: synth.disk_mesh(9, seed=3),
    "disk_unsplit": lambda: synth.disk_mesh(40, seed=4),     # enough blocks for one CTA each
    "disk_leaf": lambda: synth.disk_mesh(7, seed=6),         # 127 DoFs in one leaf
    "square": lambda: synth.square_mesh(14, jitter=0.2, seed=5),
    "graded": lambda: synth.square_mesh_graded(12, 1.5),
    "ball": lambda: synth.kuhn_ball_mesh(7),
}


@pytest.mark.parametrize("name,leaf,p", [
    ("interval", 16, 3), ("interval", 64, 8), ("interval_wide", 5, 2), ("disk", 64, 4), ("disk", 7, 8), ("disk", 3, 1),
    ("disk_unsplit", 64, 4), ("disk_unsplit", 33, 5), ("disk_leaf", 130, 3), ("square", 20, 7), ("graded", 16, 4),
    ("ball", 64, 4), ("ball", 10, 3)])
@pytest.mark.parametrize("s_range,n_sing", [((0.0, 0.1), 2), ((0.2, 0.89), 3)])
def test_fixed_point_assembly_matches_fp64(name, leaf, p, s_range, n_sing):
    import torch
    m = MESHES[name]()
    mesh = vfd.vfd_mesh(m.d, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=p, rho_leaf_m=leaf, n_sing=n_sing)
    lo, hi = s_range
    s = synth.sigmoid_field(synth.random_fourier_field(11, 1.0, d=m.d), lo, hi)
    rows = synth.random_fourier_field(12, 0.7, d=m.d).fourier
    x = torch.rand(mesh.n_dof, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) + 0.5

    def parts(shift):
        op = vfd.vfd_assemble(mesh, s, SimpleNamespace(c0=shift, fourier=rows), 0.9)
        out = {"rho": vfd.vfd_op_rho(op, torch.empty(mesh.info["n_qint"], dtype=torch.float64, device="cuda"))}
        for part in (vfd.VFD_PART_M, vfd.VFD_PART_KNEAR, vfd.VFD_PART_KFAR, vfd.VFD_PART_B):
            out[part] = vfd.vfd_apply_parts(op, part, x, torch.empty_like(x))
        return {k: v.cpu().numpy() for k, v in out.items()}

    fixed, fp64 = parts(0.0), parts(SHIFT)
    for key, tol in TOL.items():
        a, b = fixed[key], fp64[key] * math.exp(-SHIFT)
        scale = np.abs(b).max() if key in (vfd.VFD_PART_KFAR, vfd.VFD_PART_B) else np.abs(b)
        assert np.all(np.abs(a - b) <= tol * scale), (key, float(np.max(np.abs(a - b) / (scale + 1e-300))))


@pytest.mark.parametrize("name,leaf,p,n_sing", [("interval", 16, 4, 3), ("disk", 16, 4, 3), ("disk", 9, 7, 2),
                                                ("square", 64, 6, 3), ("disk_unsplit", 64, 5, 3)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 10])
def test_fixed_point_gradient_matches_fp64(name, leaf, p, n_sing, nrhs):
    """vfd_grad at fixed U and Lam scales by e^c with A; the sums change sign, so the
    1e-13 of their terms is left to grow by the cancellation of random U and Lam."""
    import torch
    m = MESHES[name]()
    mesh = vfd.vfd_mesh(m.d, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=p, rho_leaf_m=leaf, n_sing=n_sing)
    x = m.coords
    s = 0.45 + 0.3 * np.sin(2.0 * x[:, 0]) * np.cos(1.3 * x[:, -1])
    lk = 0.3 * np.cos(1.5 * x[:, -1])
    g = torch.Generator("cuda").manual_seed(3)
    U, Lam = (torch.randn(nrhs, mesh.n_dof, dtype=torch.float64, device="cuda", generator=g) for _ in range(2))

    def grads(shift):
        op = vfd.vfd_assemble(mesh, synth.nodal_field(s), synth.nodal_field(lk + shift), 0.9)
        out = [torch.empty(m.n_vert, dtype=torch.float64, device="cuda") for _ in range(2)]
        vfd.vfd_grad(op, U, Lam, *out)
        return [o.cpu().numpy() for o in out]

    for a, b in zip(grads(0.0), grads(SHIFT)):
        b = b * math.exp(-SHIFT)
        assert np.abs(a - b).max() <= 1e-11 * np.abs(b).max()
