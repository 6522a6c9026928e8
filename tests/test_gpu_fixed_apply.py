"""The fixed-point FP64 apply (vfd_apply) against the FP64 kernels, which
vfd_apply_noalloc still runs, over the forms that change its launches: one to
many columns (groups of 8, 4, 2, 1; digits on the tensor cores from a few hundred
columns on for meshes this small), odd ranks, ragged leaves, wide panels, deep trees,
leading dimensions, and vectors that its formats do not hold.
"""
import pytest

import synth
from paper_2302_02863_gb300 import vfd

pytestmark = pytest.mark.gpu

# FP64 sums of up to 4000 products differ from each other by at most some 1e-14
# of sum |a||x|, which for normal x and the panels here is below 10 max|y|
TOL = 1e-13

MESHES = {
    "interval": lambda: synth.interval_mesh(333),
    "interval_long": lambda: synth.interval_mesh(2100),
    "disk": lambda: synth.disk_mesh(13, seed=3),
    "disk_mid": lambda: synth.disk_mesh(26, seed=4),
    "square_fine": lambda: synth.square_mesh(72, jitter=0.2, seed=6),
    "square": lambda: synth.square_mesh(30, jitter=0.2, seed=5),
    "ball": lambda: synth.kuhn_ball_mesh(9),
}


def _op(name, leaf, p, lam=0.75, **kw):
    m = MESHES[name]()
    mesh = vfd.vfd_mesh(m.d, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=p, lam=lam, **kw)
    s = synth.sigmoid_field(synth.random_fourier_field(21, 1.0, d=m.d), 0.1, 0.9)
    return mesh, vfd.vfd_assemble(mesh, s, synth.random_fourier_field(22, 0.5, d=m.d), 0.95)


@pytest.mark.parametrize("name,leaf,p,lam", [
    ("interval", 16, 5, 0.75), ("interval", 64, 8, 0.75), ("interval_long", 2, 3, 0.75), ("disk", 64, 4, 0.75),
    ("disk", 11, 5, 0.75), ("disk", 7, 1, 0.75), ("disk_mid", 33, 7, 0.75), ("disk_mid", 64, 8, 0.75),
    ("disk_mid", 64, 4, 0.0), ("square", 40, 3, 0.75), ("square", 130, 6, 0.75), ("ball", 24, 3, 1.2),
    ("ball", 64, 2, 0.75), ("square_fine", 60, 4, 0.75), ("square_fine", 28, 5, 0.75), ("square_fine", 13, 3, 0.75)])
def test_fixed_point_apply_matches_fp64(name, leaf, p, lam):
    import torch
    mesh, op = _op(name, leaf, p, lam)
    n = mesh.n_dof
    g = torch.Generator("cuda").manual_seed(7)
    for nrhs, ld in ((1, n), (1, n + 3), (2, n), (3, n + 1), (5, n), (8, n), (11, n + 5), (64, n), (449, n + 1)):
        X = torch.randn(nrhs, ld, dtype=torch.float64, device="cuda", generator=g)
        X *= 10.0 ** torch.randint(-3, 4, (nrhs, 1), device="cuda", generator=g)   # columns of their own scale
        Y, R = torch.full_like(X, 7.0), torch.full_like(X, 7.0)
        vfd.vfd_apply(op, X, Y)
        for r in range(nrhs):   # column by column: the static scratch is small
            vfd.vfd_apply_noalloc(op, X[r:r + 1], R[r:r + 1])
        assert torch.all(Y[:, n:] == 7.0)
        err = (Y - R)[:, :n].abs().amax(1) / R[:, :n].abs().amax(1)
        assert float(err.max()) <= TOL, (nrhs, ld, float(err.max()))


@pytest.mark.parametrize("name,leaf,p", [("disk", 20, 4), ("square", 64, 3), ("interval", 16, 5)])
@pytest.mark.parametrize("nrhs", [1, 9, 1000])
def test_fixed_point_apply_special_values(name, leaf, p, nrhs):
    import torch
    mesh, op = _op(name, leaf, p)
    n = mesh.n_dof
    x = torch.randn(nrhs, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(8))
    cases = {v: x.clone() for v in ("nan", "inf", "-inf", "zero", "1e-290", "1e-310", "1e290")}
    for v in ("nan", "inf", "-inf"):
        cases[v][nrhs // 2, n // 3] = float(v)
    cases["zero"].zero_()
    for v in ("1e-290", "1e-310", "1e290"):
        cases[v] *= float(v)
    for v, X in cases.items():
        Y, R = torch.empty_like(X), torch.empty_like(X)
        vfd.vfd_apply(op, X, Y)
        for r in range(0, nrhs, 8):
            vfd.vfd_apply_noalloc(op, X[r:r + 8], R[r:r + 8])
        assert torch.equal(torch.isnan(Y), torch.isnan(R)), v
        inf = torch.isinf(R)
        assert torch.equal(torch.isinf(Y), inf) and torch.equal(Y[inf], R[inf]), v
        ok = torch.isfinite(R)
        scale = R[ok].abs().max() if ok.any() else 0.0
        # denormals: sums of a few hundred products, each off by a unit of 5e-324
        assert bool(((Y - R)[ok].abs() <= TOL * scale + 1e-320).all()), v
