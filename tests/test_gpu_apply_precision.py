"""Precision of the FP64 apply (vfd_apply) row by row: columns of the operator (unit
vectors) and vectors that span many decades, against the FP64 kernels, which
vfd_apply_noalloc runs, in units of |A||x|.
"""
import numpy as np
import pytest

import synth
from paper_2302_02863_gb300 import vfd

pytestmark = pytest.mark.gpu

# A row is a sum of up to 1200 products, of which a lane adds an eighth one after another:
# at most some 150 roundings of 2^-53 of its part of |A||x|, about their square root as
# roundings fall; the far field's three sums behave alike.  64 lies between.
TOL = 64 * 2.0 ** -53


def _setup(name, leaf, p, lam):
    m = synth.disk_mesh(18, seed=3) if name == "disk" else synth.square_mesh(30, jitter=0.2, seed=5)
    mesh = vfd.vfd_mesh(m.d, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=p, lam=lam)
    s = synth.sigmoid_field(synth.random_fourier_field(21, 1.0), 0.1, 0.9)
    op = vfd.vfd_assemble(mesh, s, synth.random_fourier_field(22, 0.5), 0.95)
    dof = vfd.vfd_mesh_dofs(mesh)[0]
    x = np.zeros((mesh.n_dof, 2))
    x[dof[dof >= 0]] = np.asarray(m.coords).reshape(-1, 2)[dof >= 0]
    return op, mesh.n_dof, x


def _apply(f, op, X, width):
    import torch
    Y = torch.empty_like(X)
    for i in range(0, len(X), width):
        f(op, X[i:i + width], Y[i:i + width])
    return Y


def _columns(op, n, f, width):
    import torch
    return _apply(f, op, torch.eye(n, dtype=torch.float64, device="cuda"), width)   # row j: A e_j


def _vectors(x, rows):
    """name -> (rows, n): magnitudes that vary along the mesh, from row to row of it, or in one place."""
    rng = np.random.default_rng(1)
    n, at = len(x), rng.uniform(-0.5, 0.5, (rows, 1, 2))
    sign = rng.choice([-1.0, 1.0], (rows, n))
    spike = np.zeros((rows, n))
    spike[np.arange(rows), rng.integers(0, n, rows)] = 1.0
    return {"normal": rng.standard_normal((rows, n)), "ones": np.ones((rows, n)),
            "six decades": sign * 10.0 ** (-6.0 * rng.random((rows, n))),
            "14 decades across": sign * 10.0 ** (-7.0 * (x[:, 0] + 1.0)),
            "local": np.exp(-((x - at) ** 2).sum(-1) / 0.02), "spike on 1e-18": spike + 1e-18 * sign}


SETUPS = [("disk", 64, 4, 0.0), ("disk", 32, 6, 0.75), ("square", 40, 8, 0.75), ("square", 16, 3, 0.75)]


@pytest.mark.parametrize("name,leaf,p,lam", SETUPS)
@pytest.mark.parametrize("width", [1, 5, 8])
def test_unit_vectors_give_the_entries(name, leaf, p, lam, width):
    op, n, _ = _setup(name, leaf, p, lam)
    A, B = _columns(op, n, vfd.vfd_apply_noalloc, 8), _columns(op, n, vfd.vfd_apply, width)
    if lam == 0.0:   # no far field: a panel entry plus a B + M entry, one rounding in any order
        assert bool((A == B).all())
    assert bool(((B - A).abs() <= TOL * A.abs()).all()), float(((B - A).abs() / A.abs().clamp_min(1e-300)).max())


@pytest.mark.parametrize("name,leaf,p,lam", SETUPS)
@pytest.mark.parametrize("width", [1, 3, 8])
def test_rows_keep_fp64_precision(name, leaf, p, lam, width):
    import torch
    op, n, x = _setup(name, leaf, p, lam)
    A = _columns(op, n, vfd.vfd_apply_noalloc, 8).abs()
    for kind, v in _vectors(x, 9).items():
        X = torch.tensor(v, device="cuda")
        R, Y = _apply(vfd.vfd_apply_noalloc, op, X, 3), _apply(vfd.vfd_apply, op, X, width)
        err = (Y - R).abs() / (X.abs() @ A)
        assert float(err.max()) <= TOL, (kind, float(err.max()))


@pytest.mark.parametrize("name,leaf,p,lam", SETUPS)
def test_many_columns_keep_fp64_precision(name, leaf, p, lam):
    """On the tensor cores (their digits hold normal vectors, the rest is redone)."""
    import torch
    op, n, x = _setup(name, leaf, p, lam)
    vfd.vfd_op_set_tensor_columns(op, 1)
    A = _columns(op, n, vfd.vfd_apply_noalloc, 8)
    # |A| as the sum over the parts: a near entry and one of B + M may cancel
    parts = sum(_columns(op, n, lambda o, X, Y, m=m: vfd.vfd_apply_parts(o, m, X, Y), 8).abs()
                for m in (vfd.VFD_PART_B | vfd.VFD_PART_M, vfd.VFD_PART_KNEAR, vfd.VFD_PART_KFAR))
    B = _columns(op, n, vfd.vfd_apply, n)
    assert vfd.vfd_op_apply_stats(op)["tensor_columns"] == n
    if lam == 0.0:
        assert bool((A == B).all())
    assert bool(((B - A).abs() <= TOL * A.abs()).all())
    rows = 1003
    for kind, v in _vectors(x, rows).items():
        X = torch.tensor(v, device="cuda")
        R, Y = _apply(vfd.vfd_apply_noalloc, op, X, 3), _apply(vfd.vfd_apply, op, X, rows)
        st = vfd.vfd_op_apply_stats(op)
        assert st["tensor_columns"] == rows and st["expired"] == 0
        # normal and constant columns are what the digits are for
        if kind in ("normal", "ones"):
            assert st["near_rows"] <= 0.01 * n * rows / 8 and st["projections"] == 0, (kind, st)
        if kind in ("14 decades across", "spike on 1e-18"):
            assert st["near_rows"] > 0, (kind, st)
        err = (Y - R).abs() / (X.abs() @ parts)
        assert float(err.max()) <= TOL, (kind, float(err.max()), st)


def test_unfit_columns_leave_the_others_alone():
    """Columns that the digits cannot hold at all (Inf, NaN, nearly denormal) among normal ones."""
    import torch
    op, n, x = _setup("square", 40, 8, 0.75)
    vfd.vfd_op_set_tensor_columns(op, 1)
    A = _columns(op, n, vfd.vfd_apply_noalloc, 8).abs()
    X = torch.randn(640, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    X[5, n // 2], X[77, 3], X[130], X[300] = float("nan"), float("inf"), 0.0, 1e-300 * X[300]
    R, Y = _apply(vfd.vfd_apply_noalloc, op, X, 8), torch.empty_like(X)
    vfd.vfd_apply(op, X, Y)
    st = vfd.vfd_op_apply_stats(op)
    assert st["tensor_columns"] == 640 and st["projections"] > 0 and st["leaves"] > 0
    assert torch.equal(torch.isnan(Y), torch.isnan(R)) and torch.equal(torch.isinf(Y), torch.isinf(R))
    ok = torch.isfinite(X).all(1)
    assert not Y[130].any()
    err = (Y - R).abs()[ok] / (X.abs() @ A).clamp_min(5e-324 * 2.0 ** 53)[ok]
    assert float(err.max()) <= TOL


FORMS = {
    "interval": lambda: synth.interval_mesh(333),
    "interval_long": lambda: synth.interval_mesh(2100),
    "disk": lambda: synth.disk_mesh(13, seed=3),
    "disk_mid": lambda: synth.disk_mesh(26, seed=4),
    "square": lambda: synth.square_mesh(30, jitter=0.2, seed=5),
    "graded": lambda: synth.square_mesh_graded(20, 1.5),
    "ball": lambda: synth.kuhn_ball_mesh(9),
}


@pytest.mark.parametrize("name,leaf,p,lam", [
    ("interval", 16, 5, 0.75), ("interval_long", 2, 3, 0.75), ("disk", 11, 5, 0.75), ("disk", 7, 1, 0.75),
    ("disk_mid", 33, 7, 0.75), ("disk_mid", 64, 8, 0.75), ("disk_mid", 64, 4, 0.0), ("square", 28, 5, 0.75),
    ("graded", 24, 4, 0.75), ("ball", 24, 3, 1.2), ("ball", 64, 2, 0.75)])
def test_tensor_apply_over_forms(name, leaf, p, lam):
    """Odd ranks, ragged and tiny leaves, deep trees, no far field, one to many columns in tiles of
    16, 32 and 64 and in several passes, leading dimensions."""
    import torch
    m = FORMS[name]()
    mesh = vfd.vfd_mesh(m.d, m.coords, m.cells, m.cell_is_interior, leaf_m=leaf, cheb_p=p, lam=lam)
    s = synth.sigmoid_field(synth.random_fourier_field(21, 1.0, d=m.d), 0.1, 0.9)
    op = vfd.vfd_assemble(mesh, s, synth.random_fourier_field(22, 0.5, d=m.d), 0.95)
    vfd.vfd_op_set_tensor_columns(op, 1)
    n, g = mesh.n_dof, torch.Generator("cuda").manual_seed(7)
    for nrhs, ld in ((1, n), (3, n + 1), (8, n), (17, n + 5), (40, n), (64, n + 3), (150, n + 1)):
        X = torch.randn(nrhs, ld, dtype=torch.float64, device="cuda", generator=g)
        X *= 10.0 ** torch.randint(-3, 4, (nrhs, 1), device="cuda", generator=g)
        Y, R = torch.full_like(X, 7.0), torch.full_like(X, 7.0)
        vfd.vfd_apply(op, X, Y)
        st = vfd.vfd_op_apply_stats(op)
        assert st["tensor_columns"] == nrhs and st["expired"] == 0
        for r in range(nrhs):
            vfd.vfd_apply_noalloc(op, X[r:r + 1], R[r:r + 1])
        assert torch.all(Y[:, n:] == 7.0)
        # sums of a few hundred terms of one size: a row's |A||x| is below 16 times the largest |y|
        err = (Y - R)[:, :n].abs().amax(1) / R[:, :n].abs().amax(1)
        assert float(err.max()) <= 16 * TOL, (nrhs, ld, float(err.max()), st)


def test_rule_counts_the_columns_of_a_pass():
    """Several passes of a small mesh are no reason for the tensor cores; one pass of a larger one is."""
    import torch
    op, n, _ = _setup("disk", 64, 4, 0.75)
    X = torch.ones(1024, n, dtype=torch.float64, device="cuda")
    vfd.vfd_apply(op, X, torch.empty_like(X))
    assert vfd.vfd_op_apply_stats(op)["tensor_columns"] == 0
    vfd.vfd_op_set_tensor_columns(op, 1000)
    vfd.vfd_apply(op, X, torch.empty_like(X))
    assert vfd.vfd_op_apply_stats(op)["tensor_columns"] == 1024
    m = synth.disk_mesh(37, seed=3)
    mesh = vfd.vfd_mesh(2, m.coords, m.cells, m.cell_is_interior, leaf_m=64, cheb_p=8)
    op = vfd.vfd_assemble(mesh, synth.config2_s_field(), synth.const_field(0.0), 0.9)
    X = torch.ones(64, mesh.n_dof, dtype=torch.float64, device="cuda")
    vfd.vfd_apply(op, X, torch.empty_like(X))
    assert vfd.vfd_op_apply_stats(op)["tensor_columns"] == 64


@pytest.mark.parametrize("name,leaf,p,lam", SETUPS)
def test_expired_waits_are_redone(name, leaf, p, lam):
    """A wait limit of zero: every wait of the digit kernels that is not satisfied already gives up,
    the kernels drain and return, and the apply comes from the others."""
    import torch
    op, n, _ = _setup(name, leaf, p, lam)
    vfd.vfd_op_set_tensor_columns(op, 1)
    X = torch.randn(150, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    R, Y, Z, W = (torch.full_like(X, 7.0) for _ in range(4))
    vfd.vfd_apply(op, X, R)
    assert vfd.vfd_op_apply_stats(op)["expired"] == 0
    vfd.vfd_op_set_wait_limit(op, 0.0)
    vfd.vfd_apply(op, X, Y)
    assert vfd.vfd_op_apply_stats(op)["expired"] == 1
    vfd.vfd_op_set_tensor_columns(op, 1000)   # the kernels of few columns
    vfd.vfd_apply(op, X, Z)
    assert vfd.vfd_op_apply_stats(op)["tensor_columns"] == 0
    err = (Y - Z).abs().amax(1) / Z.abs().amax(1)
    assert float(err.max()) <= 16 * TOL
    # the default limit again: the digits as before
    vfd.vfd_op_set_tensor_columns(op, 1)
    vfd.vfd_op_set_wait_limit(op, 1.0)
    vfd.vfd_apply(op, X, W)
    assert vfd.vfd_op_apply_stats(op)["expired"] == 0 and torch.equal(W, R)
    for bad in (-1.0, float("nan"), float("inf")):
        with pytest.raises(vfd.VfdError) as e:
            vfd.vfd_op_set_wait_limit(op, bad)
        assert e.value.status == vfd.VFD_EINVAL
