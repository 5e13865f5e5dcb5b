"""The residual norm from caller buffers and the fold of the coarser level's values
on boxes with short rows, where a tile takes several of them: rows of one cell
up to the longest that two fit a tile, a last tile that is not full.  The norm
against the residual by plain torch in the same precision (six additions and two
multiplications per cell, relative error of a norm far below 1e-12), with
non-finite values at active cells and none taken from inactive ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu

# (nz, ny, nx): more rows than the GPU holds warps, down to few
SHAPES = [(1024, 512, 1), (101, 151, 1), (300, 211, 2), (200, 300, 3), (512, 512, 5), (256, 257, 16), (130, 129, 33),
          (150, 150, 85), (128, 128, 127), (128, 129, 128), (5, 7, 9), (1, 1, 1), (2048, 3, 2), (3, 2048, 7)]


def _fields(shape, seed, p_active):
    nz, ny, nx = shape
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    draw = lambda s: torch.randn(s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    mask = (torch.rand(shape, generator=g, device="cuda") < p_active).to(torch.int8)
    mask[0, 0, 0] = 1
    return mask, draw(shape), draw(shape), [draw(s) for s in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))]


def reference(mask, phi, rho, h, faces):
    act = mask > 0
    a = torch.where(act, phi, torch.zeros_like(phi))
    r = -h * h * rho
    diag = torch.full_like(phi, 6.0)
    for axis in range(3):
        n = phi.shape[axis]
        for step in (-1, 1):
            inside = torch.zeros_like(act)
            near = torch.zeros_like(a)
            to, src = (slice(1, n), slice(0, n - 1)) if step < 0 else (slice(0, n - 1), slice(1, n))
            ix = lambda s: tuple(s if d == axis else slice(None) for d in range(3))  # noqa: E731
            inside[ix(to)] = act[ix(src)]
            near[ix(to)] = a[ix(src)]
            face = faces[2 - axis].narrow(axis, 0 if step < 0 else 1, n)
            r = r + torch.where(inside, near, 2.0 * face)
            diag = diag + (~inside).double()
    r = torch.where(act, r - diag * a, torch.zeros_like(a))
    return float((r.square().sum().sqrt() / (h * h)).item())


def norm(mask, phi, rho, h, faces):
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    B.mg_residual_norm_noalloc(mask, phi, rho, h, out, *faces)
    return float(out.item())


@pytest.mark.parametrize("p_active", [0.03, 0.6, 1.0])
@pytest.mark.parametrize("shape", SHAPES)
def test_norm(shape, p_active):
    mask, phi, rho, faces = _fields(shape, 11, p_active)
    phi = torch.where(mask > 0, phi, torch.full_like(phi, float("nan")))  # inactive cells are ignored
    rho = torch.where(mask > 0, rho, torch.full_like(rho, float("inf")))
    want = reference(mask, phi, torch.where(mask > 0, rho, torch.zeros_like(rho)), 0.125, faces)
    assert abs(norm(mask, phi, rho, 0.125, faces) - want) <= 1e-12 * want


@pytest.mark.parametrize("shape", [(200, 300, 3), (40, 40, 200)])
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan"), 1e200])
@pytest.mark.parametrize("where", ["phi", "rho", "face"])
def test_non_finite(shape, value, where):
    mask, phi, rho, faces = _fields(shape, 12, 1.0)
    {"phi": phi, "rho": rho, "face": faces[0]}[where][shape[0] // 2, shape[1] // 3, 0] = value
    want, got = reference(mask, phi, rho, 0.125, faces), norm(mask, phi, rho, 0.125, faces)
    assert not np.isfinite(want) and np.array_equal(got, want, equal_nan=True)


@pytest.mark.parametrize("p_active", [0.03, 0.6, 1.0])
@pytest.mark.parametrize("shape", [s for s in SHAPES if s[2] < 128] + [(100, 111, 63), (90, 100, 64), (90, 100, 65)])
def test_fold(shape, p_active):
    """Boundary values interpolated from the coarser level and folded, against the same values as face arrays."""
    nz, ny, nx = shape
    mask, rho, _, faces = _fields(shape, 13, p_active)
    g = torch.Generator(device="cuda")
    g.manual_seed(14)
    phi_c = torch.randn(tuple((n + 1) // 2 + 2 for n in shape), generator=g, device="cuda", dtype=torch.float64)
    with B.Hierarchy(mask, 0.125) as H:
        H.set_rhs(rho)
        H.set_dirichlet_from_coarse(phi_c, (-2, -2, -2))
        got = H.level_get(0, B.MG_FIELD_RHS)
        H.faces_from_coarse(phi_c, (-2, -2, -2), *faces)
        H.set_dirichlet(*faces)
        want = H.level_get(0, B.MG_FIELD_RHS)
        if p_active == 1.0:
            with pytest.raises(B.MGError):
                H.set_dirichlet_from_coarse(phi_c, (-2, 0, -2))
    # the same six terms added in another order at most: 6 roundings of values below 12 max|phi_c|
    assert np.abs(got - want).max() <= 6 * 2.0 ** -52 * 12 * float(phi_c.abs().max())


@pytest.mark.parametrize("shape", [(200, 300, 3), (20, 22, 140)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_fold_non_finite(shape, value):
    """A non-finite coarse value reaches the cells whose faces it serves, and no other."""
    nz, ny, nx = shape
    mask, rho, _, faces = _fields(shape, 15, 0.9)
    phi_c = torch.ones(tuple((n + 1) // 2 + 2 for n in shape), dtype=torch.float64, device="cuda")
    phi_c[nz // 4, ny // 4, 1] = value
    with B.Hierarchy(mask, 0.125) as H:
        H.set_rhs(rho)
        H.set_dirichlet_from_coarse(phi_c, (-2, -2, -2))
        got = H.level_get(0, B.MG_FIELD_RHS)
        H.faces_from_coarse(phi_c, (-2, -2, -2), *faces)
        H.set_dirichlet(*faces)
        want = H.level_get(0, B.MG_FIELD_RHS)
    bad = ~np.isfinite(got)
    assert 0 < bad.sum() < 2000 and np.array_equal(bad, ~np.isfinite(want))
    assert np.abs(got[~bad] - want[~bad]).max() <= 6 * 2.0 ** -52 * (12 + 0.02 * float(rho.abs().max()))
