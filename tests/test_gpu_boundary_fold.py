"""Dirichlet values from the coarser level at the sizes where the fold's tiles
(128 cells of a row per warp) and the coarse grid's cover change: the folded
right-hand side against the values handed over as face arrays (the same
interpolation, folded face by face), and the residual norm from caller buffers
on the same boxes against the hierarchy's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [0, 3])
@pytest.mark.parametrize("p_active", [0.02, 0.6, 1.0])
@pytest.mark.parametrize("shape", [(3, 4, 1), (4, 5, 127), (3, 7, 128), (5, 3, 129), (2, 3, 300), (17, 18, 33)])
def test_fold_and_norm(shape, p_active, extra):
    dev = torch.device("cuda:0")
    nz, ny, nx = shape
    m = W.random_mask(shape, seed=7, p_active=p_active)
    m[0, 0, 0] = 1
    mask = torch.from_numpy(m).to(dev)
    rho = torch.from_numpy(W.random_field(shape, seed=8)).to(dev)
    phi = torch.from_numpy(W.random_field(shape, seed=9) * m).to(dev)
    origin = tuple(-2 - 2 * extra for _ in range(3))
    phi_c = torch.from_numpy(W.random_field(tuple((n + 1) // 2 + 2 + 2 * extra for n in shape), seed=10)).to(dev)
    faces = [torch.zeros(s, dtype=torch.float64, device=dev)
             for s in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))]
    h = 0.125
    with B.Hierarchy(mask, h) as H:
        H.set_rhs(rho)
        H.set_dirichlet_from_coarse(phi_c, origin)
        got = H.level_get(0, B.MG_FIELD_RHS)
        H.set_solution(phi)
        norm = H.residual_norm()[0]
        H.faces_from_coarse(phi_c, origin, *faces)
        H.set_dirichlet(*faces)
        want = H.level_get(0, B.MG_FIELD_RHS)
    # the same six terms added in another order at most: 6 roundings of values below 2 max|phi_c| each
    assert np.abs(got - want).max() <= 6 * 2.0 ** -52 * 12 * float(phi_c.abs().max())
    out = torch.zeros(1, dtype=torch.float64, device=dev)
    B.mg_residual_norm_noalloc(mask, phi, rho, h, out, *faces)
    assert abs(out.item() - norm) <= 1e-12 * norm


def test_a_face_outside_the_coarse_centres_is_refused():
    dev = torch.device("cuda:0")
    shape = (6, 6, 6)
    mask = torch.ones(shape, dtype=torch.int8, device=dev)
    phi_c = torch.zeros((5, 5, 5), dtype=torch.float64, device=dev)
    with B.Hierarchy(mask, 1.0) as H:
        for origin in ((0, -2, -2), (-2, -2, -4), (-2, 2 ** 31 - 1, -2), (-2 ** 31, -2, -2)):
            with pytest.raises(B.MGError) as e:
                H.set_dirichlet_from_coarse(phi_c, origin)
            assert e.value.status == B.MG_ERR_INVALID_ARG
        H.set_dirichlet_from_coarse(phi_c, (-2, -2, -2))
