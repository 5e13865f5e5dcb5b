"""The coarse levels' cluster launch with deepest levels that no map solves: their
2 * coarse_sweeps half-sweeps run in one CTA or, above 256 unknowns of a colour,
over the cluster.  Masks with scattered holes end first-order hierarchies with
dozens to hundreds of unknowns; without the map (coarse_matrix = 0) the smallest
levels sweep too; and a mask whose coarser level holds more unknowns of one
colour than the finer one.  Bit for bit the launch path's V-cycles (option
coarse_cluster = 1), which runs the same levels through global memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def one_colour(nz, ny, nx):
    """Level 3: the even cells of an nz x ny x nx grid, all of one colour.  Under each, one level-2 child is wholly
    active and seven are half active (mask sum 0, no unknowns), the whole ones alternating in colour."""
    mask = np.zeros((8 * nz, 8 * ny, 8 * nx), np.int8)
    half = np.zeros((4, 4, 4), np.int8)
    half[:, :, :2] = 1  # four of the eight level-1 cells
    count = 0
    for k in range(nz):
        for j in range(ny):
            for i in range(nx):
                if (i + j + k) % 2:
                    continue
                for c in range(8):
                    z, y, x = 8 * k + 4 * (c >> 2), 8 * j + 4 * ((c >> 1) & 1), 8 * i + 4 * (c & 1)
                    mask[z:z + 4, y:y + 4, x:x + 4] = 1 if c == count % 2 else half
                count += 1
    return mask


def _masks():
    out = {"one_colour": one_colour(6, 10, 10)}
    for shape, p in (((64, 64, 64), 0.985), ((64, 64, 64), 0.995), ((48, 56, 72), 0.999), ((20, 130, 130), 0.995),
                     ((30, 30, 260), 0.998), ((260, 30, 30), 0.998)):
        out["%dx%dx%d_%g" % (*shape, p)] = W.random_mask(shape, seed=shape[0] + int(1000 * p), p_active=p)
    return out


MASKS = _masks()


def test_the_coarser_level_has_more_of_one_colour():
    with B.Hierarchy(torch.from_numpy(MASKS["one_colour"]).cuda(), 1.0 / 64) as H:
        act = [H.level_get(l, B.MG_FIELD_MASKSUM) > 0 for l in (1, 2, 3)]
    colour = [np.indices(a.shape).sum(0) % 2 for a in act]
    n = [(int((a & (c == 0)).sum()), int((a & (c == 1)).sum())) for a, c in zip(act, colour)]
    assert min(n[0]) > 256 and max(n[1]) <= 256 < max(n[2]) and min(n[2]) == 0, n


@pytest.mark.parametrize("matrix", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("name", sorted(MASKS))
def test_bitwise_the_launch_path(name, order, precision, matrix):
    mask = torch.from_numpy(MASKS[name]).cuda()
    rho = torch.from_numpy(W.random_field(MASKS[name].shape, seed=5)).cuda()
    got = []
    for cluster in (0, 1):
        with B.Hierarchy(mask, 1.0 / 64, order=order, precision=precision, coarse_cluster=cluster,
                         coarse_matrix=matrix) as H:
            H.set_rhs(rho)
            rel = [H.vcycle() for _ in range(2)]
            got.append((rel, H.get_solution()))
    assert got[0][0] == got[1][0]
    assert np.array_equal(got[0][1], got[1][1])
