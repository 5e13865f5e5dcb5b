"""The coarse levels' cluster launch (dPhi in distributed shared memory) at the
sizes where its plan changes: 2, 4, 8 and 16 CTAs, odd and flat boxes, slabs
of uneven depth, planes without unknowns, a distributed deepest level, and no
plan at all.  The arithmetic is that of the launch-per-step kernels in the same
order, so V-cycles agree bit for bit with option coarse_cluster = 1, which
runs the same levels through global memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _mask(shape, kind):
    nz, ny, nx = shape
    if kind == "full":
        return np.ones(shape, np.int8)
    if kind == "random":
        return W.random_mask(shape, seed=nx + 3 * ny + 7 * nz, p_active=0.9)
    m = np.ones(shape, np.int8)  # "gap": two slabs with empty planes between them
    m[nz // 3:nz // 3 + max(1, nz // 5)] = 0
    return m


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("kind", ["full", "random", "gap"])
@pytest.mark.parametrize("shape", [(32, 32, 32), (33, 35, 31), (62, 46, 58), (20, 70, 66), (9, 80, 64), (5, 60, 90),
                                   (140, 18, 22), (66, 64, 130), (8, 8, 8)])
def test_bitwise_the_launch_path(shape, kind, order, precision):
    dev = torch.device("cuda:0")
    mask = torch.from_numpy(_mask(shape, kind)).to(dev)
    rho = torch.from_numpy(W.random_field(shape, seed=5)).to(dev)
    got = []
    for cluster in (0, 1):
        with B.Hierarchy(mask, 1.0 / 64, order=order, precision=precision, coarse_cluster=cluster) as H:
            H.set_rhs(rho)
            rel = [H.vcycle() for _ in range(2)]
            got.append((rel, H.get_solution()))
    assert got[0][0] == got[1][0]
    assert np.array_equal(got[0][1], got[1][1])
