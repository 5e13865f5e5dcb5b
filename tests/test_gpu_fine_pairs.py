"""Restriction and prolongation of level 0 in the mixed form's FP32 cycles,
several cells per thread (restrict_pair_kernel, prolong_quad_kernel, taken with
the 16-slot segments of fine_segments = 3), against the kernels over the
compact lists (fine_segments = 0): the same arithmetic in the same order, so
whole solves are bit-identical.  The sizes put the last pair of a row on the
row's padding (31 slots in a pitch of 32), on the next row (32 slots), and
the second children of the last coarse row and plane outside the box; the
masks are full, sparse (coarse cells with one or no unknown partner) and
reach every face of the box."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import workloads as W  # noqa: E402

from test_gpu_parity import make_pair  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


@pytest.mark.parametrize("n", [(61, 27, 25), (62, 26, 25), (63, 27, 26), (64, 33, 31), (93, 14, 35)])
@pytest.mark.parametrize("fill", [1.0, 0.9, 0.3])
@pytest.mark.parametrize("order", [1, 2])
def test_pairs_match_the_lists(dev, n, fill, order):
    shape = n[::-1]
    m = np.ones(shape, np.int8) if fill == 1.0 else W.random_mask(shape, seed=7, p_active=fill)
    w = {"mask": m, "rho": W.random_field(shape, 8), "h": 0.05, "faces": W.random_faces(shape, 9)}
    res = []
    for seg in (0, 3):
        H, _ = make_pair(w, dev, fine_segments=seg, precision=1, inner_cycles=2, order=order)
        st, info = H.solve(1e-9, 60)
        res.append((st, info, H.get_solution()))
    (st0, i0, s0), (st1, i1, s1) = res
    assert st0 == st1 and i0["cycles"] == i1["cycles"]
    assert np.array_equal(i0["hist"], i1["hist"], equal_nan=True)
    assert np.array_equal(s0.view(np.uint64), s1.view(np.uint64))
