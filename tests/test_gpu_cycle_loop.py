"""A solve's cycles run as one graph with a loop on the device (use_graphs =
1) against one launch and one decision of the host per cycle (use_graphs =
0): the same cycles, the same norms and the same bits, where the loop ends by
convergence, by the order switch, by max_cycles (below, at and above the 64
cycles of one launch) and with a residual that no longer falls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import CASES, make_pair  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


@pytest.mark.parametrize("name", ["ball64", "blob48x32x40", "holes32"])
@pytest.mark.parametrize("tol,max_cycles", [(1e-8, 200), (1e-8, 1), (1e-8, 2), (1e-30, 64), (1e-30, 65), (1e-30, 130)])
@pytest.mark.parametrize("precision", [0, 1])
def test_loop_matches_single_cycles(dev, name, tol, max_cycles, precision):
    res = []
    for graphs in (0, 1):
        H, _ = make_pair(CASES[name], dev, use_graphs=graphs, precision=precision)
        first = H.solve(tol, max_cycles)
        again = H.solve(tol, max_cycles)  # the graph replayed, from the solution reached
        res.append((first, again, H.get_solution()))
    for (st0, i0), (st1, i1) in zip(res[0][:2], res[1][:2]):
        assert st0 == st1
        for k in ("cycles", "order", "switched"):
            assert i0[k] == i1[k]
        assert np.array_equal(i0["hist"], i1["hist"])
    assert np.array_equal(res[0][2].view(np.uint64), res[1][2].view(np.uint64))
