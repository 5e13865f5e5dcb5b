"""Solves that end in a few cycles run them one by one instead of in the graph's
loop: hierarchies of one level, lines of cells, loose tolerances and mixed solves
with many FP32 cycles per step.  The same cycles, norms and bits as with one host
decision per cycle and no graphs (use_graphs = 0), on both sides of the rule."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

OPTIONS = [dict(), dict(precision=1), dict(precision=1, inner_cycles=4), dict(precision=1, inner_cycles=8), dict(order=1)]


@pytest.mark.parametrize("opts", range(len(OPTIONS)))
@pytest.mark.parametrize("tol", [1e-2, 1e-5, 1e-8, 1e-30])
@pytest.mark.parametrize("shape", [(4, 4, 4), (1, 1, 70), (70, 1, 1), (16, 16, 16), (30, 33, 28)])
def test_same_as_without_graphs(shape, tol, opts):
    mask = torch.from_numpy(W.random_mask(shape, seed=3, p_active=0.97)).cuda()
    rho = torch.from_numpy(W.random_field(shape, seed=5)).cuda()
    res = []
    for graphs in (0, 1):
        with B.Hierarchy(mask, 0.1, use_graphs=graphs, **OPTIONS[opts]) as H:
            H.set_rhs(rho)
            first = H.solve(tol, 12)
            again = H.solve(tol, 70)
            res.append((first, again, H.get_solution()))
    for (st0, i0), (st1, i1) in zip(res[0][:2], res[1][:2]):
        assert st0 == st1
        assert all(i0[k] == i1[k] for k in ("cycles", "order", "switched", "cell_updates"))
        assert np.array_equal(i0["hist"], i1["hist"])
    assert np.array_equal(res[0][2].view(np.uint64), res[1][2].view(np.uint64))
