"""A patch solved on its own handle after the batch's smoothing schedule changed:
the same bits, histories and counts as a hierarchy created with those sweeps.
The patch has run cycles and solves with the earlier schedule before, so every
graph it keeps is of that one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

PATCHES = [W.ball(48), W.blob_patch((40, 32, 48), seed=104), W.holes(32)]


def _load(P, w, dev):
    P.set_rhs(torch.from_numpy(np.array(w["rho"])).to(dev))
    if "phi_c" in w:
        P.set_dirichlet_from_coarse(torch.from_numpy(np.array(w["phi_c"])).to(dev), w["origin"])
    elif w.get("bx") is not None:
        P.set_dirichlet(*(torch.from_numpy(np.array(w[k])).to(dev) for k in ("bx", "by", "bz")))


def _run(P):
    """Two bare V-cycles and a solve from zero, then a solve that goes on from there."""
    P.hold = 0
    P.set_solution(None)
    out = [P.vcycle() for _ in range(2)]
    cycled = P.get_solution()
    P.set_solution(None)
    st, info = P.solve(1e-8, 40)
    again = P.solve(1e-12, 3)
    return out, cycled, st, info, again, P.get_solution()


@pytest.mark.parametrize("first", [(2, 2), (3, 1)])
@pytest.mark.parametrize("then", [(1, 1), (3, 2)])
def test_patch_after_a_schedule_change(first, then):
    check_schedule_change(first, then)


@pytest.mark.parametrize("first,then", [((2, 2), (0, 2)), ((2, 2), (2, 0)), ((1, 1), (0, 1)), ((0, 2), (2, 2)),
                                        ((2, 0), (1, 1))])
def test_one_sided_schedules_leave_the_cluster(first, then):
    """Sweeps on one side only: the coarse levels run launch by launch, as in a hierarchy created so."""
    check_schedule_change(first, then)


def check_schedule_change(first, then):
    dev = torch.device("cuda:0")
    masks = [torch.from_numpy(w["mask"]).to(dev) for w in PATCHES]
    with_batch, fresh = [], []
    Bt = B.Batch(masks, [w["h"] for w in PATCHES], n_pre=first[0], n_post=first[1])
    for p, w in enumerate(PATCHES):
        _load(Bt.patch(p), w, dev)
        _run(Bt.patch(p))
    t = Bt.tuning
    t.n_pre, t.n_post = then
    Bt.tuning = t
    for p, w in enumerate(PATCHES):
        with_batch.append(_run(Bt.patch(p)))
        with B.Hierarchy(masks[p], w["h"], n_pre=then[0], n_post=then[1]) as H:
            _load(H, w, dev)
            fresh.append(_run(H))
    for a, b in zip(with_batch, fresh):
        assert a[0] == b[0] and a[2] == b[2]
        for x, y in ((a[3], b[3]), (a[4][1], b[4][1])):
            assert {k: x[k] for k in ("cycles", "order", "switched", "cell_updates")} == \
                   {k: y[k] for k in ("cycles", "order", "switched", "cell_updates")}
            assert np.array_equal(x["hist"], y["hist"])
        for x, y in ((a[1], b[1]), (a[5], b[5])):
            assert np.array_equal(x.view(np.uint64), y.view(np.uint64))
