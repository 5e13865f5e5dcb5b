"""Device memory of a batch: a patch holds its fields, lists and tables and no
records of the coarse levels' cluster launch, which batched cycles never use; its
first own solve allocates them once, and gives the same bits with and without
them (when the device is full)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

MB = 1 << 20


def patch_bytes(n):
    """The fields of a patch of n^3 cells in FP64 (a row of one colour padded to a multiple of 16 slots, a halo row and
    plane on each side): potential, right-hand side and codes of every level, D and 1/D and the mask sums of the coarse
    ones, level 0's h^2 rho, boundary terms, saved guess and b / D; the lists of both orders; the natural mask."""
    total, level, first = n ** 3, n, True
    while True:
        half = (level + 1) // 2
        slots = 2 * (level + 2) ** 2 * ((half + 1 + 15) // 16 * 16)
        cells = 2 * half * level * level
        total += slots * (8 + 8 + 1 + (32 if first else 16)) + cells * 4 * (1 if first else 3)
        if level <= 2:
            return total
        level, first = (level + 1) // 2, False


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_a_patch_reserves_no_cluster_records():
    n, count = 64, 24
    masks = [torch.ones((n, n, n), dtype=torch.int8, device="cuda") for _ in range(count)]
    B.Batch(masks[:1], [0.1]).close()  # the library's kernels and static memory
    before = free()
    Bt = B.Batch(masks, [0.1] * count)
    used = before - free()
    # each patch is one allocation of whole 2 MB pages; 1 MB for its tables and partial sums, 16 MB for the batch's
    assert used <= count * (patch_bytes(n) + 3 * MB) + 16 * MB, (used / count / MB, patch_bytes(n) / MB)
    rho = torch.from_numpy(W.random_field((n, n, n), seed=5)).cuda()
    for p in range(2):
        Bt.patch(p).set_rhs(rho)
    free0 = free()
    Bt.patch(0).solve(1e-6, 1)
    assert 0 < free0 - free() <= 24 * MB  # two orders' records, and the solve's graph
    free1 = free()
    Bt.patch(0).solve(1e-6, 1)
    assert free() == free1
    Bt.close()


def test_a_full_device_leaves_the_launch_path():
    shape = (40, 36, 44)
    mask = torch.from_numpy(W.random_mask(shape, seed=3, p_active=0.95)).cuda()
    rho = torch.from_numpy(W.random_field(shape, seed=5)).cuda()
    out = []
    for fail in (0, 1):
        Bt = B.Batch([mask], [0.1])
        P = Bt.patch(0)
        P.set_rhs(rho)
        B.mg_debug_fail_alloc(fail)
        st, info = P.solve(1e-8, 40)
        B.mg_debug_fail_alloc(0)
        out.append((st, info["cycles"], info["hist"], P.get_solution()))
        Bt.close()
    assert out[0][:2] == out[1][:2]
    assert np.array_equal(out[0][2], out[1][2]) and np.array_equal(out[0][3], out[1][3])
