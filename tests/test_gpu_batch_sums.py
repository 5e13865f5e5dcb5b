"""The batched residual norm and restriction with the integer neighbour sum
(fp64_sum = 1) against the plain sums (fp64_sum = 0), with chunks of one
round and of several rounds of a block: the two differ by the rounding of six
additions, so the relative norms of the first cycles agree to the bounds that
the batch's histories have against the oracle, and the chunk length changes no
cell's value at all."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_batch import HIST_FLOOR, HIST_REL, PATCHES, dev, make_batch  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,chunk", [(256, 0), (128, 4096), (512, 64)])
def test_sums_and_chunks(dev, oracle, threads, chunk):  # noqa: F811
    out = []
    for exact, c in ((1, 0), (1, chunk), (0, chunk)):
        Bt, _ = make_batch(dev, oracle, PATCHES, fp64_sum=exact)
        t = Bt.tuning
        t.threads, t.chunk = threads, c
        Bt.tuning = t
        r = [np.array(Bt.vcycle()) for _ in range(2)]
        out.append((r, [Bt.patch(p).get_solution() for p in range(len(PATCHES))]))
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
    for a, b in ((out[0], out[1]), (out[1], out[2])):
        for x, y in zip(a[0], b[0]):
            assert np.allclose(x, y, rtol=HIST_REL, atol=HIST_FLOOR)
