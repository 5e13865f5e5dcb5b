"""The FP64 prolongation of a large level 0 with short rows, on both sides of the row
length from which two unknowns per thread share their coarse cells, against the
oracle."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_prolong_pairs import dev, test_prolong_pairs as check  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,fill", [((240, 230, 6), 1.0), ((230, 220, 7), 1.0), ((230, 220, 8), 0.9),
                                        ((420, 400, 2), 1.0)])
@pytest.mark.parametrize("order", [1, 2])
def test_short_rows(dev, shape, fill, order):  # noqa: F811
    check(dev, shape, fill, order)
