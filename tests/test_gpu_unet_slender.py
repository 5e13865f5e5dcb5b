"""The network on grids one or two voxels wide, where a box of several tiles of
128 voxels is longer than a TMA copy may be (256 per axis) and the convolution
has to work on fewer tiles together: every convolution against the oracle, and
a training step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from test_gpu_unet import _input, _params, dev, flat, test_each_convolution_matches_the_oracle as check  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(100, 512, 1), (70, 513, 1), (64, 512, 2), (512, 100, 1)])
def test_slender_grids(dev, n):  # noqa: F811
    check(None, 1, n)
    net = B.UNet(1, 16, n)
    net.set_params(flat(_params(1, 16, 12)))
    x = _input(n, 6)
    y = np.random.default_rng(3).normal(size=n).astype(np.float32)
    first = net.train_step(x, y)
    assert np.isfinite(first) and np.isfinite(net.get_grads()).all() and net.train_step(x, y) != first
