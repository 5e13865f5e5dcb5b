"""The FP64 prolongation of a large level 0, two list entries per thread
(prolong_list_pairs_kernel), against the oracle: lists of odd and even length,
unknowns next to each other, apart and alone in their rows, and every corner
of the box."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

from test_gpu_parity import TOL, _level_state, active_of, dev, make_pair, relerr  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,fill", [((81, 70, 61), 1.0), ((80, 71, 62), 0.97), ((90, 81, 93), 0.6)])
@pytest.mark.parametrize("order", [1, 2])
def test_prolong_pairs(dev, shape, fill, order):  # noqa: F811
    m = np.ones(shape, np.int8) if fill == 1.0 else W.random_mask(shape, seed=31, p_active=fill)
    assert int((m > 0).sum()) >= 8 * torch.cuda.get_device_properties(dev).multi_processor_count * 256
    w = {"mask": m, "rho": W.random_field(shape, 32), "h": 0.1, "faces": W.random_faces(shape, 33)}
    H, R = make_pair(w, dev)
    _level_state(w, H, R, 0, order, seed=34)
    Sc = R.S(1)
    ec = np.where(active_of(Sc, 1, order), W.random_field(Sc.shape, 35), 0.0)
    H.level_set(1, B.MG_FIELD_PHI, ec)
    R.set_level_phi(1, ec)
    H.prolong_from(0, order)
    R.prolong_from(0, order)
    got, ref = H.level_get(0, B.MG_FIELD_PHI), R.phi(0)
    assert relerr(got, ref) < TOL
    # every cell's nine roundings, not only the largest cell's
    assert np.abs(got - ref).max() <= 16 * np.finfo(np.float64).eps * (np.abs(ref).max() + np.abs(ec).max())
