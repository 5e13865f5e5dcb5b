"""The calls that read the coarser level's potential return only once they have
read it, whatever the coarse grid's size: with work still queued on the
hierarchy's stream, nothing is left of it on return, and a potential (or a face
array) touched on another stream right after the call changes no result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1104_1703_gb300 import binding as B  # noqa: E402
from paper_1104_1703_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["set", "faces"])
@pytest.mark.parametrize("covered", [True, False])
def test_returns_after_reading(call, covered):
    dev = torch.device("cuda:0")
    n = 16
    m = np.zeros((n, n, n), np.int8)
    m[4:12, 4:12, 4:12] = 1  # away from the box's faces, so that a smaller coarse grid serves it too
    shape_c, origin = (((n + 1) // 2 + 2,) * 3, (-2, -2, -2)) if covered else ((n // 2,) * 3, (0, 0, 0))
    field = W.random_field(shape_c, seed=4)
    phi_c, kept = torch.from_numpy(field.copy()).to(dev), torch.from_numpy(field.copy()).to(dev)
    faces = [[torch.zeros(s, dtype=torch.float64, device=dev) for s in ((n, n, n + 1), (n, n + 1, n), (n + 1, n, n))]
             for _ in range(2)]
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    with B.Hierarchy(torch.from_numpy(m).to(dev), 0.1, stream=s.cuda_stream) as H:
        run = (lambda p, f: H.set_dirichlet_from_coarse(p, origin)) if call == "set" else \
              (lambda p, f: H.faces_from_coarse(p, origin, *f))
        run(kept, faces[0])
        want = H.level_get(0, B.MG_FIELD_RHS) if call == "set" else [f.clone() for f in faces[0]]
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)  # about 10 ms
        run(phi_c, faces[1])
        assert s.query()
        with torch.cuda.stream(other):
            phi_c.fill_(1e30)
            got = [f.clone() for f in faces[1]]
        torch.cuda.synchronize()
        if call == "set":
            assert np.array_equal(H.level_get(0, B.MG_FIELD_RHS), want)
        else:
            assert all(torch.equal(a, b) for a, b in zip(got, want))
