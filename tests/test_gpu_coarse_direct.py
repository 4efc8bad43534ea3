"""Forward solves on grids whose coarsest multigrid level is solved directly in
the cosine basis (odd levels of 5^3 to 15^3, lone levels) and on the relaxed
ones beside them, both operators, against the FP64 oracle's indicator."""
import numpy as np
import pytest

import synth
from oracle import pipeline as OP

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BBOX = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
SIZES = [4, 5, 9, 11, 13, 15, 16, 18, 20, 24, 28, 36, 44, 60]


@pytest.fixture(scope="module")
def W():
    import __graft_entry__ as g
    g.build()
    from paper_2609_20964_gb300 import Reconstructor
    torch.cuda.set_device(0)
    return Reconstructor


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("galerkin", [0, 1])
@pytest.mark.parametrize("res", SIZES)
def test_forward_solve_matches_the_oracle(W, res, galerkin):
    p, n = synth.sphere_cloud(1200, seed=100 + res)
    ref = OP.forward_to_mesh(p, n, BBOX, res, operator="q1" if galerkin else "lumped")
    rec = W(res, len(p), galerkin=galerkin)
    rec.reconstruct(_t(p), _t(n), BBOX, res)
    info = rec.info()
    assert info["status"] == 0, info
    chi = rec.field("chi").cpu().numpy().astype(np.float64)
    span = ref.chi.max() - ref.chi.min()
    # a relaxed solve stops at 1e-6 of ||b||; the bound of the parity tests
    assert np.abs((chi - chi.mean()) - (ref.chi - ref.chi.mean())).max() <= 1e-4 * span
    rec.close()
