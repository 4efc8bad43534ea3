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


@pytest.mark.parametrize("cloud", ["sphere", "sheet"])
@pytest.mark.parametrize("res", [4, 5, 7, 9, 11, 13, 15])
def test_a_lone_level_is_solved_to_float32_rounding(W, res, cloud):
    """The plain FP32 mode has no refinement: on a grid that is one level the
    one solve has to reach the tolerance by itself."""
    from paper_2609_20964_gb300 import PREC_FP32
    p, n = synth.sphere_cloud(4000, seed=res)
    if cloud == "sheet":
        p = np.random.default_rng(res).uniform(0.1, 0.9, p.shape).astype(np.float32)
        p[:, 2] = 0.5
        n = np.tile(np.float32([0, 0, 1]), (len(p), 1))
    rec = W(res, len(p), precision=PREC_FP32)
    rec.reconstruct(_t(p), _t(n), BBOX, res)
    info = rec.info()
    assert info["status"] == 0 and info["solver_steps"] == 1, info
    assert info["residual_rel"] <= 1e-6, info
    rec.close()
