"""The adjoint's direct solve on grids without an FFT pass (dense folded
cosine transforms): sizes with odd halves, one line tile and several, lines
that end inside a tile, reductions that end inside a staged chunk, both
operators, against the FP64 oracle's solve."""
import numpy as np
import pytest

import synth
from oracle import galerkin_q1 as Q1
from oracle import poisson as PO

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BBOX = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
SIZES = [4, 5, 9, 15, 16, 18, 24, 36, 44, 72, 88]


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
def test_adjoint_solve_matches_the_oracle(W, res, galerkin):
    p, n = synth.sphere_cloud(1200, seed=100 + res)
    rec = W(res, len(p), galerkin=galerkin)
    rec.reconstruct(_t(p), _t(n), BBOX, res)
    g = np.random.default_rng(res).standard_normal((res, res, res)).astype(np.float32)
    rec.backward(d_sdf_grid=_t(g))
    info = rec.info()
    # two FP32-exact corrections: 1e-6 of the right-hand side after the first
    # (n / 2 terms a sum), its square and the float-float limit after the second
    assert info["backward_steps"] == 2 and info["backward_residual_rel"] <= 1e-9, info
    dchi = rec.field("dchi").cpu().numpy().astype(np.float64)
    lam = rec.field("lambda").cpu().numpy().astype(np.float64)
    assert dchi.any()
    # the exported fields are the solved ones rounded to float32 (the unlumped
    # system is stored times 12)
    want = Q1.solve27(dchi) / 12.0 if galerkin else PO.solve(dchi)
    assert np.linalg.norm(lam - lam.mean() - want) <= 1e-5 * np.linalg.norm(want)
    rec.close()


def test_one_handle_over_several_grids(W):
    """A handle that changes grids rebuilds the basis tables."""
    p, n = synth.sphere_cloud(2000, seed=9)
    rec = W(72, len(p))
    for res in (72, 24, 64, 44, 72):
        g = _t(np.random.default_rng(res).standard_normal((res, res, res)).astype(np.float32))
        rec.reconstruct(_t(p), _t(n), BBOX, res, with_normals=False)
        a, _, _ = rec.backward(d_sdf_grid=g)
        one = W(res, len(p))
        one.reconstruct(_t(p), _t(n), BBOX, res, with_normals=False)
        b, _, _ = one.backward(d_sdf_grid=g)
        # equal up to the order of the FP64 atomics
        assert float((a - b).norm() / b.norm()) <= 1e-6
        one.close()
    rec.close()


def test_a_captured_solve_leaves_other_grids_their_tables(W):
    """The tables that a replay of one grid's backward writes are not taken for
    those of the grid solved before it."""
    p, n = synth.sphere_cloud(2000, seed=9)
    rec = W(72, len(p))
    P, N = _t(p), _t(n)
    seed = {res: _t(np.random.default_rng(res).standard_normal((res, res, res)).astype(np.float32)) for res in (44, 72)}

    def eager(res):
        rec.reconstruct(P, N, BBOX, res)
        return [x.clone() for x in rec.backward(d_sdf_grid=seed[res])[:2]]

    want = {res: eager(res) for res in (72, 44)}
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got44 = rec.backward(d_sdf_grid=seed[44])[:2]
    eager(72)
    rec.reconstruct(P, N, BBOX, 44)
    graph.replay()
    for a, b in zip(got44, want[44]):
        assert (a - b).norm() <= 1e-5 * b.norm()
    for a, b in zip(eager(72), want[72]):
        assert (a - b).norm() <= 1e-5 * b.norm()
    rec.close()


@pytest.mark.parametrize("res, galerkin, direct", [(320, 0, True), (576, 0, False), (576, 1, True)])
def test_adjoint_of_large_grids_against_the_v_cycles(W, res, galerkin, direct):
    """Direct up to the line where the V-cycles are faster; both ways the
    gradient is that of a handle without spectral solves."""
    p, n = synth.sphere_cloud(20_000, seed=5)
    g = torch.randn((res, res, res), device="cuda", generator=torch.Generator("cuda").manual_seed(res))
    out = []
    for spectral in (1, 0):
        rec = W(res, len(p), galerkin=galerkin, spectral=spectral)
        rec.reconstruct(_t(p), _t(n), BBOX, res, with_normals=False)
        out.append(rec.backward(d_sdf_grid=g)[0])
        steps = rec.info()["backward_steps"]
        assert (steps == 2) == (direct and spectral == 1), steps
        rec.close()
    # the V-cycles stop at 1e-7 of the right-hand side
    assert float((out[0] - out[1]).norm() / out[1].norm()) <= 1e-6
