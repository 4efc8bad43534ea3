"""The node distance search against a brute-force nearest triangle over the
library's own mesh, in FP64: grids whose lattices and blocks end inside a patch
or a block, both sides of the rules that choose the coarsest lattice, nodes
that every triangle is near to (searched one by one), with and without the
near-tie candidates, and a box far from the origin."""
import numpy as np
import pytest

import synth
from oracle import sdf as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def W():
    import __graft_entry__ as g
    g.build()
    from paper_2609_20964_gb300 import Reconstructor
    torch.cuda.set_device(0)
    return Reconstructor


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _check(rec, sdf, res, bbox, lin):
    verts, _ = rec.mesh()
    lo, h = np.asarray(bbox[:3], np.float64), float(max(bbox[3:] - bbox[:3])) / res
    k, j, i = lin // (res * res), lin // res % res, lin % res
    nodes = lo + (np.stack([i, j, k], 1) + 0.5) * h
    d, _ = S.exact_distance(nodes, verts.astype(np.float64))
    got = np.abs(sdf.cpu().numpy().reshape(-1)[lin].astype(np.float64))
    # float32 rounding of a distance and of the coordinates behind it (node and
    # vertices, the latter placed to ~48 bits where gradients are kept)
    coord = float(np.abs(np.asarray(bbox, np.float64)).max())
    assert (np.abs(got - d) <= 4e-7 * d + 3e-7 * coord).all(), np.abs(got - d).max()


@pytest.mark.parametrize("keep", [1, 0])
@pytest.mark.parametrize("res", [4, 5, 7, 9, 16, 18, 30, 36, 52, 80, 88, 160, 176])
def test_search_finds_the_nearest_triangle(W, res, keep):
    bbox = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
    p, n, _ = synth.sh_body_cloud(max(400, 3 * res * res // 2), seed=60 + res)
    rec = W(res, len(p), keep_for_backward=keep)
    sdf, _ = rec.reconstruct(_t(p), _t(n), bbox, res, with_normals=False)
    assert rec.info()["n_triangles"] > 0
    lin = np.arange(res ** 3)
    if len(lin) > 3000:
        lin = np.random.default_rng(res).choice(res ** 3, 3000, replace=False)
    _check(rec, sdf, res, bbox, np.sort(lin))
    rec.close()


@pytest.mark.parametrize("keep", [1, 0])
@pytest.mark.parametrize("res", [24, 64, 96])
def test_search_at_the_centre_of_a_sphere(W, res, keep):
    bbox = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
    p, n = synth.sphere_cloud(4096, seed=2)
    rec = W(res, len(p), keep_for_backward=keep)
    sdf, _ = rec.reconstruct(_t(p), _t(n), bbox, res, with_normals=False)
    c = np.arange(res // 2 - 3, res // 2 + 3)
    lin = ((c[:, None, None] * res + c[None, :, None]) * res + c[None, None, :]).reshape(-1)
    _check(rec, sdf, res, bbox, lin)
    again, _ = rec.reconstruct(_t(p), _t(n), bbox, res, with_normals=False)
    assert torch.equal(sdf, again)   # the candidate lists do not depend on the order of the search
    rec.close()


def test_search_in_a_box_far_from_the_origin(W):
    res = 40
    p, n = synth.sphere_cloud(3000, seed=3)
    off = np.array([64.0, -32.0, 16.0], dtype=np.float32)
    bbox = np.concatenate([off, off + 1]).astype(np.float32)
    rec = W(res, len(p))
    sdf, _ = rec.reconstruct(_t(p + off), _t(n), bbox, res, with_normals=False)
    _check(rec, sdf, res, bbox, np.random.default_rng(0).choice(res ** 3, 3000, replace=False))
    rec.close()


def test_closest_triangles_do_not_depend_on_the_capacities(W):
    """The mesh capacity and the largest grid of a handle only size its
    buffers: near-ties go the same way under any of them."""
    res, bbox = 128, np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
    p, n, _ = synth.sh_body_cloud(60_000, seed=res)
    want = None
    for max_res, cap in ((res, 0), (res, 100 * res * res), (res, 15_000_000), (res, 17_000_000), (2 * res, 0)):
        rec = W(max_res, len(p), mesh_capacity=cap)
        rec.reconstruct(_t(p), _t(n), bbox, res)
        got = [rec.field(name).clone() for name in ("closest", "phi")]
        rec.close()
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(got, want)), (max_res, cap)


@pytest.mark.parametrize("res", [72, 224])
def test_search_beside_the_lines_of_the_coarsest_lattice(W, res):
    test_search_finds_the_nearest_triangle(W, res, 1)


@pytest.mark.parametrize("res", [24, 64, 96])
def test_closest_triangles_at_the_centre_of_a_sphere(W, res):
    """The nodes that are searched one by one keep a triangle that is nearest to
    within float32 rounding, the one that their distance belongs to."""
    bbox = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
    p, n = synth.sphere_cloud(4096, seed=2)
    rec = W(res, len(p))
    sdf, _ = rec.reconstruct(_t(p), _t(n), bbox, res, with_normals=False)
    c = np.arange(res // 2 - 3, res // 2 + 3)
    lin = ((c[:, None, None] * res + c[None, :, None]) * res + c[None, None, :]).reshape(-1)
    verts, _ = rec.mesh()
    tri = verts.astype(np.float64)[rec.field("closest").cpu().numpy().reshape(-1)[lin]]
    k, j, i = lin // (res * res), lin // res % res, lin % res
    nodes = (np.stack([i, j, k], 1) + 0.5) / res
    y, _ = S.closest_point_triangle(nodes, tri[:, 0], tri[:, 1], tri[:, 2])
    own = np.linalg.norm(nodes - y, axis=1)
    nearest, _ = S.exact_distance(nodes, verts.astype(np.float64))
    bound = 4e-7 * nearest + 3e-7      # the distances' of this file
    assert (own - nearest <= bound).all()
    assert (np.abs(np.abs(sdf.cpu().numpy().reshape(-1)[lin]) - own) <= bound).all()
    rec.close()


@pytest.mark.parametrize("keep", [1, 0])
@pytest.mark.parametrize("res", [20, 64, 256])
def test_distances_scale_with_the_units_of_the_box(W, res, keep):
    """A box of 2^k gives 2^k times the distances of the unit box, whatever its
    units: scaling by a power of two is exact, and the search's fourth powers of
    a length do not leave the float range."""
    p, n = synth.sphere_cloud(3000, seed=7)
    q = np.random.default_rng(3).uniform(0, 1, (500, 3)).astype(np.float32)
    rec = W(res, len(p), keep_for_backward=keep)
    want = None
    for k in (0, -20, -24, -30, -40, 40):
        s = np.float32(2.0) ** k
        sdf, nrm = rec.reconstruct(_t(p * s), _t(n), np.array([0, 0, 0, s, s, s], np.float32), res)
        got = [sdf / float(s), nrm, rec.query_exact(_t(q * s), with_grad=False)[0] / float(s)]
        want = want or got
        for a, b in zip(got, want):
            assert bool(torch.isfinite(a).all()) and float((a - b).norm() / b.norm()) <= 1e-6, k
    rec.close()
