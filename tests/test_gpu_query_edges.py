"""Interpolated queries whose cells touch the grid's edges (one-sided stencils,
clamped positions), counts that end inside a warp's eight queries, and
non-finite positions, against the oracle's interpolation of the library's own
grid in FP64."""
import numpy as np
import pytest

import synth
from oracle import iso as I
from oracle import normals as NR

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BBOX = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)


@pytest.mark.parametrize("res,m", [(4, 1), (5, 7), (18, 8), (24, 9), (40, 1001)])
def test_query_normals_at_the_edges(res, m):
    import __graft_entry__ as g
    g.build()
    from paper_2609_20964_gb300 import Reconstructor
    p, n = synth.sphere_cloud(1500, seed=res)
    rec = Reconstructor(res, len(p))
    sdf, _ = rec.reconstruct(torch.from_numpy(p).cuda(), torch.from_numpy(n).cuda(), BBOX, res)
    rng = np.random.default_rng(m)
    q = rng.uniform(-0.1, 1.1, (m, 3)).astype(np.float32)     # a sixth of each axis is clamped
    q[: m // 2] = np.round(q[: m // 2] * 4) / 4               # faces and corners of the box
    phi = sdf.cpu().numpy().astype(np.float64)
    h = 1.0 / res
    unit, _, _ = NR.normals(phi, h)
    want = I.interpolate(phi, q.astype(np.float64), np.zeros(3), h, res)
    mv = I.interpolate(np.moveaxis(unit, 0, -1), q.astype(np.float64), np.zeros(3), h, res)
    mag = np.linalg.norm(mv, axis=1)
    got, nrm = rec.query(torch.from_numpy(q).cuda())
    alone, _ = rec.query(torch.from_numpy(q).cuda(), with_normals=False)
    # float32 weights and sums of eight values below 1: 8 * 2^-24 each
    assert np.abs(got.cpu().numpy() - want).max() <= 1e-6
    assert np.abs(alone.cpu().numpy() - want).max() <= 1e-6
    # unit corner normals from differences of float32 phi over 2 h (relative
    # 2^-23 / h), in a mean of length mag
    err = np.linalg.norm(nrm.cpu().numpy() * mag[:, None] - mv, axis=1)
    gmag = np.linalg.norm(NR.gradient(phi, h), axis=0).min()
    assert err.max() <= 1e-6 + 4 * 2.0 ** -23 * res / max(gmag, 1e-3)
    bad = q.copy()
    bad[0] = np.nan
    got2, _ = rec.query(torch.from_numpy(bad).cuda())
    assert np.isnan(got2[0].item())
    if m > 1:
        assert torch.equal(got2[1:], got[1:])
    rec.close()


@pytest.mark.parametrize("res,m", [(4, 33), (24, 1000), (64, 100_003)])
def test_query_normals_do_not_depend_on_the_order_of_the_queries(res, m):
    """Warps whose queries share cache lines take one thread a query, the others
    four lanes: the same bits either way."""
    import __graft_entry__ as g
    g.build()
    from paper_2609_20964_gb300 import Reconstructor
    p, n = synth.sphere_cloud(1500, seed=res)
    rec = Reconstructor(res, len(p))
    rec.reconstruct(torch.from_numpy(p).cuda(), torch.from_numpy(n).cuda(), BBOX, res)
    rng = np.random.default_rng(m)
    q = rng.uniform(-0.1, 1.1, (m, 3)).astype(np.float32)
    cell = (q * res).astype(int)
    rows = np.lexsort((q[:, 0], cell[:, 1], cell[:, 2]))
    sdf, nrm = rec.query(torch.from_numpy(q).cuda())
    sdf2, nrm2 = rec.query(torch.from_numpy(q[rows]).cuda())
    at = torch.from_numpy(rows).cuda()
    assert torch.equal(sdf[at], sdf2) and torch.equal(nrm[at], nrm2)
    rec.close()


def test_queries_on_a_lattice_take_less_time_than_scattered_ones():
    """2^22 queries in the order of a lattice share their cache lines; four lanes
    a query there took nearly as long (0.92 of the time) as scattered ones."""
    import __graft_entry__ as g
    g.build()
    from paper_2609_20964_gb300 import Reconstructor
    p, n = synth.sphere_cloud(20_000, seed=1)
    rec = Reconstructor(128, len(p))
    rec.reconstruct(torch.from_numpy(p).cuda(), torch.from_numpy(n).cuda(), BBOX, 128)
    k = (torch.arange(161, device="cuda") + 0.37) / 161
    lattice = torch.stack(torch.meshgrid(k, k, k, indexing="ij")[::-1], -1).reshape(-1, 3).contiguous()
    scattered = lattice[torch.randperm(len(lattice), device="cuda")].contiguous()

    def time(q):
        ms = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rec.query(q)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return sorted(ms[3:])[4]

    assert time(lattice) <= 0.75 * time(scattered)
    rec.close()
