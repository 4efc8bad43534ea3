"""D-PCA where the rows' ranges begin and end inside the groups of 16 sorted
entries, or fill them exactly: neighbour counts equal to the oracle's, and
directions within 0.1 degree.  That bound: float32 sums of at most 100 terms
leave the covariance within 100 * 2^-24 = 6e-6 of itself, which an eigen gap of
1e-2 turns into 6e-4 rad = 0.035 degree."""
import numpy as np
import pytest

from oracle import normals_pca as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BOX = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)


@pytest.mark.parametrize("sizes", [(15,), (16,), (17,), (32, 16), (31, 1, 33), (48, 16, 5), (7, 9, 16, 64)])
def test_partial_and_whole_groups(sizes):
    import __graft_entry__ as g
    g.build()
    from paper_2609_20964_gb300 import Reconstructor
    rng = np.random.default_rng(sum(sizes))
    # flat clusters in neighbouring cells (edge = R) of one row
    P = np.concatenate([np.c_[0.12 + 0.1 * k + rng.uniform(0, 0.06, m), 0.52 + rng.uniform(0, 0.06, m),
                              0.55 + 0.004 * rng.standard_normal(m)] for k, m in enumerate(sizes)])
    P = rng.permutation(P).astype(np.float32)
    R = 0.1
    eps = float(np.float32(1e-3 * R))
    rec = Reconstructor(16, len(P))
    n, c = rec.estimate_normals(torch.from_numpy(P).cuda(), BOX, R, eps, with_counts=True)
    on, olam, oc = D.dpca_normals_brute(P.astype(np.float64), R, eps)
    assert np.array_equal(c.cpu().numpy(), oc)
    gn = n.cpu().numpy().astype(np.float64)
    assert (gn.any(axis=1) == on.any(axis=1)).all()
    ok = on.any(axis=1) & (olam[:, 1] - olam[:, 0] >= 1e-2 * olam[:, 2])
    assert ok.sum() >= len(P) // 2
    ang = np.degrees(np.arccos(np.clip(np.abs(np.sum(gn[ok] * on[ok], axis=1)), 0, 1)))
    assert ang.max() <= 0.1
    rec.close()
