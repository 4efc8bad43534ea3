"""The cut of the node search's branch-free point-triangle distance: a triangle
within a node's near-tie margin is never beyond the cut of another one, so the
error of that distance, both ways, has to stay within half of the slack that
the cut adds (its constants are read from the kernel's source).  The distance
is restated here operation by operation in float32, products and sums fused
where the compiler fuses them, on the triangles of a marching-cubes cell and on
thin ones, whose face weights are the least certain."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2609_20964_gb300", "csrc", "surface.cu")
F, D = np.float32, np.float64
H = 1.0 / 128


def _constant(name):
    return float(re.search(name + r" = ([0-9.e+-]+)f;", open(SRC).read()).group(1))


def _fma(a, b, c):
    return (a.astype(D) * b.astype(D) + c.astype(D)).astype(F)


def _dot(a, b):
    return _fma(a[2], b[2], _fma(a[1], b[1], a[0] * b[0]))


def _inverse(x):
    return np.where(x > 0, F(1) / np.where(x > 0, x, F(1)), F(0)).astype(F)


def _record(a, b, c):
    ab, ac, bc = b - a, c - a, c - b
    cr = np.stack([_fma(ab[i], ac[j], -(ab[j] * ac[i])) for i, j in ((1, 2), (2, 0), (0, 1))])
    e00, e01, e11 = _dot(ab, ab), _dot(ab, ac), _dot(ac, ac)
    return a, ab, ac, e00, e01, e11, _inverse(e00), _inverse(e11), _inverse(_dot(bc, bc)), _inverse(_dot(cr, cr))


def _fast(p, rec):
    a, ab, ac, e00, e01, e11, i0, i1, ib, idet = rec
    ap = p - a
    s, d1, d2 = _dot(ap, ap), _dot(ab, ap), _dot(ac, ap)
    m1, m2 = F(-2) * d1, F(-2) * d2
    t1, t2 = np.clip(d1 * i0, F(0), F(1)), np.clip(d2 * i1, F(0), F(1))
    q1, q2 = _fma(t1, _fma(t1, e00, m1), s), _fma(t2, _fma(t2, e11, m2), s)
    g = e00 - e01
    db = (d2 - d1) + g
    t3 = np.clip(db * ib, F(0), F(1))
    q3 = _fma(t3, _fma(t3, g + (e11 - e01), F(-2) * db), (s + m1) + e00)
    v, w = _fma(e11, d1, -(e01 * d2)) * idet, _fma(e00, d2, -(e01 * d1)) * idet
    qf = _fma(v, _fma(v, e00, _fma(F(2) * w, e01, m1)), _fma(w, _fma(w, e11, m2), s))
    inside = np.minimum(np.minimum(v, w), F(1) - (v + w)) >= 0
    q = np.minimum(np.minimum(q1, q2), q3)
    return np.maximum(np.where(inside, np.minimum(q, qf), q), F(0)).astype(D)


def _exact(p, rec):
    a, ab, ac = (x.astype(D) for x in rec[:3])
    ap = p.astype(D) - a

    def edge(o, e):
        ee = (e * e).sum(0)
        t = np.clip(np.where(ee > 0, ((ap - o) * e).sum(0) / np.where(ee > 0, ee, 1), 0), 0, 1)
        return ((ap - o - t * e) ** 2).sum(0)

    n = np.cross(ab, ac, axis=0)
    nn = (n * n).sum(0)
    nn1 = np.where(nn > 0, nn, 1)
    v = (np.cross(ap, ac, axis=0) * n).sum(0) / nn1
    w = (np.cross(ab, ap, axis=0) * n).sum(0) / nn1
    best = np.minimum(np.minimum(edge(0 * ab, ab), edge(0 * ab, ac)), edge(ab, ac - ab))
    return np.where((nn > 0) & (v >= 0) & (w >= 0) & (v + w <= 1), (ap * n).sum(0) ** 2 / nn1, best)


def _thin(rng, N):
    u, w = rng.standard_normal((2, 3, N))
    u /= np.linalg.norm(u, axis=0)
    w -= u * (u * w).sum(0)
    w /= np.linalg.norm(w, axis=0)
    length = H * np.sqrt(3) * rng.uniform(0.9, 1, N)
    v = [0 * u, u * length, u * length * rng.uniform(0, 1, N) + w * length * 10 ** rng.uniform(-4, -1, N)]
    return [v[i] for i in rng.permutation(3)]


def _cell(rng, N):
    v = []
    for _ in range(3):   # a vertex on an edge of the cell, half of them close to one of its ends
        c = rng.integers(0, 2, (3, N)).astype(D)
        t = np.where(rng.random(N) < 0.5, rng.random(N), 10 ** rng.uniform(-6, 0, N))
        c[rng.integers(0, 3, N), np.arange(N)] = np.where(rng.random(N) < 0.5, t, 1 - t)
        v.append(c * H)
    return v


@pytest.mark.parametrize("shape", [_thin, _cell])
def test_error_stays_within_half_of_the_cut_slack(shape):
    rel, slack = _constant("kFastRel") - 8e-7, _constant("kFastAbs")
    rng = np.random.default_rng(5)
    N = 200_000
    for _ in range(8):
        off = rng.uniform(0.1, 0.9, (3, N))
        rec = _record(*[(x + off).astype(F) for x in shape(rng, N)])
        a, ab, ac = (x.astype(D) for x in rec[:3])
        bc = rng.dirichlet([2, 2, 2], N).T
        n = np.cross(ab, ac, axis=0)
        n /= np.maximum(np.linalg.norm(n, axis=0), 1e-30)
        n += rng.standard_normal((3, N)) * np.where(rng.random(N) < 0.5, 0, 10 ** rng.uniform(-3, 1, N))
        n /= np.maximum(np.linalg.norm(n, axis=0), 1e-30)
        p = (a + ab * bc[1] + ac * bc[2] + n * H * 10 ** rng.uniform(-1.5, 2, N)).astype(F)
        d2 = _exact(p, rec)
        assert (np.abs(_fast(p, rec) - d2) <= 0.5 * (rel * d2 + slack * H * H)).all()
