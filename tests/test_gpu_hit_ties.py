"""Hits on the shared edges of a far wall: two triangles of one plane met at
the same distance, or at distances a rounding apart, in boxes whose entry
distances differ from the hits' by rounding only.  The nearer hit, and of
equal ones the lower input id, must be found whatever order the boxes are
visited in.

The expected hit is made of the same triangle test: the wall's triangles are
loaded in eight classes of triangles that touch no other one of their class,
so that a ray meets at most one of each, and the hits of the classes are
compared by (distance, id)."""
import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu

M = 3.3  # half width of the scene, centred on the origin


def wall(rng, n):
    """n x n quads at z = M between random grid lines, two triangles each, ids
    shuffled; the class of every triangle; the grid lines."""
    x, y = (np.sort(np.concatenate([[-M, M], rng.uniform(-M, M, n - 1)])).astype(np.float32) for _ in range(2))
    verts = np.stack([np.repeat(x, n + 1), np.tile(y, n + 1), np.full((n + 1) ** 2, M, np.float32)], 1)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    v00 = i * (n + 1) + j
    t0, t1 = np.stack([v00, v00 + n + 1, v00 + n + 2], 1), np.stack([v00, v00 + n + 2, v00 + 1], 1)
    cls = (i % 2) * 2 + j % 2
    tris, cls = np.concatenate([t0, t1]).astype(np.uint32), np.concatenate([cls, cls + 4])
    p = rng.permutation(len(tris))
    return verts, tris[p], cls[p], x, y


def load(R, verts, tris, builder):
    box = scenes.tiny_box().scene
    R.load_scene(scenes.Scene(verts, tris, np.zeros(len(tris), np.uint32), box.mat_type[:1].copy(),
                              box.mat_thickness[:1].copy()), builder)


@pytest.mark.parametrize("distance", [1, 100])
@pytest.mark.parametrize("builder", [0, 1, 2])
def test_shared_edges_of_a_far_wall(builder, distance):
    from paper_1912_04000_gb300.renderer import Renderer

    R = Renderer(0)
    rng = np.random.default_rng(7)
    verts, tris, cls, x, y = wall(rng, 64)
    # rays from the other half of the scene, and from far outside it, at points
    # of the grid lines, of lengths that give every rounding of the reciprocals
    m = 1 << 20
    o = rng.uniform(-M * distance, M * distance, (m, 3)).astype(np.float32)
    o[:, 2] = -np.abs(o[:, 2])
    to = rng.uniform(-M, M, (m, 3)).astype(np.float32)
    to[:, 2] = M
    line = rng.random(m) < 0.5
    to[line, 0] = x[rng.integers(1, len(x) - 1, line.sum())]
    to[~line, 1] = y[rng.integers(1, len(y) - 1, (~line).sum())]
    d = ((to - o) * rng.uniform(0.2, 0.4, (m, 1)).astype(np.float32)).astype(np.float32)
    want_t, want_p = np.full(m, np.inf, np.float32), np.full(m, -1)
    hits = np.zeros(m, int)
    for c in range(8):
        ids = np.flatnonzero(cls == c)
        load(R, verts, tris[ids], builder)
        t, p = (a.cpu().numpy() for a in R.trace_closest(o, d))
        p = np.where(p >= 0, ids[p], -1)
        hits += p >= 0
        new = (p >= 0) & ((t < want_t) | ((t == want_t) & (p < want_p)))
        want_t[new], want_p[new] = t[new], p[new]
    load(R, verts, tris, builder)
    t, p = (a.cpu().numpy() for a in R.trace_closest(o, d))
    assert (hits >= 2).mean() > 0.05  # rays that meet two triangles or more
    bad = (t != want_t) | (p != want_p)
    assert not bad.any(), f"{int(bad.sum())} of {int((hits >= 2).sum())} rays on shared edges: another hit"
