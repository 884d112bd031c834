"""Row spans of the rasterised triangles: boxes of every shape up to the largest
that is not listed, edges along rows and columns, slivers and bands of listed
triangles, against the traversal of all rays."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _triangles(kind, rng, n, w, h):
    """n triangles of box w x h cells (unit cells) in the y-z plane at random depths."""
    o = rng.uniform(0.0, 1.0, (n, 1, 2)) * np.array([200.0, 200.0])
    if kind == "free":
        p = o + rng.uniform(0.0, 1.0, (n, 3, 2)) * np.array([w, h])
    elif kind == "right":  # an edge along a row and one along a column, both ways round
        p = o + np.array([[0.0, 0.0], [w, 0.0], [0.0, h]])
        p[::2] = p[::2, ::-1]
        p[::3, :, 1] = 2 * o[::3, :, 1] - p[::3, :, 1]
    else:  # slivers along the box's diagonal, some of no area
        p = o + np.array([[0.0, 0.0], [w, h], [0.5 * w, 0.5 * h]]) + rng.uniform(-0.02, 0.02, (n, 3, 2)) * (np.arange(n) % 3 > 0)[:, None, None]
    x = rng.uniform(-5.0, 5.0, (n, 1, 1)) + rng.uniform(-0.2, 0.2, (n, 3, 1))
    return np.concatenate([x, p], 2).reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


# boxes of one row or column, of 512 cells and a little more (listed), of 32 rows and one more, bands of a large one
@pytest.mark.parametrize("kind", ["free", "right", "sliver"])
@pytest.mark.parametrize("w,h", [(0.9, 0.9), (3, 2), (200, 0.9), (0.9, 200), (22, 22), (24, 24), (6, 33), (150, 90)])
def test_row_spans_hold_every_hit(G, kind, w, h):
    rng = np.random.default_rng(int(10 * w + h))
    xyz, tri = _triangles(kind, rng, 700, w, h)
    ang = np.array([[0.0, 0.0], [180.0, 0.0], [20.0, 35.0]])
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        res = []
        for raster in (1, 0):
            c.set_tuning(raster=raster)
            st = c.trace(ang, 1.0, eta=0.05, max_bounces=2, offset=(0.37, 0.61), flags=4 | 8)
            res.append((st, [c.get_hits(a) for a in range(3)]))
    (sr, hr), (st, ht) = res
    assert sr["raster_tests"] > 0 and st["raster_tests"] == 0 and sr["rays_launched"] > 3 * 3 * len(tri)
    assert st["valid_rays"] > 0
    for k in ("ray_bounces", "valid_rays"):
        assert sr[k] == st[k], k
    for a in range(3):
        for u, v in zip(hr[a], ht[a]):
            assert np.array_equal(u, v)
