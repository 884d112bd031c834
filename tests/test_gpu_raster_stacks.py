"""Stacks of triangles under a grid: rasterised where they are few layers deep,
traversed where they are many, with the traversal's hits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _stack(n, side=1.0, gap=0.002, seed=0):
    """n square plates of two triangles above one another, in no order."""
    h = side / 2
    p = np.array([[-h, -h, 0.0], [h, -h, 0.0], [h, h, 0.0], [-h, h, 0.0]], np.float32)
    xyz = np.tile(p, (n, 1))
    xyz[:, 2] = np.repeat(np.random.default_rng(seed).permutation(n).astype(np.float32) * np.float32(gap), 4)
    tri = np.tile(np.array([[0, 1, 2], [0, 2, 3]], np.int32), (n, 1)) + np.repeat(np.arange(n, dtype=np.int32) * 4, 2)[:, None]
    return xyz, tri


def _both(G, xyz, tri, ang, ds, **kw):
    """Trace statistics and hits, rasterised and traversed."""
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        for raster in (1, 0):
            c.set_tuning(raster=raster)
            st = c.trace(ang, ds, eta=0.05, max_bounces=1, offset=(0.37, 0.61), flags=4 | 8, **kw)
            res.append((st, [c.get_hits(a) for a in range(len(ang))]))
    (sr, hr), (st, ht) = res
    assert sr["valid_rays"] == st["valid_rays"] > 0
    for a in range(len(ang)):
        for u, v in zip(hr[a], ht[a]):
            assert np.array_equal(u, v)
    return sr, st


# two triangles of about 0.9 to 2 box cells per ray each: 4 plates stay under 20 box cells per ray, 40 do not; a grid
# whose triangles are below 2^14 cells is rasterised however deep; both kinds of aspect in one chunk, and chunks apart
@pytest.mark.parametrize("n,rays,ang,traversed", [(4, 300, [[0, 90], [20, 80]], False), (40, 300, [[0, 90], [20, 80]], True),
                                                  (40, 110, [[0, 90], [20, 80]], False),
                                                  (40, 300, [[10, 0.5], [20, 80], [30, 5]], True)])
def test_stacks_of_large_triangles(G, n, rays, ang, traversed):
    xyz, tri = _stack(n)
    sr, _ = _both(G, xyz, tri, np.array(ang, float), 1.0 / rays)
    assert (sr["node_visits"] > 0) == traversed


def _join(*meshes):
    off = np.cumsum([0] + [len(x) for x, _ in meshes])
    return np.concatenate([x for x, _ in meshes]), np.concatenate([t + o for (_, t), o in zip(meshes, off)]).astype(np.int32)


# 140,000 triangles of 81 to 100 box cells, more than the list of large ones has room for (65,536 entries), which do
# not go there; beside them a plate of 400 cells, which does; boxes of 16 to 25 cells and of 225 to 289, on both sides
# of the two limits (16 and 256); more of some 300 cells than the list holds, whose aspects traverse
@pytest.mark.parametrize("n,rays,side,plate,traversed", [(70_000, 9, 1.0, 0, False), (70_000, 20, 0.45, 1, False),
                                                         (20_000, 4, 1.0, 0, False), (3000, 11, 1.0, 0, False),
                                                         (3000, 15, 1.0, 0, False), (40_000, 17, 1.0, 0, True)])
def test_stacks_under_sparse_grids(G, n, rays, side, plate, traversed):
    mesh = _stack(n, side, gap=2.0 ** -13)
    if plate:
        x, t = _stack(1, 1.0)
        mesh = _join(mesh, (x + np.array([0, 0, 9.0], np.float32), t), (x - np.array([0, 0, 1.0], np.float32), t))
    sr, _ = _both(G, *mesh, np.array([[0.0, 90.0], [3.0, 88.0], [90.0, 90.0]]), 1.0 / rays)
    assert (sr["node_visits"] > 0) == traversed
