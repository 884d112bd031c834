"""Rasterised primary hits of grids with fewer rays than triangles against the
traversal's, ray by ray."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _with_plate(xyz, tri, side, z):
    """The mesh and a horizontal square plate of two triangles above it."""
    h = side / 2
    p = np.array([[-h, -h, z], [h, -h, z], [h, h, z], [-h, h, z]], np.float32)
    n = len(xyz)
    return np.concatenate([xyz, p]), np.concatenate([tri, np.array([[n, n + 1, n + 2], [n, n + 2, n + 3]], np.int32)])


# triangle counts around a warp's 32 (at 8 rays and more per side of theirs the grid is not sparse); one aspect, a group of 16 and one more, rows of one ray; grids of 1e-4 to 2 rays
# per triangle (triangles of more than 16 cells go to the list of large ones); a plate of more than 2^14 cells, listed
# in bands of rows
@pytest.mark.parametrize("n_tri,n_asp,rays,plate", [(33, 5, 2, 0.0), (64, 17, 3, 0.0), (33, 5, 8, 0.0), (64, 17, 11, 0.0), (20480, 1, 1, 0.0), (20480, 3, 190, 0.0),
                                                    (96_000, 17, 60, 0.0), (96_000, 16, 400, 0.0), (96_000, 4, 300, 40.0)])
def test_sparse_grids_hit_what_the_traversal_hits(G, n_tri, n_asp, rays, plate):
    import sbr_inputs as S

    if n_tri <= 64:
        xyz, tri = S.icosphere(1, 1.0)
        tri = tri[:n_tri]
    elif n_tri == 20480:
        xyz, tri = S.icosphere(5, 1.0)
    else:
        xyz, tri = S.aircraft(seed=1, target_tris=100_000)
    if plate:
        xyz, tri = _with_plate(xyz, tri, plate, 6.0)
    rng = np.random.default_rng(n_tri + n_asp)
    ang = np.stack([rng.uniform(0, 360, n_asp), rng.uniform(60 if plate else -60, 85 if plate else 60, n_asp)], 1)
    ext = float(np.max(xyz.max(0) - xyz.min(0)))
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        res = []
        for raster in (1, 0):
            c.set_tuning(raster=raster)
            st = c.trace(ang, ext / rays, eta=0.05, max_bounces=2, offset=(0.37, 0.61), flags=4 | 8)
            res.append((st, [c.get_hits(a) for a in range(n_asp)], [c.get_records(a) for a in range(n_asp)]))
    (sr, hr, rr), (st, ht, rt) = res
    assert sr["raster_tests"] > 0 and st["raster_tests"] == 0
    assert (sr["node_visits"] > 0) or sr["valid_rays"] == 0
    for k in ("rays_launched", "ray_bounces", "valid_rays"):
        assert sr[k] == st[k], k
    for a in range(n_asp):
        for u, v in zip(hr[a], ht[a]):
            assert np.array_equal(u, v)
        for k in ("ray", "coef", "L"):
            assert np.array_equal(rr[a][k], rt[a][k])


def test_more_large_triangles_than_the_list_holds(G):
    """A stack of 70,000 plates of two triangles under a 20 x 20 grid: 140,000 entries for a list of 65,536, so the
    aspect's rays traverse instead and hit the top one."""
    n = 70_000
    p = np.array([[-0.5, -0.5, 0.0], [0.5, -0.5, 0.0], [0.5, 0.5, 0.0], [-0.5, 0.5, 0.0]], np.float32)
    xyz = np.tile(p, (n, 1))
    xyz[:, 2] = np.repeat(np.arange(n, dtype=np.float32) * np.float32(2.0 ** -13), 4)
    tri = np.tile(np.array([[0, 1, 2], [0, 2, 3]], np.int32), (n, 1)) + np.repeat(np.arange(n, dtype=np.int32) * 4, 2)[:, None]
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        st = c.trace([[0.0, 90.0]], 0.05, eta=0.05, max_bounces=1, offset=(0.37, 0.61), flags=4 | 8)
        hit, _, nb = c.get_hits(0)
    assert st["node_visits"] > 0 and st["valid_rays"] > 300
    assert set(np.unique(hit[nb > 0])) == {2 * n - 2, 2 * n - 1}


@pytest.mark.parametrize("rays,n_tri", [(150, 4), (700, 4), (150, 20480)])
def test_bands_of_large_triangles(G, rays, n_tri):
    """Plates of 1e4 to 4e5 cells (whole bands and remainders, rows shorter and longer than a band) seen from above and
    at grazing incidence, beside nothing or a fine sphere: the traversal's hits."""
    import sbr_inputs as S

    xyz, tri = S.icosphere(5, 0.3) if n_tri > 4 else S.square_plate(0.2, 1)
    xyz, tri = _with_plate(xyz, tri, 1.0, 0.5)
    ang = np.array([[10.0, 80.0], [0.0, 90.0], [200.0, 3.0]])
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        for raster in (1, 0):
            c.set_tuning(raster=raster)
            st = c.trace(ang, 1.0 / rays, eta=0.05, max_bounces=1, offset=(0.37, 0.61), flags=4 | 8)
            res.append((st, [c.get_hits(a) for a in range(3)]))
    assert res[0][0]["node_visits"] == 0 < res[1][0]["node_visits"]
    assert res[0][0]["valid_rays"] == res[1][0]["valid_rays"]
    for h0, h1 in zip(res[0][1], res[1][1]):
        for u, v in zip(h0, h1):
            assert np.array_equal(u, v)
