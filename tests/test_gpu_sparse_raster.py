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
# per triangle (triangles of more than 16 cells go to the list of large ones); a plate of more than 2^14 cells, whose
# aspects traverse
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
