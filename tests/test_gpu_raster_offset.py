"""Rasterised primary hits of targets far from the coordinate origin, where the
roundings of the coordinates are a good part of a grid cell: the traversal's hits,
with rows of cells, single cells, bands of a large triangle and the silhouette mask."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


# an ellipsoid of 10 x 2 x 0.4 m and a plate behind it; grids of 8 mm and 0.2 m (with fewer rays than triangles); at
# 10 km the coordinates are 1 mm apart
@pytest.mark.parametrize("at", [(7106.0, 6220.5, -4771.0), (1484.5, 390.9, -9872.1), (0.0, 0.0, 30000.0), (150.0, -80.0, 3.0)])
@pytest.mark.parametrize("ds,sub", [(0.00822, 4), (0.2, 6)])
def test_far_targets_hit_what_the_traversal_hits(G, at, ds, sub):
    import sbr_inputs as S

    xyz, tri = S.icosphere(sub, 1.0)
    p = np.array([[-3, -3, -4], [3, -3, -4], [3, 3, -4], [-3, 3, -4]], np.float64)
    x = np.concatenate([xyz * [5, 1, 0.2], p]) + at
    n = len(xyz)
    t = np.concatenate([tri, [[n, n + 1, n + 2], [n, n + 2, n + 3]]]).astype(np.int32)
    ang = np.array([[5.7, 0.0], [87.75, 0.0], [40.0, 70.0]])
    res = []
    with G.Context(0) as c:
        c.load_mesh(x.astype(np.float32), t)
        for tune in (dict(raster=1), dict(raster=0, silhouette=1), dict(raster=0, silhouette=0)):
            c.set_tuning(**tune)
            st = c.trace(ang, ds, eta=0.3, max_bounces=1, offset=(-0.4275, -0.0015), flags=4)
            res.append((st["valid_rays"], [c.get_hits(a) for a in range(3)]))
    assert res[2][0] > 0
    for got in res[:2]:
        assert got[0] == res[2][0]
        for a in range(3):
            for u, v in zip(got[1][a], res[2][1][a]):
                assert np.array_equal(u, v)
