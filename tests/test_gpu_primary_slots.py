"""Queue and record slots of the keyed primary rays: aspects of very few tiles,
aspects that traverse among rasterised ones, and every way on from the primary
pass, against the traversal of all rays."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ESCAPE, HITS, COUNT = 2, 4, 8


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _both(G, xyz, tri, ang, spacing, bounces, flags, rx=None, width=2, chunk=0):
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        for raster in (1, 0):
            c.set_tuning(raster=raster, bvh_width=width)
            st = c.trace(ang, spacing, eta=0.05, max_bounces=bounces, offset=(0.37, 0.61), flags=flags | HITS | COUNT,
                         rx=rx, chunk_rays=chunk)
            E, R = c.po_integrate([1.0e9, 1.1e9], "HH,VV,HV,VH")
            res.append((st, [c.get_hits(a) for a in range(len(ang))], [c.get_records(a) for a in range(len(ang))], E, R))
    (sr, hr, rr, Er, Rr), (st, ht, rt, Et, Rt) = res
    for k in ("rays_launched", "ray_bounces", "valid_rays"):
        assert sr[k] == st[k], k
    for a in range(len(ang)):
        for u, v in zip(hr[a], ht[a]):
            assert np.array_equal(u, v)
        for k in ("ray", "coef", "L"):
            assert np.array_equal(rr[a][k], rt[a][k]), (a, k)
    assert np.array_equal(Er, Et) and np.array_equal(Rr, Rt, equal_nan=True)
    return sr


WAYS = [(1, 0, False, 2), (1, ESCAPE, False, 2), (1, 0, True, 2), (3, 0, False, 2), (3, 0, True, 2), (3, 0, False, 4)]


# grids of 1 to 3 tiles each, so that one step of a warp holds the starts of many aspects: fewer tiles than a warp's
# 32, one more, and more than a block's 256; chunks that end inside a step
@pytest.mark.parametrize("bounces,flags,bistatic,width", WAYS)
@pytest.mark.parametrize("n_asp,chunk", [(1, 0), (33, 0), (300, 0), (300, 1 << 11)])
def test_aspects_of_few_tiles(G, n_asp, chunk, bounces, flags, bistatic, width):
    import sbr_inputs as S

    case = S.trihedral_case()
    rng = np.random.default_rng(n_asp)
    ang = np.stack([rng.uniform(0, 360, n_asp), rng.uniform(-60, 60, n_asp)], 1)
    rx = ang[::-1].copy() if bistatic else None
    ext = float(np.max(case["xyz"].max(0) - case["xyz"].min(0)))
    _both(G, case["xyz"], case["tri"], ang, ext / 5, bounces, flags, rx, width, chunk)


# a trough of 70 m by 1 cm: at 1 mm broadside grids are wider than the 65,535 columns a cell range holds, so those
# aspects traverse; the ones along the trough are rasterised
@pytest.mark.parametrize("bounces,flags,bistatic,width", WAYS)
def test_traversed_aspects_among_rasterised_ones(G, bounces, flags, bistatic, width):
    L, w = 70.0, 0.01
    xyz = np.array([[-L / 2, -w, w], [L / 2, -w, w], [L / 2, 0, 0], [-L / 2, 0, 0], [L / 2, w, w], [-L / 2, w, w]],
                   np.float32)
    tri = np.array([[0, 1, 2], [0, 2, 3], [3, 2, 4], [3, 4, 5]], np.int32)
    ang = np.array([[0.0, 0.01], [90.0, 60.0], [0.0, 0.0], [90.0, 75.0], [180.0, 0.01]])
    rx = ang + np.array([[0.0, 10.0]]) if bistatic else None
    sr = _both(G, xyz, tri, ang, 1e-3, bounces, flags, rx, width)
    assert sr["valid_rays"] > 500_000
    if bounces == 3 and width == 2:
        assert 0 < sr["listed_hits"] < sr["valid_rays"]  # the traversed aspects' hits are not counted as rasterised
