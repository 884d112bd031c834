"""The tree of meshes above the one-block build: sizes around its limit and the
tiles of the clustering, search radii from 1 to 64, refused meshes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _mesh(n):
    import sbr_inputs as S

    xyz, tri = S.aircraft(seed=1, target_tris=60_000)
    assert len(tri) >= n
    return xyz, np.ascontiguousarray(tri[np.random.default_rng(n).permutation(len(tri))[:n]])


@pytest.mark.parametrize("n,radius", [(16384, 16), (16385, 1), (16385, 16), (16896, 64), (16897, 5), (50_001, 16)])
def test_clustered_tree_hits_what_the_karras_tree_hits(G, n, radius):
    xyz, tri = _mesh(n)
    ang = [[170.0, 4.0], [60.0, -30.0]]
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        c.set_tuning(raster=0)
        for builder, width in (("ploc", 2), ("ploc", 4), ("lbvh", 2)):
            c.build_bvh(builder=builder, ploc_radius=radius)
            info = c.bvh_info()
            assert info["n_tri"] == n and 0 < info["n_nodes4"] <= info["n_nodes"] < n
            c.set_tuning(bvh_width=width)
            st = c.trace(ang, 0.05, max_bounces=4, offset=(0.37, 0.61), flags=4 | 8)
            res.append((info, st, [c.get_hits(a) for a in range(2)]))
            c.set_tuning(bvh_width=2)
    assert res[0][0] == res[1][0]
    for _, st, hits in res[1:]:
        assert st["ray_bounces"] == res[0][1]["ray_bounces"] and st["stack_overflows"] == 0
        for h0, h1 in zip(res[0][2], hits):
            for u, v in zip(h0, h1):
                assert np.array_equal(u, v)


def test_refused_meshes_leave_the_context_usable(G):
    """A bad index, a non-finite vertex, and 70,000 coincident copies of a triangle that the clustering's ties keep
    from pairing up within its rounds: refused, and the next mesh loads and traces."""
    xyz, tri = _mesh(20_000)
    bad_tri, bad_xyz = tri.copy(), xyz.copy()
    bad_tri[12_345, 1] = len(xyz)
    bad_xyz[777, 2] = np.inf
    one = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0]], np.float32)
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        ref = c.trace([[170.0, 4.0]], 0.05, max_bounces=3)
        for x, t, code in ((xyz, bad_tri, -1), (bad_xyz, tri, -1), (one, np.tile([[0, 1, 2]], (140_000, 1)).astype(np.int32), -2)):
            with pytest.raises(G.SbrError) as e:
                c.load_mesh(x, t)
            assert e.value.code == code
            with pytest.raises(G.SbrError):
                c.trace([[170.0, 4.0]], 0.05, max_bounces=3)
            c.load_mesh(xyz, tri)
            st = c.trace([[170.0, 4.0]], 0.05, max_bounces=3)
            assert st["ray_bounces"] == ref["ray_bounces"] and st["valid_rays"] == ref["valid_rays"]


@pytest.mark.parametrize("ties", [True, False])
def test_clustering_that_ends_in_its_last_rounds_says_so(G, ties):
    """66,000 coincident triangles pair up once a round, so the limit of 65,536 rounds falls into the last ones, which
    one block runs while the others wait for it; 100 groups further apart than FP32 box areas reach stop pairing up
    there. Both are reported as the clustering's failure, not as a wait that gave up, and the next mesh loads."""
    if ties:
        x = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0]], np.float32)
        t = np.tile([[0, 1, 2]], (66_000, 1)).astype(np.int32)
    else:
        rng = np.random.default_rng(3)
        at = np.repeat(np.arange(100) * 3e20, 200)[:, None, None] + rng.uniform(0, 1e17, (20_000, 1, 3))
        x = (at + rng.uniform(0, 2e16, (20_000, 3, 3))).astype(np.float32).reshape(-1, 3)
        t = np.arange(60_000, dtype=np.int32).reshape(-1, 3)
    xyz, tri = _mesh(20_000)
    with G.Context(0) as c:
        with pytest.raises(G.SbrError) as e:
            c.load_mesh(x, t)
        assert e.value.code == -2 and "did not converge" in str(e.value)
        c.load_mesh(xyz, tri)
        assert c.trace([[170.0, 4.0]], 0.05, max_bounces=3)["valid_rays"] > 0
