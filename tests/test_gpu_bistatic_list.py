"""Bistatic traces whose primary hits are listed and rebuilt by the first bounce
pass against those whose primary rays traverse and are stored, over the
traversals and bounce limits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


@pytest.mark.parametrize("tuning", [dict(), dict(octant=1), dict(bvh_width=4), dict(packet=1)])
@pytest.mark.parametrize("bounces,flags", [(1, 0), (2, 0), (6, 0), (3, 2)])
def test_listed_and_stored_bistatic_states_agree(G, tuning, bounces, flags):
    import sbr_inputs as S

    xyz, tri = S.aircraft(seed=1, target_tris=6000)
    rng = np.random.default_rng(bounces)
    tx = np.stack([rng.uniform(0, 360, 5), rng.uniform(-20, 20, 5)], 1)
    rx = tx + np.stack([rng.uniform(-60, 60, 5), rng.uniform(-10, 10, 5)], 1)
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        for t in (dict(raster=0), dict(raster=1, **tuning)):
            c.set_tuning(**t)
            st = c.trace(tx, 0.05, max_bounces=bounces, offset=(0.37, 0.61), flags=flags | 4, rx=rx)
            E, _ = c.po_integrate([1e9, 2e9], "HH,VV,HV,VH")
            res.append((st, E, [c.get_hits(a) for a in range(5)], [c.get_records(a) for a in range(5)]))
    (s0, E0, h0, r0), (s1, E1, h1, r1) = res
    for k in ("rays_launched", "ray_bounces", "valid_rays", "stack_overflows"):
        assert s0[k] == s1[k], k
    assert np.array_equal(E0, E1)
    for a in range(5):
        for u, v in zip(h0[a], h1[a]):
            assert np.array_equal(u, v)
        for k in ("ray", "coef", "L"):
            assert np.array_equal(r0[a][k], r1[a][k])
