"""Rays that stay trapped for many bounces, followed by half a warp each, against
the pass-by-pass transport (a stack depth of 128 entries keeps it)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


# fewer rays than half warps and more; one bounce under and at the line where they are handed over (16 after pass 2);
# pooled chunks, the octant copies, bistatic; leaves of 1 and of 16 triangles, a deep tree
@pytest.mark.parametrize("spacing,bounces,kw", [(0.1, 17, {}), (0.1, 18, {}), (0.02, 70, {}), (0.05, 70, dict(flags=2)),
                                                (0.05, 40, dict(chunk_rays=1 << 17)), (0.05, 40, dict(octant=1)),
                                                (0.1, 40, dict(rx=1)), (0.05, 40, dict(leaf_max=1)),
                                                (0.05, 40, dict(leaf_max=16)), (0.05, 40, dict(builder="lbvh"))])
def test_trapped_rays_equal_pass_by_pass(G, spacing, bounces, kw):
    import sbr_inputs as S

    xyz, tri = S.aircraft(seed=1, target_tris=20_000)
    ang = np.array([[180.0, 0.0], [175.0, 3.0], [184.0, -2.0]])
    kw = dict(kw)
    rx = ang + [20.0, 5.0] if kw.pop("rx", None) else None
    octant, flags = kw.pop("octant", 0), kw.pop("flags", 0)
    tree = {k: kw.pop(k) for k in ("leaf_max", "builder") if k in kw}
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        if tree:
            c.build_bvh(**tree)
        for depth in (64, 128):
            c.set_tuning(stack_depth=depth, octant=octant)
            st = c.trace(ang, spacing, max_bounces=bounces, offset=(0.37, 0.61), flags=flags | 4, rx=rx, **kw)
            E, _ = c.po_integrate([1e9], "HH,VV,HV,VH")
            res.append((st, E, [c.get_hits(a) for a in range(3)], [c.get_records(a) for a in range(3)]))
    (s0, E0, h0, r0), (s1, E1, h1, r1) = res
    assert max(int(h[2].max()) for h in h0) > 8  # some rays go on after they have been handed over
    for k in ("rays_launched", "ray_bounces", "valid_rays", "stack_overflows"):
        assert s0[k] == s1[k], k
    assert np.array_equal(E0, E1)
    for a in range(3):
        for u, v in zip(h0[a], h1[a]):
            assert np.array_equal(u, v)
        for k in ("ray", "coef", "L"):
            assert np.array_equal(r0[a][k], r1[a][k])


def test_more_trapped_rays_than_warps_take(G):
    """5 mm grids into the inlets: more trapped rays than two per warp (9,728), which a lane each follows."""
    import sbr_inputs as S

    xyz, tri = S.aircraft(seed=1, target_tris=20_000)
    ang = np.array([[180.0, 0.0], [178.0, 0.0], [182.0, 0.0], [180.0, 2.0]])
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        for depth in (64, 128):
            c.set_tuning(stack_depth=depth)
            st = c.trace(ang, 0.005, max_bounces=40)
            E, _ = c.po_integrate([1e9], "HH,VV")
            res.append((st, E, c.get_records(0)))
    (s0, E0, r0), (s1, E1, r1) = res
    for k in ("rays_launched", "ray_bounces", "valid_rays", "stack_overflows"):
        assert s0[k] == s1[k], k
    assert np.array_equal(E0, E1)
    for k in ("ray", "coef", "L"):
        assert np.array_equal(r0[k], r1[k])
