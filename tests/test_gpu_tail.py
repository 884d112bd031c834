"""Bounce passes with few rays, which one launch follows to their end, against
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


# few rays from the start (20 cm grid) and more than one per thread until a late pass (1 cm); one chunk and pooled
# chunks; B = 2 (no pass after the first), 3 (one) and many; the escape rule; the octant copies; bistatic
@pytest.mark.parametrize("spacing,bounces,kw", [(0.2, 2, {}), (0.2, 3, {}), (0.2, 60, {}), (0.05, 20, dict(flags=2)),
                                                (0.01, 12, {}), (0.05, 12, dict(chunk_rays=1 << 17)),
                                                (0.05, 12, dict(octant=1)), (0.1, 9, dict(rx=1))])
def test_tail_equals_pass_by_pass(G, spacing, bounces, kw):
    import sbr_inputs as S

    xyz, tri = S.aircraft(seed=1, target_tris=20_000)
    ang = np.array([[180.0, 0.0], [175.0, 3.0], [40.0, -5.0]])
    kw = dict(kw)
    rx = ang + [20.0, 5.0] if kw.pop("rx", None) else None
    octant, flags = kw.pop("octant", 0), kw.pop("flags", 0)
    res = []
    with G.Context(0) as c:
        c.load_mesh(xyz, tri)
        for depth in (64, 128):
            c.set_tuning(stack_depth=depth, octant=octant)
            st = c.trace(ang, spacing, max_bounces=bounces, offset=(0.37, 0.61), flags=flags | 4, rx=rx, **kw)
            E, _ = c.po_integrate([1e9], "HH,VV,HV,VH")
            res.append((st, E, [c.get_hits(a) for a in range(3)], [c.get_records(a) for a in range(3)]))
    (s0, E0, h0, r0), (s1, E1, h1, r1) = res
    assert (s0["kernel_launches"] > s1["kernel_launches"]) == (bounces > 2 or flags != 0)
    for k in ("rays_launched", "ray_bounces", "valid_rays", "stack_overflows"):
        assert s0[k] == s1[k], k
    assert np.array_equal(E0, E1)
    for a in range(3):
        for u, v in zip(h0[a], h1[a]):
            assert np.array_equal(u, v)
        for k in ("ray", "coef", "L"):
            assert np.array_equal(r0[a][k], r1[a][k])
