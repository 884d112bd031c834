"""Which way rays take that stay between two facing plates for many bounces: handed
over after ten bounces of the tail and followed by a warp each or by a lane each.
How many there are follows from the recorded hits, so that each way is shown to run;
the results are those of the pass-by-pass transport (a stack depth of 128 entries
keeps it)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LOOKS = [2, 3, 4] + [m << s for s in range(1, 6) for m in (3, 4)]  # passes whose rays the tail may take
HAND_AFTER, HAND_BOUNCES, PER_WARP = 10, 16, 2


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _corridor(length=40.0, half=1.0, n=24):
    """Two facing plates 1 m apart: rays that enter at 45 degrees are reflected once a metre."""
    x, y = np.meshgrid(np.linspace(0, length, n + 1), np.linspace(-half, half, 5), indexing="ij")
    i, j = np.meshgrid(np.arange(n), np.arange(4), indexing="ij")
    a = (i * 5 + j).ravel()
    t = np.concatenate([np.stack([a, a + 5, a + 6], 1), np.stack([a, a + 6, a + 1], 1)])
    v = np.stack([x, y, np.full_like(x, 0.5)], -1).reshape(-1, 3)
    return (np.concatenate([v, v * [1, 1, -1]]).astype(np.float32),
            np.concatenate([t, t + len(v)]).astype(np.int32))


@pytest.mark.parametrize("way,ds,kw", [("warp", 0.05, {}), ("lane", 0.008, {}), ("lane", 0.008, dict(flags=2)),
                                       ("warp", 0.05, dict(flags=2)), ("warp", 0.03, dict(rx=1)),
                                       ("lane", 0.008, dict(rx=1)), ("passes", 0.0025, {})])
def test_trapped_rays_take_the_way_their_number_asks_for(G, way, ds, kw):
    torch = pytest.importorskip("torch")
    bounces = 30
    ang = np.array([[180.0, 45.0]])
    kw = dict(kw)
    rx = ang + [0.0, 20.0] if kw.pop("rx", None) else None
    flags = kw.pop("flags", 0)
    xyz, tri = _corridor()
    res = []
    with G.Context(0) as c:
        blocks = torch.cuda.get_device_properties(0).multi_processor_count * c.tuning()["blocks_per_sm"]
        c.load_mesh(xyz, tri)
        for depth in (64, 128):
            c.set_tuning(stack_depth=depth)
            st = c.trace(ang, ds, eta=0.02, max_bounces=bounces, offset=(0.37, 0.61), flags=flags | 4, rx=rx)
            E, _ = c.po_integrate([1e9], "HH,VV,HV,VH")
            res.append((st, E, c.get_hits(0), c.get_records(0)))
    (s0, E0, h0, r0), (s1, E1, h1, r1) = res
    nb = h0[2]
    look = next((b for b in LOOKS if 0 < np.sum(nb >= b) <= 256 * blocks), None)
    handed = int(np.sum(nb >= look + HAND_AFTER)) if look and bounces - look >= HAND_BOUNCES else 0
    per_warp = handed / (8 * (blocks + 1 & ~1))
    assert way == ("passes" if handed == 0 else "lane" if per_warp > PER_WARP else "warp"), (look, handed, per_warp)
    for k in ("rays_launched", "ray_bounces", "valid_rays", "stack_overflows"):
        assert s0[k] == s1[k], k
    assert np.array_equal(E0, E1)
    for u, v in zip(h0, h1):
        assert np.array_equal(u, v)
    for k in ("ray", "coef", "L"):
        assert np.array_equal(r0[k], r1[k])
