"""The work that users of this framework have it do, as cases that can be timed one by one.

A case is a dict of plain values. ``prepare`` makes what a program holds before the call (a context
with its mesh loaded, the aspect angles, requests, training samples), ``run`` makes one pass through
the public entry points and returns its results whole, ``work`` counts what the pass cannot do
without, and ``exact`` gives the same results in 64 bits from plain torch where that is practical.
Angles, grid offsets, samples and requests come from the seed; the meshes are those of ``sbr_inputs``.

Every context runs with the default tuning, and every size is one of the repository's own
configurations (icosphere, triangular trihedral, procedural aircraft, batched requests, surrogate)
or lies between them.
"""
import functools
import math

import numpy as np
import torch

import paper_2604_09243_gb300 as G
import sbr_inputs as S

C0 = 299_792_458.0
ETA = 0.05  # aperture margin of the traces


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # one look at a canonical target: the smallest call, where launches and host waits count
        dict(name="sphere_one_aspect", kind="trace", mesh="sphere", size=5, ghz=3.0, aspects=1, bounces=1, freqs=1,
             pols="HH,VV", form="scalar", phase="compensated", escape=False, bistatic=False),
        # a calibration target swept in azimuth: small mesh, coherent triple bounces, many aspects in one call
        dict(name="trihedral_sweep", kind="trace", mesh="trihedral", size=32, ghz=10.0, aspects=181, bounces=3, freqs=1,
             pols="HH,VV", form="vector", phase="compensated", escape=False, bistatic=False),
        # a range profile: a few aspects over a wide band in all four polarisations, where the PO sum carries the time
        dict(name="trihedral_wideband", kind="trace", mesh="trihedral", size=32, ghz=12.0, aspects=9, bounces=3,
             freqs=201, pols="HH,VV,HV,VH", form="vector", phase="compensated", escape=False, bistatic=False),
        # a full azimuth cut of a large mesh at a low frequency: few rays per triangle
        dict(name="aircraft_1ghz_cut", kind="trace", mesh="aircraft", size=1_000_000, ghz=1.0, aspects=360, bounces=10,
             freqs=1, pols="HH,VV", form="vector", phase="compensated", escape=False, bistatic=False),
        # the headline workload, thinned in azimuth: many rays per triangle, several chunks
        dict(name="aircraft_10ghz_sweep", kind="trace", mesh="aircraft", size=1_000_000, ghz=10.0, aspects=37,
             bounces=10, freqs=1, pols="HH,VV", form="vector", phase="compensated", escape=False, bistatic=False),
        # engine inlets with the escape rule: a long tail of bounces over few rays
        dict(name="aircraft_deep_cavity", kind="trace", mesh="aircraft", size=1_000_000, ghz=3.0, aspects=45,
             bounces=100, freqs=1, pols="HH,VV", form="vector", phase="compensated", escape=True, bistatic=False),
        # transmitter and receiver apart: a visibility query for every ray's last hit
        dict(name="aircraft_bistatic", kind="trace", mesh="aircraft", size=250_000, ghz=3.0, aspects=33, bounces=6,
             freqs=3, pols="HH,VV,HV,VH", form="vector", phase="compensated", escape=False, bistatic=True),
        # mixed requests of uneven ray counts, each with its own list of 1 to 64 frequencies
        dict(name="batch_aircraft", kind="batch", mesh="aircraft", size=1_000_000, requests=23, bounces=10,
             graph=False),
        # the same form on a small target, submitted asynchronously to device outputs
        dict(name="batch_submitted", kind="batch", mesh="trihedral", size=32, requests=61, bounces=3, graph=True),
        # a new geometry and the first look at it: upload, tree build, one aspect
        dict(name="new_aircraft_mesh", kind="mesh", size=1_000_000, ghz=1.0, bounces=10),
        # an epoch of ensemble training: forward, backward and Adam
        dict(name="surrogate_epoch", kind="train", n=50_000, batch=8192, epochs=1, members=4, width=512, depth=6,
             fourier=256),
        # dense sweep answered by the ensemble
        dict(name="surrogate_lattice", kind="predict", n=300_000, members=4, width=512, depth=6, fourier=256),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["sphere", "trihedral", "trihedral", "aircraft", "aircraft", "aircraft", "batch", "submitted",
                       "mesh", "train", "predict"])
    if kind in ("sphere", "trihedral", "aircraft"):
        c = dict(kind="trace", mesh=kind)
        c["bistatic"] = rng.random() < 0.2
        if kind == "sphere":
            c.update(size=rng.randint(2, 5), ghz=round(_log(rng, 0.5, 6.0), 3), bounces=1)
            c["aspects"] = int(_log(rng, 1, 130))
        elif kind == "trihedral":
            c.update(size=int(_log(rng, 4, 90)), ghz=round(_log(rng, 3.0, 12.0), 3), bounces=rng.randint(2, 4))
            c["aspects"] = int(_log(rng, 1, 182))
        else:
            c.update(size=int(_log(rng, 20_000, 1_000_000)), ghz=round(_log(rng, 1.0, 10.0), 3),
                     bounces=int(_log(rng, 2, 100)))
            most = min(360.0, 37 * (10.0 / c["ghz"]) ** 2)
            c["aspects"] = int(_log(rng, 1, most))
        c["phase"] = "fp64" if kind != "aircraft" and rng.random() < 0.2 else "compensated"
        # a band over every aspect of a long sweep would cost more than any listed case: fewer frequencies then
        most = 4 if kind == "aircraft" else min(202, max(2, 1809 // (c["aspects"] * (8 if c["phase"] == "fp64" else 1))))
        c["freqs"] = int(_log(rng, 1, most)) if rng.random() < 0.5 else 1
        c["pols"] = rng.choice(["HH,VV", "HH,VV", "VV", "HH,VV,HV,VH"])
        c["form"] = "scalar" if kind == "sphere" and not c["bistatic"] and rng.random() < 0.5 else "vector"
        c["escape"] = kind == "aircraft" and rng.random() < 0.3
        return c
    if kind in ("batch", "submitted"):
        mesh = rng.choice(["sphere", "trihedral", "aircraft"])
        size = 5 if mesh == "sphere" else (32 if mesh == "trihedral" else int(_log(rng, 100_000, 1_000_000)))
        return dict(kind="batch", mesh=mesh, size=size, requests=int(_log(rng, 1, 24 if mesh == "aircraft" else 90)),
                    bounces={"sphere": 1, "trihedral": 3, "aircraft": 10}[mesh], graph=kind == "submitted")
    if kind == "mesh":
        return dict(kind="mesh", size=int(_log(rng, 2_000, 1_000_000)), ghz=round(rng.uniform(0.5, 2.0), 3),
                    bounces=rng.randint(2, 10))
    net = dict(members=rng.randint(1, 4), width=128 * rng.randint(1, 4), depth=rng.randint(2, 6),
               fourier=128 * rng.randint(1, 2))
    if kind == "train":
        batch = 128 * int(_log(rng, 2, 65))
        return dict(kind="train", n=batch * rng.randint(1, 6) + rng.randint(0, 127), batch=batch, epochs=1, **net)
    return dict(kind="predict", n=int(_log(rng, 1_000, 300_000)), **net)


# --------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=8)
def _mesh(kind, size):
    if kind == "sphere":
        return S.icosphere(size, 1.0)
    if kind == "trihedral":
        return S.trihedral(1.0, size)
    return S.aircraft(seed=1, target_tris=size)


@functools.lru_cache(maxsize=8)
def _aircraft_smooth(size):
    """The aircraft before any jitter, for cases that bring a new geometry each time."""
    return S.aircraft(seed=1, target_tris=size, jitter_sigma=0.0)


def _aspects(case, rng):
    """Aspect angles [n, 2] (az, el) and, for a bistatic case, the receivers' [n, 2]."""
    n = case["aspects"]
    if case["mesh"] == "sphere":
        ang = np.stack([rng.uniform(0, 360, n), np.degrees(np.arcsin(rng.uniform(-1, 1, n)))], 1)
    elif case["mesh"] == "trihedral":
        step = 90.0 / n
        ang = np.stack([step * (np.arange(n) + rng.uniform()), np.full(n, 35.26 + rng.uniform(-2, 2))], 1)
    elif case.get("escape"):
        # the inlets' mouths face -x: aspects around the nose
        step = 60.0 / n
        ang = np.stack([150.0 + step * (np.arange(n) + rng.uniform()), np.full(n, rng.uniform(-3, 3))], 1)
    else:
        step = 360.0 / n
        ang = np.stack([(step * (np.arange(n) + rng.uniform())) % 360.0, np.full(n, rng.uniform(-3, 3))], 1)
    rx = None
    if case.get("bistatic"):
        rx = ang + np.stack([rng.uniform(5, 60, n), rng.uniform(-10, 10, n)], 1)
    return ang, rx


def _freqs(case, rng):
    """One frequency, or an evenly stepped band whose top is the case's frequency (a third of it wide)."""
    top = case["ghz"] * 1e9
    n = case["freqs"]
    return np.array([top]) if n == 1 else np.linspace(top * (2.0 / 3.0), top, n)


def _requests(case, rng):
    """Aspect requests as a mixed queue has them: random aspect, 5 to 10 rays per wavelength of the highest
    frequency, 1 to 64 frequencies between 1 and 12 GHz."""
    out = []
    counts = np.random.default_rng(case["requests"]).integers(1, 65, case["requests"])  # the queue's shape
    for nf in counts:
        f = np.sort(rng.uniform(1e9, 12e9, int(nf)))
        d = float(rng.uniform(5.0, 10.0))
        out.append(dict(az=float(rng.uniform(0, 360)), el=float(rng.uniform(-30, 30)), freqs=f,
                        spacing=C0 / (float(f[-1]) * d)))
    return out


def _field_samples(n, rng):
    """(az, el, f) points of a nose-on sweep patch and the complex field of a few scattering centres there, the
    shape of the data that a trace gives the surrogate."""
    az = rng.uniform(178.0, 182.0, n)
    el = rng.uniform(-1.0, 1.0, n)
    f = rng.uniform(1.0e9, 1.2e9, n)
    a, e = np.radians(az), np.radians(el)
    r = np.stack([np.cos(e) * np.cos(a), np.cos(e) * np.sin(a), np.sin(e)], 1)
    pos = rng.uniform(-1.0, 1.0, (12, 3)) * np.array([7.0, 3.0, 1.0])
    ph = (2.0 * 2.0 * np.pi / C0) * f[:, None] * (r @ pos.T)
    w = rng.normal(size=(2, 12, 2))
    hh = np.exp(1j * ph) @ (w[0, :, 0] + 1j * w[0, :, 1])
    vv = np.exp(1j * ph) @ (w[1, :, 0] + 1j * w[1, :, 1])
    return np.stack([az, el, f], 1), np.stack([hh.real, hh.imag, vv.real, vv.imag], 1)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    k = case["kind"]
    if k == "mesh":
        xyz, tri = _aircraft_smooth(case["size"])
        # another airframe: every vertex displaced by the build tolerance
        new = (xyz + rng.normal(0.0, 1e-3, xyz.shape)).astype(np.float32)
        ctx = G.Context(0)
        return dict(case=case, ctx=ctx, xyz=new, tri=tri, ang=np.array([[rng.uniform(0, 360), rng.uniform(-5, 5)]]),
                    freqs=np.array([case["ghz"] * 1e9]), spacing=C0 / (case["ghz"] * 1e9 * 10.0))
    if k in ("train", "predict"):
        s = G.Surrogate(0, n_members=case["members"], width=case["width"], depth=case["depth"],
                        n_fourier=case["fourier"], seed=1 + seed % 1000)
        n = case["n"]
        x, y = _field_samples(n if k == "train" else 2048, rng)
        if k == "train":
            return dict(case=case, s=s, x=x, y=y)
        # a short fit first, so that the members differ as trained ones do
        s.train(x, y, epochs=1, batch=1024, lr=1e-3)
        q = np.stack([rng.uniform(178.0, 182.0, n), rng.uniform(-1.0, 1.0, n), rng.uniform(1.0e9, 1.2e9, n)], 1)
        return dict(case=case, s=s, x=q)
    ctx = G.Context(0)
    xyz, tri = _mesh(case["mesh"], case["size"])
    ctx.load_mesh(xyz, tri)
    if k == "batch":
        reqs = _requests(case, rng)
        st = dict(case=case, ctx=ctx, reqs=reqs)
        if case["graph"]:
            rows = sum(len(r["freqs"]) for r in reqs)
            st["E"] = torch.zeros((rows, 2, 2), dtype=torch.float64, device="cuda")
            st["R"] = torch.zeros((rows, 2), dtype=torch.float64, device="cuda")
        return st
    ang, rx = _aspects(case, rng)
    return dict(case=case, ctx=ctx, ang=ang, rx=rx, freqs=_freqs(case, rng), spacing=C0 / (case["ghz"] * 1e9 * 10.0),
                offset=(float(rng.uniform()), float(rng.uniform())))


# --------------------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "mesh":
        ctx = st["ctx"]
        ctx.load_mesh(st["xyz"], st["tri"])
        t = ctx.trace(st["ang"], st["spacing"], eta=ETA, max_bounces=case["bounces"])
        E, R = ctx.po_integrate(st["freqs"], "HH,VV")
        return dict(E=E, rcs=R, box=ctx.get_bbox(), valid=t["valid_rays"], bounces=t["ray_bounces"])
    if k == "train":
        s = st["s"]
        loss = s.train(st["x"], st["y"], epochs=case["epochs"], batch=case["batch"], lr=1e-3)
        return dict(loss=loss, params=[s.params(e) for e in range(case["members"])])
    if k == "predict":
        mean, spread = st["s"].predict(st["x"])
        return dict(mean=mean, spread=spread)
    ctx = st["ctx"]
    if k == "batch":
        if case["graph"]:
            ctx.submit_batch(st["reqs"], E_out=st["E"], rcs_out=st["R"], eta=ETA, max_bounces=case["bounces"])
            t = ctx.sync()
            return dict(E=st["E"], rcs=st["R"], valid=t["valid_rays"], bounces=t["ray_bounces"])
        E, R, t = ctx.run_batch(st["reqs"], eta=ETA, max_bounces=case["bounces"])
        return dict(E=np.concatenate(E), rcs=np.concatenate(R), valid=t["valid_rays"], bounces=t["ray_bounces"])
    flags = G.sbr.TRACE_REQUIRE_ESCAPE if case["escape"] else 0
    t = ctx.trace(st["ang"], st["spacing"], eta=ETA, max_bounces=case["bounces"], offset=st["offset"], flags=flags,
                  rx=st["rx"])
    E, R = ctx.po_integrate(st["freqs"], case["pols"], mode=case["form"], phase=case["phase"])
    return dict(E=E, rcs=R, valid=t["valid_rays"], bounces=t["ray_bounces"])


# --------------------------------------------------------------------------- what a pass cannot do without
#: per mesh: the box, the share of the grid's rays that hit, closest-hit queries after the first per hit ray
_SHAPE = {"sphere": ((2.0, 2.0, 2.0), 0.71, 0.0), "trihedral": ((1.0, 1.0, 1.0), 0.45, 1.6),
          "aircraft": ((15.0, 17.0, 4.6), 0.25, 1.2)}
_RAY, _QUERY, _TUBE = 60, 200, 30  # FLOP per launched ray (origin, one decision), later query with its update, tube x frequency


def _rays(mesh, spacing, el=0.0):
    """Rays of one aspect's grid, averaged over azimuth."""
    bx, by, bz = _SHAPE[mesh][0]
    az = np.radians(np.arange(0, 360, 5.0))
    lu = bx * np.abs(np.sin(az)) + by * np.abs(np.cos(az))
    ce, se = math.cos(math.radians(el)), abs(math.sin(math.radians(el)))
    lv = bz * ce + (bx * np.abs(np.cos(az)) + by * np.abs(np.sin(az))) * se
    return float(np.mean(lu * lv)) * (1 + ETA) ** 2 / spacing**2


def work(case):
    k = case["kind"]
    if k in ("train", "predict"):
        p = case["width"] * (case["fourier"] + (case["depth"] - 1) * case["width"] + 4)
        n = case["n"] if k == "predict" else (case["n"] // case["batch"]) * case["batch"] * case["epochs"]
        flops = 2.0 * p * n * case["members"] * (1 if k == "predict" else 3)
        io = case["n"] * (24 + 36 if k == "predict" else 24 + 32) + 4.0 * p * case["members"] * (1 if k == "predict" else 6)
        return {"bytes": io, "flops": flops}
    if k == "mesh":
        n, spacing = case["size"], C0 / (case["ghz"] * 1e10)
        rays = _rays("aircraft", spacing)
        return {"bytes": 18.0 * n + 48, "flops": 100.0 * n + rays * (_RAY + 0.25 * (1.2 * _QUERY + _TUBE))}
    tris = {"sphere": 20 * 4 ** case["size"], "trihedral": 3 * case["size"] ** 2, "aircraft": case["size"]}[case["mesh"]]
    _, share, later = _SHAPE[case["mesh"]]
    if k == "batch":
        # mean over the request distribution: highest frequency about 11.5 GHz, 7.5 rays per wavelength, 32 frequencies
        rays = case["requests"] * _rays(case["mesh"], C0 / (11.5e9 * 7.5), 15.0)
        return {"bytes": 18.0 * tris + case["requests"] * 32 * 2 * 24.0,
                "flops": rays * (_RAY + share * (later * _QUERY + 32 * _TUBE))}
    rays = case["aspects"] * _rays(case["mesh"], C0 / (case["ghz"] * 1e10), 35.26 if case["mesh"] == "trihedral" else 0.0)
    npol = len(case["pols"].split(","))
    later = min(later, case["bounces"] - 1) + (1.0 if case["bistatic"] else 0.0)
    return {"bytes": 18.0 * tris + case["aspects"] * case["freqs"] * npol * 24.0,
            "flops": rays * (_RAY + share * (later * _QUERY + case["freqs"] * _TUBE))}


# --------------------------------------------------------------------------- the same results in 64 bits
def _angles64(az, el):
    a, e = math.radians(az), math.radians(el)
    ca, sa, ce, se = math.cos(a), math.sin(a), math.cos(e), math.sin(e)
    r = torch.tensor([ce * ca, ce * sa, se], dtype=torch.float64, device="cuda")
    v = torch.tensor([se * ca, se * sa, -ce], dtype=torch.float64, device="cuda")
    h = torch.tensor([-sa, ca, 0.0], dtype=torch.float64, device="cuda")
    return r, v, h


def _closest64(tri, o, d, skip):
    """Closest hit (index or -1, distance) of rays o + t d on triangles tri [m, 3, 3], by testing them all."""
    v0, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    n = o.shape[0]
    best_t = torch.full((n,), math.inf, dtype=torch.float64, device=o.device)
    best_k = torch.full((n,), -1, dtype=torch.int64, device=o.device)
    step = max(1, 60_000_000 // tri.shape[0])
    for a in range(0, n, step):
        oo, dd = o[a:a + step, None, :], d[a:a + step, None, :]
        p = torch.linalg.cross(dd, e2[None])
        det = (e1[None] * p).sum(-1)
        s = oo - v0[None]
        u = (s * p).sum(-1) / det
        q = torch.linalg.cross(s, e1[None])
        v = (dd * q).sum(-1) / det
        t = (e2[None] * q).sum(-1) / det
        ok = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0)
        if skip is not None:
            ok[torch.arange(ok.shape[0], device=o.device), skip[a:a + step]] = False
        t = torch.where(ok, t, math.inf)
        bt, bk = t.min(1)
        best_t[a:a + step] = bt
        best_k[a:a + step] = torch.where(torch.isfinite(bt), bk, -1)
    return best_k, best_t


def _aspect64(tri, box, az, el, spacing, offset, bounces, form):
    """Tube coefficients [n, 4] (HH, VV, HV, VH) and paths [n] of one aspect's valid rays."""
    r, vh, hh = _angles64(az, el)
    kd = -r
    lo, hi = box[0], box[1]
    diag = float(torch.linalg.vector_norm(hi - lo))
    mid = 0.5 * (lo + hi)
    pts = torch.stack([torch.where(torch.tensor([bool(m & 1), bool(m & 2), bool(m & 4)], device="cuda"), hi, lo)
                       for m in range(8)])
    lu, lv = float((pts @ hh).max() - (pts @ hh).min()), float((pts @ vh).max() - (pts @ vh).min())
    nu = max(1, math.ceil((1 + ETA) * lu / spacing - 1e-9))
    nv = max(1, math.ceil((1 + ETA) * lv / spacing - 1e-9))
    au = (torch.arange(nu, dtype=torch.float64, device="cuda") + 0.5 - 0.5 * nu + offset[0]) * spacing
    av = (torch.arange(nv, dtype=torch.float64, device="cuda") + 0.5 - 0.5 * nv + offset[1]) * spacing
    base = mid - (0.5 * diag + 1.0) * kd
    o = (base[None, None] + au[None, :, None] * hh + av[:, None, None] * vh).reshape(-1, 3)
    d = kd.expand_as(o).clone()
    path = o @ kd
    ev = vh.expand_as(o).clone()
    nrm = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    nrm = nrm / torch.linalg.vector_norm(nrm, dim=1, keepdim=True)
    dA = spacing * spacing
    out_c, out_l = [], []
    last, cand, nb, cos0 = None, None, 0, None
    while True:
        if nb == bounces:
            out_c.append(cand[0])
            out_l.append(cand[1])
            break
        k, t = _closest64(tri, o, d, last)
        hit = k >= 0
        if nb:
            out_c.append(cand[0][~hit])
            out_l.append(cand[1][~hit])
        if not bool(hit.any()):
            break
        o, d, path, ev, k, t = o[hit], d[hit], path[hit], ev[hit], k[hit], t[hit]
        x = o + t[:, None] * d
        path = path + t
        n = nrm[k]
        dn = (d * n).sum(-1)
        nf = torch.where((dn < 0)[:, None], n, -n)
        cos0 = (nf @ r) if nb == 0 else cos0[hit]
        nb += 1
        eh = (1.0 if (nb - 1) % 2 else -1.0) * torch.linalg.cross(d, ev)
        if form == "scalar":
            a = -2.0 * dA * cos0 * (-1.0 if nb % 2 else 1.0)
            c = torch.stack([a, a, torch.zeros_like(a), torch.zeros_like(a)], 1)
        else:
            w = []
            for e in (eh, ev):
                j = 2.0 * (d * (nf * e).sum(-1, keepdim=True) - e * (nf * d).sum(-1, keepdim=True))
                w.append((dA / dn.abs())[:, None] * (j - (j @ r)[:, None] * r))
            c = torch.stack([w[0] @ hh, w[1] @ vh, w[1] @ hh, w[0] @ vh], 1)
        cand = (c, path + x @ kd)
        ev = 2.0 * (n * ev).sum(-1, keepdim=True) * n - ev
        d = d - 2.0 * dn[:, None] * n
        o = x + 1e-5 * diag * nf
        last = k
    return torch.cat(out_c), torch.cat(out_l)


def _field64(c, path, freqs, sel):
    E = np.empty((len(freqs), len(sel)), np.complex128)
    for i, f in enumerate(freqs):
        kk = 2.0 * math.pi * float(f) / C0
        ph = torch.polar(torch.ones_like(path), -kk * path)
        for j, s in enumerate(sel):
            E[i, j] = (-1j * kk / (4 * math.pi)) * complex((c[:, s] * ph).sum().item())
    return E


def exact(case, seed):
    if case["kind"] not in ("trace", "batch") or case["mesh"] == "aircraft" or case.get("bistatic") or case.get("escape"):
        return None  # a full aircraft grid against a million triangles, or a network from the library's own draws
    rng = np.random.default_rng(seed)
    xyz, tri = _mesh(case["mesh"], case["size"])
    box = torch.tensor(np.stack([xyz.min(0), xyz.max(0)]).astype(np.float64), device="cuda")
    if case["mesh"] == "trihedral":
        # the plates as one triangle each: the same surface
        o, ex, ey, ez = (0.0, 0.0, 0.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0)
        T = torch.tensor([[o, ex, ey], [o, ey, ez], [o, ez, ex]], dtype=torch.float64, device="cuda")
    else:
        T = torch.tensor(xyz[tri].astype(np.float64), device="cuda")
    pol = {"HH": 0, "VV": 1, "HV": 2, "VH": 3}
    if case["kind"] == "batch":
        items = [(r["az"], r["el"], r["spacing"], r["freqs"]) for r in _requests(case, rng)]
        offset, form, sel = (0.0, 0.0), "vector", [0, 1]
    else:
        ang, _ = _aspects(case, rng)
        f, sp = _freqs(case, rng), C0 / (case["ghz"] * 1e9 * 10.0)
        offset = (float(rng.uniform()), float(rng.uniform()))
        items = [(a, e, sp, f) for a, e in ang]
        form, sel = case["form"], [pol[p] for p in case["pols"].split(",")]
    n = sum(_rays(case["mesh"], sp, e) for a, e, sp, f in items)
    if n * T.shape[0] > 1.5e10 or sum(_rays(case["mesh"], sp, e) * len(f) for a, e, sp, f in items) > 3e9:
        return None
    E = []
    for az, el, sp, f in items:
        c, path = _aspect64(T, box, az, el, sp, offset, case["bounces"], form)
        E.append(_field64(c, path, f, sel))
    # cross-polarised and shadowed sums cancel to rounding: their dB value says nothing, the field does
    rcs = None
    if case["kind"] == "batch":
        return dict(E=np.concatenate(E), rcs=rcs, valid=None, bounces=None)
    return dict(E=np.stack(E), rcs=rcs, valid=None, bounces=None)
