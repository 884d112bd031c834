"""The PO sums of synthetic records against FP64 numpy: tube counts around the
edges of a thread block's items and of the final sum's slices, frequency and
polarisation counts around those a block reduction carries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C0 = 299_792_458.0


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


@pytest.mark.parametrize("counts", [(1, 0, 255), (1024, 1025, 31 * 1024), (33 * 1024 + 7, 5, 257 * 1024)])
@pytest.mark.parametrize("n_freq,pols", [(1, "HH,VV"), (2, "VV"), (3, "HH,VV,HV"), (4, "HH,VV"), (5, "HH,VV,HV,VH"),
                                         (9, "HV,VH")])
def test_po_sums_match_fp64(G, counts, n_freq, pols):
    """Each term's phase is within about 3 half-units of the FP32 fraction of a cycle (2 pi 3 2^-25 rad) and sine and
    cosine within 2 units, each product and the 20 additions a term passes through round once in FP32: 40 2^-24 of
    the sum of |c| per aspect bounds the error."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n_freq + counts[0])
    n = sum(counts)
    rec = np.zeros((n, 8), np.float32)
    rec[:, :5] = rng.normal(0, 1e-3, (n, 5))
    L = rng.uniform(-40.0, 40.0, n)
    rec[:, 5] = L
    rec[:, 6] = L - rec[:, 5].astype(np.float64)
    d = torch.from_numpy(rec).cuda()
    f = np.linspace(2e9, 11e9, n_freq)
    names = pols.split(",")
    E = torch.full((len(counts), n_freq, len(names), 2), float("nan"), dtype=torch.float64, device="cuda")
    off = np.concatenate([[0], np.cumsum(counts)])
    torch.cuda.synchronize()
    G.sbr.po_integrate_noalloc(d.data_ptr(), off, f, pols, E_ptr=E.data_ptr())
    torch.cuda.synchronize()
    got = E.cpu().numpy()
    path = rec[:, 5].astype(np.float64) + rec[:, 6].astype(np.float64)
    sel = [("HH", "VV", "HV", "VH").index(p) for p in names]
    for a in range(len(counts)):
        s = slice(off[a], off[a + 1])
        for q in range(n_freq):
            k = 2 * np.pi * f[q] / C0
            ph = np.exp(-1j * k * path[s])
            for p, c in enumerate(sel):
                cc = rec[s, c].astype(np.float64)
                ref = -1j * k / (4 * np.pi) * np.sum(cc * ph)
                err = abs(got[a, q, p, 0] + 1j * got[a, q, p, 1] - ref)
                assert err <= k / (4 * np.pi) * 40 * 2.0 ** -24 * np.abs(cc).sum(), (a, q, p, err)
