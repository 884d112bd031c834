"""Every phase mode of the PO sum at every item size, with one to four polarisations
and with frequency counts around those a reduction carries, against FP64 numpy over
the trace's own records."""
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


@pytest.mark.parametrize("phase", ["compensated", "fp32", "fp64"])
@pytest.mark.parametrize("item", [512, 1024, 2048])
def test_phase_modes_match_fp64(G, phase, item):
    """As in test_po_sums_match_fp64 each term is within 40 2^-24 of its size; the FP32 phase adds the roundings of k,
    of the path and of their product: 3 2^-24 k |L|."""
    import sbr_inputs as S

    xyz, tri = S.icosphere(4, 1.0)
    with G.Context(0) as c:
        c.set_tuning(po_item=item)
        c.load_mesh(xyz, tri)
        c.trace([[20.0, 10.0]], 0.02, eta=0.05, max_bounces=1, offset=(0.37, 0.61))
        r = c.get_records(0)
        assert len(r["L"]) > 2 * item
        for n_freq, pols in ((1, "HH,VV"), (2, "VV"), (3, "HH,VV,HV"), (4, "HH,VV"), (5, "HH,VV,HV,VH"), (9, "HV,VH")):
            f = np.linspace(2e9, 11e9, n_freq)
            E, _ = c.po_integrate(f, pols, phase=phase)
            sel = [("HH", "VV", "HV", "VH").index(p) for p in pols.split(",")]
            cc = r["coef"].astype(np.float64)[:, sel]
            for q in range(n_freq):
                k = 2 * np.pi * f[q] / C0
                ref = -1j * k / (4 * np.pi) * np.sum(cc * np.exp(-1j * k * r["L"])[:, None], 0)
                term = 40.0 + (3.0 * k * np.abs(r["L"]).max() if phase == "fp32" else 0.0)
                assert np.all(np.abs(E[0, q] - ref) <= k / (4 * np.pi) * term * 2.0 ** -24 * np.abs(cc).sum(0)), (n_freq, q)
