"""The tensor-core GEMM at the tile widths its rule picks: the numbers of tiles on
both sides of each line, for 152 SMs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


# 128 x 128 tiles: 76 and 77 (64 or 128 columns), 152 (one wave of 128), 160 and 304 (one and two waves of 256), 456
# (three waves of 128 or two of 256), an odd number of tile columns (no 256)
@pytest.mark.parametrize("M,N,K,pad", [(128 * 38, 256, 128, 0), (128 * 77, 128, 64, 8), (128 * 38, 512, 64, 0), (2048, 1280, 192, 0),
                                       (128 * 76, 512, 64, 8), (128 * 114, 512, 128, 0), (128 * 51, 384, 64, 0)])
def test_gemm_tile_widths(G, M, N, K, pad):
    torch = pytest.importorskip("torch")
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randn(M, K + pad, generator=g).to(torch.bfloat16).cuda()
    B = torch.randn(N, K + pad, generator=g).to(torch.bfloat16).cuda()
    C = torch.full((M, N + pad), float("nan"), device="cuda")
    G.gemm_bf16_tn(A.data_ptr(), K + pad, B.data_ptr(), K + pad, M, N, K, C.data_ptr(), N + pad)
    ref = (A[:, :K].double() @ B[:, :K].double().T).cpu().numpy()
    got = C.cpu().numpy()
    assert np.isnan(got[:, N:]).all() and not np.isnan(got[:, :N]).any()
    # exact BF16 products, FP32 accumulation
    assert np.max(np.abs(got[:, :N] - ref)) <= 2e-6 * np.sqrt(K) * np.abs(ref).max()
