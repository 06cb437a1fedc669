"""Weighted sums of lines that hold one infinity are infinite, not NaN (every weight is
positive): the encoded rows of A, and the residuals that the verify reports for a column line
of a re-read result, in the first and in a later 64-row segment of a verify block."""
import numpy as np
import pytest

from paper_0806_3121_gb300 import abft

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0806_3121_gb300 import build
    build.build()
    return abft.load()


def run(dtype, m, n, k, vb):
    g = torch.Generator(device="cuda").manual_seed(m + vb)
    dt = torch.float64 if dtype == "f64" else torch.bfloat16
    A = torch.randn(m, k, generator=g, device="cuda").to(dt)
    B = torch.randn(k, n, generator=g, device="cuda").to(dt)
    d = abft.make_desc(m, n, k, dtype, vb, 64)
    ws = torch.zeros(abft.abft_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    C = torch.zeros(m, n, device="cuda",
                    dtype=torch.float64 if dtype == "f64" else torch.float32)
    return A, B, C, d, ws


@pytest.mark.parametrize("vb,row", [(32, 3), (200, 5), (200, 130), (600, 599)])
def test_encoded_rows(vb, row):
    A, B, C, d, ws = run("f64", 600, 128, 96, vb)
    A[row, 7] = float("-inf")
    abft.abft_encode(d, A, B, ws)
    L = abft.abft_workspace_layout(d)
    acs = ws[L.acs:L.acs + 8 * L.R * 96].view(torch.float64).view(L.R, 96).cpu().numpy()
    at = acs[2 * (row // vb):2 * (row // vb) + 2, 7]
    assert np.all(at == -np.inf), at
    acs[2 * (row // vb):2 * (row // vb) + 2, 7] = 0
    assert np.all(np.isfinite(acs))


@pytest.mark.parametrize("dtype", ["f64", "bf16"])
@pytest.mark.parametrize("vb,row", [(32, 3), (200, 5), (200, 130), (600, 599)])
def test_reported_residuals(dtype, vb, row):
    A, B, C, d, ws = run(dtype, 600, 128, 96, vb)
    abft.abft_encode(d, A, B, ws)
    abft.abft_gemm(d, A, B, C, ws)
    want = C.clone()
    C[row, 70] = float("inf")
    st, rep, count = abft.abft_verify_correct(d, C, ws, reread_C=1)
    assert st == abft.OK and count == 1
    f = rep[0]
    assert (f["row"], f["col"]) == (row, 70)
    assert f["r_e"] == np.inf and f["r_w"] == np.inf, f
    assert torch.allclose(C, want, rtol=1e-4, atol=1e-3)
