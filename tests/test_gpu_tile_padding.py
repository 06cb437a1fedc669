"""Checksum rows and columns in the padding of the last data tiles (taken where that saves a
wave of tiles) and the choice between regular and tall tiles: C, E and F against binary64,
a fault-free verify, and a flip in the tile that holds data, checksum rows and columns.

Tolerance: elementwise 2 k u32 (|A||B|) plus what the operands' split drops; E and F further
2^-16 of the checksums' pieces and 256 u32 of their sums."""
import pytest

from paper_0806_3121_gb300 import abft

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U32 = 2.0 ** -24
DROPPED = {"bf16": 0.0, "bf16x3": 2.0 ** -16, "bf16x6": 2.0 ** -25}


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0806_3121_gb300 import build
    build.build()
    return abft.load()


def sums(x, vb):
    """Plain and weighted sums of x's rows per block of vb rows."""
    m, n = x.shape
    nb = -(-m // vb)
    x = torch.cat([x, x.new_zeros(nb * vb - m, n)]).view(nb, vb, n)
    w = torch.arange(1, vb + 1, device=x.device).double() / 2.0 ** (vb - 1).bit_length()
    return torch.stack([x.sum(1), (w[:, None] * x).sum(1)], 1).view(2 * nb, n)


@pytest.mark.parametrize("dtype", ["bf16", "bf16x3", "bf16x6"])
@pytest.mark.parametrize("m,n,k,vb_r", [
    (3001, 2999, 130, 128),   # columns ride in the last tile column, rows have tiles
    (2820, 3072, 130, 256),   # rows ride in the last tile row, columns have tiles
    (2820, 3240, 130, 256),   # both
    (4100, 4000, 2112, 128)]) # bf16: tall tiles, three checksum halves below one of data
def test_mixed_tiles(dtype, m, n, k, vb_r, monkeypatch):
    for name in ("ABFT_PAIR_TILES", "ABFT_TALL_TILES", "ABFT_PROMOTE_KSTEPS"):
        monkeypatch.delenv(name, raising=False)
    g = torch.Generator(device="cuda").manual_seed(m + n)
    lda, ldb = (k + 7) // 8 * 8, (n + 7) // 8 * 8
    A = torch.randn(m, lda, generator=g, device="cuda")
    B = torch.randn(k, ldb, generator=g, device="cuda")
    if dtype == "bf16":
        A, B = A.bfloat16(), B.bfloat16()
    d = abft.make_desc(m, n, k, dtype, vb_r, 256, lda=lda, ldb=ldb)
    L = abft.abft_workspace_layout(d)
    ws = torch.zeros(L.total, dtype=torch.uint8, device="cuda")
    C = torch.full((m, n), float("nan"), device="cuda")
    abft.abft_encode(d, A, B, ws)
    abft.abft_gemm(d, A, B, C, ws)
    st, rep, count = abft.abft_verify_correct(d, C, ws, reread_C=0)
    assert st == abft.OK and count == 0, rep
    a, b = A[:, :k].double(), B[:, :n].double()
    dot = (2 * k * U32 + DROPPED[dtype])
    assert bool(((C.double() - a @ b).abs() <= dot * (a.abs() @ b.abs())).all())
    cs = dot + 2.0 ** -16 + 256 * U32
    E = ws[L.E:L.E + 8 * L.R * n].view(torch.float64).view(L.R, n)
    F = ws[L.F:L.F + 8 * L.Cc * m].view(torch.float64).view(m, L.Cc)
    assert bool(((E - sums(a, vb_r) @ b).abs() <= cs * (sums(a.abs(), vb_r) @ b.abs())).all())
    assert bool(((F - a @ sums(b.T, 256).T).abs() <= cs * (a.abs() @ sums(b.T.abs(), 256).T)).all())
    abft.abft_set_epilogue_faults(d, ws, [(m - 1, n - 1, 30)])
    abft.abft_gemm(d, A, B, C, ws)
    st, rep, count = abft.abft_verify_correct(d, C, ws, reread_C=0)
    assert st == abft.OK and [(r["row"], r["col"]) for r in rep] == [(m - 1, n - 1)]
    assert bool(((C.double() - a @ b).abs()[-1, -1] <= 2 * cs * n * (a.abs() @ b.abs()).max()))
