"""CTA-pair tiles of the long split and FP8 products, kept in step through one workspace
word, against one-CTA tiles: the rule takes pairs at these sizes (k at and above its
limits; one wave of pairs and several, the last one partly filled; ragged tiles).

Tolerance: elementwise 2 k u32 (|A||B|), the bound of any order of k binary32
multiply-adds, plus what the split of the operands drops (bf16x3 2^-16, bf16x6 2^-25)."""
import pytest

from paper_0806_3121_gb300 import abft

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U32 = 2.0 ** -24
DROPPED = {"bf16x3": 2.0 ** -16, "bf16x6": 2.0 ** -25, "fp8": 0.0}


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0806_3121_gb300 import build
    build.build()
    return abft.load()


@pytest.mark.parametrize("dtype,k", [("bf16x6", 5120), ("bf16x3", 8200), ("fp8", 9300)])
@pytest.mark.parametrize("m,n", [(300, 720), (2590, 9200)])
def test_long_products(dtype, k, m, n, monkeypatch):
    for name in ("ABFT_PAIR_TILES", "ABFT_TALL_TILES", "ABFT_PROMOTE_KSTEPS"):
        monkeypatch.delenv(name, raising=False)
    g = torch.Generator(device="cuda").manual_seed(m + k)
    ld = (k + 15) // 16 * 16
    A = torch.zeros(m, ld, device="cuda")
    A[:, :k] = torch.randn(m, k, generator=g, device="cuda")
    B = torch.randn(k, n, generator=g, device="cuda")
    sc = ()
    if dtype == "fp8":
        A, B = A.to(torch.float8_e4m3fn), B.to(torch.float8_e4m3fn)
        sc = (2.0 ** torch.randint(-3, 3, (-(-m // 128), -(-k // 128)), generator=g,
                                   device="cuda").float(),
              2.0 ** torch.randint(-3, 3, (-(-k // 128), -(-n // 128)), generator=g,
                                   device="cuda").float())
    d = abft.make_desc(m, n, k, dtype, 128, 256, lda=ld)
    ws = torch.zeros(abft.abft_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    out = []
    for pair in (None, "0"):
        if pair:
            monkeypatch.setenv("ABFT_PAIR_TILES", pair)
        C = torch.full((m, n), float("nan"), device="cuda")
        for _ in range(2):  # the second product starts from a used workspace
            abft.abft_encode(d, A, B, ws, *sc)
            abft.abft_gemm(d, A, B, C, ws, *sc)
        st, rep, count = abft.abft_verify_correct(d, C, ws, reread_C=1)
        assert st == abft.OK and count == 0, rep
        out.append(C.double())
    a, b = A[:, :k].double(), B.double()
    if dtype == "fp8":
        a *= sc[0].double().repeat_interleave(128, 0)[:m].repeat_interleave(128, 1)[:, :k]
        b *= sc[1].double().repeat_interleave(128, 0)[:k].repeat_interleave(128, 1)[:, :n]
    ref, bound = a @ b, (2 * k * U32 + DROPPED[dtype]) * (a.abs() @ b.abs())
    for C in out:
        assert bool(((C - ref).abs() <= bound).all())
