"""Which of the two binary64 products takes a shape: short K loops and planes without room
run on the FP64 pipe (the same bits as a call without a workspace), planes with room for a
part of K run in panels (the 64-wide one and a remainder of one here).

Tolerance of the panels: 0.7 sqrt(k) u (|A||B|) for what the operands' rounding drops, one
rounding of each panel's sum and of its addition, u = 2^-53."""
import pytest

from paper_0806_3121_gb300 import abft

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0806_3121_gb300 import build
    build.build()
    return abft.load()


def run(m, n, k):
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A = torch.randn(m, k, generator=g, dtype=torch.float64, device="cuda")
    B = torch.randn(k, n, generator=g, dtype=torch.float64, device="cuda")
    d = abft.make_desc(m, n, k, "f64", min(128, m), min(128, n))
    ws = torch.zeros(abft.abft_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    C, C0 = torch.full((2, m, n), 7.0, dtype=torch.float64, device="cuda")
    abft.abft_encode(d, A, B, ws)
    abft.abft_gemm(d, A, B, C, ws)
    abft.abft_gemm_plain(d, A, B, C0)
    st, rep, count = abft.abft_verify_correct(d, C, ws)
    assert st == abft.OK and count == 0, rep
    return A, B, C, C0


@pytest.mark.parametrize("shape", [(1500, 1500, 1), (2048, 2100, 47), (64, 65536, 16),
                                   (1 << 21, 1, 48)])
def test_fp64_pipe(shape):
    _, _, C, C0 = run(*shape)
    assert torch.equal(C, C0)


@pytest.mark.parametrize("shape", [(1, 200000, 65), (200000, 1, 65), (1500, 1500, 48)])
def test_tensor_cores_in_panels(shape):
    A, B, C, _ = run(*shape)
    # the exact products of two 53-bit numbers as a sum of two binary64 ones, by splitting
    # each operand in 26 and 27 bits; summed in order of k with the rounding errors kept
    hi = lambda x: (x * 134217729.0) - (x * 134217729.0 - x)
    ref = torch.zeros_like(C)
    low = torch.zeros_like(C)
    for l in range(A.shape[1]):
        a, b = A[:, l:l + 1], B[l:l + 1]
        p = a * b
        ah, bh = hi(a), hi(b)
        low += ((ah * bh - p) + ah * (b - bh) + (a - ah) * bh) + (a - ah) * (b - bh)
        s = ref + p
        t = s - ref
        low += (ref - (s - t)) + (p - t)
        ref = s
    err = ((C - ref) - low).abs()
    mag = A.abs() @ B.abs()
    panels = -(-A.shape[1] // 64)
    bound = 0.7 * A.shape[1] ** 0.5 * U * mag + 2 * panels * U * mag
    # the reference itself: its corrections add up with one rounding each
    bound += 4 * A.shape[1] ** 2 * U * U * mag + U * ref.abs() * 2.0 ** -40
    assert bool((err <= bound).all())
