"""The binary64 product on the tensor cores (abft_gemm / abft_gemm_plain with a
workspace) against the exact product of sampled rows and columns in extended precision.

Tolerance: elementwise 2 k u (|A||B|), u = 2^-53, the rounding bound of any order of k
multiply-adds.  The product meets it by construction: the operands are rounded at most
2^-(b+1) of their row's and column's scale (b = 58 or 59), so a term errs by at most
2^-b + 2^-2b in those units, and an element is only taken where |A||B| is at least
1.52 2^(53-b) sqrt(k) of them: the error is at most 0.7 sqrt(k) u (|A||B|).  Its Frobenius
error is also at most that of the DFMA kernel (the same call without a workspace) or one
rounding."""
import numpy as np
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


def operands(kind, m, n, k):
    r = np.random.default_rng(m + 7 * n + 31 * k)
    A, B = r.standard_normal((m, k)), r.standard_normal((k, n))
    if kind == "rows":       # one magnitude per row of A and of B
        A *= 10.0 ** r.uniform(-2, 2, (m, 1))
        B *= 10.0 ** r.uniform(-2, 2, (k, 1))
    elif kind == "graded":   # large columns of A meet small rows of B
        d = 10.0 ** r.uniform(-8, 8, k)
        A, B = A * d, B / d[:, None]
    elif kind == "outlier":  # a large column of A meets zeros of B in every other column
        A[:, k // 2] = 1e9
        B[k // 2, ::2] = 0
    elif kind == "int":
        A, B = r.integers(-999, 1000, (m, k)) * 1.0, r.integers(-999, 1000, (k, n)) * 1.0
    elif kind == "eye":
        A = np.eye(m, k)
    elif kind == "sparse":
        A *= r.random((m, k)) < 0.01
        B *= r.random((k, n)) < 0.01
    elif kind == "equal":    # one value everywhere: residues add up with one sign
        A[:] = B[:] = -(128 * (256 ** 8 - 1) // 255) / 2.0 ** 63
    elif kind == "wide":     # exponents outside the range of the lines' scales
        A *= 10.0 ** r.uniform(-200, -100, (m, 1))
    elif kind == "zero":
        A[::2] = 0
        B[:, ::3] = 0
    return A, B


def product(A, B, ws=True, vb=(64, 48), pad=0):
    (m, k), n = A.shape, B.shape[1]
    d = abft.make_desc(m, n, k, "f64", min(vb[0], m), min(vb[1], n), lda=k + pad, ldb=n + pad,
                       ldc=n + pad)
    dev = [torch.zeros(x.shape[0], x.shape[1] + pad, dtype=torch.float64, device="cuda")
           for x in (A, B)]
    for t, x in zip(dev, (A, B)):
        t[:, :x.shape[1]] = torch.from_numpy(x)
    C = torch.full((m, n + pad), 7.0, dtype=torch.float64, device="cuda")
    w = torch.zeros(abft.abft_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    if ws:
        abft.abft_encode(d, *dev, w)
        abft.abft_gemm(d, *dev, C, w)
    else:
        abft.abft_gemm_plain(d, *dev, C)
    torch.cuda.synchronize()
    assert pad == 0 or bool((C[:, n:] == 7.0).all())
    return C[:, :n].cpu().numpy(), d, w


def sample(x, count=24):
    r = np.random.default_rng(x)
    return np.unique(np.r_[0, x - 1, r.integers(0, x, min(x, count))])


def check(A, B, C, C0=None):
    rows, cols = sample(A.shape[0]), sample(B.shape[1])
    a, b = A[rows].astype(np.longdouble), B[:, cols].astype(np.longdouble)
    ref, mag = a @ b, np.abs(a) @ np.abs(b)
    err = C[np.ix_(rows, cols)] - ref
    assert np.all(np.abs(err) <= 2 * A.shape[1] * U * mag)
    if C0 is not None:
        e0 = C0[np.ix_(rows, cols)] - ref
        assert np.linalg.norm(err.astype(float)) <= max(
            np.linalg.norm(e0.astype(float)), U * np.linalg.norm(ref.astype(float)))


# edges of the 128-row tiles, the 64-column boxes, the 64-wide k-steps, the 1024-term
# accumulators and the 16320-wide panels; one, two and four boxes per tile, CTA pairs
SHAPES = [(128, 128, 128), (129, 127, 129), (1, 2500, 1000), (300, 3, 3000), (257, 65, 1023),
          (127, 193, 1025), (640, 2600, 64), (2000, 2100, 100), (130, 200, 16321), (2800, 3000, 130)]


@pytest.mark.parametrize("shape", SHAPES)
def test_edges(shape):
    A, B = operands("normal", *shape)
    C, _, _ = product(A, B)
    check(A, B, C, product(A, B, ws=False)[0])
    A, B = operands("int", *shape)
    assert np.array_equal(product(A, B, pad=1)[0], A @ B)


@pytest.mark.parametrize("kind", ["rows", "graded", "outlier", "eye", "sparse", "equal", "wide",
                                  "zero"])
def test_operand_kinds(kind):
    A, B = operands(kind, 300, 330, 1100)
    C, d, ws = product(A, B, pad=3)
    check(A, B, C, product(A, B, ws=False)[0])
    if kind == "eye":
        assert np.array_equal(C, B[:300])


def test_checksum_rows_and_columns():
    """E = acs B and F = A bcs of the same launch, and a fault located from them."""
    A, B = operands("normal", 270, 400, 500)
    C, d, ws = product(A, B)
    L = abft.abft_workspace_layout(d)

    def region(off, r, c):
        return ws[off:off + 8 * r * c].view(torch.float64).view(r, c).cpu().numpy()

    check(region(L.acs, L.R, 500), B, region(L.E, L.R, 400))
    check(A, region(L.bcs, 500, L.Cc), region(L.F, 270, L.Cc))
    Cd = torch.from_numpy(C).cuda()
    abft.abft_inject_bitflips(d, Cd, [(130, 77, 61)])
    st, rep, n = abft.abft_verify_correct(d, Cd, ws)
    assert st == abft.OK and n == 1 and (rep[0]["row"], rep[0]["col"]) == (130, 77)
    assert np.allclose(Cd.cpu().numpy(), C, rtol=1e-11, atol=1e-11)


def test_non_finite_operands_match_the_dfma_kernel():
    A, B = operands("normal", 300, 330, 700)
    A[5, 7], A[200, 600], B[3, 300] = np.nan, np.inf, -np.inf
    C, C0 = product(A, B)[0], product(A, B, ws=False)[0]
    assert np.array_equal(np.isnan(C), np.isnan(C0))
    assert np.array_equal(C[np.isinf(C0)], C0[np.isinf(C0)])


def test_bounded_wait_reports_a_timeout(monkeypatch):
    """A stalled producer's waits run out; the verify reports it and leaves C alone, and
    the next product on the workspace is good again."""
    A, B = operands("normal", 256, 256, 256)
    monkeypatch.setenv("ABFT_TEST_STALL_PRODUCER", "1")
    C, d, ws = product(A, B)
    monkeypatch.delenv("ABFT_TEST_STALL_PRODUCER")
    Cd = torch.from_numpy(C).cuda()
    with pytest.raises(abft.AbftError) as e:
        abft.abft_verify_correct(d, Cd, ws)
    assert e.value.status == abft.ERR_TIMEOUT
    assert np.array_equal(Cd.cpu().numpy(), C, equal_nan=True)
    dev = [torch.from_numpy(x).cuda() for x in (A, B)]
    abft.abft_gemm(d, *dev, Cd, ws)
    st, _, n = abft.abft_verify_correct(d, Cd, ws)
    assert st == abft.OK and n == 0
    check(A, B, Cd.cpu().numpy())
