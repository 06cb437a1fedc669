"""Rounding of the binary64 product on the tensor cores, on operands made for it, against
exact integer sums.

Ties: rows whose largest element (1.0, which meets a zero) makes the integers' unit 2^-58
and whose other elements lie in [2^-7, 2^-6), multiples of 2^-59: every odd multiple is a tie.
Odd and even multiples alternate against +1, -1, so the k / 2 errors of 2^-59 add up with one
sign unless ties go to the even neighbour.  Then they are independent signs: 6 sqrt(k / 2) of
them bounds a row's error but for one row in 10^9, and one rounding of the result.

Bound: |err| <= 0.7 sqrt(k) u (|A||B|) + 2 u (|A||B|) per panel of K (16320), u = 2^-53, on
operands of which no element is left to the FP64 pipe: what the rounding of the operands
drops, at most 0.66 sqrt(k) u, with the roundings of a panel's sum and of its addition.
Cancelling: neighbours that agree to 1e-3 against +1, -1, in rows whose largest element meets a
zero, so the operands keep fewer bits than a binary64 and the sums are far below |A||B|."""
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


def product(A, B, vb=64):
    (m, k), n = A.shape, B.shape[1]
    d = abft.make_desc(m, n, k, "f64", min(vb, m), min(vb, n))
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A, B)]
    C = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    ws = torch.zeros(abft.abft_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    abft.abft_encode(d, *dev, ws)
    abft.abft_gemm(d, *dev, C, ws)
    return C.cpu().numpy()


@pytest.mark.parametrize("m,k", [(300, 256), (128, 1024), (70, 4096)])
def test_ties_do_not_add_up(m, k):
    r = np.random.default_rng(k)
    odd = r.integers(2 ** 52, 2 ** 53, (m, k // 2)) | 1
    even = np.clip(odd + 1 + 2 * r.integers(-2 ** 41, 2 ** 41, odd.shape), 2 ** 52, 2 ** 53 - 2)
    X = np.stack([odd, even & ~np.int64(1)], axis=2).reshape(m, k)  # multiples of 2^-59
    sign = np.where(np.arange(k) % 2 == 0, 1, -1)
    A = np.concatenate([np.ones((m, 1)), np.ldexp(X.astype(np.float64), -59)], axis=1)
    n = 2 ** 21 // (m * k) + 130
    B = np.zeros((k + 1, n))
    B[1:] = sign[:, None]
    B[1:, 1::2] *= -1  # columns of both signs
    C = product(A, B)
    exact = (X * sign).sum(axis=1)  # in 2^-59, below 2^53
    err = np.ldexp(C, 59) - np.where(np.arange(n) % 2, -1, 1) * exact[:, None].astype(np.float64)
    assert np.all(np.abs(err) <= 6 * (k / 2) ** 0.5 + U * np.abs(exact[:, None]) + 1)


def bounded(kind, m, n, k):
    r = np.random.default_rng(m + k)
    if kind == "uniform":
        return r.uniform(-1, 1, (m, k)), r.uniform(-1, 1, (k, n))
    if kind == "rows":
        return (r.uniform(-1, 1, (m, k)) * 10.0 ** r.uniform(-2, 2, (m, 1)),
                r.standard_normal((k, n)))
    x = np.exp2(r.uniform(-8, -6, (m, k)))
    x[:, 2::2] = x[:, 1:-1:2] * (1 + r.uniform(-1e-3, 1e-3, x[:, 2::2].shape))
    B = np.where(np.arange(k) % 2 == 0, 1.0, -1.0)[:, None] * np.ones((1, n))
    x[:, 0], B[0] = 1.0, 0.0
    return x, B


@pytest.mark.parametrize("kind", ["uniform", "rows", "cancelling"])
@pytest.mark.parametrize("m,n,k", [(130, 129, 129), (256, 200, 1025), (140, 65, 4097),
                                   (64, 300, 12001), (33, 65, 16400)])
def test_error_stays_within_the_stated_bound(kind, m, n, k):
    A, B = bounded(kind, m, n, k)
    C = product(A, B)
    rows, cols = np.unique(np.r_[0, m - 1, 17 % m, m // 2]), np.unique(np.r_[0, n - 1, n // 3])
    a, b = A[rows].astype(np.longdouble), B[:, cols].astype(np.longdouble)
    # long double keeps the exact products of binary64 numbers to 64 bits or more: its own
    # error, k 2^-63 of |A||B|, is added
    ref, mag = a @ b, np.abs(a) @ np.abs(b)
    bound = (0.7 * k ** 0.5 + 2 * -(-k // 16320) + k * 2.0 ** -10) * U * mag
    assert np.all(np.abs(C[np.ix_(rows, cols)] - ref) <= bound)
