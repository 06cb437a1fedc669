"""Rounding of the binary64 product on the tensor cores, on operands made for it, against
exact integer sums.

Ties: rows whose largest element (1.0, which meets a zero) makes the integers' unit 2^-58
and whose other elements lie in [2^-7, 2^-6), multiples of 2^-59: every odd multiple is a tie.
Odd and even multiples alternate against +1, -1, so the k / 2 errors of 2^-59 add up with one
sign unless ties go to the even neighbour.  Then they are independent signs: 6 sqrt(k / 2) of
them bounds a row's error but for one row in 10^9, and one rounding of the result."""
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
