"""The encode of the split dtypes (bf16x3, bf16x6) against binary64: first operand planes,
checksum rows and columns and the norms.  The warps of a CTA share a verify block's rows in
batches of eight, a CTA takes 256 columns: sizes at and around those edges.

Tolerance: a checksum is a binary32 sum of vb terms (vb u32 sum |terms|) split in pieces
that drop 2^-16 (bf16x3) or 2^-24 (bf16x6) of it; a norm is the root of a binary32 sum of
squares (at most (terms + 2) u32 of it)."""
import numpy as np
import pytest

from paper_0806_3121_gb300 import abft

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U32 = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0806_3121_gb300 import build
    build.build()
    return abft.load()


def blocks(x, vb):
    """Plain and weighted sums of x's rows per block of vb, and the same sums of |x|."""
    w = np.arange(1, vb + 1)[:, None] / 2.0 ** int(np.ceil(np.log2(vb)))
    out = [[], []]
    for i in range(0, len(x), vb):
        b = x[i:i + vb]
        for o, v in zip(out, (b, np.abs(b))):
            o += [v.sum(0), (w[:len(b)] * v).sum(0)]
    return np.array(out[0]), np.array(out[1])


@pytest.mark.parametrize("dtype", ["bf16x3", "bf16x6"])
@pytest.mark.parametrize("m,n,k,vb_r,vb_c", [
    (1, 8, 1, 1, 8), (7, 255, 129, 7, 16), (129, 257, 255, 64, 256), (300, 520, 264, 130, 128),
    (65, 2056, 2049, 65, 8)])
def test_planes_checksums_norms(dtype, m, n, k, vb_r, vb_c):
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A = torch.randn(m, k, generator=g, device="cuda")
    B = torch.randn(k, n, generator=g, device="cuda")
    d = abft.make_desc(m, n, k, dtype, vb_r, vb_c)
    L = abft.abft_workspace_layout(d)
    ws = torch.full((L.total,), 0x7f, dtype=torch.uint8, device="cuda")
    abft.abft_encode(d, A, B, ws)

    def region(off, shape, ld, dt):
        size = torch.empty(0, dtype=dt).element_size()
        x = ws[off:off + shape[0] * ld * size].view(dt).view(shape[0], ld)
        return x[:, :shape[1]].double().cpu().numpy()

    bf = torch.bfloat16
    assert np.array_equal(region(L.op_a, (m, k), L.op_a_ld, bf), A.to(bf).double().cpu().numpy())
    assert np.array_equal(region(L.op_b, (k, n), L.op_b_ld, bf), B.to(bf).double().cpu().numpy())
    a, b = A.double().cpu().numpy(), B.double().cpu().numpy()
    drop = 2.0 ** -16 if dtype == "bf16x3" else 2.0 ** -24
    sides = ((a, vb_r, L.acs, L.acs_plane, (L.acs_rows, k), L.acs_ld, L.nArow, L.nAblk, False),
             (b.T, vb_c, L.bcs, L.bcs_plane, (k, L.bcs_cols), L.bcs_ld, L.nBcol, L.nBblk, True))
    for x, vb, off, plane, shape, ld, nline, nblk, turn in sides:
        cs = sum(region(off + i * plane, shape, ld, bf) for i in range(L.planes))
        cs = cs.T if turn else cs
        ref, mag = blocks(x, vb)
        assert np.all(np.abs(cs - ref) <= (vb * U32 + drop) * mag)
        line = region(nline, (len(x), 1), 1, torch.float64)[:, 0]
        np.testing.assert_allclose(line, np.sqrt((x * x).sum(1)), rtol=(k + 2) * U32)
        norm = region(nblk, (len(ref) // 2, 4), 4, torch.float64)[:, 2:].reshape(-1)
        err = (vb * U32 + drop) * np.sqrt((mag * mag).sum(1))  # of the checksum rows' norms
        want = np.sqrt((ref * ref).sum(1))
        assert np.all(np.abs(norm - want) <= (k + 2) * U32 * want + err)
