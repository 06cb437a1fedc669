"""Size of the binary64 workspace, from the plan alone (no GPU is touched): the residue planes
of the tensor-core product stay within their budget for every shape, and short K loops keep
none, so a problem that the FP64 pipe alone could hold still fits."""
import pytest

from paper_0806_3121_gb300 import abft, build

DEVICE = 284208 << 20
MIB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return abft.load()


def sizes(m, n, k, vb=128, p=0):
    """(bytes of A, B and C; bytes of the planes' regions: the workspace below the scratch
    that is not checksums, norms or carried bounds)."""
    d = abft.make_desc(m, n, k, "f64", min(vb, m), min(vb, n), p, p)
    L = abft.abft_workspace_layout(d)
    return 8 * (m * k + k * n + m * n), L.scratch - (L.car_b + 16 * -(-n // min(vb, n))), L.total


# beside the planes: the residues of each CTA's tile, scales, maxima, chunk masks
BESIDE = 170 * MIB


@pytest.mark.parametrize("shape", [
    (128, 128, 128), (300, 3, 3000), (1, 1 << 20, 300), (1 << 22, 8, 64), (8, 1 << 22, 100), (1 << 20, 1, 60),
    (1 << 22, 1, 48), (400000, 8, 64), (16, 16, 1 << 20), (1, 1, 1 << 22), (4096, 4096, 4096),
    (20000, 20000, 20000), (60000, 60000, 60000), (100000, 100000, 100000)])
def test_planes_stay_within_the_budget(shape):
    held, planes, _ = sizes(*shape)
    # per-row records and masks of the longest sides: 8 + 1 bytes and maxima (4 bytes per 256)
    lines = sum(shape[:2]) + 1024
    assert planes <= min(12 << 30, 5 * held + 256 * MIB) + BESIDE + 320 * lines


@pytest.mark.parametrize("shape", [(1 << 22, 8, 16), (1 << 21, 1, 1), (2048, 2048, 47),
                                   (64, 65536, 32), (1 << 22, 1, 48)])
def test_no_planes_for_short_k_or_mostly_padding(shape):
    _, planes, _ = sizes(*shape)
    assert planes <= MIB


def test_operands_that_nearly_fill_the_device_keep_their_room():
    for s in (105000, 107000, 108500):
        held, _, total = sizes(s, s, s, vb=512)
        free = sizes(s, s, 1, vb=512)  # k = 1: checksums of C alone, no planes
        assert free[1] <= MIB
        assert held + total <= DEVICE


def test_ordinary_sizes_keep_one_panel():
    """Planes of the whole K: 18 planes of 2 bytes for (rows + columns) x K."""
    for m, n, k, p in ((512, 512, 512, 0), (1000, 1501, 777, 0), (4096, 4096, 4096, 8),
                       (300, 300, 4096, 0), (256, 4096, 4096, 0), (11264, 11264, 11264, 22)):
        _, planes, _ = sizes(m, n, k, vb=512 if p else 32, p=p)
        assert planes >= 36 * (m + n) * k
