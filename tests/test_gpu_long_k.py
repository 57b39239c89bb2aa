"""Products with a very long inner dimension: past the 65535 blocks of 32 and
256 entries that one grid covers, and past the 2^26 that one launch of the
digit-sliced product sums.  Operands of small integers at a few places
(the ends of blocks, grids and launches among them): the result is exact."""
import pytest

pytestmark = pytest.mark.gpu

PLACES = [0, 31, 255, 511, 32 * 65535 - 1, 32 * 65535, 256 * 65535 - 1, 256 * 65535, (1 << 26) - 1, 1 << 26]


def _operands(k, dtype):
    import torch
    a = torch.zeros(k, dtype=dtype, device="cuda")      # 1 x k
    b = torch.zeros(2 * k, dtype=dtype, device="cuda")   # k x 2, column-major
    at = sorted({p for p in PLACES if p < k} | {k - 1})
    want = [0j, 0j]
    for i, p in enumerate(at):
        x, y = complex(i + 1, 3 - i), [complex(2 * i - 5, 1), complex(-i, i + 2)]
        a[p], b[p], b[k + p] = x, y[0], y[1]
        want = [w + x * v for w, v in zip(want, y)]
    return a, b, want


@pytest.mark.parametrize("k", [2_097_120, 2_100_000, 16_776_960, 16_800_000, (1 << 26) + 1000])
def test_digit_sliced(k):
    import torch
    import paper_1404_1768_gb300 as fg
    a, b, want = _operands(k, torch.complex128)
    c = torch.full((2,), 10 - 1j, dtype=torch.complex128, device="cuda")
    lib = fg.load()
    nb = int(lib.feast_zgemm_oz_work_bytes(1, 2, k))
    work = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = lib.feast_zgemm_oz(1, 2, k, 2.0, 0.0, a.data_ptr(), 1, b.data_ptr(), k, 0.0, 1.0, c.data_ptr(), 1,
                            (work.data_ptr() + 255) // 256 * 256, nb, err.data_ptr(), 0)
    torch.cuda.synchronize()
    assert st == 0 and int(err.item()) == 0
    assert c.tolist() == [2 * w + 1j * (10 - 1j) for w in want]


@pytest.mark.parametrize("k", [2_097_120, 2_100_000, 16_800_000])
def test_complex64(k):
    import torch
    import paper_1404_1768_gb300 as fg
    a, b, want = _operands(k, torch.complex64)
    c = torch.zeros(2, dtype=torch.complex64, device="cuda")
    lib = fg.load()
    nb = int(lib.feast_cgemm_tc_scratch_bytes(1, 2, k, 1))
    work = torch.empty(nb, dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = lib.feast_cgemm_tc(1, 2, k, 1.0, 0.0, a.data_ptr(), 1, k, b.data_ptr(), k, 2 * k, 0.0, 0.0, c.data_ptr(), 1, 2, 1,
                            work.data_ptr(), nb, err.data_ptr(), 0)
    torch.cuda.synchronize()
    assert st == 0 and int(err.item()) == 0
    assert c.tolist() == want
