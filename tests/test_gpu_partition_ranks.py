"""The partition pass's stable ranks where they can go wrong: few distinct digits (whole warps on one
match word), partial tiles, one element, every digit width, payloads that tell equal keys apart."""
import numpy as np
import pytest

from helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402


@pytest.mark.parametrize("dtype", [np.uint32, np.uint64, np.float32, np.float64])
@pytest.mark.parametrize("kind", ["one", "two", "sorted", "reversed", "random"])
@pytest.mark.parametrize("n", [1, 31, 33, 4095, 4096, 4097, 70_001])
def test_radix_sort_is_stable(dtype, kind, n):
    rs = np.random.RandomState(n)
    if kind == "one":
        k = np.full(n, 0x01020304)
    elif kind == "two":
        k = np.where(rs.rand(n) < 0.5, 7, 0x7F000007)
    elif kind == "random":
        k = rs.randint(0, 1 << 31, n)
    else:
        k = np.arange(n) // 3 * 257
        k = k[::-1] if kind == "reversed" else k
    k = np.ascontiguousarray(k.astype(dtype))
    if dtype in (np.float32, np.float64) and kind == "random":
        k *= np.where(rs.rand(n) < 0.5, -1, 1).astype(dtype)
    order = np.argsort(k, kind="stable")
    for pay in (False, True):
        dk, kt = to_dev(k)
        dp = torch.arange(n, dtype=torch.int32, device="cuda") if pay else None
        nns.radix_sort(dk, dp, key_type=kt)
        np.testing.assert_array_equal(from_dev(dk, k), k[order])
        if pay:
            np.testing.assert_array_equal(dp.cpu().numpy(), order)


@pytest.mark.parametrize("bucket_log2", [9, 10, 11, 12])
@pytest.mark.parametrize("n", [400, 6_000, 90_001, 1_500_000])
def test_bucket_digit_widths(bucket_log2, n):
    """Positions straight from the keys: one to two passes of 1 to 9 bits, stable inside a bucket."""
    g = torch.Generator(device="cuda").manual_seed(n)
    k = torch.randint(0, 50_000, (n,), generator=g, device="cuda").to(torch.float32)
    L = int(n * 1.25) + 1
    slots = (k.double() / 50_000 * (L - 1)).to(torch.int32)
    work = k.clone()
    pay = torch.arange(n, dtype=torch.int32, device="cuda")
    nns.sort(work, pay, slots=slots, eps=1, bucket_log2=bucket_log2)
    want = torch.sort(k, stable=True)
    assert torch.equal(work, want.values)
    assert torch.equal(pay, want.indices.to(torch.int32))
