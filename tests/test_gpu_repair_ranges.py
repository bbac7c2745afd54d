"""Seam repairs at the sizes where they change hands: a block on chip, the multi-block sort; in arrays of at
most 65,536 elements, whose blocks take as much as one alone on its SM can hold, and in larger ones."""
import numpy as np
import pytest

from helpers import bits, from_dev, to_dev
from oracle import oracle as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402
from paper_1907_08817_gb300 import _lib as L  # noqa: E402


def _sort(dtype, n, length):
    """n keys at their positions but for `length` consecutive ones, whose positions run backward: one range
    of exactly that many elements. Returns the launches of the sort."""
    rs = np.random.RandomState(length)
    v = np.arange(n, dtype=np.int64) * 37 + 5
    keys = (v + (1 << 40 if dtype.itemsize == 8 else 0)).astype(dtype)  # ascending
    a = (n - length) // 2
    rank = np.arange(n)
    rank[a:a + length] = rank[a:a + length][::-1]
    order = rs.permutation(n)
    shuffled = keys[order]
    Lp, _, _ = orc.nm_split(n)
    slots = np.minimum(np.floor(rank * 1.25), Lp - 1).astype(np.int64)[order]
    dk, kt = to_dev(shuffled)
    ds = torch.from_numpy(slots.astype(np.uint32).view(np.int32)).cuda()
    before = L.lib().nnsort_launch_count()
    st = nns.sort(dk, None, None, eps=1, tau=0, slots=ds, key_type=kt, bucket_log2=12)
    count = L.lib().nnsort_launch_count() - before
    np.testing.assert_array_equal(bits(from_dev(dk, shuffled)), bits(keys))
    assert (st["repair_ranges"], st["repaired"]) == (1, length)
    return count


@pytest.mark.parametrize("dtype", [np.uint32, np.float32, np.uint64, np.float64])
def test_ranges_around_a_blocks_capacity(dtype):
    dtype = np.dtype(dtype)
    # what a block holds: alone on its SM, and with a second one beside it (and at most 8,192)
    alone, beside = (18_848, 8_192) if dtype.itemsize == 4 else (13_808, 5_984)
    for n, cap in ((40_000, alone), (65_536, alone), (65_537, beside)):
        few = [_sort(dtype, n, m) for m in (cap - 1, cap)]
        many = [_sort(dtype, n, m) for m in (cap + 1, cap + 1_000)]
        assert max(few) < min(many)


@pytest.mark.parametrize("dtype", [np.float32, np.uint64])
def test_many_ranges_with_rows(dtype):
    """Hundreds of repairs with rows carried, each a sort by row and then by key over the same tables: the
    output, with its payload and fates, is the stable sort run after run."""
    n, rs = 3_000_001, np.random.RandomState(77)
    rank = rs.permutation(n)
    keys = (rank // 2).astype(dtype)  # pairs of equal keys, which the rows order
    lim, _, _ = orc.nm_split(n)
    slots = (rank * 5 // 4 + rs.randint(-1, 2, n)).astype(np.int64)
    idx = rs.choice(n, 300, replace=False)
    slots[idx] += rs.randint(-3000, 3000, 300)
    slots = np.clip(slots, 0, lim - 1)
    src, kt = to_dev(keys)
    ds = torch.from_numpy(slots.astype(np.uint32).view(np.int32)).cuda()
    order = torch.from_numpy(np.argsort(keys, kind="stable").astype(np.int32)).cuda()
    want = src[order.long()]
    for _ in range(24):
        dk, pay = src.clone(), torch.arange(n, dtype=torch.int32, device="cuda")
        st, _ = nns.sort(dk, pay, None, slots=ds, eps=3, tau=0, fate=True, key_type=kt, bucket_log2=9)
        assert st["repair_ranges"] > 200
        assert torch.equal(dk, want) and torch.equal(pay, order)
