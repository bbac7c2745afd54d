"""Buckets whose keys crowd into few bins, in blocks of 128, 256 and 512 threads: what the first bins hold,
what the finer bins cut by their counts hold, and what only the radix sort takes. The path of each input
follows from the bins' arithmetic, restated here."""
import numpy as np
import pytest

from helpers import bits, from_dev, stats_core, to_dev
from oracle import oracle as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402

BIN_MAX = 24


def _path(keys, threads):
    """Which of the three sorts a bucket of these keys takes."""
    width = keys.dtype.itemsize * 8
    k = [int(v) for v in keys]
    n, lo = len(k), min(k)
    br, ib = (max(k) - lo).bit_length(), (n - 1).bit_length()
    nlog = {128: 10, 256: 11, 512: 12}[threads]
    drop = max(br + ib - 32, 0)
    bs = max(br + ib - drop - nlog, 0)
    word = [((v - lo) >> (drop - ib)) if drop >= ib else ((((v - lo) << (ib - drop)) & 0xFFFFFFFF) | (i >> drop))
            for i, v in enumerate(k)]
    c = np.bincount([w >> bs for w in word], minlength=1 << nlog).reshape(threads, 8)
    if c.max() <= BIN_MAX and (c.astype(np.int64) ** 2).sum(1).max() <= BIN_MAX ** 2:
        return "bins"
    sh, fine = br - nlog, (1 << nlog) // 2
    if n > 8192 or sh <= 0 or br + ib <= nlog:
        return "radix"
    start = np.concatenate([[0], np.cumsum(c.ravel())[:-1]]) * fine // n
    start = [int(s) for s in start] + [fine]
    low = min(sh, 16)
    f = []
    for v in k:
        d = v - lo
        b = d >> sh
        part = (d >> (sh - low)) & ((1 << low) - 1)
        f.append(min(start[b] + ((start[b + 1] - start[b]) * part >> low), fine - 1))
    assert width >= br
    return "fine" if np.bincount(f).max() <= BIN_MAX else "radix"


def _keys(kind, dtype, n, nlog, rs):
    br = 8 * dtype.itemsize - 2  # the outlier sets the range
    one = 1 << (br - nlog)       # keys a first bin holds
    if kind == "even":           # every first bin its share
        v = (np.arange(n) * ((1 << br) // n)).astype(np.uint64)
    elif kind == "sixteen":      # sixteen keys in each of a few first bins
        v = (np.arange(n) * (one // 16)).astype(np.uint64)
    elif kind == "one":          # one first bin, spread over all of it
        v = (np.arange(n) * (one // n)).astype(np.uint64)
    else:                        # dense: neither first nor finer bins tell the keys apart
        v = np.arange(n).astype(np.uint64)
    v[-1] = np.uint64((1 << br) - 1)
    return rs.permutation(v).astype(dtype)


@pytest.mark.parametrize("kind,want", [("even", "bins"), ("sixteen", "fine"), ("one", "fine"), ("dense", "radix")])
@pytest.mark.parametrize("dtype,wlog,threads", [(np.uint32, 10, 128), (np.uint32, 11, 256), (np.uint32, 12, 512),
                                                (np.uint64, 9, 128), (np.uint64, 10, 256), (np.uint64, 12, 512)])
def test_crowded_buckets(kind, want, dtype, wlog, threads):
    dtype = np.dtype(dtype)
    rs = np.random.RandomState(wlog)
    n = 2 << wlog if threads < 512 else 5_900  # about what the block holds
    keys = _keys(kind, dtype, n, {128: 10, 256: 11, 512: 12}[threads], rs)
    assert _path(keys, threads) == want
    L, _, _ = orc.nm_split(n)
    slots = rs.randint(0, 1 << wlog, n).astype(np.int64)  # all of them in the first bucket
    dk, kt = to_dev(keys)
    ds = torch.from_numpy(slots.astype(np.uint32).view(np.int32)).cuda()
    st = nns.sort(dk, None, None, eps=3, tau=0, slots=ds, key_type=kt, bucket_log2=wlog)
    order, _, ost, _ = orc.nnsort(keys, slots, L, 3, 0, None)
    np.testing.assert_array_equal(bits(from_dev(dk, keys)), bits(order))
    assert stats_core(st) == stats_core(ost)


@pytest.mark.parametrize("eps", [0, 1, 3])
@pytest.mark.parametrize("n,traced", [(5_000, False), (40_000, False), (140_000, False), (140_000, True)])
def test_oversized_buckets_are_counted_without_rounds(eps, n, traced):
    """Every key in one bucket, above the polish's capacity from 5,000 u64 keys on, whichever form sorts it."""
    keys = np.random.RandomState(n).permutation(n).astype(np.uint64)
    dk, kt = to_dev(keys)
    ds = torch.zeros(n, dtype=torch.int32, device="cuda")
    r = nns.sort(dk, None, None, eps=eps, tau=0, slots=ds, key_type=kt, bucket_log2=12, fate=traced)
    st = r[0] if traced else r
    assert st["oversized_buckets"] == 1
    np.testing.assert_array_equal(from_dev(dk, keys), np.sort(keys))
