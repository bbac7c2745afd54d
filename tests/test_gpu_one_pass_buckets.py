"""One-pass buckets (rounds, run split and sorted output in one block) against the oracle: outputs and
per-round counts, for key widths, payloads, round limits and buckets of one element up to ones that no
block holds; the same call with a row trace takes the two-kernel path and has to agree."""
import numpy as np
import pytest

from helpers import bits, from_dev, stats_core, to_dev
from oracle import oracle as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402


def _distinct(dtype, n, kind, rs):
    """n distinct keys (the tie rule of equal keys in different buckets is not the oracle's)."""
    if kind == "dense":          # words hold the whole composite key
        v = rs.permutation(n).astype(np.uint64) + np.uint64(1 << 20)
    elif kind == "wide":         # ranges of nearly the key's width: words drop index and key bits
        top = 31 if dtype in ("f32", "u32") else 62
        v = np.unique(rs.randint(0, 1 << top, 2 * n + 8).astype(np.uint64))
        v = rs.permutation(v)[:n]
    else:                        # clusters far apart: crowded bins, the radix sort
        v = (rs.randint(0, 3, n).astype(np.uint64) << np.uint64(28)) + rs.permutation(n).astype(np.uint64)
    if dtype == "u32":
        return v.astype(np.uint32)
    if dtype == "u64":
        return v
    if dtype == "f32":
        return (v.astype(np.uint32) & np.uint32(0x7F7FFFFF)).view(np.float32)  # finite
    return (v & np.uint64(0x7FEFFFFFFFFFFFFF)).view(np.float64)


def _check(keys, slots, L, eps, bucket_log2, fate):
    dk, kt = to_dev(keys)
    ds = torch.from_numpy(slots.astype(np.uint32).view(np.int32)).cuda()
    r = nns.sort(dk, None, None, eps=eps, tau=0, slots=ds, fate=fate, key_type=kt, bucket_log2=bucket_log2)
    return from_dev(dk, keys), (r[0] if fate else r)


@pytest.mark.parametrize("dtype", ["f32", "f64", "u32", "u64"])
@pytest.mark.parametrize("kind", ["dense", "wide", "clusters"])
@pytest.mark.parametrize("n,spread", [(1, 1.0), (2, 1.0), (513, 1.0), (4_097, 1.0), (9_001, 0.5), (30_011, 0.3),
                                      (30_011, 1.0)])
def test_counts_and_order_match_the_oracle(dtype, kind, n, spread):
    rs = np.random.RandomState(n)
    keys = np.unique(_distinct(dtype, n, kind, rs))
    keys = keys[rs.permutation(keys.size)]
    n = keys.size
    L, _, _ = orc.nm_split(n)
    rank = np.argsort(np.argsort(keys, kind="stable"), kind="stable")
    # positions near the order, noisy, squeezed into a share of the buckets (collisions, large buckets)
    slots = np.clip(rank * 1.25 * spread + rs.normal(0, 40, n), 0, L - 1).astype(np.int64)
    for eps, wlog in ((0, 12), (1, 12), (3, 12), (8, 9)):
        got, st = _check(keys, slots, L, eps, wlog, False)
        want, _, ost, _ = orc.nnsort(keys, slots, L, eps, 0, None)
        np.testing.assert_array_equal(bits(got), bits(want))
        assert stats_core(st) == stats_core(ost)
        traced, st2 = _check(keys, slots, L, eps, wlog, True)
        np.testing.assert_array_equal(bits(traced), bits(want))
        assert (st["repaired"], st["repair_ranges"]) == (st2["repaired"], st2["repair_ranges"])


@pytest.mark.parametrize("dtype", ["f32", "u32", "u64", "f64"])
@pytest.mark.parametrize("n", [700, 20_000, 140_000])
def test_equal_keys_keep_their_payload_order(dtype, n):
    """A model that sends everything to a few buckets: up to buckets that no block holds, all keys equal
    or nearly so, payload in input order."""
    rs = np.random.RandomState(n)
    np_t = {"f32": np.float32, "u32": np.uint32, "u64": np.uint64, "f64": np.float64}[dtype]
    code = {"f32": orc.F32, "f64": orc.F64, "u32": orc.U32, "u64": orc.U64}[dtype]
    for distinct in (1, 2, 300):
        keys = rs.randint(0, distinct, n).astype(np_t)
        f = nns.Model.create(code, 1, 8, 0, np.zeros(25, np.float32), translate="ordbits")
        dk, kt = to_dev(keys)
        pay = torch.arange(n, dtype=torch.int32, device="cuda")
        nns.sort(dk, pay, f, eps=2, key_type=kt)
        order = np.argsort(keys, kind="stable")
        np.testing.assert_array_equal(from_dev(dk, keys), keys[order])
        np.testing.assert_array_equal(pay.cpu().numpy(), order)


@pytest.mark.parametrize("n,spread", [(40_000, 1.0), (140_000, 0.02), (1_400_000, 0.01), (1_400_000, 1.0)])
@pytest.mark.parametrize("payload", [False, True])
def test_refused_calls_leave_the_arrays_untouched(n, spread, payload):
    """A NaN key, or a position out of range: buckets of every size, those that no block holds included."""
    rs = np.random.RandomState(n)
    keys = rs.standard_normal(n).astype(np.float32)
    L, _, _ = orc.nm_split(n)
    good = (rs.uniform(0, spread, n) * (L - 1)).astype(np.int64)
    for fault in ("nan", "slot"):
        k, sl = keys.copy(), good.copy()
        if fault == "nan":
            k[n // 3] = np.nan
        else:
            sl[n // 3] = L
        dk, kt = to_dev(k)
        pay = torch.arange(n, dtype=torch.int32, device="cuda") if payload else None
        ds = torch.from_numpy(sl.astype(np.uint32).view(np.int32)).cuda()
        f = nns.Model.create(orc.F32, 1, 8, 0, np.zeros(25, np.float32), translate="ordbits")
        before = dk.clone().view(torch.int32)
        for kw in ({"slots": ds}, {}) if fault == "nan" else ({"slots": ds},):
            with pytest.raises(nns.NNSortError):
                nns.sort(dk, pay, None if kw else f, eps=2, key_type=kt, **kw)
            assert torch.equal(dk.view(torch.int32), before)
            if payload:
                assert torch.equal(pay, torch.arange(n, dtype=torch.int32, device="cuda"))
