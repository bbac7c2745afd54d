"""Arrays of few buckets, whose per-bucket steps share launches of one block (up to 1,024 buckets), on both
sides of that limit; and the compiled form's 32-bit search at the ends of the keys' range."""
import numpy as np
import pytest

from helpers import bits, from_dev, lib_model, stats_core, to_dev
from oracle import oracle as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402


@pytest.mark.parametrize("dtype", [np.uint32, np.uint64])
@pytest.mark.parametrize("buckets", [1, 2, 31, 32, 33, 1023, 1024, 1025])
@pytest.mark.parametrize("noise", [0, 400, 40_000])
def test_bucket_counts_around_one_block(dtype, buckets, noise):
    """Positions off by up to `noise`: no seam to repair, neighbouring buckets, nearly the whole array.
    Half of the buckets stay empty in the middle of the range."""
    n = (512 * buckets - 1) * 4 // 5
    L, _, _ = orc.nm_split(n)
    assert (L + 511) // 512 == buckets
    rs = np.random.RandomState(buckets)
    keys = rs.permutation(n).astype(dtype) * dtype(37)
    rank = np.argsort(np.argsort(keys))
    pos = np.where(rank < n // 2, rank * 0.625, L - 1 - (n - 1 - rank) * 0.625)
    slots = np.clip(pos + rs.uniform(-noise, noise, n), 0, L - 1).astype(np.int64)
    dk, kt = to_dev(keys)
    ds = torch.from_numpy(slots.astype(np.uint32).view(np.int32)).cuda()
    for eps in (1, 3):
        dk.copy_(to_dev(keys)[0])
        st = nns.sort(dk, None, None, eps=eps, tau=0, slots=ds, key_type=kt, bucket_log2=9)
        want, _, ost, _ = orc.nnsort(keys, slots, L, eps, 0, None)
        np.testing.assert_array_equal(bits(from_dev(dk, keys)), bits(want))
        assert stats_core(st) == stats_core(ost)


@pytest.mark.parametrize("dtype", ["u32", "f32"])
@pytest.mark.parametrize("n", [7, 2_047, 2_049, 40_000])
def test_compiled_positions_at_the_ends_of_32_bit_keys(dtype, n):
    """Within one position of the binary64 model's, and equal but for rounding at half-positions (at most
    one key in 10,000, or one): the compiled form's stated accuracy."""
    rs = np.random.RandomState(n)
    keys = rs.randint(0, 1 << 32, n).astype(np.uint32)
    keys[:4] = [0, 1, 0xFFFFFFFF, 0xFFFFFFFE]
    if dtype == "f32":
        keys[:4] = [0xFF7FFFFF, 0x80000000, 0x7F7FFFFF, 0]       # lowest, -0, largest, +0
        keys = keys.view(np.float32)
        keys[np.isnan(keys)] = 1.5
    for h in (1, 24):
        om, _, _ = orc.train(keys, 1, h, 0, orc.ORDBITS, sample_n=max(7, n // 10), steps=40, seed=3)
        dk, kt = to_dev(keys)
        got = nns.predict(dk, lib_model(om), precision="pwl", key_type=kt, want_y=False)[0].cpu().numpy()
        L, hi, lo = orc.nm_split(n, 1.25)
        y = orc.mlp_forward_f64(1, h, 0, om.params, orc.translate_f64(keys, om.norm))
        s = np.floor(np.minimum(y, 1.0) * (float(np.float32(hi)) + float(np.float32(lo))) + 0.5)
        want = np.clip(np.where(y > 0, s, 0), 0, L - 1).astype(np.int64)
        d = np.abs(got - want)
        assert d.max() <= 1 and (d != 0).sum() <= max(1, n // 10_000)
