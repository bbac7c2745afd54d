"""F(x) and positions where a model's numbers are far from a trained one's: weights that the split form's
FP16 part cannot hold, weights whose half is not a binary32 number, and slopes so steep that the low part
of the compiled form's pair carries many positions."""
from fractions import Fraction

import numpy as np
import pytest

from helpers import to_dev
from oracle import oracle as orc
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402


@pytest.mark.parametrize("h", [16, 32, 64])
@pytest.mark.parametrize("w2", [65_504.0, 65_520.0, 1e5, -1e5])
def test_wide_second_layer_weights_do_not_depend_on_the_warp(h, w2):
    """A second-layer weight beyond FP16's range makes the split form's product with the low part infinite
    or NaN; the epilogues must agree on it: a key's F(x) may not depend on its warp's other keys."""
    n = 4096
    near = (np.uint64(1 << 40) + W.uniform_u64(n, 5) % np.uint64(1 << 30)).astype(np.uint64)
    near[1::7] = np.uint64(1 << 40)  # x = 0: activations without a low part
    mixed = near.copy()
    far = np.arange(0, n, 32)  # one in every warp
    mixed[far] = np.uint64((1 << 63) + 12345)
    p = orc.init_params(2, h, h, 3)
    p[2 * h:2 * h + h * h:h + 1] = w2  # the diagonal
    f = nns.Model.create(orc.U64, 2, h, h, p, translate="ordbits", lo_bits=1 << 40, scale=2.0 ** -30)
    keep = np.ones(n, bool)
    keep[far] = False
    got = []
    for keys in (near, mixed):
        dk, kt = to_dev(keys)
        s, y = nns.predict(dk, f, precision="bf16x2", key_type=kt)
        got.append((s.cpu().numpy()[keep], y.cpu().numpy()[keep].view(np.uint32)))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("h", [16, 32, 64])
def test_output_weights_below_the_normal_range(h):
    """W3 = 2^-149 has no half; with z = 2^126 every unit adds exactly 2^-23."""
    p = np.zeros(h * h + 4 * h + 1, np.float32)
    p[2 * h + h * h:3 * h + h * h] = 2.0 ** 126  # b2
    p[3 * h + h * h:4 * h + h * h] = np.float32(2.0 ** -149)  # W3
    f = nns.Model.create(orc.U64, 2, h, h, p, translate="ordbits", lo_bits=0, scale=2.0 ** -30)
    dk, kt = to_dev(W.uniform_u64(1000, 7) % np.uint64(1 << 30))
    for precision in ("bf16", "bf16x2"):
        _, y = nns.predict(dk, f, precision=precision, key_type=kt)
        assert torch.equal(y, torch.full_like(y, h * 2.0 ** -23))


@pytest.mark.parametrize("log_slope", [1, 10, 20, 26])
@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("m", [1.25, 4294000.0])
def test_compiled_positions_of_steep_models(log_slope, dtype, m):
    """F = slope (x - c) around one key c, with few positions and with nearly 2^32. The pair of binary32
    holds A d, of magnitude slope * n m, to 47 bits and adds C of the same magnitude: positions are within
    2^-46 of that of the exact line's, and one of rounding."""
    n, slope = 1000, 2 ** log_slope
    step = max(1, 2 ** 32 // slope // n)
    b1 = np.float32(-((1 << 31) + 12345) / 2.0 ** 32)
    c = int(-Fraction(float(b1)) * 2 ** 32)  # the key where F leaves 0
    keys = np.minimum(c - 20 + step * np.arange(n, dtype=np.int64), (1 << 32) - 1).astype(
        np.uint32 if dtype == "u32" else np.uint64)
    f = nns.Model.create(getattr(orc, dtype.upper()), 1, 1, 0, np.array([1.0, b1, slope, 0.0], np.float32),
                         translate="ordbits", lo_bits=0, scale=2.0 ** -32)
    dk, kt = to_dev(keys)
    got = nns.predict(dk, f, m=m, precision="pwl", key_type=kt, want_y=False)[0].cpu().numpy()
    nm = Fraction(n) * Fraction(float(np.float32(m)))
    want = [min(max(int(nm * slope * (int(k) - c) / 2 ** 32 + Fraction(1, 2)), 0), int(nm)) if k > c else 0
            for k in keys]
    bound = 1 + int(nm * slope / 2 ** 46)
    assert np.abs(got - np.array(want)).max() <= bound
