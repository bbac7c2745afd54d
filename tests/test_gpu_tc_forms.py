"""The tensor-core predict's two epilogues and its ragged ends: a warp that holds a key far outside the
training range takes the general epilogue, and must give its other keys the very same F(x) and positions
as the plain one; sizes around a sub-tile agree with longer calls."""
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


def _model(h, scale=2.0 ** -30, seed=3):
    return nns.Model.create(orc.U64, 2, h, h, orc.init_params(2, h, h, seed), translate="ordbits",
                            lo_bits=1 << 40, scale=scale)


@pytest.mark.parametrize("h", [16, 32, 64])
@pytest.mark.parametrize("precision", ["bf16", "bf16x2"])
def test_epilogues_agree(h, precision):
    n = 4096
    near = (np.uint64(1 << 40) + W.uniform_u64(n, 5) % np.uint64(1 << 30)).astype(np.uint64)
    mixed = near.copy()
    far = np.arange(0, n, 32)  # one in every warp
    mixed[far] = np.uint64((1 << 63) + 12345)
    f = _model(h)
    dk, kt = to_dev(near)
    s0, y0 = nns.predict(dk, f, precision=precision, key_type=kt)
    dk, kt = to_dev(mixed)
    s1, y1 = nns.predict(dk, f, precision=precision, key_type=kt)
    keep = np.ones(n, bool)
    keep[far] = False
    np.testing.assert_array_equal(s0.cpu().numpy()[keep], s1.cpu().numpy()[keep])
    np.testing.assert_array_equal(y0.cpu().numpy()[keep].view(np.uint32), y1.cpu().numpy()[keep].view(np.uint32))


@pytest.mark.parametrize("h", [16, 32, 64])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 257, 100_003])
def test_ragged_ends(h, n):
    keys = (np.uint64(1 << 40) + W.uniform_u64(200_000, 6) % np.uint64(1 << 30)).astype(np.uint64)
    f = _model(h)
    dk, kt = to_dev(keys)
    _, y = nns.predict(dk, f, precision="bf16x2", key_type=kt)
    slots, yn = nns.predict(dk[:n], f, precision="bf16x2", key_type=kt)
    assert torch.equal(y[:n].view(torch.int32), yn.view(torch.int32))
    # the positions' arithmetic, from the oracle
    nm_hi, nm_lo = np.float32(n * 1.25), np.float32(n * 1.25 - np.float64(np.float32(n * 1.25)))
    L = orc.nm_split(n)[0]
    some = range(0, n, max(1, n // 50))
    want = [orc.slot1(float(yn[i]), float(nm_hi), float(nm_lo), L) for i in some]
    assert [int(slots[i]) for i in some] == want
