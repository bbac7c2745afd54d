"""Launches of a sort: paths for buckets that an array does not hold are not launched."""
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

# f(x) = x on u32 keys: positions as even as the keys
LINE = np.array([1.0, 0.0, 1.0, 0.0], np.float32)


def _launches(call):
    before = L.lib().nnsort_launch_count()
    call()
    return L.lib().nnsort_launch_count() - before


@pytest.mark.parametrize("payload", [False, True])
@pytest.mark.parametrize("n", [9_000, 13_000, 20_000, 40_000, 65_536, 65_537, 200_000])
def test_an_even_array_takes_one_launch_a_stage(n, payload):
    """Predict, one partition pass of three kernels (four from 65,537 keys on), bounds and order, buckets,
    finalize, seam, repairs: also for arrays that could hold a bucket no block holds. Arrays that one block
    can hold (at most 18,848 keys) do not wait for the counts, and launch the two kernels of heavy buckets."""
    keys = np.random.RandomState(n).randint(0, 1 << 32, n).astype(np.uint32)
    f = nns.Model.create(orc.U32, 1, 1, 0, LINE, translate="ordbits", lo_bits=0, scale=2.0 ** -32)
    dk, kt = to_dev(keys)
    pay = torch.arange(n, dtype=torch.int32, device="cuda") if payload else None
    assert _launches(lambda: nns.sort(dk, pay, f, key_type=kt, bucket_log2=12)) <= (11 if n <= 18_848 else 9 if n <= 65_536 else 10)
    order = np.argsort(keys, kind="stable")
    np.testing.assert_array_equal(bits(from_dev(dk, keys)), keys[order])
    if payload:
        np.testing.assert_array_equal(pay.cpu().numpy(), order)
