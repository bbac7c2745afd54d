"""Statistics of a refused sort (a NaN key, a position out of range): the conflict arrays' sizes that the
positions give, for buckets of every size."""
import ctypes as C

import numpy as np
import pytest

from helpers import to_dev
from oracle import oracle as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402
from paper_1907_08817_gb300 import _lib as L  # noqa: E402


@pytest.mark.parametrize("fault,want", [("nan", -2), ("slot", -1)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,spread", [(1, 1.0), (300, 1.0), (40_000, 1.0), (140_000, 0.02), (1_400_000, 0.01),
                                      (1_400_000, 1.0)])
def test_refused_sorts_count_their_conflicts(fault, want, dtype, n, spread):
    if fault == "slot" and dtype == np.float64:
        pytest.skip("the position check does not depend on the key")
    rs = np.random.RandomState(n)
    keys = rs.standard_normal(n).astype(dtype)
    lim, _, _ = orc.nm_split(n)
    slots = (rs.uniform(0, spread, n) * (lim - 1)).astype(np.int64)
    eps = 3
    if fault == "nan":
        keys[n // 3] = np.nan
        held = np.bincount(slots)
    else:
        slots[n // 3] = lim  # counted at position 0
        held = np.bincount(np.where(slots == lim, 0, slots))
    # each iteration stores one element of every position that holds any; it ends after eps or with none left
    w = [int(np.maximum(held - r, 0).sum()) for r in range(eps + 1)]
    t = next((r for r in range(eps) if w[r] == 0), eps)
    dk, _ = to_dev(keys)
    ds = torch.from_numpy(slots.astype(np.uint32).view(np.int32)).cuda()
    o = nns._sopts(1.25, eps, 0, "fp32", 12, ds, None, False)
    st = L.Stats()
    rc = L.lib().nnsort_sort(C.c_void_p(dk.data_ptr()), None, n, orc.F32 if dtype == np.float32 else orc.F64, None,
                             C.byref(o), C.byref(st), nns._stream())
    assert rc == want
    got = st.as_dict()
    assert (got["t"], got["w_size"]) == (t, w[:t + 1])
    assert got["placed"] == [w[r] - w[r + 1] for r in range(t)]
    assert got["repaired"] == 0 and not any(got["out_of_order"])
