"""Training that is refused (a NaN in the sample, an unknown translate): the caller's loss array is left as it
was, and the steps are not run."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle as orc
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402
from paper_1907_08817_gb300 import _lib as L  # noqa: E402

# every route of the steps: one cluster launch, one cooperative launch, launches per step
ARCHS = [(1, 16, 0, 0), (1, 64, 0, 70_000), (2, 64, 64, 0), (2, 32, 32, 0), (2, 8, 8, 0)]


def _train(keys, steps, layers, h1, h2, batch, translate="ordbits"):
    """(status, loss array filled with -1 before the call, launches)"""
    o = nns._topts(layers=layers, h1=h1, h2=h2, sample_n=4000, steps=steps, batch=batch, seed=3, translate=translate)
    loss = np.full(steps, -1.0, np.float32)
    h = C.c_void_p()
    before = L.lib().nnsort_launch_count()
    rc = L.lib().nnsort_train(C.c_void_p(keys.data_ptr()), keys.numel(), orc.F32, C.byref(o), C.byref(h),
                              loss.ctypes.data_as(C.c_void_p), nns._stream())
    assert (rc == 0) == bool(h.value)
    if h.value:
        L.lib().nnsort_model_free(h)
    return rc, loss, L.lib().nnsort_launch_count() - before


@pytest.mark.parametrize("layers,h1,h2,batch", ARCHS)
def test_refused_training_leaves_the_losses_and_stops(layers, h1, h2, batch):
    keys = torch.from_numpy(W.lognormal_f32(20_000, 1)).cuda()
    bad = keys.clone()
    bad[5_000:15_000] = float("nan")  # half of the sample
    steps = 4000
    for k, translate, want in ((bad, "ordbits", -2), (keys, 7, -1)):
        rc, loss, launches = _train(k, steps, layers, h1, h2, batch, translate)
        assert rc == want
        np.testing.assert_array_equal(loss, np.full(steps, -1.0, np.float32))
        # launched ahead of the sample's status, if at all: a small part of two launches a step
        assert launches < steps, launches
    rc, loss, _ = _train(keys, 3, layers, h1, h2, batch)  # the next call is none the worse
    assert rc == 0 and (loss >= 0).all()


def test_a_refused_model_leaves_the_others_of_a_batch_alone():
    """The models beside it end as when trained by themselves: the same counts in the sort."""
    reqs = [W.lognormal_f32(n, n).astype(np.float64) for n in (30_000, 20_000, 25_000)]
    reqs[1][2_000:12_000] = np.nan
    opts = dict(layers=2, h1=32, h2=32, sample_n=2000, steps=20)
    with nns.Server(workers=1, max_batch=4, train=opts) as srv:
        work = [r.copy() for r in reqs]
        tickets = [srv.submit(r, seed=j) for j, r in enumerate(work)]
        for j, t in enumerate(tickets):
            if j == 1:
                with pytest.raises(nns.NNSortError) as e:
                    srv.wait(t)
                assert e.value.status == -2
                continue
            st, _ = srv.wait(t)
            dk = torch.from_numpy(reqs[j]).cuda()
            f, _ = nns.train(dk, seed=j, **opts)
            alone = nns.sort(dk, None, f)
            assert {k: st[k] for k in ("w_size", "placed", "out_of_order")} == \
                {k: alone[k] for k in ("w_size", "placed", "out_of_order")}
            np.testing.assert_array_equal(work[j], np.sort(reqs[j]))
