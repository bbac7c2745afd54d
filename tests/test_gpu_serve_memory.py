"""The server's memory while a batch's models train side by side, each with its rows of partial gradients."""
import threading
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402

# 262,144 samples a step of a 1-32-32-1 model: 1,024 rows of 1,153 binary32 sums, 4.7 MB
TRAIN = dict(layers=2, h1=32, h2=32, sample_n=300, steps=10, batch=1 << 18)


def test_models_side_by_side_stay_within_the_budget():
    """256 requests of 1,000 keys: the batch that would take all of them
    takes 1.2 GB for the sums alone. Allowed: the budget, what the pool keeps (256 MB), and as much again."""
    rs = np.random.RandomState(0)
    arrays = [rs.standard_normal(1000).astype(np.float32) for _ in range(256)]
    nns.release()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    low, stop = [free0], threading.Event()

    def watch():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])
            time.sleep(2e-4)

    t = threading.Thread(target=watch)
    with nns.Server(workers=1, max_batch=256, hbm_budget=384 << 20, train=TRAIN) as srv:
        t.start()
        tickets = [srv.submit(a, seed=i) for i, a in enumerate(arrays)]
        for tk in tickets:
            srv.wait(tk)
    stop.set()
    t.join()
    assert all((np.diff(a) >= 0).all() for a in arrays)
    assert free0 - low[0] <= (384 + 2 * 256) << 20


def test_a_request_that_fits_without_its_models_sums_is_served():
    a = np.random.RandomState(1).standard_normal(50_000).astype(np.float32)
    want = np.sort(a)
    # its arrays, its share of the sort's workspace and its sample
    fits = a.nbytes + nns.workspace_bytes(a.size, nns.F32) + 300 * 24 + (1 << 20)
    with nns.Server(hbm_budget=fits, train=TRAIN) as srv:
        srv.wait(srv.submit(a, seed=2))
    np.testing.assert_array_equal(a, want)
    with nns.Server(hbm_budget=fits - 1, train=TRAIN) as srv:
        with pytest.raises(nns.NNSortError) as e:
            srv.submit(a)
        assert e.value.status == -4
