"""Models trained side by side in a server's batch are the models that each request gets alone: the conflict,
placed and out-of-order counts of its sort (which follow every parameter's bits) are the same."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402

COUNTS = ("t", "w_size", "placed", "out_of_order", "repaired")


@pytest.mark.parametrize("train,sizes", [
    # the cooperative launches of width 64 follow one another on one meeting counter
    (dict(layers=2, h1=64, h2=64, sample_n=9_000, batch=4096), [30_000, 9_500, 3_000, 1, 45_000]),
    (dict(layers=2, h1=50, h2=40, sample_n=500, batch=0), [700, 30_000, 64, 20_000]),
    # samples on both sides of 65,536: alone the small ones take one cluster launch
    (dict(layers=1, h1=32, h2=0, sample_n=70_000, batch=0), [80_000, 3_000, 65_536, 65_537, 17]),
    (dict(layers=1, h1=16, h2=0, sample_n=2_000, batch=333), [30_000, 1_000, 2, 25_000]),
    (dict(layers=2, h1=32, h2=32, sample_n=20_000, batch=0), [40_000, 16_384, 16_385, 500]),
    (dict(layers=2, h1=8, h2=5, sample_n=1_500, batch=0, monotone=1), [9_000, 1_500, 3, 70_000]),
])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_batched_models_are_the_models_trained_alone(train, sizes, dtype):
    train = dict(train, steps=12)
    dists = (W.lognormal_f32, W.uniform_f32, W.normal_f32)
    reqs = [dists[j % 3](n, 7 + n).astype(dtype) for j, n in enumerate(sizes)]
    with nns.Server(workers=1, max_batch=16, train=train) as srv:
        # the worker is busy with the first request while the others arrive, so that they share a batch
        first = W.lognormal_f32(4_000_000, 5).astype(dtype)
        work = [first] + [r.copy() for r in reqs]
        tickets = [srv.submit(a, seed=100 + j) for j, a in enumerate(work)]
        stats = [srv.wait(t)[0] for t in tickets]
    for j, r in enumerate(reqs):
        np.testing.assert_array_equal(work[j + 1], np.sort(r))
        dk = torch.from_numpy(r).cuda()
        f, _ = nns.train(dk, seed=101 + j, **dict(train, sample_n=min(train["sample_n"], r.size)))
        alone = nns.sort(dk, None, f, bucket_log2=12)
        assert {k: stats[j + 1][k] for k in COUNTS} == {k: alone[k] for k in COUNTS}, sizes[j]
