"""Calls of different sizes side by side in several threads, each on a stream of its own: kernels whose
launches take different amounts of shared memory must not meet in the function's limit."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402


def _side_by_side(makers, rounds):
    """Every maker's call, `rounds` times, in a thread of its own; the first failures."""
    failures, ready = [], threading.Barrier(len(makers))

    def body(make):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                call = make(stream)
                ready.wait(60)
                for _ in range(rounds):
                    call()
        except Exception as e:  # noqa: BLE001
            failures.append(f"{type(e).__name__}: {e}")

    threads = [threading.Thread(target=body, args=(m,)) for m in makers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures[:3]


def _sort(n, bucket_log2=0, precision="fp32", h=8, fate=False):
    keys = W.lognormal_f32(n, 3)
    want = torch.from_numpy(np.sort(keys)).cuda()
    src = torch.from_numpy(keys).cuda()
    model, _ = nns.train(src, layers=2 if h > 8 else 1, h1=h, h2=h if h > 8 else 0, sample_n=500, steps=10)
    torch.cuda.synchronize()

    def make(stream):
        work = torch.empty_like(src)

        def call():
            work.copy_(src)
            nns.sort(work, None, model, precision=precision, bucket_log2=bucket_log2, fate=fate, stream=stream)
            assert torch.equal(work, want)

        return call

    return make


def _train(sample, batch):
    keys = torch.from_numpy(W.lognormal_f32(20_000, 5)).cuda()
    torch.cuda.synchronize()

    def make(stream):
        if batch:
            return lambda: nns.train_batch([keys], sample_n=sample, h1=8, steps=1, stream=stream)
        return lambda: nns.train(keys, layers=1, h1=8, sample_n=sample, steps=1, stream=stream)

    return make


@pytest.mark.parametrize("case", ["repairs", "two kernels", "compiled", "training", "batched training"])
def test_calls_of_different_sizes_side_by_side(case):
    makers = {
        "repairs": lambda: [_sort(n) for n in (12_000, 18_000, 13_000, 17_000, 14_000, 30_000, 9_000, 16_000)],
        "two kernels": lambda: [_sort(3_000, w, fate=w < 13) for w in (9, 14, 10, 13, 9, 14, 11, 13)],
        "compiled": lambda: [_sort(3_000, 12, "pwl", h) for h in (8, 64, 16, 48, 8, 64, 24, 32)],
        "training": lambda: [_train(s, False) for s in (100, 18_000, 1_500, 12_000, 200, 16_000, 3_000, 9_000)],
        "batched training": lambda: [_train(s, True) for s in (20, 1_000, 2_000, 4_000, 5_000, 16_000, 60, 500)],
    }[case]()
    _side_by_side(makers, 250)
