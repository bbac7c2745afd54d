"""The gradient sums of the batched small-model training against binary64, through one step whose update is
a power of two times the gradient: full batches of one chunk, and mini-batches of several chunks.

The bound. u = 2^-24. One rounding of a binary32 sum is some 0.43 u of it in the mean square. The samples go
to 64 rows of four lanes, each holding every 256th sample of the sorted sample, so that each partial sum is
about its share of the whole; a tree then adds the 256 lanes. With terms of one sign, the roundings of the
tree's levels add up to sqrt(1 + 1/2 + ...) < sqrt(2) of one, the lanes' own to less than 0.3, the factor W3
and the update to one each: at most 2.1 x 0.43 u, 0.9 u, of the sum of the terms' magnitudes. A sum that runs
through 64 rows one after another adds 64 / 3 such roundings in the square, 2 u."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402

def _errors(S, h, seed, batch):
    """|gradient - its binary64 value| over the sum of its terms' magnitudes, per parameter."""
    keys = torch.from_numpy(W.lognormal_f32(200_000, 3, sigma=2.0)).cuda()
    kw = dict(sample_n=S, h1=h, batch=batch, seed=seed)
    p0 = nns.train_batch([keys], steps=0, **kw)[0][0].describe()[1].astype(np.float64)
    # moments off and an epsilon far above |g|: the step is lr / eps = 2^30 times the gradient
    f, _ = nns.train_batch([keys], steps=1, lr=2.0 ** 70, beta1=0.0, beta2=0.0, adam_eps=2.0 ** 40, **kw)
    got = (p0 - f[0].describe()[1].astype(np.float64)) / 2.0 ** 30
    x, lab, _, _ = nns.sample_labels(keys, S, seed)
    x, lab = x.cpu().numpy(), lab.cpu().numpy()
    if batch:
        draws = W.rng_u64(W.stream_seed(seed, 3), 0, batch)  # the mini-batch stream
        at = np.array([int(v) * S >> 64 for v in draws])
        x, lab = x[at], lab[at]
    w1, b1, w3, b3 = p0[:h], p0[h:2 * h], p0[2 * h:3 * h], p0[3 * h]
    # activations and residuals in binary32, as the kernel rounds them: only the sums are compared
    y = np.full(x.size, np.float32(b3), np.float32)
    act = np.empty((x.size, h))
    for j in range(h):
        act[:, j] = np.maximum((w1[j] * x.astype(np.float64) + b1[j]).astype(np.float32), 0)
        y = (w3[j] * act[:, j] + y.astype(np.float64)).astype(np.float32)
    g = ((np.float32(2) * (y - lab)) * np.float32(1.0 / np.float32(x.size))).astype(np.float64)[:, None]
    on = (act > 0) * w3
    terms = np.concatenate([g * on * x[:, None], g * on, g * act, g], 1)
    size = np.abs(terms).sum(0)
    return (np.abs(got - terms.sum(0)) / np.where(size > 0, size, 1.0))[size > 0]


@pytest.mark.parametrize("S,batch", [(1000, 0), (4096, 0), (10_000, 0), (16_384, 0), (1000, 3000), (9000, 20_001)])
def test_gradient_sums_round_no_more_than_a_tree(S, batch):
    e = np.concatenate([_errors(S, h, seed, batch) for h in (8, 16, 32) for seed in range(6)])
    u = 2.0 ** -24
    assert np.sqrt((e ** 2).mean()) <= u, (np.sqrt((e ** 2).mean()) / u)
    assert e.max() <= 4 * u, e.max() / u
