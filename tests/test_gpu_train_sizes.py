"""Training at the edges of its batches' rows: one-hidden-layer models whose steps run in one cluster
launch (rows of 64 samples dealt to 16 blocks) and, beyond 65,536 samples a step, in the per-step
kernels, against binary64 training; and models trained side by side in a server's batch."""
import numpy as np
import pytest

from oracle import oracle as orc
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402

# a step moves a weight by about lr; binary32 gradients of a sum of B terms are within B ulps of a term
# of the binary64 ones, which Adam's normalisation carries into the step: 2e-3 bounds 20 steps at lr 1e-2
TOL = 2e-3


@pytest.mark.parametrize("h1", [3, 16, 32, 64])
@pytest.mark.parametrize("S,batch", [(1, 0), (63, 0), (64, 0), (65, 0), (1023, 0), (1025, 0), (16_385, 0),
                                     (2000, 65), (2000, 5000), (66_000, 0)])
def test_one_layer_training_tracks_binary64(h1, S, batch):
    keys = W.lognormal_f32(30_000, 11)
    om, _, oloss = orc.train(keys, 1, h1, 0, orc.ORDBITS, sample_n=S, steps=20, batch=batch, lr=1e-2, seed=4)
    m, loss = nns.train(torch.from_numpy(keys).cuda(), layers=1, h1=h1, sample_n=S, steps=20, batch=batch,
                        lr=1e-2, seed=4)
    d, p = m.describe()
    assert d["lo_bits"] == om.norm.lo_bits and d["scale"] == om.norm.scale
    np.testing.assert_allclose(p, om.params, atol=TOL, rtol=0)
    np.testing.assert_allclose(loss, oloss, atol=TOL, rtol=TOL)


@pytest.mark.parametrize("arch", [(1, 32, 0), (2, 32, 32), (2, 8, 5)])
def test_server_trains_side_by_side_and_fails_alone(arch):
    layers, h1, h2 = arch
    sizes = [1, 2, 700, 20_001, 40_000]
    reqs = [W.lognormal_f32(n, 20 + n).astype(np.float64) for n in sizes]
    reqs[3][5_000:15_000] = np.nan  # half its sample: its model fails, the others train
    want = [np.sort(r) for r in reqs]
    with nns.Server(workers=1, max_batch=8, train=dict(layers=layers, h1=h1, h2=h2, sample_n=1500, steps=5)) as srv:
        work = [r.copy() for r in reqs]
        tickets = [srv.submit(r, seed=j) for j, r in enumerate(work)]
        for j, t in enumerate(tickets):
            if j == 3:
                with pytest.raises(nns.NNSortError) as e:
                    srv.wait(t)
                assert e.value.status == -2
                np.testing.assert_array_equal(work[j].view(np.uint64), reqs[j].view(np.uint64))
            else:
                srv.wait(t)
                np.testing.assert_array_equal(work[j].view(np.uint64), want[j].view(np.uint64))


@pytest.mark.parametrize("h", [5, 32])  # padded and exact widths
def test_captured_passes_replay_the_same_bits(h):
    """Buffers of a captured call belong to its graph, not to the library's pool."""
    rs = np.random.RandomState(h)
    p, x, gy = (torch.from_numpy(rs.uniform(-1, 1, n).astype(np.float32)).cuda() for n in (3 * h + 1, 4097, 4097))

    def both():
        return (nns.mlp_forward(p, x, 1, h, 0),) + nns.mlp_backward(p, x, gy, 1, h, 0)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = both()
    want = both()
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        for a, b in zip(got, want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("n", [1, 63, 65, 4096, 16_384, 16_385, 32_768, 32_769])
def test_block_product_gradient_at_the_edges_of_its_split(n):
    """Batches of up to 256 chunks, 512 and beyond take one, two and four chunks of 64 samples per block.
    Bound: the gradient's stated 1e-4 of the largest component against binary64."""
    rs = np.random.RandomState(n)
    h = 32
    p, x, lab = (torch.from_numpy(rs.uniform(-1, 1, m).astype(np.float32)).cuda() for m in (h * h + 4 * h + 1, n, n))
    loss, gp = nns.mlp_loss_grad(p, x, lab, 2, h, h)
    q = p.double().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(q, [h, h, h * h, h, h, 1])
    a = torch.relu(x.double()[:, None] * w1 + b1)
    y = torch.relu(a @ w2.view(h, h).T + b2) @ w3 + b3
    want = (y - lab.double()).square().mean()
    want.backward()
    assert abs(loss.item() - want.item()) <= 1e-5 * want.item()
    assert (gp.double() - q.grad).abs().max().item() <= 1e-4 * q.grad.abs().max().item()
