"""The binary32 forward kernels at the edges of their tiles: positions and F(x) bit for bit the
oracle's for every padded width, both key widths, sizes around a step and a tile, keys far outside
the training range, and normalisers that do and do not fit 32 bits."""
import numpy as np
import pytest

from helpers import lib_model, to_dev
from oracle import oracle as orc
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)
import paper_1907_08817_gb300 as nns  # noqa: E402


def _keys(dtype, n):
    k = W.lognormal_f32(n, n + 1, sigma=2.0)
    k[: n // 3] *= np.float32(-1.0)
    if n > 4:
        k[:4] = [np.inf, -np.inf, 0.0, -0.0]
    if dtype == "f64":
        return k.astype(np.float64) * 1.0000001
    if dtype == "u32":
        return k.view(np.uint32).copy()
    return k if dtype == "f32" else (k.view(np.uint32).astype(np.uint64) << np.uint64(31))


@pytest.mark.parametrize("arch", [(1, 3, 0), (1, 16, 0), (1, 32, 0), (1, 50, 0),
                                  (2, 6, 2), (2, 16, 9), (2, 32, 32), (2, 64, 64)])
@pytest.mark.parametrize("dtype", ["f32", "f64", "u32", "u64"])
def test_positions_at_tile_edges(arch, dtype):
    layers, h1, h2 = arch
    for n in (1, 127, 129, 257, 1023, 2048, 2049, 6161):
        keys = _keys(dtype, n)
        _, nm, _, _ = orc.sample_labels(keys[n // 4:] if n > 8 else keys, max(2, n // 2), 3, orc.ORDBITS)
        om = orc.Model(layers, h1, h2, nm, orc.init_params(layers, h1, h2, n))
        dk, kt = to_dev(keys)
        slots, y = nns.predict(dk, lib_model(om), key_type=kt)
        want, want_y = orc.predict_slots(keys, om)
        np.testing.assert_array_equal(slots.cpu().numpy().astype(np.uint32), want)
        np.testing.assert_array_equal(y.cpu().numpy().view(np.uint32), want_y.view(np.uint32))


def test_normaliser_beyond_32_bits():
    keys = W.uniform_f32(3000, 5)
    nm = orc.Norm(orc.F32, orc.ORDBITS, (1 << 33) + 5, 0.0, 2.0 ** -34, np.float32(0.0), np.float32(2.0 ** -34))
    om = orc.Model(1, 32, 0, nm, orc.init_params(1, 32, 0, 1))
    dk, _ = to_dev(keys)
    slots, y = nns.predict(dk, lib_model(om))
    want, want_y = orc.predict_slots(keys, om)
    np.testing.assert_array_equal(slots.cpu().numpy().astype(np.uint32), want)
    np.testing.assert_array_equal(y.cpu().numpy().view(np.uint32), want_y.view(np.uint32))
