"""Per-component networks with pre-activations far outside the range of the exponential (|z| up to 1e30,
and around +-88, where 2^(-z log2 e) leaves FP32's normal range), against FP64."""
import numpy as np
import pytest

from oracle import fnet
from tests.helpers import TOL_F32, assert_parity
from tests.test_gpu_fnet import _configs, _flat

pytestmark = pytest.mark.gpu

BIAS = [-1e30, -1e4, -200.0, -104.0, -90.0, -89.0, -88.5, -88.0, -87.5, -87.0, -50.0, 0.0, 50.0, 88.0, 200.0, 1e4]


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("width,depth", [(16, 1), (32, 2), (64, 1)])
def test_saturated_activations(width, depth):
    import torch

    from paper_2402_12199_gb300 import api

    flat = _flat(width, depth, 5)
    n = fnet.net_size(width, depth)
    wo = n - 3 - width
    for c in range(5):
        o = c * n
        b = np.resize(np.array(BIAS), width)
        flat[o + 8 + 4 * width:o + 8 + 5 * width] = b
        # the next weights by 1 / silu: every unit's contribution is of the same size
        scale = 1.0 / np.maximum(1.0, b)
        if depth > 1:
            flat[o + 8 + 5 * width:o + 8 + 5 * width + width * width] *= np.tile(scale, width)
        else:
            flat[o + wo:o + wo + width] *= scale
    f = api.FNet(width, depth)
    f.set_params(flat)
    s, q = _configs(700, 41)
    cfg = np.zeros((len(s), 8), np.float32)
    cfg[:, :3], cfg[:, 4:] = s, q
    out = f.pairs(torch.from_numpy(cfg).cuda()).double().cpu().numpy()
    assert np.isfinite(out).all()
    with np.errstate(over="ignore"):
        Fj, ti, tj, _ = fnet.predict(fnet.unpack(flat.astype(np.float64), width, depth), s.astype(np.float64),
                                     q.astype(np.float64))
    for a, ref in ((0, Fj), (4, ti), (8, tj)):
        assert_parity(out[:, a:a + 3], ref, TOL_F32)
