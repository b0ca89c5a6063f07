"""The FP32 network kernel's two tile sizes at width 128: the same bits for every pair, at the edges of
the tiles and of the rule that chooses between them (a tile per SM, partly filled last rounds)."""
import numpy as np
import pytest

from paper_2402_12199_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("depth", [1, 2, 3, 4])
def test_tile_sizes_give_the_same_bits(depth):
    import torch

    from paper_2402_12199_gb300 import api

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mu, isd = inputs.feature_normalisation(5.0, 9.43)
    m = api.MLP(128, depth)
    m.set_params(inputs.mlp_params(128, depth, depth, mu=mu, inv_sd=isd, e_scale=1.3, e_shift=0.2))
    whole = 64 * sms  # exactly a 64-pair tile per SM
    c7 = inputs.pair_configs(2 * whole, depth, 5.0, 9.4)
    cfg = np.zeros((2 * whole, 8), np.float32)
    cfg[:, :3], cfg[:, 4:] = c7[:, :3], c7[:, 3:]
    cfg = torch.from_numpy(cfg).cuda()
    ref = [torch.cat(x) for x in zip(*(m.pairs(c, "fp32", grad=True) for c in cfg.split(whole)))]
    for n in (1, 31, 32, 33, 32 * sms, 32 * sms + 1, whole + 1, 96 * sms - 31, 96 * sms, 96 * sms + 1):
        out, g = m.pairs(cfg[:n].contiguous(), "fp32", grad=True)
        assert torch.equal(out, ref[0][:n]) and torch.equal(g, ref[1][:n])
