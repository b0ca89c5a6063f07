"""The fused training gradients against the FP64 oracle at the edges of their tiles: batches of one
sample, one below, at and above a tile, and beyond one tile per CTA; every width, depths 1 to 4 (both
tile forms of the energy network), the per-component networks' widths and depths.  The bound is the
one of the FP32 gradients elsewhere in these tests, 1e-5 of the gradient's norm: sums of up to 10^4
FP32 terms in fixed partial sums of at most 64 samples lose a few 2^-24 each."""
import numpy as np
import pytest

from oracle import fnet, nn
from paper_2402_12199_gb300 import inputs
from tests.helpers import rel_err
from tests.test_gpu_fnet import _flat, _sampled

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("width,depth,batch", [
    (64, 1, 31), (64, 2, 64), (64, 4, 33), (128, 1, 17), (128, 2, 16), (128, 3, 15), (128, 4, 100),
    (128, 3, 2433), (128, 3, 4897), (256, 1, 9), (256, 3, 8), (256, 3, 1300), (256, 4, 7),
])
def test_energy_network_gradient(width, depth, batch):
    import torch

    from paper_2402_12199_gb300 import api

    mu, isd = inputs.feature_normalisation(5.0, 9.43)
    flat = inputs.mlp_params(width, depth, width + depth, mu=mu, inv_sd=isd, e_scale=1.3, e_shift=0.2)
    c7 = inputs.pair_configs(batch, batch, 5.0, 9.4)
    lab = np.random.default_rng(batch + 1).standard_normal((batch, 10)).astype(np.float32)
    c8 = np.zeros((batch, 8), np.float32)
    c8[:, :3], c8[:, 4:] = c7[:, :3], c7[:, 3:]
    l12 = np.zeros((batch, 12), np.float32)
    l12[:, :3], l12[:, 3], l12[:, 4:7], l12[:, 8:11] = lab[:, 1:4], lab[:, 0], lab[:, 4:7], lab[:, 7:10]
    m = api.MLP(width, depth)
    m.set_params(flat)
    tr = api.Trainer(m, batch)
    cfg, labels = torch.from_numpy(c8).cuda(), torch.from_numpy(l12).cuda()
    loss, g = tr.grad(cfg, labels, 0.5, 0.1, 1.5, 0.7)
    L_ref, g_ref = nn.force_matching_loss(flat.astype(np.float64), width, depth, c7.astype(np.float64),
                                          lab.astype(np.float64), 0.5, 0.1, 1.5, 0.7)
    assert loss == pytest.approx(L_ref, rel=1e-5)
    assert rel_err(g.double().cpu().numpy(), g_ref) < 1e-5
    # a step's parameters are used by the next gradient and by evaluations
    tr.step(cfg, labels, 0.5, 0.1, f_scale=1.5, kT_w=0.7)
    w = m.get_params()
    fresh = api.MLP(width, depth)
    fresh.set_params(w)
    assert torch.equal(m.pairs(cfg, "fp32"), fresh.pairs(cfg, "fp32"))
    assert torch.equal(tr.grad(cfg, labels, 0.5, 0.1)[1], api.Trainer(fresh, batch).grad(cfg, labels, 0.5, 0.1)[1])


@pytest.mark.parametrize("width,depth,batch", [
    (16, 1, 1), (16, 3, 255), (16, 2, 257), (32, 1, 127), (32, 3, 129), (32, 8, 300), (64, 2, 63), (64, 3, 65),
    (64, 8, 200), (32, 3, 9000),
])
def test_per_component_gradient(width, depth, batch):
    import torch

    from paper_2402_12199_gb300 import api

    flat = _flat(width, depth, 7 * width + depth)
    f = api.FNet(width, depth)
    f.set_params(flat)
    cfg, lab = _sampled(batch + 300, 42)
    cfg, lab = cfg[:batch].contiguous(), lab[:batch].contiguous()
    assert len(cfg) == batch
    tr = api.FNetTrainer(f, batch)
    tr.set_cap(5.0, 1.5)
    loss, g = tr.grad(cfg, lab)
    c, lb = cfg.double().cpu().numpy(), lab.double().cpu().numpy()
    d, t = fnet.targets(c[:, :3], c[:, 4:8], lb[:, 0:3], lb[:, 4:7], cap=5.0)
    L_ref, g_ref = fnet.loss_and_grad(flat.astype(np.float64), width, depth, d, t, f_scale=1.5)
    assert loss == pytest.approx(L_ref, rel=1e-5)
    assert rel_err(g.double().cpu().numpy(), g_ref) < 1e-5
    tr.step(cfg, lab)
    w = f.get_params()
    fresh = api.FNet(width, depth)
    fresh.set_params(w)
    assert torch.equal(f.pairs(cfg), fresh.pairs(cfg))
    assert torch.equal(tr.grad(cfg, lab)[1], _grad(fresh, batch, cfg, lab))


def _grad(f, batch, cfg, lab):
    from paper_2402_12199_gb300 import api

    tr = api.FNetTrainer(f, batch)
    tr.set_cap(5.0, 1.5)
    return tr.grad(cfg, lab)[1]
