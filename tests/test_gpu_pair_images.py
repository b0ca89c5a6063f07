"""The pair list for centres stored as any image: centred on the box's middle, or shifted by whole box
lengths, in a box with cell blocks away from every face (at least 18 x 10 x 10 cells, blocks of 8 x 4 x 4), where
the build leaves the minimum image out for centres in [0, L).  List and forces against brute force, as in
test_gpu_pair_list."""
import numpy as np
import pytest

from paper_2402_12199_gb300 import inputs
from tests.test_gpu_pair_list import OCTA, RC, _brute

pytestmark = pytest.mark.gpu

BOX = np.array([71.0, 40.0, 40.0])
N = 4000


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _stored(images):
    rng = np.random.default_rng(23)
    x = rng.uniform(0.0, 1.0, (N, 3)) * BOX
    if images == "centred":
        x -= BOX * (x >= 0.5 * BOX)
    elif images == "shifted":  # some bodies only
        x += BOX * (rng.integers(-2, 3, (N, 3)) * (rng.random((N, 1)) < 0.2))
    elif images == "all shifted":
        x += BOX
    pos = np.zeros((N, 4), np.float32)
    pos[:, :3] = x
    return pos


@pytest.mark.parametrize("images", ["inside", "centred", "shifted", "all shifted"])
@pytest.mark.parametrize("skin", [0.0, 0.4])
def test_list_and_forces_for_any_image(images, skin):
    import torch

    from paper_2402_12199_gb300 import api

    pos = _stored(images)
    x = pos[:, :3].astype(np.float64)
    quat = np.zeros((N, 4), np.float32)
    quat[:, 0] = 1.0
    s = api.System(N, BOX.tolist(), "custom", template=OCTA)
    if skin > 0.0:
        s.set_skin(skin)
    s.set_state(torch.from_numpy(pos).cuda(), torch.from_numpy(quat).cuda())
    s.build_pairs()
    p = s.pairs()
    d = x[p[:, 1]] - x[p[:, 0]]
    d -= BOX * np.rint(d / BOX)
    r = np.sqrt((d * d).sum(1))
    ref = _brute(x, BOX)
    got = set(map(tuple, p[r < RC].tolist()))
    assert r.max() < RC + skin + 1e-4
    assert got <= set(ref) and all(v > RC - 1e-4 for k, v in ref.items() if k not in got)
    # every body's force is the sum over exactly its pairs
    mu, isd = inputs.feature_normalisation(0.5, RC)
    m = api.MLP(64, 2)
    m.set_params(inputs.mlp_params(64, 2, 3, mu=mu, inv_sd=isd))
    F = s.forces_nn(m, "fp32")["force"][:, :3].double().cpu().numpy()
    s.sync()
    cfg = np.zeros((len(p), 8), np.float32)
    cfg[:, :3] = d
    cfg[:, 4] = 1.0
    f = m.pairs(torch.from_numpy(cfg).cuda(), "fp32")[:, :3].double().cpu().numpy()
    f[r >= RC] = 0.0
    want = np.zeros((N, 3))
    np.add.at(want, p[:, 1], f)
    np.add.at(want, p[:, 0], -f)
    # the tolerance of test_gpu_pair_list, and separations of centres up to 3 box lengths away
    scale = np.abs(f).max() * np.sqrt(2.0 * len(p) / N)
    assert np.abs(F - want).max() < 3 * 2e-4 * scale
