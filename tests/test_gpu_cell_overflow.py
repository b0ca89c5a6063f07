"""More bodies in one cell than a cell's list holds: reported, and the bodies left out have no
neighbours in the list that is built all the same (a system's first list, or one after another, whose
rows must not be taken up again)."""
import numpy as np
import pytest

from tests.test_gpu_pair_list import OCTA, RC, _brute

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("earlier_list", [False, True])
@pytest.mark.parametrize("crowd", [33, 60])  # a cell holds 2 x max_neighbors = 32
def test_bodies_left_out_of_a_full_cell(crowd, earlier_list):
    import torch

    from paper_2402_12199_gb300 import api

    n, L = 343, 28.0  # 8 x 8 x 8 cells
    rng = np.random.default_rng(7)
    g = np.stack(np.meshgrid(*[np.arange(7)] * 3, indexing="ij"), -1).reshape(-1, 3)
    good = np.zeros((n, 4), np.float32)
    good[:, :3] = rng.permutation((g + 0.5) * 3.3)  # up to six neighbours each
    bad = np.zeros((n, 4), np.float32)
    bad[:, :3] = rng.permutation((g + 0.5) * 4.0)
    bad[:crowd, :3] = 1.75 + rng.uniform(-0.3, 0.3, (crowd, 3))
    quat = np.zeros((n, 4), np.float32)
    quat[:, 0] = 1.0
    quat = torch.from_numpy(quat).cuda()
    s = api.System(n, [L] * 3, "custom", template=OCTA, max_neighbors=16)
    if earlier_list:
        s.set_state(torch.from_numpy(good).cuda(), quat)
        assert s.build_pairs() > 0
    s.set_state(torch.from_numpy(bad).cuda(), quat)
    with pytest.raises(api.RBError, match="cell capacity"):
        s.build_pairs()
    p = s.pairs()
    d = bad[p[:, 1], :3].astype(np.float64) - bad[p[:, 0], :3]
    d -= L * np.rint(d / L)
    assert len(p) > 0 and np.all(p[:, 0] < p[:, 1]) and p.min() >= 0 and p.max() < n
    assert np.sqrt((d * d).sum(1)).max() < RC + 1e-4
    # the next list is complete
    s.set_state(torch.from_numpy(good).cuda(), quat)
    s.build_pairs()
    ref = _brute(good[:, :3].astype(np.float64), [L] * 3)
    got = set(map(tuple, s.pairs().tolist()))
    assert got <= set(ref) and all(r > RC - 1e-4 for k, r in ref.items() if k not in got)
