"""Both forms of the list's row build (a warp per body; blocks of cells) around the lines of their rule:
by size (24000 bodies), by mean bodies per cell (0.4 and 2.4), and a system crowded in a part of its box,
which the block form finds out itself.  Lists against a periodic k-d tree; a dense list must not take the
block form's way around its limits."""
import numpy as np
import pytest

from tests.helpers import TOL_F32, assert_parity, make_state
from tests.test_gpu_pair_list import OCTA, RC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _system(n, per_cell, part, max_neighbors, seed=5):
    """n bodies at random in the corner of a cube of which they take the part `part` of each side."""
    import torch

    from paper_2402_12199_gb300 import api

    L = (n / per_cell) ** (1 / 3) * RC
    x = np.random.default_rng(seed).uniform(0.0, L * part, (n, 3))
    pos = np.zeros((n, 4), np.float32)
    pos[:, :3] = x
    quat = np.zeros((n, 4), np.float32)
    quat[:, 0] = 1.0
    s = api.System(n, [float(np.float32(L))] * 3, "custom", template=OCTA, max_neighbors=max_neighbors)
    s.set_state(torch.from_numpy(pos).cuda(), torch.from_numpy(quat).cuda())
    return s, pos[:, :3].astype(np.float64), float(np.float32(L))


@pytest.mark.parametrize("n,per_cell,part,max_neighbors", [
    (23999, 1.0, 1.0, 64), (24001, 1.0, 1.0, 64),    # the line by size
    (30000, 0.39, 1.0, 64), (30000, 0.42, 1.0, 64),  # sparse cells
    (30000, 2.2, 1.0, 64), (30000, 2.5, 1.0, 64),    # dense cells
    (30000, 1.0, 0.5, 160),                          # crowded in an eighth of the box (8 a cell)
    (700, 12.0, 1.0, 160), (700, 1.0, 0.5, 160),     # rows of more than 32 neighbours
])
def test_list_is_the_trees(n, per_cell, part, max_neighbors):
    spatial = pytest.importorskip("scipy.spatial")
    s, x, L = _system(n, per_cell, part, max_neighbors)
    for _ in range(2):  # the second build finds the counters that the first one left
        count = s.build_pairs()
    p = s.pairs()
    assert len(p) == count
    key = p[:, 0].astype(np.int64) * n + p[:, 1]
    assert np.all(p[:, 0] < p[:, 1]) and np.all(np.diff(key) > 0)
    tree = spatial.cKDTree(np.mod(x, L), boxsize=L)
    inner = np.sort(tree.query_pairs(RC - 1e-4, output_type="ndarray"), 1)
    outer = np.sort(tree.query_pairs(RC + 1e-4, output_type="ndarray"), 1)
    assert np.isin(inner[:, 0].astype(np.int64) * n + inner[:, 1], key).all()
    assert np.isin(key, outer[:, 0].astype(np.int64) * n + outer[:, 1]).all()
    # every pair is found again from its second body's row: forces sum to zero
    f = s.forces_beads()["force"][:, :3].double().cpu().numpy()
    if np.isfinite(f).all():
        assert np.abs(f.sum(0)).max() <= 1e-4 * np.abs(f).sum()
    s2, _, _ = _system(n, per_cell, part, max_neighbors)
    assert s2.build_pairs() == count and np.array_equal(s2.pairs(), p)


@pytest.mark.parametrize("n,per_cell,part,limit_ms", [
    (4000, 24.0, 1.0, 3.0),    # 100 neighbours each: 0.27 ms; by blocks of cells 37 ms
    (30000, 24.0, 1.0, 8.0),   # 0.9 ms; 83 ms
    (30000, 2.0, 0.4, 12.0),   # crowded in a sixteenth of the box: found out by the block form
])
def test_dense_lists_take_the_form_for_them(n, per_cell, part, limit_ms):
    import torch

    from paper_2402_12199_gb300 import api

    s, _, _ = _system(n, per_cell, part, 320)
    build = lambda: api.check(api.load().rb_build_pairs(s.handle, None))
    build()
    s.sync()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(5):
        build()
    b.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(b) / 5 < limit_ms


def test_dense_replica_in_a_batch():
    """A replica with four bodies a cell (rows by warps inside the batched kernel) beside a dilute one:
    the trajectory of the system stepped alone, to FP32 rounding (the batched kernels' fused
    multiply-adds may be formed differently)."""
    import torch

    from paper_2402_12199_gb300 import api

    n, L = 512, 52.0
    rng = np.random.default_rng(3)
    g = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), -1).reshape(-1, 3)
    st = {k: np.zeros((n, 4), np.float32) for k in ("pos", "quat", "vel", "angmom")}
    st["pos"][:, :3] = rng.permutation((g + 0.5) * 6.5)
    st["quat"][:, 0] = 1.0
    st["vel"][:, :3] = 0.1 * rng.standard_normal((n, 3))
    st["angmom"][:, :3] = 20.0 * rng.standard_normal((n, 3))
    other, L2, _ = make_state(700, 0.15, 9)
    srv = api.Server(4 << 30, 2, None, steps_per_tick=4)
    t = [srv.submit(st, [L] * 3, "cube", api.RB_PATH_BEADS, "fp32", 40),
         srv.submit(other, [L2] * 3, "cube", api.RB_PATH_BEADS, "fp32", 40)]
    for k in t:
        r = srv.wait(k)
        assert r["status"] == 0 and r["steps_done"] == 40, r
    got = srv.fetch_state(t[0])
    srv.close()
    s = api.System(n, [L] * 3, "cube")
    s.set_state(*(torch.from_numpy(st[k]).cuda() for k in ("pos", "quat", "vel", "angmom")))
    s.step(40, 0.002)
    ref = s.get_state(to_host=True)
    assert s.build_pairs() > 3 * n
    for k in ("pos", "quat", "vel", "angmom"):
        assert_parity(got[k][:, :3].astype(np.float64), ref[k][:, :3].astype(np.float64), TOL_F32, k)
