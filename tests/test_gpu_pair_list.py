"""The pair list against a brute-force search, over the forms the list build distinguishes: box
sides of 2, 3, 8 and 9 cells (stencils that wrap onto themselves, whole and partial cell blocks),
bodies with more neighbours than a shared row holds, and cells too crowded for a block's shared
memory.  The bodies' orientations are the identity, so the per-body network forces must be the sums
of the pairs' own (rb_nn_pairs): that checks every body's pair indices.  Pairs within 1e-4 of the
list's radius may fall on either side in FP32 and are left out of the comparison."""
import numpy as np
import pytest

from paper_2402_12199_gb300 import inputs

pytestmark = pytest.mark.gpu

# six beads: principal axes along x, y, z; r_circ 0.5, Rc = 2 x 0.5 + 2.5 = 3.5
OCTA = np.array([[0.5, 0, 0], [-0.5, 0, 0], [0, 0.4, 0], [0, -0.4, 0], [0, 0, 0.3], [0, 0, -0.3]], np.float32)
RC = 3.5


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _system(n, box, seed, max_neighbors, cluster=1.0):
    import torch

    from paper_2402_12199_gb300 import api

    rng = np.random.default_rng(seed)
    pos = np.zeros((n, 4), np.float32)
    pos[:, :3] = rng.uniform(0.0, 1.0, (n, 3)) * np.array(box) * cluster
    quat = np.zeros((n, 4), np.float32)
    quat[:, 0] = 1.0
    s = api.System(n, box, "custom", template=OCTA, max_neighbors=max_neighbors)
    s.set_state(torch.from_numpy(pos).cuda(), torch.from_numpy(quat).cuda())
    return s, pos[:, :3].astype(np.float64)


def _brute(x, box):
    d = x[None] - x[:, None]
    d -= np.array(box) * np.rint(d / np.array(box))
    r = np.sqrt((d * d).sum(-1))
    i, j = np.nonzero(np.triu(r < RC + 1e-4, 1))
    return {(a, b): r[a, b] for a, b in zip(i, j)}


@pytest.mark.parametrize("n,box,max_neighbors,cluster", [
    (1, (7.5, 7.5, 7.5), 0, 1.0),
    (40, (7.5, 7.1, 8.0), 64, 1.0),        # two cells a side
    (150, (10.6, 7.5, 31.8), 64, 1.0),     # 3 x 2 x 9 cells
    (257, (28.5, 28.5, 32.0), 0, 1.0),     # 8 x 8 x 9 cells, one body past a segment
    (300, (14.0, 14.0, 14.0), 128, 1.0),   # rows longer than a shared row
    (900, (14.0, 14.0, 14.0), 256, 1.0),   # cells too crowded for a block's shared memory
    (1500, (64.0, 33.0, 15.0), 256, 0.35),  # a cluster in an empty box, several segments
])
def test_list_is_the_brute_force_list(n, box, max_neighbors, cluster):
    import torch

    from paper_2402_12199_gb300 import api

    s, x = _system(n, box, 11 + n, max_neighbors, cluster)
    count = s.build_pairs()
    p = s.pairs()
    assert len(p) == count
    assert np.all(p[:, 0] < p[:, 1])
    key = p[:, 0].astype(np.int64) * n + p[:, 1]
    assert np.all(np.diff(key) > 0)  # ascending, each pair once
    ref = _brute(x, box)
    got = set(map(tuple, p.tolist()))
    assert got <= set(ref)
    assert all(r > RC - 1e-4 for k, r in ref.items() if k not in got)
    if count == 0:
        return
    # every body's sum runs over exactly its pairs
    mu, isd = inputs.feature_normalisation(0.5, RC)
    m = api.MLP(64, 2)
    m.set_params(inputs.mlp_params(64, 2, 3, mu=mu, inv_sd=isd))
    F = s.forces_nn(m, "fp32")["force"][:, :3].double().cpu().numpy()
    s.sync()
    d = x[p[:, 1]] - x[p[:, 0]]
    d -= np.array(box) * np.rint(d / np.array(box))
    cfg = np.zeros((count, 8), np.float32)
    cfg[:, :3] = d
    cfg[:, 4] = 1.0
    f = m.pairs(torch.from_numpy(cfg).cuda(), "fp32")[:, :3].double().cpu().numpy()
    f[(d * d).sum(1) >= RC * RC] = 0.0
    want = np.zeros((n, 3))
    np.add.at(want, p[:, 1], f)
    np.add.at(want, p[:, 0], -f)
    # FP32 separations (relative 2^-22 of the box) through the network, and FP32 sums over a row
    scale = np.abs(f).max() * np.sqrt(max(1.0, 2.0 * count / n))
    assert np.abs(F - want).max() < 2e-4 * scale


@pytest.mark.parametrize("n,max_neighbors", [(300, 12), (900, 32)])
def test_too_many_neighbours_is_reported_and_the_next_list_is_right(n, max_neighbors):
    import torch

    from paper_2402_12199_gb300 import api

    box = (42.0, 42.0, 42.0)
    s, x = _system(n, box, 5, max_neighbors, cluster=1.0 / 3.0)
    with pytest.raises(api.RBError) as e:
        s.build_pairs()
    assert e.value.status == 4
    s.forces_beads()  # sums over a truncated list: no invalid pair index may be left in it
    with pytest.raises(api.RBError):
        s.sync()
    # the same bodies spread out: 27 times fewer neighbours
    spread = np.zeros((n, 4), np.float32)
    spread[:, :3] = 3.0 * x
    s.set_state(torch.from_numpy(spread).cuda())
    s.build_pairs()
    ref = _brute(spread[:, :3].astype(np.float64), box)
    got = set(map(tuple, s.pairs().tolist()))
    assert got <= set(ref) and all(r > RC - 1e-4 for k, r in ref.items() if k not in got)


def test_more_segments_than_one_pass_adds_up():
    """130^3 bodies on a lattice with six neighbours each: more offset segments than a CTA of the
    emitting kernel adds up by itself."""
    import torch

    from paper_2402_12199_gb300 import api

    m, a = 130, 3.3
    n = m ** 3
    rng = np.random.default_rng(3)
    site = rng.permutation(n)  # body -> lattice site
    ijk = np.stack([site // (m * m), site // m % m, site % m], 1)
    pos = np.zeros((n, 4), np.float32)
    pos[:, :3] = (ijk + 0.5) * a
    quat = np.zeros((n, 4), np.float32)
    quat[:, 0] = 1.0
    s = api.System(n, [m * a] * 3, "custom", template=OCTA, max_neighbors=8)
    s.set_state(torch.from_numpy(pos).cuda(), torch.from_numpy(quat).cuda())
    assert s.build_pairs() == 3 * n
    p = s.pairs().astype(np.int64)
    assert np.all(p[:, 0] < p[:, 1]) and np.all(np.diff(p[:, 0] * n + p[:, 1]) > 0)
    d = np.abs(ijk[p[:, 0]] - ijk[p[:, 1]])
    d = np.minimum(d, m - d)
    assert np.all(d.sum(1) == 1)
