"""Bead sums and sampled pairs of templates other than the cube's and the cylinder's, against the FP64
oracle: grids of beads whose columns of 5 or 8 fill one, two or more rows of the column kernel's lanes
(up to 128, 160 and 256 beads), and grids without such columns (every distance computed).  The bounds
are those of the same comparisons on the cube and the cylinder."""
import numpy as np
import pytest

import oracle
from oracle import bodies, fnet, sampler
from paper_2402_12199_gb300 import inputs
from tests.helpers import TOL_F32, assert_parity, oracle_beads
from tests.test_gpu_fnet import _configs, _flat
from tests.test_gpu_hphc import H
from tests.test_gpu_train import cfg7, lab10

pytestmark = pytest.mark.gpu

COLUMNS = [(2, 1, 5), (4, 4, 5), (5, 6, 5), (6, 6, 5), (7, 7, 5), (4, 4, 8), (5, 4, 8), (5, 5, 8), (8, 4, 8)]
OTHER = [(2, 2, 2), (5, 5, 4), (6, 7, 6)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _grid(n):
    return np.stack(np.meshgrid(*(np.arange(k) - 0.5 * (k - 1) for k in n), indexing="ij"), -1).reshape(-1, 3)


def _state(t, n, seed):
    rng = np.random.default_rng(seed)
    r = bodies.circumradius(t)
    L = round(n ** (1 / 3)) * (2.0 * r + 1.2)
    f4 = np.zeros((n, 4), np.float32)
    f4[:, :3] = inputs.place_bodies(n, L, r, rng)
    return f4, inputs.random_quaternions(n, rng).astype(np.float32), L


def _system(t, pos, quat, L, **kw):
    import torch

    from paper_2402_12199_gb300 import api

    s = api.System(len(pos), [L] * 3, "custom", template=t, **kw)
    z = torch.zeros((len(pos), 4), device="cuda")
    s.set_state(torch.from_numpy(pos).cuda(), torch.from_numpy(quat).cuda(), z, z.clone())
    return s


@pytest.mark.parametrize("grid,potential", [(g, "lj") for g in COLUMNS + OTHER] + [(g, "hphc") for g in COLUMNS])
def test_bead_forces(grid, potential):
    t = _grid(grid)
    pos, quat, L = _state(t, 125, len(t))
    if potential == "lj":
        s = _system(t, pos, quat, L)
        F, T, E, _, pairs = oracle_beads(dict(pos=pos, quat=quat), L, t)
    else:
        s = _system(t, pos, quat, L, potential="hphc", hphc=H)
        pot = oracle.pot_hphc(H["A"], H["b"], H["c"], H["p"], False)
        p64 = pos[:, :3].astype(np.float64)
        pairs = oracle.pairs_bruteforce(p64, np.array([L] * 3), bodies.pair_cutoff(t, oracle.pot_cutoff(pot)))
        F, T, E, _ = oracle.forces_beads(p64, quat.astype(np.float64), np.array([L] * 3), t, pairs, pot=pot)
    res = s.forces_beads(energy=True)
    s.sync()
    assert np.abs(F).max() > 0
    assert_parity(res["force"][:, :3].double().cpu().numpy(), F, TOL_F32, "force")
    assert_parity(res["torque"][:, :3].double().cpu().numpy(), T, TOL_F32, "torque")
    assert res["energy"] == pytest.approx(E, rel=TOL_F32)


@pytest.mark.parametrize("grid", [(2, 1, 5), (5, 6, 5), (7, 7, 5), (4, 4, 8), (8, 4, 8), (2, 2, 2), (6, 7, 6)])
def test_sampled_pairs(grid):
    import torch

    from paper_2402_12199_gb300 import api

    t = _grid(grid)
    s = api.System(8, [80.0] * 3, "custom", template=t)
    u = inputs.sampler_uniforms(25, 7)
    cfg, lab, rc = (x.cpu().numpy() for x in api.sample_pairs(s, torch.from_numpy(u).cuda()))
    d, q = sampler.draws_to_config(u.astype(np.float64))
    Rc = bodies.pair_cutoff(t)
    for b in range(0, 25, 4):
        assert rc[b] == pytest.approx(sampler.contact_distance(d[b], q[b], t, Rc, 1.0), abs=2e-5)
    ref, got = sampler.label_pairs(cfg7(cfg), t), lab10(lab)
    for a in (1, 4, 7):
        assert_parity(got[:, a:a + 3], ref[:, a:a + 3], TOL_F32)
    assert np.abs(got[:, 0] - ref[:, 0]).max() <= TOL_F32 * max(1.0, np.abs(ref[:, 0]).max())


@pytest.mark.parametrize("width,depth,n", [(32, 4, 1), (32, 6, 257), (64, 2, 1023), (16, 4, 3)])
def test_per_component_pairs(width, depth, n):
    """Both ways the networks are held (all five resident, or one after the other), two pairs per
    thread with an odd number of pairs."""
    import torch

    from paper_2402_12199_gb300 import api

    flat = _flat(width, depth, width + depth)
    f = api.FNet(width, depth)
    f.set_params(flat)
    c, q = (x[:n] for x in _configs(1500, 3 + n))
    assert len(c) == n
    cfg = np.zeros((n, 8), np.float32)
    cfg[:, :3], cfg[:, 4:] = c, q
    out = f.pairs(torch.from_numpy(cfg).cuda()).double().cpu().numpy()
    Fj, ti, tj, _ = fnet.predict(fnet.unpack(flat.astype(np.float64), width, depth), c.astype(np.float64),
                                 q.astype(np.float64))
    for a, ref in ((0, Fj), (4, ti), (8, tj)):
        assert_parity(out[:, a:a + 3], ref, TOL_F32)


@pytest.mark.parametrize("offset", [0, 1])
def test_force_rows_of_any_alignment(offset):
    """Rows that start on a 16-byte boundary are written by the reduction, others are copied: the same."""
    import torch

    from paper_2402_12199_gb300 import api

    t = _grid((4, 4, 5))
    pos, quat, L = _state(t, 125, 11)
    s = _system(t, pos, quat, L)
    ref = s.forces_beads()
    buf = torch.zeros(2, 4 * 125 + 4, device="cuda")
    rows = [b[offset:offset + 500] for b in buf]
    api.check(api.load().rb_forces_beads(s.handle, rows[0].data_ptr(), rows[1].data_ptr(), None, None))
    s.sync()
    assert torch.equal(rows[0].view(-1, 4), ref["force"]) and torch.equal(rows[1].view(-1, 4), ref["torque"])
    assert buf[:, :offset].abs().sum() == 0 and buf[:, offset + 500:].abs().sum() == 0
