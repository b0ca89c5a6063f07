"""The workloads this library is timed on, each through its public Python API.

Kinds of case (a case is a dict of plain values):
  md      MD steps of one system from a given state: set_state, step(n), the new state back
  forces  forces, torques of one system at a new state, with its pair list rebuilt
  pairs   the pair network on explicit configurations, with its input gradient
  train   force matching of the pair network: a monitored gradient, Adam steps, the parameters
  fntrain regression of the per-component cylinder networks, the same sequence
  sample  training pairs drawn and labelled by the bead sum
  serve   MD replicas through the server, to their final states

Inputs come from the seed alone: bodies on a lattice, displaced at random as far as contact
allows (bead distances from 0.9 sigma), uniform orientations, Maxwell momenta, networks with
N(0, 1 / fan_in) weights, the body's point group and the smooth cutoff attached, as
train_net.train_network sets them up.  exact() restates every computation in FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2402_12199_gb300 import api

V_PARTICLE = {"cube": 125.0, "cylinder": math.pi * 2.5 ** 2 * 9.0}
HPHC = {"A": 0.00035, "b": 1.46375, "c": 3.3833, "p": 2.5}  # the paper's Eq. 1 workload
F64 = torch.float64


def listed():
    return [
        # a small replica, where launches and one tile's latency are the step
        dict(name="md_bf16_512", kind="md", path="bf16", shape="cube", n=512, phi=0.10, steps=20),
        # the headline: 32768 cubes on the BF16 network, list kept by the skin
        dict(name="md_bf16_32768", kind="md", path="bf16", shape="cube", n=32768, phi=0.20, steps=20),
        # the same workload on the exact bead sum
        dict(name="md_beads_32768", kind="md", path="beads", shape="cube", n=32768, phi=0.20, steps=20),
        # the paper's cylinder method: five per-component networks
        dict(name="md_fnet_cyl_30000", kind="md", path="fnet", shape="cylinder", n=30000, phi=0.15,
             steps=10),
        # one force call on a large system without a skin (list rebuilt)
        dict(name="forces_bf16_524288", kind="forces", path="bf16", shape="cube", n=524288, phi=0.20),
        # FP32 accuracy on the tensor cores, an odd size
        dict(name="forces_f16x3_20011", kind="forces", path="f16x3", shape="cube", n=20011, phi=0.18),
        # the width-256 network of the cylinders
        dict(name="forces_w256_cyl_32768", kind="forces", path="w256", shape="cylinder", n=32768,
             phi=0.15),
        # explicit configurations at the API's default precision, as evaluation and autograd call it
        dict(name="pairs_fp32_50003", kind="pairs", precision="fp32", width=128, n=50003),
        # force matching at the repository's batch size
        dict(name="train_w128_4096", kind="train", width=128, batch=4096, steps=8),
        # the per-component networks' training at their batch size
        dict(name="fntrain_w32_4096", kind="fntrain", width=32, batch=4096, steps=4),
        # training pairs with contact bisection and bead labels
        dict(name="sample_cube_65536", kind="sample", shape="cube", n=65536, contact=0.85),
        # serving a mix of small replicas on the network and on the beads
        dict(name="serve_6_small", kind="serve", replicas=6, n_max=4096, steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "forces", "forces", "pairs", "train", "fntrain", "sample",
                       "serve"])
    if kind == "md":
        path = rng.choice(["bf16", "bf16", "beads", "beads", "f16x3", "hphc_nvt", "fnet"])
        shape = "cylinder" if path == "fnet" else rng.choice(["cube", "cylinder"]) if path == "beads" else "cube"
        return dict(kind=kind, path=path, shape=shape, n=_log_int(rng, 400, 65536),
                    phi=round(rng.uniform(0.05, 0.22 if shape == "cube" else 0.16), 4),
                    steps=rng.choice([8, 10, 16, 20]))
    if kind == "forces":
        path = rng.choice(["bf16", "bf16", "beads", "f16x3", "w256"])
        shape = "cylinder" if path == "w256" else "cube"
        return dict(kind=kind, path=path, shape=shape,
                    n=_log_int(rng, 1000, 400000 if path == "bf16" else 100000),
                    phi=round(rng.uniform(0.05, 0.22 if shape == "cube" else 0.16), 4))
    if kind == "pairs":
        precision = rng.choice(["fp32", "fp32", "bf16", "f16x3"])
        width = 128 if precision == "f16x3" else rng.choice([128, 256])
        return dict(kind=kind, precision=precision, width=width, n=_log_int(rng, 100, 200000))
    if kind == "train":
        return dict(kind=kind, width=rng.choice([128, 128, 256]), batch=_log_int(rng, 500, 10000),
                    steps=rng.choice([4, 8]))
    if kind == "fntrain":
        return dict(kind=kind, width=rng.choice([16, 32, 64]), batch=_log_int(rng, 500, 10000),
                    steps=rng.choice([2, 4]))
    if kind == "sample":
        return dict(kind=kind, shape=rng.choice(["cube", "cylinder"]), n=_log_int(rng, 1000, 65536),
                    contact=rng.choice([0.85, 1.0]))
    return dict(kind=kind, replicas=rng.choice([3, 4, 6, 7, 8]), n_max=_log_int(rng, 1000, 8000),
                steps=rng.choice([40, 60, 100]))


# ------------------------------------------------------------------ bodies and inputs

def _template(shape):
    if shape == "cube":
        g = np.arange(5.0) - 2.0
        return np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    disc = [(a + 0.5 * c, c * math.sqrt(3.0) / 2.0) for a in range(-4, 5) for c in range(-4, 5)]
    disc = [p for p in disc if p[0] ** 2 + p[1] ** 2 <= 4.0 + 1e-9]
    return np.array([(x, y, (k - 3.5) * 8.0 / 7.0) for k in range(8) for x, y in disc])


def _body(shape):
    t = _template(shape)
    inertia = (t ** 2).sum() - (t ** 2).sum(0)
    return t, float(len(t)), inertia, float(np.sqrt((t ** 2).sum(1)).max())


def _rcut(pot):
    return HPHC["b"] + math.pi / HPHC["c"] if pot == "hphc" else 2.5


def _rot(q):
    """Rotation matrices of unit quaternions (..., 4) in the order (s, i, j, k)."""
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                       -1).reshape(q.shape[:-1] + (3, 3))


def _qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _conj(q):
    return q * q.new_tensor([1.0, -1.0, -1.0, -1.0])


def _mv(R, v):
    return (R @ v[..., None])[..., 0]


def _squared_distances(t, b):
    """|b_l - t_k|^2 (pairs, k, l) of the beads t of body i and b (pairs, l, 3) of body j."""
    t2, b2 = (t * t).sum(1), (b * b).sum(2)
    return torch.baddbmm(t2[:, None] + b2[:, None, :], t.expand(len(b), -1, -1), b.transpose(1, 2), alpha=-2.0)


def _min_bead_distance(s, R, t):
    """Smallest bead distance per pair (s: centre of j, R: its rotation, in i's frame), by chunks."""
    out = []
    for a in range(0, len(s), 16384):
        b = s[a:a + 16384, None, :] + t @ R[a:a + 16384].transpose(1, 2)
        out.append(_squared_distances(t, b).amin((1, 2)).clamp(min=0.0).sqrt())
    return torch.cat(out) if out else s.new_zeros(0)


def _fluid(shape, n, phi, seed, kT=1.0):
    """State (4, n, 4) float32 on the GPU (pos, quat, vel, angmom rows), the box side and the
    candidate pairs i < j (bodies on neighbouring lattice sites, a superset of those in range)."""
    rng = np.random.default_rng(seed)
    t, mass, inertia, rc = _body(shape)
    m = math.ceil(n ** (1.0 / 3.0) - 1e-9)
    side = max((n * V_PARTICLE[shape] / phi) ** (1.0 / 3.0), m * (2.0 * rc + 0.95))
    L = float(np.float32(side))
    a = L / m
    site = rng.permutation(m ** 3)[:n]
    ijk = np.stack([site // (m * m), site // m % m, site % m], 1)
    amp = 0.5 * (a - 5.2)
    disp = torch.from_numpy(rng.uniform(-amp, amp, (n, 3))).cuda()
    q = rng.standard_normal((n, 4))
    q = torch.from_numpy((q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)).cuda()
    v = rng.standard_normal((n, 3)) * math.sqrt(kT / mass)
    ang = rng.standard_normal((n, 3)) * np.sqrt(kT * inertia)
    grid = np.full(m ** 3, -1, dtype=np.int64)
    grid[site] = np.arange(n)
    pairs = []
    for o in [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)][14:]:
        k = (ijk + np.array(o)) % m
        j = grid[(k[:, 0] * m + k[:, 1]) * m + k[:, 2]]
        i = np.arange(n)
        pairs.append(np.stack([np.minimum(i, j), np.maximum(i, j)], 1)[j >= 0])
    pairs = torch.from_numpy(np.concatenate(pairs)).cuda()
    i, j = pairs.unbind(1)
    base = torch.from_numpy((ijk + 0.5) * a).cuda()
    tt = torch.from_numpy(t).float().cuda()
    for _ in range(8):  # bodies that overlap move back towards their sites
        x = base + disp
        d = x[j] - x[i]
        d = d - L * torch.round(d / L)
        near = torch.nonzero((d * d).sum(1) < (2.0 * rc + 0.9) ** 2)[:, 0]
        ni, nj = i[near], j[near]
        Ri = _rot(q[ni])
        s = _mv(Ri.transpose(1, 2), d[near].float())
        bad = near[_min_bead_distance(s, Ri.transpose(1, 2) @ _rot(q[nj]), tt) < 0.9]
        shrink = torch.ones(n, dtype=torch.bool, device="cuda")
        shrink[i[bad]] = False
        shrink[j[bad]] = False
        disp = torch.where(shrink[:, None], disp, disp * 0.7)
    st = torch.zeros((4, n, 4), dtype=torch.float32, device="cuda")
    st[0, :, :3] = (base + disp).float()
    st[1] = q
    st[2, :, :3] = torch.from_numpy((v - v.mean(0)).astype(np.float32)).cuda()
    st[3, :, :3] = torch.from_numpy(ang.astype(np.float32)).cuda()
    return st, L, pairs


def _mlp_flat(width, seed, Rc, depth=3):
    """Flat parameters (the library's layout) with the canonical features' rough moments."""
    rng = np.random.default_rng(seed)
    mu = [5.0, 3.0, 1.5, 0.85, 0.0, 0.0, 0.0, 7.5, 0.14, 58.0]
    sd = [1.5, 1.3, 1.0, 0.1, 0.25, 0.25, 0.25, 1.5, 0.03, 22.0]
    parts, fan = [np.array(mu), 1.0 / np.array(sd)], 10
    for _ in range(depth):
        parts += [rng.standard_normal(width * fan) / math.sqrt(fan), 0.1 * rng.standard_normal(width)]
        fan = width
    parts += [rng.standard_normal(width) / math.sqrt(width), 0.1 * rng.standard_normal(1), np.array([1.5, -0.2])]
    return np.concatenate(parts).astype(np.float32)


def _fnet_flat(width, seed, Rc, depth=3):
    rng = np.random.default_rng(seed)
    parts = []
    for _ in range(5):
        parts.append(np.array([Rc / 2, Rc / 2, math.pi / 4, 0.0, 2 / Rc, 2 / Rc, 4 / math.pi, 1 / math.pi]))
        fan = 4
        for _l in range(depth):
            parts += [rng.standard_normal(width * fan) / math.sqrt(fan), 0.1 * rng.standard_normal(width)]
            fan = width
        parts += [rng.standard_normal(width) / math.sqrt(width), np.array([0.05, 1.25, 0.0])]
    return np.concatenate(parts).astype(np.float32)


def _net(width, seed, shape):
    """A pair network as train_network leaves it: point group and smooth cutoff attached."""
    Rc = 2.0 * _body(shape)[3] + 2.5
    m = api.MLP(width, 3)
    m.set_params(_mlp_flat(width, seed, Rc))
    m.set_symmetry(*api.template_symmetry(_template(shape)))
    m.set_cutoff(Rc - 1.0, Rc)
    return m


RHO_MIN = {"cube": 5.0, "cylinder": 4.9}  # closer pairs take the bead sum (training contact)


def _configs(shape, n, seed):
    """n pair configurations (n, 8) float32 on the GPU in the frame of body i: separations from
    contact (0.85 sigma) to Rc, and their bead labels (n, 12)."""
    rng = np.random.default_rng(seed)
    t, _, _, rc = _body(shape)
    Rc = 2.0 * rc + 2.5
    tt = torch.from_numpy(t).float().cuda()
    got, have = [], 0
    while have < n:
        k = 2 * n + 64
        d = rng.standard_normal((k, 3))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        q = rng.standard_normal((k, 4))
        q /= np.linalg.norm(q, axis=1, keepdims=True)
        c = np.zeros((k, 8), np.float32)
        c[:, :3] = d * rng.uniform(4.2, Rc, (k, 1))
        c[:, 4:] = q
        c = torch.from_numpy(c).cuda()
        c = c[_min_bead_distance(c[:, :3], _rot(c[:, 4:]), tt) >= 0.85]
        got.append(c)
        have += len(c)
    return torch.cat(got)[:n].contiguous()


def _labels(shape, cfg):
    c = cfg.double()
    E, F, ti, tj = _bead_pairs(shape, "lj", c[:, :3], _rot(c[:, 4:]))
    out = torch.zeros((len(c), 12), dtype=torch.float32, device="cuda")
    out[:, :3], out[:, 3], out[:, 4:7], out[:, 8:11] = F.float(), E.float(), ti.float(), tj.float()
    return out


def _train_inputs(case, seed):
    shape = "cube" if case["kind"] == "train" and case["width"] == 128 else "cylinder"
    n = case["batch"] * (case["steps"] + 1)
    cfg = _configs(shape, n, seed)
    lab = _labels(shape, cfg)
    b = case["batch"]
    return shape, [(cfg[k * b:(k + 1) * b].contiguous(), lab[k * b:(k + 1) * b].contiguous())
                   for k in range(case["steps"] + 1)]


LR = 2e-5  # the end of the repository's cosine schedules


def _replicas(case, seed):
    """(path, state, box side, candidate pairs) of each served replica."""
    out, last = [], case["replicas"] - 1
    for k in range(case["replicas"]):  # sizes spread over 512 .. n_max, densities over 0.06 .. 0.18
        n = int(round(512.0 * (case["n_max"] / 512.0) ** ((5 * k % (last + 1)) / last)))
        st, L, pairs = _fluid("cube", n, 0.06 + 0.12 * k / last, seed * 31 + k)
        out.append(("beads" if k % 3 == 2 else "bf16", st, L, pairs))
    return out


# ------------------------------------------------------------------ prepare and run

def _system(case, st, L):
    pot = "hphc" if case["path"] == "hphc_nvt" else "lj"
    s = api.System(st.shape[1], [L] * 3, case["shape"], skin=0.4 if case["kind"] == "md" else 0.0,
                   potential=pot, hphc=HPHC if pot == "hphc" else None)
    s.set_state(st[0], st[1], st[2], st[3])
    return s


def prepare(case, seed):
    kind, x = case["kind"], {"case": case}
    if kind in ("md", "forces"):
        st, L, _ = _fluid(case["shape"], case["n"], case["phi"], seed)
        s = _system(case, st, L)
        x.update(state=st, system=s, out={k: torch.empty_like(st[0]) for k in ("pos", "quat", "vel", "angmom")})
        if case["path"] in ("bf16", "f16x3", "w256"):
            x["net"] = _net(256 if case["path"] == "w256" else 128, seed + 1, case["shape"])
            s.set_nn_fallback(RHO_MIN[case["shape"]])
        elif case["path"] == "fnet":
            x["net"] = api.FNet(32, 3)
            x["net"].set_params(_fnet_flat(32, seed + 1, s.pair_cutoff))
        elif case["path"] == "hphc_nvt":
            s.set_thermostat(0.7, 1.0)
    elif kind == "pairs":
        x["net"] = _net(case["width"], seed + 1, "cube")
        x["cfg"] = _configs("cube", case["n"], seed)
    elif kind == "train":
        shape, x["batches"] = _train_inputs(case, seed)
        x["net"] = _net(case["width"], seed + 1, shape)
        x["trainer"] = api.Trainer(x["net"], case["batch"], lr=LR)
    elif kind == "fntrain":
        shape, x["batches"] = _train_inputs(case, seed)
        x["net"] = api.FNet(case["width"], 3)
        x["net"].set_params(_fnet_flat(case["width"], seed + 1, 2.0 * _body(shape)[3] + 2.5))
        x["trainer"] = api.FNetTrainer(x["net"], case["batch"], lr=LR)
        x["trainer"].set_cap(5.0, 1.0)
    elif kind == "sample":
        x["system"] = api.System(8, [70.0] * 3, case["shape"])
        u = np.random.default_rng(seed).random((case["n"], 6), dtype=np.float32)
        x["u"] = torch.from_numpy(u).cuda()
    else:
        x["net"] = _net(128, seed + 1, "cube")
        x["server"] = api.Server(2 << 30, 8, x["net"])
        x["server"].set_network("cube", x["net"], RHO_MIN["cube"])
        x["requests"] = [(path, {k: st[r].cpu().numpy() for r, k in enumerate(("pos", "quat", "vel", "angmom"))}, L)
                         for path, st, L, _ in _replicas(case, seed)]
    return x


def run(x):
    case = x["case"]
    kind = case["kind"]
    if kind == "md":
        s, st, path = x["system"], x["state"], case["path"]
        s.set_state(st[0], st[1], st[2], st[3])
        if path == "fnet":
            s.step_fnet(x["net"], case["steps"], 0.002)
        elif path == "beads":
            s.step(case["steps"], 0.002)
        elif path == "hphc_nvt":
            s.step(case["steps"], 0.005)
        else:
            s.step(case["steps"], 0.002, path=api.RB_PATH_NN, mlp=x["net"], precision=path)
        return s.get_state(out=x["out"])
    if kind == "forces":
        s, st = x["system"], x["state"]
        s.set_state(st[0], st[1], st[2], st[3])
        if case["path"] == "beads":
            return s.forces_beads()
        return s.forces_nn(x["net"], "f16x3" if case["path"] == "f16x3" else "bf16")
    if kind == "pairs":
        out, grad = x["net"].pairs(x["cfg"], case["precision"], grad=True)
        return {"out": out, "grad": grad}
    if kind == "train":
        tr, bs = x["trainer"], x["batches"]
        loss, grad = tr.grad(*bs[0], 1.0, 0.1, f_scale=2.0)
        for cfg, lab in bs[1:]:
            tr.step(cfg, lab, 1.0, 0.1, want_loss=False, f_scale=2.0)
        return {"loss": loss, "grad": grad, "params": x["net"].get_params()}
    if kind == "fntrain":
        tr, bs = x["trainer"], x["batches"]
        loss, grad = tr.grad(*bs[0])
        for cfg, lab in bs[1:]:
            tr.step(cfg, lab)
        return {"loss": loss, "grad": grad, "params": x["net"].get_params()}
    if kind == "sample":
        cfg, lab, rho = api.sample_pairs(x["system"], x["u"], case["contact"])
        return {"cfg": cfg, "labels": lab, "rho_contact": rho}
    srv = x["server"]
    tickets = [srv.submit(st, [L] * 3, "cube", api.RB_PATH_NN if path == "bf16" else api.RB_PATH_BEADS,
                          "bf16", case["steps"], skin=0.4) for path, st, L in x["requests"]]
    for t in tickets:
        if srv.wait(t)["status"] != 0:
            raise RuntimeError("a replica failed")
    return [srv.fetch_state(t) for t in tickets]


# ------------------------------------------------------------------ work

def _pairs_expected(shape, n, phi, pot="lj"):
    Rc = 2.0 * _body(shape)[3] + _rcut(pot)
    return 0.5 * n * n * 4.0 / 3.0 * math.pi * Rc ** 3 * phi / (n * V_PARTICLE[shape])


def _pair_flops(path, shape):
    """Per body pair: the network's GEMMs forward and for the input gradient; for the beads the
    rotation of one body's beads, their distances to the nearest column and ten bead terms."""
    if path in ("bf16", "f16x3", "w256"):
        w = 256 if path == "w256" else 128
        return 4.0 * (10 * w + 2 * w * w + w)
    if path == "fnet":
        return 10.0 * (4 * 32 + 2 * 32 * 32 + 32)
    b = len(_template(shape))
    return 18.0 * b + 8.0 * b * (5 if shape == "cube" else 8) + 160.0


def work(case):
    kind = case["kind"]
    if kind in ("md", "forces"):
        pot = "hphc" if case["path"] == "hphc_nvt" else "lj"
        p = _pairs_expected(case["shape"], case["n"], case["phi"], pot) * _pair_flops(case["path"], case["shape"])
        steps = case.get("steps", 1)
        return {"bytes": 128.0 * case["n"], "flops": p * steps}
    if kind == "pairs":
        w = case["width"]
        return {"bytes": 112.0 * case["n"], "flops": 4.0 * (10 * w + 2 * w * w + w) * case["n"]}
    if kind in ("train", "fntrain"):
        w = case["width"]
        # train: value and tangent forward, the plain and the two-stream reverse, two weight products
        gemm = 16.0 * (10 * w + 2 * w * w) if kind == "train" else 5 * 6.0 * (4 * w + 2 * w * w)
        n = case["batch"] * (case["steps"] + 1)
        return {"bytes": 80.0 * n, "flops": gemm * n}
    if kind == "sample":
        # per sample one exact contact distance (every bead pair once) and one label
        b = len(_template(case["shape"]))
        return {"bytes": 108.0 * case["n"], "flops": (8.0 * b * b + 18.0 * b) * case["n"]}
    n = case["replicas"] * (case["n_max"] - 512) / math.log(case["n_max"] / 512.0)
    return {"bytes": 128.0 * n,
            "flops": _pairs_expected("cube", n, 0.12) * _pair_flops("bf16", "cube") * case["steps"]}


# ------------------------------------------------------------------ exact: FP64 torch

def _bead_pairs(shape, pot, s, R):
    """(E, F_j, tau_i, tau_j) of body pairs in the frame of body i (s: centre of j, R: its
    rotation): the plain double sum, over the bead pairs within the cutoff."""
    t = torch.from_numpy(_template(shape)).to(s.device)
    rc = float(np.float32(_rcut(pot)))
    E, F, ti, tj = [], [], [], []
    for a in range(0, len(s), 4096):
        b = s[a:a + 4096, None, :] + t @ R[a:a + 4096].transpose(1, 2)
        k, x, y = torch.nonzero(_squared_distances(t, b) < rc * rc, as_tuple=True)
        d = b[k, y] - t[x]
        r2 = (d * d).sum(1)
        if pot == "lj":
            s6 = r2 ** -3
            c6 = rc ** -6
            u, f = 4.0 * (s6 * s6 - s6) - 4.0 * (c6 * c6 - c6), 24.0 * (2.0 * s6 * s6 - s6) / r2
        else:
            A, bb, c, p = (float(np.float32(HPHC[z])) for z in ("A", "b", "c", "p"))
            r1 = r2.sqrt()
            h = (bb - r1).clamp(min=0.0)
            u = torch.where(r1 <= bb, h ** p - 2 * A, -A * (1 + torch.cos(c * (r1 - bb))))
            f = torch.where(r1 <= bb, p * h ** (p - 1), -A * c * torch.sin(c * (r1 - bb))) / r1
        fv = f[:, None] * d
        z = lambda v: torch.zeros((len(b),) + v.shape[1:], dtype=F64, device=s.device).index_add_(0, k, v)
        E.append(z(u))
        F.append(z(fv))
        ti.append(-z(torch.linalg.cross(t[x], fv)))
        tj.append(z(torch.linalg.cross(b[k, y] - s[a:a + 4096][k], fv)))
    cat = lambda v, w: torch.cat(v) if v else s.new_zeros(w)
    return cat(E, (0,)), cat(F, (0, 3)), cat(ti, (0, 3)), cat(tj, (0, 3))


def _group(shape):
    """Proper rotations of the body (unit quaternions); its inversion is a symmetry as well."""
    if shape == "cube":
        h = math.sqrt(0.5)
        e = np.eye(4)
        q = [e[k] for k in range(4)]
        q += [h * (e[a] + sg * e[b]) for a in range(4) for b in range(a + 1, 4) for sg in (1, -1)]
        q += [0.5 * np.array([1, x, y, z]) for x in (1, -1) for y in (1, -1) for z in (1, -1)]
    else:
        q = [[math.cos(k * math.pi / 6), 0, 0, math.sin(k * math.pi / 6)] for k in range(6)]
        q += [[0, math.cos(k * math.pi / 6), math.sin(k * math.pi / 6), 0] for k in range(6)]
    return torch.tensor(np.array(q), dtype=F64, device="cuda")


def _canonical(shape, s, q):
    """(s', q', Q_k, Q_j, sign): s' = sign R(Q_k) s, q' = Q_k q Q_j, the representative that puts
    s' closest to (3, 2, 1) and q' closest to the identity, with a non-negative scalar part."""
    g = _group(shape)
    u = torch.tensor([3.0, 2.0, 1.0], dtype=F64, device="cuda")
    dots = s @ torch.einsum("kab,a->kb", _rot(g), u).T
    k = dots.abs().argmax(1)
    sg = torch.where(dots.gather(1, k[:, None])[:, 0] < 0, -1.0, 1.0).to(F64)
    qk = g[k]
    q1 = _qmul(qk, q)
    qj = g[(q1 @ _conj(g).T).abs().argmax(1)]
    q2 = _qmul(q1, qj)
    return sg[:, None] * _mv(_rot(qk), s), q2, qk, qj, sg


def _mlp_unpack(flat, width, depth=3):
    p, o = {}, 0
    for name, shp in ([("mu", (10,)), ("isd", (10,))]
                      + [x for l in range(depth) for x in (("W%d" % l, (width, 10 if l == 0 else width)), ("b%d" % l, (width,)))]
                      + [("wo", (width,)), ("bo", (1,)), ("es", (1,)), ("et", (1,))]):
        n = int(np.prod(shp))
        p[name] = flat[o:o + n].reshape(shp)
        o += n
    return p


def _mlp_energy(p, s, q, Rc, depth=3):
    qc = torch.where(q[:, :1] < 0, -q, q)
    rho = torch.sqrt((s * s).sum(1, keepdim=True))
    h = (torch.cat([s, qc, rho, 1.0 / rho, rho * rho], 1) - p["mu"]) * p["isd"]
    for l in range(depth):
        h = torch.nn.functional.silu(h @ p["W%d" % l].T + p["b%d" % l])
    E = p["es"] * (h @ p["wo"] + p["bo"]) + p["et"]
    r_on = float(np.float32(Rc - 1.0))
    t = ((rho[:, 0] - r_on) / (float(np.float32(Rc)) - r_on)).clamp(0.0, 1.0)
    return E * (1.0 - t ** 3 * (10.0 - 15.0 * t + 6.0 * t * t))


def _nn_pairs(p, shape, s, q, create_graph=False):
    """(E, F_j, tau_i, tau_j, dE/ds, dE/dq) in the frame of body i."""
    Rc = 2.0 * _body(shape)[3] + 2.5
    sc, qc, qk, qj, sg = _canonical(shape, s, q)
    sc, qc = sc.detach().requires_grad_(), qc.detach().requires_grad_()
    E = _mlp_energy(p, sc, qc, Rc)
    Gs, Gq = torch.autograd.grad(E.sum(), (sc, qc), create_graph=create_graph)
    if not create_graph:
        E = E.detach()
    Gs = sg[:, None] * _mv(_rot(qk).transpose(1, 2), Gs)
    Gq = _qmul(_qmul(_conj(qk), Gq), _conj(qj))
    # a small rotation theta of body j: dq = (0, theta) q / 2
    tj = -0.5 * _qmul(Gq, _conj(q))[:, 1:]
    ti = torch.linalg.cross(s, Gs) - tj
    return E, -Gs, ti, tj, Gs, Gq


def _chunked(f, s, q, step=65536):
    parts = [f(s[a:a + step], q[a:a + step]) for a in range(0, len(s), step)]
    return [torch.cat(z) for z in zip(*parts)]


def _fnet_frame(s, q):
    sz = torch.where(s[:, 2] < 0, -1.0, 1.0).to(F64)
    pr = torch.sqrt(s[:, 0] ** 2 + s[:, 1] ** 2)
    zero = torch.zeros_like(pr)
    xh = torch.stack([s[:, 0] / pr, s[:, 1] / pr, zero], 1)
    zh = torch.stack([zero, zero, sz], 1)
    yh = torch.linalg.cross(zh, xh)
    ax = _rot(q)[:, :, 2]
    u = torch.stack([(ax * e).sum(1) for e in (xh, yh, zh)], 1)
    u = torch.where(u[:, 2:] < 0, -u, u)
    d = torch.stack([pr, s[:, 2].abs(), torch.atan2(torch.hypot(u[:, 0], u[:, 1]), u[:, 2]),
                     torch.atan2(u[:, 1], u[:, 0])], 1)
    return xh, yh, zh, d


def _fnet_values(flat, width, d, depth=3):
    out = []
    for net in flat.reshape(5, -1):
        h, o = (d - net[:4]) * net[4:8], 8
        for l in range(depth):
            fan = 4 if l == 0 else width
            W = net[o:o + width * fan].reshape(width, fan)
            b = net[o + width * fan:o + width * (fan + 1)]
            h = torch.nn.functional.silu(h @ W.T + b)
            o += width * (fan + 1)
        out.append(net[o + width + 1] * (h @ net[o:o + width] + net[o + width]) + net[o + width + 2])
    return torch.stack(out, 1)


def _fnet_pairs(flat, width, s, q):
    xh, yh, zh, d = _fnet_frame(s, q)
    y = _fnet_values(flat, width, d)
    F = y[:, :1] * xh + y[:, 1:2] * yh + y[:, 2:3] * zh
    ti = y[:, 3:4] * xh + y[:, 4:5] * yh
    return torch.zeros_like(y[:, 0]), F, ti, -ti - torch.linalg.cross(s, F)


def _forces(path, shape, pairs, x, q, L, flat):
    """Per-body (F, half energies) and torque rows (n, 4) in FP64."""
    pot = "hphc" if path == "hphc_nvt" else "lj"
    Rc = float(np.float32(2.0 * _body(shape)[3] + _rcut(pot)))
    i, j = pairs.unbind(1)
    d = x[j] - x[i]
    d = d - L * torch.round(d / L)
    on = (d * d).sum(1) < Rc * Rc
    i, j, d = i[on], j[on], d[on]
    Ri = _rot(q[i])
    s = _mv(Ri.transpose(1, 2), d)
    qr = _qmul(_conj(q[i]), q[j])
    beads = lambda m: _bead_pairs(shape, pot, s[m], _rot(qr[m]))
    if path in ("beads", "hphc_nvt"):
        E, F, ti, tj = beads(slice(None))
    elif path == "fnet":
        E, F, ti, tj = _fnet_pairs(flat, 32, s, qr)
    else:
        p = _mlp_unpack(flat, 256 if path == "w256" else 128)
        E, F, ti, tj = _chunked(lambda a, b: _nn_pairs(p, shape, a, b)[:4], s, qr)
        m = (s * s).sum(1) < RHO_MIN[shape] ** 2
        E, F, ti, tj = (z.index_put((m,), w) for z, w in zip((E, F, ti, tj), beads(m)))
    F, ti, tj = _mv(Ri, F), _mv(Ri, ti), _mv(Ri, tj)
    out = x.new_zeros((2, len(x), 4))
    e = 0.5 * E[:, None]
    out[0].index_add_(0, j, torch.cat([F, e], 1)).index_add_(0, i, torch.cat([-F, e], 1))
    z = torch.zeros_like(e)
    out[1].index_add_(0, j, torch.cat([tj, z], 1)).index_add_(0, i, torch.cat([ti, z], 1))
    return out[0], out[1]


def _md(path, shape, st, L, pairs, flat, steps, dt):
    """Velocity Verlet with the NO_SQUISH rotation; Nose-Hoover halves around it for hphc_nvt."""
    _, M, I, _ = _body(shape)
    I = torch.tensor(I, dtype=F64, device="cuda")
    x, q, v, w = (st[k].double() for k in range(4))
    x, v, w = x[:, :3], v[:, :3], w[:, :3]
    dt = float(np.float32(dt))
    n = len(x)
    xi, kT = 0.0, float(np.float32(0.7))
    gkT = (6.0 * n - 3.0) * kT
    kin = lambda: float(0.5 * (M * (v * v).sum() + (w * w / I).sum()))
    F, T = _forces(path, shape, pairs, x, q, L, flat)
    for _ in range(steps):
        if path == "hphc_nvt":
            xi, v, w = _nose_hoover(xi, v, w, kin(), gkT, dt / 2)
        v = v + 0.5 * dt * F[:, :3] / M
        w = w + 0.5 * dt * _mv(_rot(q).transpose(1, 2), T[:, :3])
        x = torch.remainder(x + dt * v, L)
        for ax, frac in ((2, 0.5), (1, 0.5), (0, 1.0), (1, 0.5), (2, 0.5)):
            a, b = (ax + 1) % 3, (ax + 2) % 3
            phi = frac * dt * w[:, ax] / I[ax]
            r = torch.zeros_like(q)
            r[:, 0], r[:, 1 + ax] = torch.cos(0.5 * phi), torch.sin(0.5 * phi)
            q = _qmul(q, r)
            wa, wb = w[:, a].clone(), w[:, b].clone()
            w = w.clone()
            w[:, a] = torch.cos(phi) * wa + torch.sin(phi) * wb
            w[:, b] = torch.cos(phi) * wb - torch.sin(phi) * wa
        q = q / q.norm(dim=1, keepdim=True)
        F, T = _forces(path, shape, pairs, x, q, L, flat)
        v = v + 0.5 * dt * F[:, :3] / M
        w = w + 0.5 * dt * _mv(_rot(q).transpose(1, 2), T[:, :3])
        if path == "hphc_nvt":
            xi, v, w = _nose_hoover(xi, v, w, kin(), gkT, dt / 2)
    pad = lambda z: torch.cat([z, torch.zeros_like(z[:, :1])], 1)
    return {"pos": pad(x), "quat": q, "vel": pad(v), "angmom": pad(w)}


def _nose_hoover(xi, v, w, K, gkT, h, tau=1.0):
    Q = gkT * tau * tau
    xi += 0.5 * h * (2.0 * K - gkT) / Q
    sc = math.exp(-xi * h)
    xi += 0.5 * h * (2.0 * K * sc * sc - gkT) / Q
    return xi, v * sc, w * sc


def _adam(params, grads, mask, m, v, t):
    m.mul_(0.9).add_(grads, alpha=0.1)
    v.mul_(0.999).add_(grads * grads, alpha=0.001)
    step = LR * (m / (1.0 - 0.9 ** t)) / ((v / (1.0 - 0.999 ** t)).sqrt() + 1e-8)
    return torch.where(mask, params - step, params)


def _fit(flat, mask, batches, loss_of):
    """The monitored loss and gradient on the first batch, then Adam over the others."""
    def grad(f, batch):
        f = f.detach().requires_grad_()
        loss = loss_of(f, *batch)
        g, = torch.autograd.grad(loss, f)
        return float(loss.detach()), torch.where(mask, g, torch.zeros_like(g))
    loss, first = grad(flat, batches[0])
    m, v = torch.zeros_like(flat), torch.zeros_like(flat)
    for t, b in enumerate(batches[1:], 1):
        flat = _adam(flat, grad(flat, b)[1], mask, m, v, t)
    return {"loss": np.float64(loss), "grad": first, "params": flat}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("md", "forces"):
        if kind == "md" and case["path"] in ("beads", "hphc_nvt") and case["n"] * case["steps"] > 800000:
            return None  # the FP64 bead sums would take over 20 s
        shape, path = case["shape"], case["path"]
        st, L, pairs = _fluid(shape, case["n"], case["phi"], seed)
        Rc = 2.0 * _body(shape)[3] + 2.5
        flat = {"fnet": lambda: _fnet_flat(32, seed + 1, float(np.float32(Rc))),
                "w256": lambda: _mlp_flat(256, seed + 1, Rc)}.get(path, lambda: _mlp_flat(128, seed + 1, Rc))()
        flat = torch.from_numpy(flat).double().cuda()
        if kind == "md":
            return _md(path, shape, st, L, pairs, flat, case["steps"], 0.005 if path == "hphc_nvt" else 0.002)
        F, T = _forces(path, shape, pairs, st[0, :, :3].double(), st[1].double(), L, flat)
        return {"force": F, "torque": T}
    if kind == "pairs":
        c = _configs("cube", case["n"], seed).double()
        Rc = 2.0 * _body("cube")[3] + 2.5
        p = _mlp_unpack(torch.from_numpy(_mlp_flat(case["width"], seed + 1, Rc)).double().cuda(), case["width"])
        E, F, ti, tj, Gs, Gq = _chunked(lambda a, b: _nn_pairs(p, "cube", a, b), c[:, :3], c[:, 4:])
        z = torch.zeros_like(E[:, None])
        return {"out": torch.cat([F, E[:, None], ti, z, tj, z], 1), "grad": torch.cat([Gs, z, Gq], 1)}
    if kind in ("train", "fntrain"):
        shape, batches = _train_inputs(case, seed)
        w, Rc = case["width"], 2.0 * _body(shape)[3] + 2.5
        batches = [(c.double(), l.double()) for c, l in batches]
        if kind == "train":
            flat = torch.from_numpy(_mlp_flat(w, seed + 1, Rc)).double().cuda()
            mask = torch.ones_like(flat, dtype=torch.bool)
            mask[:20] = False
            mask[-2:] = False

            def loss_of(f, c, lab):
                E, F, ti, tj, _, _ = _nn_pairs(_mlp_unpack(f, w), shape, c[:, :3], c[:, 4:], True)
                F0, ti0, tj0 = lab[:, :3], lab[:, 4:7], lab[:, 8:11]
                sq = lambda z: (z * z).sum(1)
                wt = 1.0 / (1.0 + (sq(F0) + sq(ti0) + sq(tj0)) / 4.0)
                lam = float(np.float32(0.1))
                return (wt * (sq(F - F0) + sq(ti - ti0) + sq(tj - tj0) + lam * (E - lab[:, 3]) ** 2)).mean()
            return _fit(flat, mask, batches, loss_of)
        flat = torch.from_numpy(_fnet_flat(w, seed + 1, Rc)).double().cuda()
        mask = torch.ones((5, len(flat) // 5), dtype=torch.bool, device="cuda")
        mask[:, :8] = False
        mask[:, -2:] = False

        def loss_fn(f, c, lab):
            xh, yh, zh, d = _fnet_frame(c[:, :3], c[:, 4:])
            dot = lambda a, b: (a * b).sum(1)
            F0, t0 = lab[:, :3], lab[:, 4:7]
            t = torch.stack([dot(F0, xh), dot(F0, yh), dot(F0, zh), dot(t0, xh), dot(t0, yh)], 1).clamp(-5.0, 5.0)
            wt = 1.0 / (1.0 + (t * t).sum(1))
            return (wt * ((_fnet_values(f, w, d) - t) ** 2).sum(1)).mean()
        return _fit(flat, mask.reshape(-1), batches, loss_fn)
    if kind == "sample":
        u = torch.from_numpy(np.random.default_rng(seed).random((case["n"], 6), dtype=np.float32)).double().cuda()
        shape = case["shape"]
        Rc = float(np.float32(2.0 * _body(shape)[3] + 2.5))
        t = torch.from_numpy(_template(shape)).cuda()
        z, tp = 2.0 * u[:, 0] - 1.0, 2.0 * math.pi
        xy = torch.sqrt((1.0 - z * z).clamp(min=0.0))
        dr = torch.stack([xy * torch.cos(tp * u[:, 1]), xy * torch.sin(tp * u[:, 1]), z], 1)
        a, b = torch.sqrt(1.0 - u[:, 2]), torch.sqrt(u[:, 2])
        q = torch.stack([a * torch.sin(tp * u[:, 3]), a * torch.cos(tp * u[:, 3]),
                         b * torch.sin(tp * u[:, 4]), b * torch.cos(tp * u[:, 4])], 1)
        R = _rot(q)
        lo, hi = torch.zeros_like(z), torch.full_like(z, Rc)
        contact = float(np.float32(case["contact"]))
        for _ in range(40):
            mid = 0.5 * (lo + hi)
            close = _min_bead_distance(mid[:, None] * dr, R, t) < contact
            lo, hi = torch.where(close, mid, lo), torch.where(close, hi, mid)
        rc = 0.5 * (lo + hi)
        s = (rc + u[:, 5] * (Rc - rc))[:, None] * dr
        E, F, ti, tj = _bead_pairs(shape, "lj", s, R)
        zero = torch.zeros_like(E[:, None])
        return {"cfg": torch.cat([s, zero, q], 1),
                "labels": torch.cat([F, E[:, None], ti, zero, tj, zero], 1), "rho_contact": rc}
    if case["replicas"] * case["n_max"] * case["steps"] > 3000000:
        return None
    Rc = 2.0 * _body("cube")[3] + 2.5
    flat = torch.from_numpy(_mlp_flat(128, seed + 1, Rc)).double().cuda()
    return [_md(path, "cube", st, L, pairs, flat, case["steps"], 0.002)
            for path, st, L, pairs in _replicas(case, seed)]
