"""A trainer destroyed after its network (as the end of a Python process may order it): the trainer's
memory is freed without looking at the network."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np
import torch
import __graft_entry__ as g
g.build()
from oracle import fnet
from paper_2402_12199_gb300 import api, inputs
for i in range(20):
    mu, isd = inputs.feature_normalisation(5.0, 9.43)
    m = api.MLP(64, 2)
    m.set_params(inputs.mlp_params(64, 2, 3, mu=mu, inv_sd=isd))
    f = api.FNet(16, 2)
    f.set_params(np.zeros(5 * fnet.net_size(16, 2), np.float32))
    pairs = []
    for net, make in ((m, api.Trainer), (f, api.FNetTrainer)):
        t = make(net, 64)
        t.grad(torch.ones(64, 8, device="cuda"), torch.ones(64, 12, device="cuda"))
        pairs.append((net, t))
    for net, t in pairs:
        net.__del__()
        junk = [bytearray(b"\\xff" * 400) for _ in range(2000)]  # the network's memory in other hands
        t.__del__()
torch.cuda.synchronize()
print("destroyed in either order")
"""


def test_trainer_outlives_its_network():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "either order" in r.stdout, r.stderr[-2000:]
