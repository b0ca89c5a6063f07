"""Tensor-core networks of growing depth in one process (a process of its own: the kernels' shared-memory
limits are set once in it): a deeper network after a shallower one of the same width and precision."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch
import __graft_entry__ as g
g.build()
from paper_2402_12199_gb300 import api, inputs
from tests.helpers import gpu_system, make_state
mu, isd = inputs.feature_normalisation(5.0, 9.43)
st, L, _ = make_state(64, 0.2, 3)
s = gpu_system(st, L, "cube")
q = torch.randn(300, 8, device="cuda")
q[:, 4:] /= q[:, 4:].norm(dim=1, keepdim=True)
for width, precision in ((128, "bf16"), (128, "f16x3"), (256, "bf16")):
    for depth in (1, 2, 3):
        m = api.MLP(width, depth)
        m.set_params(inputs.mlp_params(width, depth, 3, mu=mu, inv_sd=isd))
        assert torch.isfinite(m.pairs(q, precision)).all()
        assert torch.isfinite(s.forces_nn(m, precision)["force"]).all()
        s.sync()
print("all depths ran")
"""


def test_deeper_networks_after_shallower_ones():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "all depths ran" in r.stdout, r.stderr[-2000:]
