"""Force and torque rows in memory of other kinds than this device's own (page-locked host memory, managed
memory): the rows of a call are those of the same call into device memory."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_templates import _grid, _state, _system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("kind", ["page-locked", "managed"])
def test_rows_in_memory_of_another_kind(kind):
    import torch

    from paper_2402_12199_gb300 import api

    n = 125
    pos, quat, L = _state(_grid((4, 4, 5)), n, 11)
    s = _system(_grid((4, 4, 5)), pos, quat, L)
    ref = s.forces_beads()
    s.sync()
    if kind == "page-locked":
        rows = torch.zeros((2, n, 4)).pin_memory()
        at, view = rows.data_ptr(), rows.numpy()
    else:
        cuda = ctypes.CDLL("libcuda.so.1")
        p = ctypes.c_uint64()
        assert cuda.cuMemAllocManaged(ctypes.byref(p), ctypes.c_size_t(2 * n * 16), ctypes.c_uint(1)) == 0
        at = p.value
        view = np.ctypeslib.as_array(ctypes.cast(at, ctypes.POINTER(ctypes.c_float)), (2, n, 4))
        view[:] = 0.0
    api.check(api.load().rb_forces_beads(s.handle, at, at + 16 * n, None, None))
    s.sync()
    assert np.array_equal(view[0], ref["force"].cpu().numpy())
    assert np.array_equal(view[1], ref["torque"].cpu().numpy())
    if kind == "managed":
        assert cuda.cuMemFree_v2(p) == 0
