"""The learned fallback's evaluation when one thread's wait runs out and the
others' do not: every thread reaches the group's vote, so the launch ends, with
the error word set, whatever thread it is and whether tiles are left or not."""
import ctypes
import time

import pytest
import torch

from mlp_cases import random_weights
from paper_1902_05942_gb300 import pps
from test_gpu_launch_shapes import _vertices


@pytest.mark.parametrize("row,tiles", [(-1, 1), (128, 1), (0, 0), (0, 4)])
def test_arguments(row, tiles):
    w = ctypes.c_uint32(7)
    assert pps.lib().pps_selftest_infer(row, tiles, ctypes.byref(w)) == pps.PPS_EINVAL
    assert pps.lib().pps_selftest_infer(0, 1, None) == pps.PPS_EINVAL


@pytest.mark.gpu
@pytest.mark.parametrize("row", [0, 1, 31, 32, 95, 127])
@pytest.mark.parametrize("tiles", [1, 2, 3])
def test_a_thread_that_gives_up_alone(row, tiles):
    from paper_1902_05942_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    t0 = time.perf_counter()
    assert pps.pps_selftest_infer(row, tiles) == 1
    assert time.perf_counter() - t0 < 10.0
    # the context, and the tensor memory, are still usable
    net = pps.MLP(pps.mlp_params(), init=random_weights(5))
    v = _vertices(2000, 3)
    a, b = net.forward(v), net.forward(v)
    assert all(torch.equal(a[c], b[c]) and torch.isfinite(a[c]).all() for c in "rgb")
    net.close()
