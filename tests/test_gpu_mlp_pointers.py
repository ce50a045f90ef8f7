"""Targets and loss pointers that kernels cannot use in place: the training step copies
them, and a pointer that the copy refuses is an error of the call, not a fault.  Targets in
device memory, pinned host memory and at an address off the 4-byte grid give the same step;
ordinary host memory gives the same step or MPM_ECUDA, after which the network goes on.
"""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2507_04192_gb300 import mpm

pytestmark = pytest.mark.gpu

WIDTHS, BATCH = [24, 40, 16], 32


def network(stream):
    rng = np.random.default_rng(3)
    net = mpm.MLP(WIDTHS, BATCH, stream=stream.cuda_stream)
    net.set_params((0.2 * rng.standard_normal(net.num_params)).astype(np.float32))
    return net, torch.tensor(rng.standard_normal((BATCH, 24)), dtype=torch.float32), \
        torch.tensor(rng.uniform(0.1, 0.6, (BATCH, 16)), dtype=torch.float32)


def step(net, x, t_ptr, loss_ptr, stream):
    net.train_step_async(BATCH, x.data_ptr(), t_ptr, 1e-3, loss_ptr)
    stream.synchronize()
    return net.get_params(1), net.get_params(0)


@pytest.fixture(scope="module")
def reference():
    stream = torch.cuda.Stream()
    net, x, t = network(stream)
    xd, td, loss = x.cuda(), t.cuda(), torch.zeros(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    g, p = step(net, xd, td.data_ptr(), loss.data_ptr(), stream)
    net.close()
    return g, p, float(loss.item())


@pytest.mark.parametrize("where", ["pinned", "off the grid", "host"])
def test_targets_in_other_memory(reference, where):
    stream = torch.cuda.Stream()
    net, x, t = network(stream)
    xd, loss = x.cuda(), torch.zeros(1, dtype=torch.float64, device="cuda")
    if where == "pinned":
        keep = t.pin_memory()
        ptr = keep.data_ptr()
    elif where == "off the grid":
        raw = np.zeros(4 * t.numel() + 4, dtype=np.uint8)
        raw[1:-3] = np.frombuffer(t.numpy().tobytes(), dtype=np.uint8)
        keep = torch.from_numpy(raw).cuda()
        ptr = keep.data_ptr() + 1
    else:
        keep = t.numpy().copy()
        ptr = keep.ctypes.data
    torch.cuda.synchronize()
    try:
        g, p = step(net, xd, ptr, loss.data_ptr(), stream)
    except mpm.MPMError as e:
        assert where == "host" and e.code == mpm.MPM_ECUDA
        td = t.cuda()
        torch.cuda.synchronize()
        g, p = step(net, xd, td.data_ptr(), loss.data_ptr(), stream)
    net.close()
    np.testing.assert_array_equal(g, reference[0])
    np.testing.assert_array_equal(p, reference[1])
    assert float(loss.item()) == pytest.approx(reference[2], rel=1e-12)


@pytest.mark.parametrize("where", ["pinned", "off the grid", "host", "none"])
def test_loss_pointers_in_other_memory(reference, where):
    stream = torch.cuda.Stream()
    net, x, t = network(stream)
    xd, td = x.cuda(), t.cuda()
    host = C.c_double(0.0)
    pinned, raw = torch.zeros(1, dtype=torch.float64).pin_memory(), torch.zeros(12, dtype=torch.uint8, device="cuda")
    ptr = {"pinned": pinned.data_ptr(), "off the grid": raw.data_ptr() + 4, "host": C.addressof(host), "none": 0}[where]
    torch.cuda.synchronize()
    refused = False
    try:
        g, p = step(net, xd, td.data_ptr(), ptr, stream)
    except mpm.MPMError as e:
        assert where == "host" and e.code == mpm.MPM_ECUDA
        refused = True
        stream.synchronize()
        g, p = net.get_params(1), net.get_params(0)
    net.close()
    np.testing.assert_array_equal(g, reference[0])
    np.testing.assert_array_equal(p, reference[1])
    got = {"pinned": lambda: float(pinned[0]), "host": lambda: host.value, "none": lambda: reference[2],
           "off the grid": lambda: np.frombuffer(raw.cpu().numpy().tobytes()[4:12], dtype=np.float64)[0]}[where]()
    assert refused or got == pytest.approx(reference[2], rel=1e-12)
