"""lpdf_set_state / lpdf_get_state with on_device = 1 and arrays that a kernel cannot use as they are: odd
addresses, host memory. They are copied, or the call returns an error and leaves the ensemble as it was; a
kernel never touches them. (Arrays of another GPU take the same way.)"""
import ctypes

import numpy as np
import pytest

from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_state_layout import KEYS, _state, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu
N, NS = 1003, 3


def _context():
    return lpdf.Context(lpdf.Mesh(wl.channel_mesh(5, 4, 3)), lpdf.make_params(ns=NS), 2 * N)


def _call(ctx, name, n, pointers):
    p = [ctypes.c_void_p(q) for q in pointers]
    f = getattr(lpdf.lib(), name)
    return f(ctx.h, n, *p, 1, lpdf._stream(None)) if name == "lpdf_set_state" else f(ctx.h, *p, 1, lpdf._stream(None))


def _same(ctx, st):
    got = ctx.get_state(device=False)
    return all(np.array_equal(got[k].view(np.uint32), st[k].view(np.uint32)) for k in KEYS)


@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_device_arrays_at_odd_addresses(torch_cuda, offset):  # noqa: F811
    torch = torch_cuda
    ctx, st = _context(), _state(N, NS, 3)
    bufs = []
    for k in KEYS:
        raw = st[k].reshape(-1).view(np.uint8)
        b = torch.zeros(raw.size + 16, dtype=torch.uint8, device="cuda")
        b[offset:offset + raw.size] = torch.from_numpy(raw.copy()).cuda()
        bufs.append(b)
    assert _call(ctx, "lpdf_set_state", N, [b.data_ptr() + offset for b in bufs]) == lpdf.LPDF_OK
    assert _same(ctx, st)
    for b in bufs:
        b.zero_()
    assert _call(ctx, "lpdf_get_state", N, [b.data_ptr() + offset for b in bufs]) == lpdf.LPDF_OK
    for k, b in zip(KEYS, bufs):
        raw = st[k].reshape(-1).view(np.uint8)
        assert np.array_equal(b.cpu().numpy()[offset:offset + raw.size], raw), k
        assert int(b[:offset].sum()) == 0 and int(b[offset + raw.size:].sum()) == 0


@pytest.mark.parametrize("pinned", [False, True])
def test_host_memory_given_as_device_memory(torch_cuda, pinned):  # noqa: F811
    torch = torch_cuda
    ctx, first, st = _context(), _state(N - 3, NS, 4), _state(N, NS, 5)
    ctx.set_state(first)
    host = {}
    for k in KEYS:
        t = torch.zeros(st[k].shape, dtype=torch.int32, pin_memory=pinned)
        host[k] = t.numpy().view(st[k].dtype)
        host[k][...] = st[k]
    rc = _call(ctx, "lpdf_set_state", N, [host[k].ctypes.data for k in KEYS])
    torch.cuda.synchronize()
    assert rc in (lpdf.LPDF_OK, lpdf.LPDF_ERR_CUDA)          # as cudaMemcpyAsync takes such addresses
    assert _same(ctx, st if rc == lpdf.LPDF_OK else first)
