"""lpdf_set_state / lpdf_get_state when device memory is short (a memory pool of the test's own, small and,
where asked, all in use, stands in for a full GPU): a failed set leaves the ensemble usable."""
import contextlib
import ctypes

import numpy as np
import pytest

from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests import gpu_common as gc
from tests.test_gpu_state_layout import KEYS, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu
MB = 1 << 20


class PoolProps(ctypes.Structure):      # CUmemPoolProps: pinned memory of device 0
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("loc_type", ctypes.c_int),
                ("loc_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def small_pool(torch, size, in_use):
    """Stream-ordered allocations of the device from a pool of at most `size` bytes."""
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(rc):
        assert rc == 0, rc

    pool, old, p = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    props = PoolProps(alloc_type=1, loc_type=1, loc_id=0, max_size=size)
    ok(cu.cuDeviceGetMemPool(ctypes.byref(old), 0))
    ok(cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)))
    held = []
    if in_use:
        step = size
        while step >= 512:
            if cu.cuMemAllocFromPoolAsync(ctypes.byref(p), ctypes.c_size_t(step), pool, None) == 0:
                held.append(p.value)
            else:
                step //= 2
    ok(cu.cuDeviceSetMemPool(0, pool))
    try:
        yield
    finally:
        torch.cuda.synchronize()
        ok(cu.cuDeviceSetMemPool(0, old))
        for q in held:
            ok(cu.cuMemFreeAsync(ctypes.c_void_p(q), None))
        torch.cuda.synchronize()
        ok(cu.cuMemPoolDestroy(pool))


def test_a_failed_set_leaves_the_ensemble(torch_cuda):  # noqa: F811
    torch = torch_cuda
    mesh = wl.channel_mesh(25, 20, 3)
    ns = 2
    params = lpdf.make_params(ns=ns)
    ctx = lpdf.Context(lpdf.Mesh(mesh), params, mesh.n_tri * 60)
    F = torch.from_numpy(wl.synthetic_node_fields(mesh, ns, seed=5)).cuda()
    st, more = wl.synthetic_state(mesh, 20, ns, seed=7), wl.synthetic_state(mesh, 60, ns, seed=8)
    ctx.set_state(gc.torch_state(st))
    before = ctx.get_state()
    with small_pool(torch, 32 * MB, True):
        with pytest.raises(lpdf.LpdfError) as e:
            ctx.set_state(more)
        assert e.value.code == lpdf.LPDF_ERR_CUDA
    assert ctx.n == mesh.n_tri * 20
    after = ctx.get_state()
    assert all(torch.equal(after[k].view(torch.int32), before[k].view(torch.int32)) for k in KEYS)
    ctx.pdf_step(F, 1)
    ctx.status()
    ctx.set_state(more)
    assert ctx.n == mesh.n_tri * 60 and np.array_equal(ctx.get_state(device=False)["x"], more.x)
