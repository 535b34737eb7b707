"""Host arrays of lpdf_set_state / lpdf_get_state: page-locked ones, which a kernel moves itself, and pageable
ones through the staging buffer that the context keeps: with little memory left, and from several streams."""
import numpy as np
import pytest

from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_state_layout import KEYS, _state, torch_cuda  # noqa: F401
from tests.test_gpu_state_no_memory import MB, small_pool

pytestmark = pytest.mark.gpu


def _context(n, ns):
    return lpdf.Context(lpdf.Mesh(wl.channel_mesh(5, 4, 3)), lpdf.make_params(ns=ns), n)


def _equal(got, st):
    return all(np.array_equal(got[k].view(np.uint32), st[k].view(np.uint32)) for k in KEYS)


@pytest.mark.parametrize("ns,n", [(1, 1), (2, 33), (3, 1021), (4, 100003)])
def test_page_locked_arrays(torch_cuda, ns, n):  # noqa: F811
    torch = torch_cuda
    ctx, st = _context(n, ns), _state(n, ns, 11)
    pinned = {}
    for k in KEYS:
        pinned[k] = torch.zeros(st[k].shape, dtype=torch.int32, pin_memory=True).numpy().view(st[k].dtype)
        pinned[k][...] = st[k]
    ctx.set_state(pinned)
    torch.cuda.synchronize()
    for k in KEYS:
        pinned[k].view(np.uint32)[...] = 0
    p = lpdf._ptr
    assert lpdf.lib().lpdf_get_state(ctx.h, *[p(pinned[k]) for k in KEYS], 0, lpdf._stream(None)) == lpdf.LPDF_OK
    torch.cuda.synchronize()
    assert _equal(pinned, st)


def test_little_memory(torch_cuda):  # noqa: F811
    n, ns = (1 << 22) + 5, 2
    ctx, st = _context(n, ns), _state(n, ns, 12)
    with small_pool(torch_cuda, 32 * MB, False):             # the whole staging buffer would take 168 MB
        ctx.set_state(st)
        assert _equal(ctx.get_state(device=False), st)
        del ctx


def test_streams_take_turns(torch_cuda):  # noqa: F811
    torch = torch_cuda
    n, ns = 200001, 2
    ctx = _context(n, ns)
    streams = [torch.cuda.Stream() for _ in range(3)]
    last = torch.cuda.Event()
    for k in range(6):
        s = streams[k % 3]
        st = _state(n, ns, 20 + k)
        s.wait_event(last) if k else None                     # the ensemble itself is the caller's to order
        ctx.set_state(st, stream=s)
        last.record(s)
        t = streams[(k + 1) % 3]
        t.wait_event(last)
        assert _equal(ctx.get_state(stream=t, device=False), st)
        last.record(t)
