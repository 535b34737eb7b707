"""lpdf_set_state / lpdf_get_state against the context's own particle layout: every scalar count, host and
device arrays, more particles than one staging block, rows that the caller leaves out."""
import numpy as np
import pytest

from paper_1006_0549_gb300 import lpdf, workloads as wl

pytestmark = pytest.mark.gpu
KEYS = ("x", "y", "u", "v", "w", "omega", "psi", "elem", "pid")


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1006_0549_gb300 import _build
    _build.build()
    return torch


def _state(n, ns, seed):
    rng = np.random.default_rng(seed)
    st = {k: rng.standard_normal(n).astype(np.float32) for k in KEYS[:6]}
    st["psi"] = rng.random((ns, n)).astype(np.float32)
    st["elem"] = rng.integers(0, 40, n).astype(np.int32)
    st["pid"] = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)     # every bit pattern: NaNs too
    return st


@pytest.mark.parametrize("ns,n", [(1, 1), (1, 1000), (2, 257), (3, 4097), (4, 333), (2, (1 << 22) + 5)])
def test_round_trip(torch_cuda, ns, n):
    torch = torch_cuda
    mesh = lpdf.Mesh(wl.channel_mesh(5, 4, 3))
    ctx = lpdf.Context(mesh, lpdf.make_params(ns=ns), n)
    st = _state(n, ns, n + ns)
    ctx.set_state(st)
    for device in (False, True):
        got = ctx.get_state(device=device)
        for k in KEYS:
            g = got[k].cpu().numpy() if device else got[k]
            assert np.array_equal(g.view(np.uint32), st[k].view(np.uint32)), (k, device)
    dev = {k: torch.from_numpy(v.view(np.int32) if v.dtype == np.uint32 else v).cuda() for k, v in _state(n, ns, 7).items()}
    ctx.set_state(dev)
    back = ctx.get_state()
    assert all(torch.equal(back[k].view(torch.int32), dev[k].view(torch.int32)) for k in KEYS)
    # only x and psi wanted
    x, psi = torch.zeros(n, device="cuda"), torch.zeros((ns, n), device="cuda")
    p = lpdf._ptr
    rc = lpdf.lib().lpdf_get_state(ctx.h, p(x), None, None, None, None, None, p(psi), None, None, 1, lpdf._stream(None))
    assert rc == lpdf.LPDF_OK and torch.equal(x, dev["x"]) and torch.equal(psi, dev["psi"])
    hx = np.zeros(n, dtype=np.float32)
    rc = lpdf.lib().lpdf_get_state(ctx.h, p(hx), None, None, None, None, None, None, None, None, 0, lpdf._stream(None))
    torch.cuda.synchronize()
    assert rc == lpdf.LPDF_OK and np.array_equal(hx, dev["x"].cpu().numpy())
