"""The network kernels at the edges of their tiles: one and several rows, a tile's remainder, as many
tiles as SMs (one tile per CTA), one more (two tiles in flight per SM, an odd number of them), and a
gradient of more tiles than CTAs, against the oracle. Bounds as in test_gpu_mlp."""
import numpy as np
import pytest

from oracle import mlp as om
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_mlp import FWD_MAX, FWD_MEAN, GRAD_REL, _blocks, _net, _norm_for, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles,extra", [(0, 2), (1, -1), (1, 1), ("sms", 0), ("sms", 1), ("sms", 129)])
def test_forward_tiles(torch_cuda, tiles, extra):  # noqa: F811
    torch = torch_cuda
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = 128 * (sms if tiles == "sms" else tiles) + extra
    feat, tgt = wl.mlp_random_data(B, 50 + B)
    p, norm = _net(B), _norm_for(feat, tgt)
    net = lpdf.MLP(1)
    net.set_params(p, norm)
    out = torch.full((B + 1, 7), 5.0, dtype=torch.float32, device="cuda")
    net.forward(torch.from_numpy(feat).cuda(), out[:B])
    got = out.cpu().numpy().astype(np.float64)
    d = np.abs(got[:B] - om.forward_user(p.astype(np.float64), norm.astype(np.float64), feat)) / norm[30:37]
    assert d.max() <= FWD_MAX and d.mean() <= FWD_MEAN, (d.max(), d.mean())
    assert np.all(got[B] == 5.0)                       # nothing past the last row


@pytest.mark.parametrize("B", [1, 129, 152 * 128 + 130])
def test_gradient_tiles(torch_cuda, B):  # noqa: F811
    torch = torch_cuda
    feat, tgt = wl.mlp_random_data(max(B, 8), 60 + B)
    p, norm = _net(3 + B), _norm_for(feat, tgt)
    feat, tgt = feat[:B], tgt[:B]
    net = lpdf.MLP(B)
    net.set_params(p, norm)
    g, L = net.gradient(torch.from_numpy(feat).cuda(), torch.from_numpy(tgt).cuda())
    want, Lw = om.gradient(p.astype(np.float64), norm.astype(np.float64), feat, tgt, bf16_ops=True)
    assert L == pytest.approx(Lw, rel=1e-3)
    for a, b in _blocks():
        e = np.linalg.norm(g[a:b] - want[a:b]) / np.linalg.norm(want[a:b])
        assert e <= GRAD_REL, (a, b, e)
