"""The re-bucketing of a step on both sides of its dispatch lines (one cluster for small ensembles, several
launches above; one scan launch for few tiles of elements, three for many): the order that a step
leaves is the stable counting sort of its elements, so the next step's listing is known exactly; the
sums agree with the oracle's reduction."""
import numpy as np
import pytest

import oracle
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests import gpu_common as gc
from tests.test_gpu_state_layout import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

# (nx, ny), particles: one block; a block's remainder; the cluster's limit and one more; its limit of
# elements and above; more tiles of elements than one scan launch takes
CASES = [((3, 2), 1), ((3, 2), 257), ((25, 20), 1 << 17), ((25, 20), (1 << 17) + 1), ((89, 46), 40000),
         ((64, 64), 40000), ((300, 120), 30000)]


@pytest.mark.parametrize("cells,n", CASES)
@pytest.mark.parametrize("order", ["sorted", "random"])
def test_order_after_a_step(torch_cuda, cells, n, order):  # noqa: F811
    torch = torch_cuda
    mesh = wl.channel_mesh(*cells, 9)
    st = wl.synthetic_state(mesh, -(-n // mesh.n_tri), 1, 4)
    pick = np.sort(np.random.default_rng(n).choice(st.n, n, replace=False))
    if order == "random":
        np.random.default_rng(1).shuffle(pick)
    st = gc.reorder(st, pick)
    gm = lpdf.Mesh(mesh)
    ctx = lpdf.Context(gm, lpdf.make_params(seed=3), n)
    F = torch.from_numpy(wl.synthetic_node_fields(mesh, 1, seed=5)).cuda()
    ctx.set_state(gc.torch_state(st))
    for step in (1, 2, 3):
        before = gc.host_state(ctx.get_state(), 1)
        ctx.pdf_step(F, step)
        after = gc.host_state(ctx.get_state(), 1)
        # the first step lists the input order, a later one the previous listing sorted by element
        want = before.pid if step == 1 else before.pid[np.argsort(before.elem, kind="stable")]
        assert np.array_equal(after.pid, want)
    ctx.status()
    S = torch.empty((gm.n_nodes, 13), dtype=torch.float64, device="cuda")
    ctx.grid_statistics(S, raw=True)
    gc.compare_moments(oracle.OracleMesh(mesh), after, S.cpu().numpy(), 1)
