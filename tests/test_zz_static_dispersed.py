"""The no-allocation step on ensembles in no order: sub-tiles of 512 particles over fewer elements than
bins, over more (the direct path for the rest), and over as many as the bin hash holds and more (no bins
at all). States against the oracle's step, sums against its reduction."""
import numpy as np
import pytest

import oracle
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests import gpu_common as gc
from tests.test_gpu_state_layout import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [1, 4])
@pytest.mark.parametrize("elements", [40, 200, 256, 1600])
def test_static_step_of_a_dispersed_ensemble(torch_cuda, elements, ns):  # noqa: F811
    torch = torch_cuda
    mesh = wl.channel_mesh(40, 20, 9)
    rng = np.random.default_rng(elements + ns)
    st = wl.synthetic_state(mesh, 30, ns, 4, speed=0.1)
    keep = np.isin(st.elem, rng.choice(mesh.n_tri, elements, replace=False))
    pick = rng.permutation(np.nonzero(keep)[0])[:512 * 2 + 77]
    st = gc.reorder(st, pick)
    om = oracle.OracleMesh(mesh)
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(ns=ns, seed=11)
    F = wl.synthetic_node_fields(mesh, ns, seed=5)
    state = gc.torch_state(st)
    S = torch.full((gm.n_nodes, 11 + 2 * ns), float("nan"), dtype=torch.float64, device="cuda")
    rc, status = lpdf.pdf_step_static(gm, params, state, torch.from_numpy(F).cuda(), 3, S)
    assert rc == lpdf.LPDF_OK, status
    g = gc.host_state(state, ns)
    gc.compare_step(mesh, om, params, F, st, 3, g)
    gc.compare_moments(om, g, S.cpu().numpy(), ns)
    first = S.clone()
    again = gc.torch_state(st)
    rc, _ = lpdf.pdf_step_static(gm, params, again, torch.from_numpy(F).cuda(), 3, S)
    assert rc == lpdf.LPDF_OK and torch.equal(S, first)      # the same bits every time
