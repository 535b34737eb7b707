"""The no-allocation step of particles that end far outside the walls (further than eight mirrorings take them
back): reported as lost, each after the hops of the oracle's walk, which leaves through a wall only where
no interior edge is crossed."""
import numpy as np
import pytest

import oracle
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests import gpu_common as gc
from tests.test_gpu_state_layout import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["channel", "cavity"])
def test_hops_of_lost_particles(torch_cuda, kind):  # noqa: F811
    torch = torch_cuda
    mesh = wl.channel_mesh(25, 20, 5) if kind == "channel" else wl.cavity_mesh(20, 20, 5)
    om = oracle.OracleMesh(mesh)
    st = wl.synthetic_state(mesh, 1, 1, 6)
    out = np.random.default_rng(7).random(st.n) < 0.5
    st.v[out] = np.where(st.pid[out] % 2 == 0, 3.0e4, -3.0e4).astype(np.float32)
    state = gc.torch_state(st)
    S = torch.zeros((mesh.n_nodes, 13), dtype=torch.float64, device="cuda")
    F = torch.from_numpy(wl.synthetic_node_fields(mesh, 1, seed=5)).cuda()
    rc, status = lpdf.pdf_step_static(lpdf.Mesh(mesh), lpdf.make_params(ns=1, dt=1e-3), state, F, 0, S)
    assert rc == lpdf.LPDF_ERR_LOST_PARTICLE
    g = gc.host_state(state, 1)
    walks = [om.locate_walk(e, x, y) for e, x, y in zip(st.elem, g.x, g.y)]
    owner, hops = np.array([w[0] for w in walks]), np.array([w[1] for w in walks])
    assert (owner < 0).sum() > 50
    assert status[1] == (owner < 0).sum()
    assert np.array_equal(g.elem, np.where(owner < 0, st.elem, owner))
    assert status[3] == hops.sum()
