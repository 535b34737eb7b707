"""A CG whose thread block gives up a wait: the solve returns LPDF_ERR_CUDA and leaves the caller's fields
and the warm start alone, whether or not the first block saw every system converge; the next solve is
right. Nothing hangs: every wait is bounded, here to a few ms. Bounds as in test_gpu_fields."""
import numpy as np
import pytest

from oracle import fields as of
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_cg import MESHES
from tests.test_gpu_fields import _compare, _solve, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


# the block that gives up: a unit of the small kernel's first component; one that collects no sums
@pytest.mark.parametrize("scale", [1.0, 2.0])   # the kept solution converges at once, or not
@pytest.mark.parametrize("name,quit_cta", [("258-rows", 3), ("2046-rows", 200), ("2077-rows", 40),
                                           ("several-rows-per-thread", 100), ("matrix-in-global-memory", 150)])
def test_a_wait_that_gives_up(torch_cuda, name, quit_cta, scale):  # noqa: F811
    torch = torch_cuda
    mesh = MESHES[name]()
    stats = wl.synthetic_statistics(mesh, 1, 61)
    S = torch.from_numpy(stats).cuda()
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1, cg_warm_start=1)
    _solve(torch, gm, params, stats)
    gm.set_cg_wait(1 << 13, quit_cta)
    out = torch.full((gm.n_nodes, 24), 7.0, dtype=torch.float32, device="cuda")
    with pytest.raises(lpdf.LpdfError) as e:
        gm.elliptic_relax_solve(params, scale * S, out, 1e-8)
    assert e.value.code == lpdf.LPDF_ERR_CUDA
    assert bool((out == 7.0).all())
    gm.set_cg_wait()
    F, its = _solve(torch, gm, params, stats, 1e-10)
    assert max(its) <= 8                                     # from the solution before
    _compare(F, of.node_fields(mesh, stats, 1, nu=params.nu, gmodel=0, pressure_solve=1), 1, name)
    with pytest.raises(lpdf.LpdfError) as e:
        gm.set_cg_wait(0)
    assert e.value.code == lpdf.LPDF_ERR_ARG
