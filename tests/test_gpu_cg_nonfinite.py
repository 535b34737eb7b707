"""A solve whose statistics hold a value that is not finite: reported as not converged, the caller's fields
and the warm start left alone, the next solve right. Every CG kernel; bounds as in test_gpu_fields."""
import numpy as np
import pytest

from oracle import fields as of
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_cg import MESHES
from tests.test_gpu_fields import _compare, _solve, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("column", [4, 1])     # <u'u'>: both systems; <u>: the pressure's alone
@pytest.mark.parametrize("name", ["258-rows", "2077-rows", "many-entries", "several-rows-per-thread"])
def test_nonfinite_statistics_do_not_converge(torch_cuda, name, column, value):  # noqa: F811
    torch = torch_cuda
    mesh = MESHES[name]()
    stats = wl.synthetic_statistics(mesh, 1, 41)
    S = torch.from_numpy(stats).cuda()
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1, cg_warm_start=1)
    F, _ = _solve(torch, gm, params, stats)
    bad = S.clone()
    bad[int(gm.masters()[mesh.n_nodes // 2]), column] = value
    out = torch.full((gm.n_nodes, 24), 7.0, dtype=torch.float32, device="cuda")
    with pytest.raises(lpdf.LpdfError) as e:
        gm.elliptic_relax_solve(params, bad, out, 1e-10)
    assert e.value.code == lpdf.LPDF_ERR_CG_NOCONV
    assert bool((out == 7.0).all())
    again, its = _solve(torch, gm, params, stats, 1e-10)
    assert max(its) <= 8                                     # from the solution before
    _compare(again, of.node_fields(mesh, stats, 1, nu=params.nu, gmodel=0, pressure_solve=1), 1, name)
    assert np.isfinite(F).all()
