"""The CG kernels of the gridpoint solve at the edges of their layouts, against the FP64 oracle: fewer
rows than a warp, the small kernel's blocks of 256 rows, rows with many entries, one and several rows
per thread, the matrix in shared memory and out of it. Bounds as in test_gpu_fields."""
import numpy as np
import pytest

from oracle import fields as of
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_fields import _compare, _solve, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _wheel(spokes):
    """A polygon of `spokes` triangles about one vertex: a matrix row of spokes + 1 entries."""
    t = 2.0 * np.pi * np.arange(spokes) / spokes
    xy = np.vstack([[0.5, 0.5], np.stack([0.5 + 0.5 * np.cos(t), 0.5 + 0.5 * np.sin(t)], 1)])
    xy = xy.astype(np.float32).astype(np.float64)
    tri = np.array([(0, 1 + k, 1 + (k + 1) % spokes) for k in range(spokes)], dtype=np.int32)
    tag = np.tile(np.array([0, wl.EDGE_WALL, 0], dtype=np.int32), (spokes, 1))
    box = (float(xy[:, 0].min()), float(xy[:, 0].max()), float(xy[:, 1].min()), float(xy[:, 1].max()))
    return wl.Mesh(xy, tri, tag, 0.0, box, "cavity", 0, 0)


MESHES = {
    "9-rows": lambda: wl.channel_mesh(3, 2, 11),
    "256-rows": lambda: wl.channel_mesh(32, 7, 12),
    "258-rows": lambda: wl.channel_mesh(43, 5, 13),
    "2046-rows": lambda: wl.channel_mesh(66, 30, 14),
    "2077-rows": lambda: wl.channel_mesh(67, 30, 15),
    "many-entries": lambda: _wheel(20),
    "several-rows-per-thread": lambda: wl.channel_mesh(330, 101, 16),
    "matrix-in-global-memory": lambda: wl.channel_mesh(520, 215, 17),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_cg_layouts_match_the_oracle(torch_cuda, name):  # noqa: F811
    mesh = MESHES[name]()
    stats = wl.synthetic_statistics(mesh, 1, 21)
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1)
    F, its = _solve(torch_cuda, gm, params, stats)
    O = of.node_fields(mesh, stats, 1, nu=params.nu, gmodel=0, pressure_solve=1)
    _compare(F, O, 1, name)
    again, its2 = _solve(torch_cuda, gm, params, stats)
    assert its == its2 and np.array_equal(F, again)          # a fixed order of every sum


@pytest.mark.parametrize("nx,ny", [(25, 20), (67, 30)])
def test_a_solve_that_does_not_converge_leaves_the_fields_and_the_warm_start(torch_cuda, nx, ny):  # noqa: F811
    torch = torch_cuda
    mesh = wl.channel_mesh(nx, ny, 18)
    S = torch.from_numpy(wl.synthetic_statistics(mesh, 1, 22)).cuda()
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1, cg_warm_start=1)
    out = torch.full((gm.n_nodes, 24), 7.0, dtype=torch.float32, device="cuda")
    its = gm.elliptic_relax_solve(params, S, out, 1e-10)
    want = out.clone()
    out.fill_(7.0)
    with pytest.raises(lpdf.LpdfError) as e:
        gm.elliptic_relax_solve(params, 2.0 * S, out, 1e-10, maxit=11)
    assert e.value.code == lpdf.LPDF_ERR_CG_NOCONV
    assert bool((out == 7.0).all())
    warm = gm.elliptic_relax_solve(params, S, out, 1e-10)    # from the last converged solution
    assert max(warm) <= 8 < min(its)
    assert torch.allclose(out, want, rtol=2e-5, atol=2e-5 * float(want.abs().max()))
