"""The polynomial preconditioner of the gridpoint solve where its layout can go wrong: rows numbered at
random (every CTA's halo is nearly as large as it gets), a halo that does not fit shared memory (the
plain path), a closed box, the most rows of the one-row-per-thread layout, and the 32-bit epochs
running out. Bounds as in test_gpu_fields."""
import numpy as np
import pytest

from oracle import fields as of
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_cg import _wheel
from tests.test_gpu_fields import _compare, _solve, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _shuffled(mesh, seed):
    """The same mesh with its nodes numbered at random."""
    new = np.random.default_rng(seed).permutation(mesh.n_nodes).astype(np.int32)
    xy = np.empty_like(mesh.node_xy)
    xy[new] = mesh.node_xy
    return wl.Mesh(xy, new[mesh.tri], mesh.edge_tag, mesh.period_x, mesh.box, mesh.kind, mesh.nx, mesh.ny)


MESHES = {
    "random-numbering": lambda: _shuffled(wl.channel_mesh(90, 50, 31), 32),
    "halo-too-large": lambda: _wheel(2600),
    "cavity": lambda: wl.cavity_mesh(61, 47, 33),
    "192-rows-per-cta": lambda: wl.channel_mesh(288, 100, 34),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_polynomial_matches_the_oracle(torch_cuda, name):  # noqa: F811
    mesh = MESHES[name]()
    stats = wl.synthetic_statistics(mesh, 1, 35)
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1)
    F, its = _solve(torch_cuda, gm, params, stats)
    O = of.node_fields(mesh, stats, 1, nu=params.nu, gmodel=0, pressure_solve=1)
    _compare(F, O, 1, name)
    again, its2 = _solve(torch_cuda, gm, params, stats)
    assert its == its2 and np.array_equal(F, again)          # a fixed order of every sum


def test_epochs_run_out(torch_cuda):  # noqa: F811
    torch = torch_cuda
    mesh = wl.channel_mesh(67, 30, 36)
    S = torch.from_numpy(wl.synthetic_statistics(mesh, 1, 37)).cuda()
    gm = lpdf.Mesh(mesh)
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1)
    out = torch.zeros((gm.n_nodes, 24), dtype=torch.float32, device="cuda")
    want = None
    for _ in range(40):   # each takes 16 x 2^24 of the 2^32 epochs off, at most
        its = gm.elliptic_relax_solve(params, S, out, 1e-8, maxit=(1 << 24) - 1)
        if want is None:
            want = (its, out.clone())
        assert its == want[0] and torch.equal(out, want[1])
