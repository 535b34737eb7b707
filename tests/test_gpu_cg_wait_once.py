"""A CG with several rows per thread whose neighbour block is lost waits once, not once per row. The rows are
numbered at random, so that most warps have a row of the lost block beside each of theirs."""
import time

import pytest

from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_cg_polynomial import _shuffled
from tests.test_gpu_fields import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def test_a_lost_block_costs_one_wait(torch_cuda):  # noqa: F811
    torch = torch_cuda
    mesh = _shuffled(wl.channel_mesh(580, 249, 81), 82)      # 145,000 rows: 954 a block
    S = torch.from_numpy(wl.synthetic_statistics(mesh, 1, 83)).cuda()
    gm = lpdf.Mesh(mesh)
    out = torch.zeros((gm.n_nodes, 24), dtype=torch.float32, device="cuda")

    def lost(gmodel):
        params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=gmodel, pressure_solve=1)
        best = 1e9
        for _ in range(3):
            torch.cuda.synchronize()
            t = time.perf_counter()
            with pytest.raises(lpdf.LpdfError) as e:
                gm.elliptic_relax_solve(params, S, out, 1e-8)
            best = min(best, time.perf_counter() - t)
            assert e.value.code == lpdf.LPDF_ERR_CUDA
        return best

    gm.set_cg_wait(1 << 15, 100)
    one, five = lost(1), lost(0)     # one row per thread (the pressure alone), five (all components)
    print("one row", one, "five rows", five)
    assert five < one                # as many threads poll in both; a wait per row took 1.6 times as long
