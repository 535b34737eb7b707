"""The gridpoint solve where its matrix is finite in FP64 only: nearly laminar statistics in small units (a
large k, an epsilon below its floor) give relaxation lengths whose square exceeds FP32's range. Every CG
kernel; bounds as in test_gpu_fields."""
import numpy as np
import pytest

from oracle import fields as of
from paper_1006_0549_gb300 import lpdf, workloads as wl
from tests.test_gpu_cg import MESHES
from tests.test_gpu_fields import _compare, _solve, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["258-rows", "2077-rows", "many-entries", "several-rows-per-thread"])
def test_relaxation_lengths_beyond_fp32(torch_cuda, name):  # noqa: F811
    mesh = MESHES[name]()
    stats = wl.synthetic_statistics(mesh, 1, 51)
    stats[:, 1:4] *= 3e3
    stats[:, 4:10] *= 1e7
    stats[:, 10] *= 1e-20
    params = lpdf.make_params(nu=1.0 / 180.0, ns=1, gmodel=0, pressure_solve=1)
    F, _ = _solve(torch_cuda, lpdf.Mesh(mesh), params, stats)
    O = of.node_fields(mesh, stats, 1, nu=params.nu, gmodel=0, pressure_solve=1)
    assert np.isfinite(O).all()
    _compare(F, O, 1, name)
