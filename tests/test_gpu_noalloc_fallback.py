"""The allocation-free electrostatic solve where the mesh's multigrid hierarchy
does not pay: it goes on with the diagonal as its preconditioner and meets the
same tolerance.
"""
import numpy as np
import pytest

from paper_2102_06248_gb300 import workloads as W
from test_gpu_parity import F   # noqa: F401
from test_gpu_small_solves import node_laplacian, relative_residual

pytestmark = pytest.mark.gpu


# 12,167 interior nodes.  Moved by a tenth of a cell: the hierarchy alone; by
# 0.6 of a cell, tangled: more than its 100 iterations, so the solve has the
# launches of the second one (D^-1, its barrier, itself) besides.
@pytest.mark.parametrize("jitter,more", [(0.1, 0), (0.6, 3)])
@pytest.mark.parametrize("tol", [1e-8, 1e-11])
def test_tangled_mesh(F, jitter, more, tol):                                                    # noqa: F811
    import torch
    box = W.kuhn_box((24, 24, 24), (1.0, 1.0, 1.0), jitter=jitter, seed=2)
    L, inside = node_laplacian(box)
    assert inside.size >= 8192
    mesh = F.Mesh(box.xyz, box.tets)
    sim = F.Sim(mesh, 1e-12)         # the device copy of the mesh
    b = np.zeros(mesh.n_nodes)
    b[inside] = 1e-12 * np.random.default_rng(6).normal(size=inside.size)
    phi = torch.full((len(b),), float("nan"), dtype=torch.float64, device="cuda")
    n0 = F.launch_count()
    F.electrostatic_solve_noalloc(mesh, torch.tensor(b, device="cuda"), phi, tol=tol)
    assert F.launch_count() - n0 == 4 + more      # gather, barrier, solve, scatter
    res, slack = relative_residual(L, b[inside], phi.cpu().numpy()[inside])
    assert res <= tol + slack, (res / tol, slack / tol)
    # no charge, no potential
    F.electrostatic_solve_noalloc(mesh, torch.zeros_like(phi), phi, tol=tol)
    assert not phi.any()
    del sim
