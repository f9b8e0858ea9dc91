"""Allocation-free electrostatic solves from several host threads, each on its
own stream: the calls share one device array (vectors, partial sums, the grid
barrier's counter) and take turns on it, so every result is bit for bit that of
the call made alone.
"""
import threading

import numpy as np
import pytest

from paper_2102_06248_gb300 import workloads as W
from test_gpu_parity import F   # noqa: F401

pytestmark = pytest.mark.gpu


# a system of one launch of the small solve, a streamed one (tolerance 1e-14)
# and one with a multigrid hierarchy, each solved by two threads at once
@pytest.mark.parametrize("cells,tol", [(9, 1e-12), (16, 1e-14), (24, 1e-12)])
def test_calls_from_threads_take_turns(F, cells, tol):                                          # noqa: F811
    import torch
    box = W.kuhn_box((cells,) * 3, (1.0,) * 3, jitter=0.15, seed=3)
    mesh = F.Mesh(box.xyz, box.tets)
    sim = F.Sim(mesh, 1e-12)         # the device copy of the mesh
    rng = np.random.default_rng(4)
    rho = [torch.tensor(1e-12 * rng.normal(size=mesh.n_nodes), device="cuda") for _ in range(4)]
    nan = torch.full((mesh.n_nodes,), float("nan"), dtype=torch.float64, device="cuda")
    alone = [F.electrostatic_solve_noalloc(mesh, r, nan.clone(), tol=tol).cpu() for r in rho]
    streams = [torch.cuda.Stream() for _ in rho]
    out = [[nan.clone() for _ in range(12)] for _ in rho]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            for phi in out[k]:
                F.electrostatic_solve_noalloc(mesh, rho[k], phi, tol=tol, stream=streams[k])
        except Exception as e:       # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for k in range(4):
        for phi in out[k]:
            assert torch.equal(phi.cpu(), alone[k]), k
    del sim
