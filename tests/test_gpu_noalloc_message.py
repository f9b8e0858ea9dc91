"""pic_last_error keeps the message of the last call that failed: the
allocation-free solve leaves it alone where its multigrid solve stops short
and the second solve reaches the tolerance.
"""
import numpy as np
import pytest

from paper_2102_06248_gb300 import workloads as W
from test_gpu_parity import F   # noqa: F401

pytestmark = pytest.mark.gpu


def test_message_of_a_call_that_succeeds(F):                                                    # noqa: F811
    import torch
    box = W.kuhn_box((24, 24, 24), (1.0, 1.0, 1.0), jitter=0.6, seed=2)   # tangled: the second solve
    mesh = F.Mesh(box.xyz, box.tets)
    sim = F.Sim(mesh, 1e-12)         # the device copy of the mesh
    with pytest.raises(F.PicError):
        F.Sim(mesh, -1.0)
    lib = F.load()
    before = lib.pic_last_error()
    assert b"invalid configuration" in before
    b = 1e-12 * np.random.default_rng(6).normal(size=mesh.n_nodes)
    phi = torch.zeros(mesh.n_nodes, dtype=torch.float64, device="cuda")
    n0 = F.launch_count()
    F.electrostatic_solve_noalloc(mesh, torch.tensor(b, device="cuda"), phi, tol=1e-8)
    assert F.launch_count() - n0 == 7        # gather, barrier, solve; D^-1, barrier, solve; scatter
    assert lib.pic_last_error() == before
    del sim
