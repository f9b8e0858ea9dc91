"""Small systems (one slice of the matrix per warp): what the one-launch solve
returns meets the stopping rule, also where its pipelined recurrence cannot
reach it -- stretched cells, time steps far above the explicit limit, tight
tolerances, runs without any charge to scale the completion's tolerance.

The systems are the ones at which a NumPy model of that recurrence stopped
falling above the tolerance, or ended with a residual of its own below it and a
true one above, while PCG with two inner products of the current residual
converged.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2102_06248_gb300 import workloads as W
from test_gpu_parity import F, rel_err   # noqa: F401

pytestmark = pytest.mark.gpu

DT_CFL_6 = 1.3017565848335032e-10   # tests/golden/dt_cfl.json, thermal_plasma_cube_6^3


def node_laplacian(box):
    """G^T M G on all nodes (M the Whitney-1 mass: eps0 times P1 stiffness), and the interior nodes."""
    t, n = np.sort(box.tets, 1).astype(np.int64), len(box.xyz)
    d = box.xyz[t][:, 1:] - box.xyz[t][:, :1]
    inv = np.linalg.inv(d)
    g = np.concatenate([-inv.sum(2)[:, None, :], inv.transpose(0, 2, 1)], 1)
    vol = np.abs(np.linalg.det(d)) / 6.0
    k = W.EPS0 * vol[:, None, None] * np.einsum("tid,tjd->tij", g, g)
    L = sp.csr_matrix((k.ravel(), (np.repeat(t, 4, 1).ravel(), np.tile(t, (1, 4)).ravel())), shape=(n, n))
    lo, hi = box.ref_xyz.min(0), box.ref_xyz.max(0)
    eps = 1e-9 * (hi - lo)
    inside = np.where(((box.ref_xyz > lo + eps) & (box.ref_xyz < hi - eps)).all(1))[0]
    return L[inside][:, inside].tocsr(), inside


def relative_residual(L, b, x):
    """|b - L x| / |b|, and the rounding it carries: each of a row's products and
    sums to half an ulp of its terms, in this matrix and in the library's own
    (a dozen operations a row each)."""
    r = b - L @ x
    slack = 24 * np.finfo(float).eps * np.linalg.norm(np.abs(L) @ np.abs(x) + np.abs(b))
    return np.linalg.norm(r) / np.linalg.norm(b), slack / np.linalg.norm(b)


LAPLACIANS = [((10, 10, 10), (1.0, 1.0, 1.0)), ((20, 20, 20), (1.0, 1.0, 1.0)), ((20, 20, 20), (1.0, 30.0, 30.0)),
              ((18, 18, 18), (1.0, 10.0, 100.0)), ((24, 24, 24), (1.0, 10.0, 100.0))]


@pytest.mark.parametrize("tol", [1e-10, 1e-12, 1e-13])
@pytest.mark.parametrize("cells,size", LAPLACIANS)
@pytest.mark.parametrize("rhs", ["random", "smooth"])
def test_initial_potential_meets_its_tolerance(F, cells, size, tol, rhs):                       # noqa: F811
    box = W.kuhn_box(cells, size)
    L, inside = node_laplacian(box)
    b = np.zeros(len(box.xyz))
    b[inside] = 1e-12 * (np.random.default_rng(5).normal(size=inside.size) if rhs == "random" else 1.0)
    sim = F.Sim(F.Mesh(box.xyz, box.tets), 1e-12, init_tol=tol)
    sim.set_background_charge(b)
    sim.init()
    res, slack = relative_residual(L, b[inside], sim.field("PHI")[inside])
    assert res <= tol + slack, (res / tol, slack / tol)


@pytest.mark.parametrize("tol", [1e-10, 1e-12, 1e-13, 1e-14])
@pytest.mark.parametrize("cells,size", [c for c in LAPLACIANS if c[0][0] <= 20])   # below the multigrid sizes
def test_allocation_free_potential_meets_its_tolerance(F, cells, size, tol):                    # noqa: F811
    import torch
    box = W.kuhn_box(cells, size)
    L, inside = node_laplacian(box)
    assert inside.size < 8192
    b = np.zeros(len(box.xyz))
    b[inside] = 1e-12 * np.random.default_rng(6).normal(size=inside.size)
    mesh = F.Mesh(box.xyz, box.tets)
    sim = F.Sim(mesh, 1e-12)         # the device copy of the mesh
    phi = torch.full((len(b),), float("nan"), dtype=torch.float64, device="cuda")
    F.electrostatic_solve_noalloc(mesh, torch.tensor(b, device="cuda"), phi, tol=tol)
    res, slack = relative_residual(L, b[inside], phi.cpu().numpy()[inside])
    assert res <= tol + slack, (res / tol, slack / tol)
    del sim


# steps of 2, 30 and 300 times the explicit limit: condition numbers of about
# 10, 10^3 and 10^5, so that FP64 leaves 1e-11 of the residual at most
@pytest.mark.parametrize("cells,factor,tol", [(8, 2, 1e-13), (8, 30, 1e-10), (12, 30, 1e-12), (8, 300, 1e-10),
                                              (12, 300, 1e-10)])
def test_newmark_solve_at_large_steps(F, cells, factor, tol):                                   # noqa: F811
    wl = W.thermal_plasma_cube(n_cells=cells, n_particles=2000, seed=9)
    mesh = F.Mesh(wl.mesh.xyz, wl.mesh.tets)
    sim = F.Sim(mesh, factor * DT_CFL_6 * 6 / cells, cg_tol=tol)
    sim.init()
    e = np.random.default_rng(10).normal(size=mesh.n_edges)
    sim.set_field("E", e)            # (wall edges are kept at zero)
    for step in range(2):
        sim.step()
        d = sim.diag()
        # the residual is formed after the completion, which takes its
        # gradient part out along M (a well-shaped mesh: norm below 2)
        assert d["cg_relres"] <= 2 * (tol + 1e-11), (step, d)


@pytest.mark.parametrize("cells", [4, 6, 16])
def test_completion_without_charge(F, oracle_lib, cells):                                       # noqa: F811
    """No charge anywhere: the completion's absolute rule has no scale, and its
    relative one asks for init_tol (1e-14)."""
    wl = W.thermal_plasma_cube(n_cells=cells, n_particles=100, seed=11)
    dt = 2 * DT_CFL_6 * 6 / cells
    om = oracle_lib.OracleMesh(wl.mesh.xyz, wl.mesh.tets)
    osim = oracle_lib.OracleSim(om, oracle_lib.OracleConfig(dt=dt, cg_tol=1e-13))
    osim.init()
    gsim = F.Sim(F.Mesh(wl.mesh.xyz, wl.mesh.tets), dt, cg_tol=1e-13)
    gsim.init()
    e = np.random.default_rng(12).normal(size=om.n_edges)
    eb, _, _ = om.flags()
    e[eb == 1] = 0.0
    for s in (osim, gsim):
        s.set_field("E", e)
    for step in range(2):
        osim.step()
        gsim.step()
        assert rel_err(gsim.field("E"), osim.field("E")) <= 1e-10, step


def test_iteration_limit_is_kept(F):                                                            # noqa: F811
    """A solve that reaches cg_max_iters reports it (a rule that it cannot meet
    in four iterations, pipelined)."""
    wl = W.thermal_plasma_cube(n_cells=8, n_particles=2000, seed=13)
    sim = F.sim_from_workload(wl, 2 * DT_CFL_6 * 6 / 8, cg_tol=1e-12, cg_max_iters=4)
    with pytest.raises(F.PicError) as ei:
        sim.step()
    assert ei.value.code == 6
