"""Sizes at which the kernels change what they do: tiles and warps that are
nearly empty or just full, the largest system of the one-launch solve and the
smallest streamed one, meshes whose node numbering gives no small column
offsets, record counts on both sides of the one-launch ranking.

Each case is compared with the FP64 oracle.  Tolerances: particle phase PLAIN
1e-12 and MIXED 2e-5 of a field's largest value (FP32 positions: eps32 over
the ~0.3 cells that a particle moves, as in the frozen-field comparisons);
steps PLAIN 1e-10 (both solves stop at a relative residual of 1e-13, and the
Newmark matrix at twice the stable step has a condition number below 1e3).
"""
import numpy as np
import pytest

from paper_2102_06248_gb300 import workloads as W
from test_gpu_parity import F, compare_particles, continuity_host, frozen_field_case, rel_err   # noqa: F401

pytestmark = pytest.mark.gpu

DT_CFL_6 = 1.3017565848335032e-10   # tests/golden/dt_cfl.json, thermal_plasma_cube_6^3


# sort tiles hold 2,048 keys, push blocks 256 particles, warps 32; 311,297
# particles give each MIXED warp two rounds and a remainder, and in the
# 2^3 mesh (48 tets) runs of equal keys that span warps and blocks; 60,000
# fast particles in 6^3 cells leave more than 16,384 crossing records
@pytest.mark.parametrize("n,cells,speed", [(1, 3, 0.3), (31, 3, 0.3), (33, 3, 0.3), (2047, 3, 0.3), (2048, 3, 0.3),
                                           (2049, 3, 0.3), (60_000, 6, 1.0), (311_297, 2, 0.1)])
@pytest.mark.parametrize("precision", ["plain", "mixed"])
def test_particle_counts(F, oracle_lib, precision, n, cells, speed):                            # noqa: F811
    box, om, osim, gsim = frozen_field_case(F, oracle_lib, precision=precision, n=n, cells=cells, speed=speed, seed=9)
    for it in range(2):
        rho0, wall0 = gsim.field("RHO"), gsim.field("WALL")
        osim.particle_phase()
        gsim.particle_phase()
        if precision == "plain":
            compare_particles(gsim.particles(), osim.particles(), 1.0)
        for name in ("DG", "RHO"):
            assert rel_err(gsim.field(name), osim.field(name)) <= (1e-12 if precision == "plain" else 2e-5), (it, name)
        cont = continuity_host(gsim.mesh, gsim.field("RHO"), rho0, gsim.field("WALL"), wall0, gsim.field("DG"))
        assert cont <= (1e-12 if precision == "plain" else 1e-14), cont
    assert gsim.diag()["status"] == 0


def renumbered(wl, seed):
    """The same workload with its nodes in random order."""
    perm = np.random.default_rng(seed).permutation(len(wl.mesh.xyz))
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))
    wl.mesh.xyz = np.ascontiguousarray(wl.mesh.xyz[perm])
    wl.mesh.tets = np.ascontiguousarray(inv[wl.mesh.tets].astype(wl.mesh.tets.dtype))
    return wl


# interior edges 7 n^3 - 9 n^2 + 3 n: 26 (one slice), 117, 52,460 (1,640
# slices, one launch), 60,921 (1,904 slices, streamed)
@pytest.mark.parametrize("cells,shuffled", [(2, False), (3, False), (3, True), (20, False), (21, False), (21, True)])
def test_newmark_sizes(F, oracle_lib, cells, shuffled):                                         # noqa: F811
    wl = W.thermal_plasma_cube(n_cells=cells, n_particles=3000, seed=51)
    if shuffled:
        wl = renumbered(wl, 52)
    dt = 2 * DT_CFL_6 * 6 / cells
    osim = oracle_lib.from_workload(wl, dt, cg_tol=1e-13)
    gsim = F.sim_from_workload(wl, dt, precision="plain", cg_tol=1e-13)
    for step in range(2):
        osim.step()
        gsim.step()
        for name in ("E", "G", "RHO"):
            assert rel_err(gsim.field(name), osim.field(name)) <= 1e-10, (step, name)
        d = gsim.diag()
        assert d["cg_relres"] <= 1e-12, d
        assert d["continuity_abs"] <= 1e-12 * d["rho_max"], d
        assert d["gauss_abs"] <= 1e-12 * d["rho_max"], d


# 512 and 9,261 interior nodes: one launch of the pipelined recurrence, and the
# multigrid one; against the potential of the allocating path.  Both stop at
# 1e-14 of the right side and the node Laplacian's condition number is below
# 1e3 at these sizes, so they agree to 2e-11.
@pytest.mark.parametrize("cells,shuffled", [(9, True), (22, False), (22, True)])
def test_electrostatic_sizes(F, cells, shuffled):                                               # noqa: F811
    import torch
    wl = W.thermal_plasma_cube(n_cells=cells, n_particles=20000, seed=53)
    if shuffled:
        wl = renumbered(wl, 54)
    sim = F.sim_from_workload(wl, 2 * DT_CFL_6 * 6 / cells)
    rho = torch.tensor(sim.field("RHO") + sim.field("RHO_BG"), dtype=torch.float64, device="cuda")
    phi = torch.full((sim.mesh.n_nodes,), float("nan"), dtype=torch.float64, device="cuda")
    F.electrostatic_solve_noalloc(sim.mesh, rho, phi, tol=1e-14)
    torch.cuda.synchronize()
    ref = sim.field("PHI")
    assert rel_err(phi.cpu().numpy(), ref) <= 2e-11


# 26 rows (two tiles, one of 10 rows; every backward batch past the end), 117,
# 665 rows, regular and shuffled numberings; the tolerances of the network's
# comparison with its oracle (FP32 sums)
@pytest.mark.parametrize("cells,shuffled", [(2, False), (3, True), (5, False), (5, True)])
def test_network_sizes(F, oracle_lib, cells, shuffled):                                         # noqa: F811
    from oracle import gnn_oracle as GO
    from test_gpu_gnn import random_weights
    wl = W.thermal_plasma_cube(n_cells=cells, n_particles=500, seed=61)
    if shuffled:
        wl = renumbered(wl, 62)
    dt = 2 * DT_CFL_6 * 6 / cells
    sim = F.sim_from_workload(wl, dt, precision="plain")
    A, ids = GO.interior_system(oracle_lib.OracleMesh(wl.mesh.xyz, wl.mesh.tets), dt)
    w = random_weights(63)
    sim.gnn_set_weights(w)
    r = np.zeros(sim.mesh.n_edges)
    r[ids] = np.random.default_rng(64).normal(size=ids.size)
    net = GO.EdgeNet(A)
    z, (zo, _) = sim.gnn_apply(r), net.forward(r[ids], GO.bf16(w))
    assert np.abs(z[ids] - zo).max() <= 1e-5 * np.abs(zo).max()
    L, g = sim.gnn_loss_grad(r)
    Lo, go, _ = net.loss_and_grad(r[ids], GO.bf16(w))
    assert L == pytest.approx(Lo, rel=1e-5, abs=1e-6)
    for name, (o, s) in GO.OFFSETS.items():
        if name == "_size":
            continue
        sl = slice(o, o + int(np.prod(s)))
        scale = max(np.abs(go[sl]).max(), 1e-3 * np.abs(go).max())
        assert np.abs(g[sl] - go[sl]).max() <= 1e-3 * scale, name
