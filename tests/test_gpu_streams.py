"""The streamed matrix products of the persistent solvers, in every form a
record takes: FP64 and FP32 values, one-byte and 32-bit columns (a regular and
a random node numbering), alone and batched.

The ring's stages are rewritten while other warps still load: a stage reused
too early would give sums that differ from run to run, so results are compared
bit by bit between runs, and the residual of the solution is the one the
diagnostics form from the matrix as it is stored, without the stream.
"""
import numpy as np
import pytest

from paper_2102_06248_gb300 import workloads as W
from test_gpu_edges import renumbered
from test_gpu_parity import F, rel_err   # noqa: F401

pytestmark = pytest.mark.gpu

DT_CFL_6 = 1.3017565848335032e-10   # tests/golden/dt_cfl.json, thermal_plasma_cube_6^3


def workload(cells, shuffled, n=3000, seed=71):
    wl = W.thermal_plasma_cube(n_cells=cells, n_particles=n, seed=seed)
    return renumbered(wl, seed + 1) if shuffled else wl


# interior edges 7 n^3 - 9 n^2 + 3 n: 26 (one slice), 665, 60,921 (more records
# than a ring has stages in every warp), 91,816 (multigrid completion).  The
# refinement of the MIXED solve stops at 1e-13; FP64 rounding of the residual
# that the diagnostics form, at a condition number below 1e3: another 1e-13.
@pytest.mark.parametrize("cells", [2, 5, 21, 24])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("precision", ["mixed", "plain"])
def test_streamed_solves_repeat_and_reach_the_tolerance(F, precision, shuffled, cells):         # noqa: F811
    fields = []
    for _ in range(3):
        wl = workload(cells, shuffled)
        sim = F.sim_from_workload(wl, 2 * DT_CFL_6 * 6 / cells, precision=precision, cg_tol=1e-13)
        for step in range(3):
            sim.step()
            d = sim.diag()
            assert d["cg_relres"] <= 2e-13, (step, d)
            assert d["gauss_abs"] <= 1e-12 * d["rho_max"], (step, d)
        fields.append({f: sim.field(f) for f in ("PHI", "E", "B", "G", "RHO")})
    for other in fields[1:]:
        for name, a in fields[0].items():
            np.testing.assert_array_equal(a, other[name], err_msg=name)


# members with 26 to 91,816 unknowns: two regular, two with 32-bit columns, one
# of these (24^3) with a multigrid completion; solves at 1e-13, so batched and
# solo fields agree to 1e-9 (PLAIN), or to the FP32 state (MIXED), as in the
# batch test of a multigrid member
@pytest.mark.parametrize("multigrid", [False, True])
@pytest.mark.parametrize("precision", ["mixed", "plain"])
def test_batch_of_regular_and_irregular_meshes(F, precision, multigrid):                        # noqa: F811
    cases = [(2, False, 200), (8, True, 20000), (21, False, 20000), (24 if multigrid else 14, True, 20000)]
    wls = [(workload(c, sh, n, 80 + k), 2 * DT_CFL_6 * 6 / c) for k, (c, sh, n) in enumerate(cases)]
    solo = [F.sim_from_workload(wl, dt, precision=precision, cg_tol=1e-13) for wl, dt in wls]
    memb = [F.sim_from_workload(wl, dt, precision=precision, cg_tol=1e-13) for wl, dt in wls]
    assert (memb[3].mesh.n_int_nodes >= 8192) == multigrid
    batch = F.Batch(memb)
    batch.step(8)         # one eager step, a six-step graph, one more
    assert batch.info()["graph_launches"] == 1
    tol = 1e-9 if precision == "plain" else 1e-6
    for (a, b), (c, sh, _) in zip(zip(solo, memb), cases):
        a.step(8)
        for f in ("E", "RHO", "G"):
            assert rel_err(b.field(f), a.field(f)) <= tol, (c, sh, f)
        d = b.diag()
        assert d["cg_relres"] <= 2e-13, (c, sh, d)
        assert d["continuity_abs"] <= 1e-12 * d["rho_max"], (c, sh, d)
        assert d["gauss_abs"] <= 1e-12 * d["rho_max"], (c, sh, d)
