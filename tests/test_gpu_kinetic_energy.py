"""The kinetic energy of a MIXED push is summed in pairs of floats; a particle
whose energy leaves the FP32 range makes the sum infinite, not undefined.
"""
import numpy as np
import pytest

from paper_2102_06248_gb300 import workloads as W
from test_gpu_parity import F   # noqa: F401

pytestmark = pytest.mark.gpu


# 40 particles: two rounds of a warp, the last one partly empty; 1e20 m/s
# squares past the FP32 range (3.4e38), 1e18 does not
@pytest.mark.parametrize("speed,finite", [(1e18, True), (1e20, False)])
@pytest.mark.parametrize("fast", [1, 40])
def test_energy_past_the_fp32_range(F, speed, finite, fast):                                    # noqa: F811
    n, m = 40, 9.1e-31
    box = W.kuhn_box((3, 3, 3), (1.0, 1.0, 1.0))
    v = np.zeros((n, 3))
    v[n - fast:, 0] = speed
    sim = F.Sim(F.Mesh(box.xyz, box.tets), 1e-4 / speed, precision="mixed")
    sim.particles_load(0, 1.6e-19, m, 1.0, np.array([0.37, 0.43, 0.21]) + 1e-3 * np.arange(n)[:, None], v)
    sim.init()
    sim.step()
    d = sim.diag()
    assert d["status"] == 0 and d["n_alive"] == n
    if finite:
        # FP32 terms (charges of 1.6e-19 C do not change such a speed)
        assert d["energy_k"] == pytest.approx(fast * 0.5 * m * speed ** 2, rel=1e-6)
    else:
        assert d["energy_k"] == np.inf
