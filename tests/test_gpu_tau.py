"""FP64 populations away from tau = 1 and without a body force, where the collision
keeps a part of the old populations, against the oracle (1e-12): periodic and walled
boxes with a moving body, both cells-a-thread shapes and the row-staged one."""
import numpy as np
import pytest

import oracle
from paper_1108_0786_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.mark.parametrize("shape", [(1, 0), (2, 0), (-1, 1)])
@pytest.mark.parametrize("bc", [7, wl.PERIODIC_Y])
@pytest.mark.parametrize("tau", [0.55, 2 / 3, 0.8, 1.7])
def test_fp64_unforced_matches_the_oracle(tau, bc, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    sc = wl.Scenario("tau", 32, 23, 25, tau, bc=bc)
    sc.bodies.append(wl.Body(wl.SPHERE, 3.1, 0.0, 900.0, (14.2, 11.3, 12.1)))
    gpu, ref = lbm.from_scenario(sc, precision="f64"), oracle.from_scenario(sc)
    gpu.tune(*shape)
    pop = W[:, None] * (1 + 0.01 * np.random.default_rng(4).standard_normal((19, sc.cells)))
    for sim in (gpu, ref):
        s = sim.bodies()[0].copy()
        s[7:10] = (0.03, -0.02, 0.01)
        sim.set_body_state(0, s)
        sim.set_pop(pop)
        sim.step(14)
    assert np.abs(gpu.pop() - ref.pop()).max() < 1e-12
    gpu.close()
