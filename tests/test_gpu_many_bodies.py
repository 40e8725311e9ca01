"""More bodies than one block of the reversed rigid-body step, or of the
rigid-body step without fluid, takes: gradients and trajectories against the
oracle's at the bars of the few-body tests (1e-9 of each array's largest
magnitude; 1e-12)."""
import numpy as np
import pytest

import oracle
from paper_1108_0786_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()


def chain(bodies, n=(48, 32, 32), pitch=(12, 11, 16)):
    """Spheres and capsules joined by springs along a chain and across it, each driven."""
    sc = wl.Scenario("chain", *n, 0.8, g=(1e-6, -2e-6, 0.0))
    rng = wl.SplitMix64(5)
    for b in range(bodies):
        site = (b % 4, b // 4 % 3, b // 12)
        pos = tuple((s + 0.5) * p + rng.uniform(-0.3, 0.3) for s, p in zip(site, pitch))
        if b % 3 == 2:
            q = (0.9, 0.2, -0.3, 0.25)
            norm = sum(v * v for v in q) ** 0.5
            sc.bodies.append(wl.Body(wl.CAPSULE, 1.8, 2.0, 2.0 * wl.capsule_volume(1.8, 2.0), pos,
                                     tuple(v / norm for v in q)))
        else:
            sc.bodies.append(wl.Body(wl.SPHERE, 2.2, 0.0, 2.0 * wl.sphere_volume(2.2), pos))
        sc.drives.append(wl.Drive(b, 3e-3 * (1 + 0.1 * b), 1 / 50.0, 0.2 * b))
        for other in (b - 1, b - 5):
            if other >= 0:
                sc.springs.append(wl.Spring(other, b, 0.004, 11.0 + 0.1 * b, 0.003))
    return sc


def moving(sim):
    st = sim.bodies()
    for b in range(len(st)):
        st[b, 7:10] = (0.012 * (1 - b % 3), 0.01 * (b % 2), -0.008 + 0.004 * (b % 5))
        st[b, 10:13] = (0.003, -0.002 * (b % 4), 0.001)
        sim.set_body_state(b, st[b])
    return sim


@pytest.mark.parametrize("options", [0, lbm.OPT_NO_FLUID])
@pytest.mark.parametrize("bodies", [9, 20])
def test_gradients_of_many_bodies(bodies, options):
    sc = chain(bodies)
    seed = np.random.default_rng(2).standard_normal((bodies, 13))
    lat = moving(lbm.from_scenario(sc, precision="f64", options=options))
    lat.adjoint_record(24, 7)
    got = lat.adjoint_backward(seed)
    final = lat.bodies()
    lat.close()
    ref_run = moving(oracle.from_scenario(sc, options))
    ref = ref_run.adjoint(24, seed)
    np.testing.assert_allclose(final, ref_run.bodies(), rtol=1e-10, atol=1e-12)
    for k in ("state", "prev", "drive", "spring", "body"):
        assert np.abs(got[k] - ref[k]).max() <= 1e-9 * max(np.abs(ref[k]).max(), 1e-300), k


@pytest.mark.parametrize("bodies", [4, 5, 24, 254])
def test_rigid_bodies_without_fluid(bodies):
    """Every body steps once a step and the clock advances once."""
    sc = chain(bodies)
    lat, ref = (moving(lbm.from_scenario(sc, precision="f64", options=lbm.OPT_NO_FLUID)),
                moving(oracle.from_scenario(sc, lbm.OPT_NO_FLUID)))
    for n in (1, 3, 40):
        lat.step(n)
        ref.step(n)
        np.testing.assert_allclose(lat.bodies(), ref.bodies(), rtol=1e-10, atol=1e-12)
    lat.close()
