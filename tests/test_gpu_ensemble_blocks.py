"""Batches with 64 bodies and more in a launch, where the force kernel takes one
block for each body of an ordinary member: the bits of members stepped alone."""
import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


def box(k):
    sc = wl.Scenario("box", 32 + 2 * (k % 3), 24, 28, 0.8)
    rng = wl.SplitMix64(900 + k)
    wl.add_swimmer(sc, (16.3 + rng.uniform(-0.4, 0.4), 11.7, 14.2 + rng.uniform(-0.4, 0.4)), (1.0, 0.0, 0.0, 0.0),
                   (wl.SPHERE,) * 3, 2.4, 0.0, 9.0, 0.02, 0.01, 2e-3, 64.0, density=2.0)
    return sc


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16"])
def test_one_force_block_a_body(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    scs = [box(k) for k in range(46)]           # 23 boxes, 69 bodies in each of the two launches
    lats = [lbm.from_scenario(sc, precision=precision) for sc in scs]
    ens = lbm.Ensemble(lats)
    ens.step(18)
    ens.sync()
    got = [(lat.bodies(), lat.forces(), lat.pop()) for lat in lats]
    ens.close()
    for lat in lats:
        lat.close()
    for sc, (b, f, p) in zip(scs, got):
        lat = lbm.from_scenario(sc, precision=precision)
        lat.step(18)
        assert np.array_equal(lat.bodies(), b) and np.array_equal(lat.forces(), f) and np.array_equal(lat.pop(), p)
        lat.close()


@pytest.mark.parametrize("order", [(48, 33), (33, 48)])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
def test_even_and_odd_rows_in_separate_launches(precision, order):
    """Members of one storage type whose launches take different bulk shapes (two
    cells a thread where every row of the launch is even, one where a row is odd)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")

    def lattice(nx):
        sc = wl.Scenario("rows", nx, 24, 26, 0.8, g=(1e-6, 0.0, 2e-6))
        sc.bodies.append(wl.Body(wl.SPHERE, 2.6, 0.0, 200.0, (nx / 2 + 0.3, 11.8, 12.6)))
        lat = lbm.from_scenario(sc, precision=precision)
        w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
        lat.set_pop(w[:, None] * (1 + 0.01 * np.random.default_rng(nx).standard_normal((19, sc.cells))))
        return lat

    lats = [lattice(nx) for nx in order]
    ens = lbm.Ensemble(lats)
    ens.step(32)
    ens.sync()
    for nx, lat in zip(order, lats):
        ref = lattice(nx)
        ref.step(32)
        assert np.array_equal(lat.pop(), ref.pop()) and np.array_equal(lat.bodies(), ref.bodies())
        ref.close()
    ens.close()
    for lat in lats:
        lat.close()
