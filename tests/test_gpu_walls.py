"""No-slip walls (Eq. 4) in every launch shape of the bulk kernel, at rows and
row ends where its lanes cross: each shape gives the bits of one cell a thread,
whose FP64 populations match the oracle at the parity bar (1e-12), and so does
the same lattice stepped in an ensemble beside a periodic one."""
import numpy as np
import pytest

import oracle
from paper_1108_0786_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = {"f64": ((2, 0), (-1, 1)), "f32": ((2, 0), (2, 4), (4, 0), (-1, 1), (-1, 2)),
          "f16": ((2, 0), (4, 0), (4, 3), (8, 0), (-1, 2), (-1, 4)), "bf16": ((2, 4), (4, 2), (8, 2), (-1, 3))}


@pytest.fixture(scope="module", autouse=True)
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()


def scenario(nx, bc):
    sc = wl.Scenario("walls", nx, 23, 25, 0.8, bc=bc, g=(1e-5, -2e-5, 1.5e-5))
    if nx >= 19:
        sc.bodies.append(wl.Body(wl.SPHERE, 2.3, 0.0, 400.0, (8.1, 9.7, 4.2)))
    return sc


def run(sc, precision, shape=None, steps=9):
    lat = lbm.from_scenario(sc, precision=precision)
    rng = np.random.default_rng(3)
    if shape:
        lat.tune(*shape)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    lat.set_pop(w[:, None] * (1 + 0.01 * rng.standard_normal((19, sc.cells))))
    lat.step(steps)
    out = lat.pop()
    lat.close()
    return out


@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("nx", [1, 21, 32, 48])
@pytest.mark.parametrize("bc", [0, wl.PERIODIC_X, wl.PERIODIC_Y | wl.PERIODIC_Z, wl.PERIODIC_Z])
def test_walls_in_every_launch_shape(precision, nx, bc):
    sc = scenario(nx, bc)
    ref = run(sc, precision, (1, 0))
    if precision == "f64":
        o = oracle.from_scenario(sc)
        rng = np.random.default_rng(3)
        w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
        o.set_pop(w[:, None] * (1 + 0.01 * rng.standard_normal((19, sc.cells))))
        o.step(9)
        assert np.abs(ref - o.pop()).max() < 1e-12
    for v, blocks in SHAPES[precision]:
        if (v > 0 and nx % v) or (v < 0 and nx % 16):
            continue
        assert np.array_equal(run(sc, precision, (v, blocks)), ref), (v, blocks)


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
def test_walled_and_periodic_members_together(precision):
    scs = [scenario(21, 0), scenario(32, wl.PERIODIC_ALL), scenario(24, wl.PERIODIC_Z)]
    alone = []
    for sc in scs:
        lat = lbm.from_scenario(sc, precision=precision)
        lat.step(32)
        alone.append(lat.pop())
        lat.close()
    lats = [lbm.from_scenario(sc, precision=precision) for sc in scs]
    ens = lbm.Ensemble(lats)
    ens.step(32)
    ens.sync()
    for lat, pop in zip(lats, alone):
        assert np.array_equal(lat.pop(), pop)
    ens.close()
