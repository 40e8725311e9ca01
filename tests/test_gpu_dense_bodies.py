"""Many bodies: rods whose remap cubes overlap (every fluid cell near a body is
listed once for the boundary kernel, so the list holds however many cubes cover
a cell), and lists long enough for the boundary kernel to take a thread a cell.
FP64 storage matches the oracle at the parity bars (populations 1e-12, positions
1e-10 relative); a lattice gives the same bits whichever way its list is taken
(alone a warp a cell, in an ensemble a thread a cell)."""
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


def rods():
    """18 parallel rods of radius 2 and length 30 in 48^3 cells (remap cubes of
    43 cells a side), moving."""
    sc = wl.Scenario("rods", 48, 48, 48, 0.8)
    for i in range(18):
        sc.bodies.append(wl.Body(wl.CAPSULE, 2.0, 30.0, 2.0 * wl.capsule_volume(2.0, 30.0),
                                 (23.3 + 0.7 * (i % 3), 7.6 + 16 * (i % 3), 4.2 + 8 * (i // 3))))
    return sc


def moving(sim, sc):
    for b in range(len(sc.bodies)):
        s = sim.bodies()[b].copy()
        s[7:10] = (4e-3 * (1 - b % 3), 3e-3 * (b % 2), -2e-3 + 1e-3 * (b % 5))
        sim.set_body_state(b, s)


def listed_cells(sc, reach=1.5):
    """fluid cells within `reach` of a rod's surface"""
    z, y, x = np.meshgrid(*(np.arange(n) for n in (sc.nz, sc.ny, sc.nx)), indexing="ij")
    near = np.zeros(x.shape, bool)
    for b in sc.bodies:
        d = [p - c for p, c in zip((x, y, z), b.pos)]
        d = [v - n * np.round(v / n) for v, n in zip(d, (sc.nx, sc.ny, sc.nz))]
        ax = np.clip(d[0], -b.length / 2, b.length / 2)
        d2 = (d[0] - ax) ** 2 + d[1] ** 2 + d[2] ** 2
        near |= (d2 < (b.radius + reach) ** 2) & (d2 > b.radius ** 2)
    return int(near.sum())


def test_rods_step_and_match_the_oracle():
    sc = rods()
    gpu, ref = lbm.from_scenario(sc, precision="f64"), oracle.from_scenario(sc)
    for sim in (gpu, ref):
        moving(sim, sc)
    for _ in range(3):
        gpu.step(6)
        ref.step(6)
        assert np.array_equal(gpu.flags(), ref.flags())
        assert np.abs(gpu.pop() - ref.pop()).max() < 1e-12
        b, rb = gpu.bodies(), ref.bodies()
        assert np.abs(b[:, :3] - rb[:, :3]).max() < 1e-10 * np.abs(rb[:, :3]).max()
    gpu.close()


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16"])
def test_rods_alone_and_in_an_ensemble(precision):
    """The batched remap (listed candidates) gives the bits of the single one."""
    sc = rods()
    lat = lbm.from_scenario(sc, precision=precision)
    moving(lat, sc)
    lat.step(17)
    want = (lat.bodies(), lat.pop())
    lat.close()
    lats = [lbm.from_scenario(sc, precision=precision) for _ in range(2)]
    for m in lats:
        moving(m, sc)
    ens = lbm.Ensemble(lats)
    ens.step(17)
    ens.sync()
    for m in lats:
        assert np.array_equal(m.bodies(), want[0]) and np.array_equal(m.pop(), want[1])
    ens.close()
    for m in lats:
        m.close()


def test_list_holds_each_cell_once():
    """A list limited to the number of cells within reach of a rod (with a tenth to
    spare for cells a rod has just left) is enough."""
    sc = rods()
    lat = lbm.from_scenario(sc, precision="f32")
    lat.debug_set(lbm.DEBUG_CELL_LIST_CAP, int(1.1 * listed_cells(sc)))
    moving(lat, sc)
    lat.step(16)
    lat.sync()
    lat.close()


def suspension(bodies, bc, seed=0):
    """Spheres of radius 3 on a loose grid of 44 x 40 x 48 cells, fast enough to
    cover and uncover cells."""
    sc = wl.Scenario("suspension", 44, 40, 48, 0.8, bc=bc, g=(2e-6, -1e-6, 3e-6))
    rng = wl.SplitMix64(77 + seed)
    sites = [(i, j, k) for k in range(4) for j in range(3) for i in range(4)]
    for s in sites[:bodies]:
        pos = tuple((v + 0.5) * p + rng.uniform(-0.4, 0.4) for v, p in zip(s, (11, 13, 12)))
        sc.bodies.append(wl.Body(wl.SPHERE, 3.0, 0.0, 2.0 * wl.sphere_volume(3.0), pos))
    return sc


def swept(sim, sc):
    for b in range(len(sc.bodies)):
        s = sim.bodies()[b].copy()
        s[7:10] = (0.04 * (1 - b % 3), 0.03 * (b % 2), -0.03 + 0.015 * (b % 5))
        s[10:13] = (0.01, -0.005 * (b % 3), 0.0)
        sim.set_body_state(b, s)


@pytest.mark.parametrize("bc", [7, wl.PERIODIC_X, 0])
def test_long_list_matches_the_oracle(bc):
    sc = suspension(36, bc)                     # about 9,600 cells listed
    gpu, ref = lbm.from_scenario(sc, precision="f64"), oracle.from_scenario(sc)
    for sim in (gpu, ref):
        swept(sim, sc)
    for _ in range(4):
        gpu.step(4)
        ref.step(4)
        assert np.array_equal(gpu.flags(), ref.flags())
        assert np.abs(gpu.pop() - ref.pop()).max() < 1e-12
        fr = ref.forces()
        assert np.abs(gpu.forces() - fr).max() < 1e-12 + 1e-10 * np.abs(fr).max()
    gpu.close()


@pytest.mark.parametrize("bc", [7, wl.PERIODIC_Z])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
def test_bits_of_a_warp_and_a_thread_a_cell(precision, bc):
    n = 18 if precision == "f64" else 36        # about 4,800 and 9,600 cells a lattice
    scs = [suspension(n, bc, k) for k in range(6)]
    lats = [lbm.from_scenario(sc, precision=precision) for sc in scs]
    for m, sc in zip(lats, scs):
        swept(m, sc)
    ens = lbm.Ensemble(lats)
    ens.step(16)                                # in two launches: 14,400 and 28,900 cells each
    ens.sync()
    for m, sc in zip(lats, scs):
        lat = lbm.from_scenario(sc, precision=precision)
        swept(lat, sc)
        lat.step(16)
        assert np.array_equal(m.bodies(), lat.bodies()) and np.array_equal(m.pop(), lat.pop())
        lat.close()
    ens.close()
    for m in lats:
        m.close()
