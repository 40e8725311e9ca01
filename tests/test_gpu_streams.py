"""Step graphs on streams of different priorities: a lattice moved from stream to
stream between steps, its graphs captured anew where the priority changes, gives
the bits of one that stays."""
import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()
    return torch


def swimmer():
    sc = wl.Scenario("swimmer", 48, 32, 32, 0.8, g=(1e-6, 0.0, 0.0))
    wl.add_swimmer(sc, (23.6, 15.8, 16.1), (1.0, 0.0, 0.0, 0.0), (wl.SPHERE,) * 3, 3.0, 0.0, 11.0, 0.02, 0.01, 2e-3,
                   64.0, density=2.0)
    return sc


@pytest.mark.parametrize("options", [0, lbm.OPT_OVERLAP])
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
def test_streams_of_other_priorities(cuda, precision, options):
    torch = cuda
    ref = lbm.from_scenario(swimmer(), precision=precision, options=options)
    ref.step(57)
    want = (ref.bodies(), ref.pop())
    ref.close()
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1, -5, 0)]
    lat = lbm.from_scenario(swimmer(), precision=precision, options=options)
    lat.step(3)
    for s, n in zip(streams, (17, 16, 20, 1)):
        lat.sync()
        lat.set_stream(s.cuda_stream)
        lat.step(n)
    assert np.array_equal(lat.bodies(), want[0]) and np.array_equal(lat.pop(), want[1])
    lat.sync()
    lat.set_stream(0)
    lat.close()


def test_ensemble_on_a_stream_of_greatest_priority(cuda):
    torch = cuda
    ref = lbm.from_scenario(swimmer())
    ref.step(35)
    want = ref.pop()
    ref.close()
    with torch.cuda.stream(torch.cuda.Stream(priority=-5)):
        lats = [lbm.from_scenario(swimmer()) for _ in range(3)]
        ens = lbm.Ensemble(lats)
        ens.step(35)
        ens.sync()
        for lat in lats:
            assert np.array_equal(lat.pop(), want)
        ens.close()
        for lat in lats:
            lat.close()
