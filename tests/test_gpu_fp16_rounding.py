"""FP16 storage: the stored values of a bulk step, bit for bit.

In a slow flow FP16 populations are a few units in the last place, and many
exact results lie half way between two FP16 values: an FP32 result that
misses the half-way value breaks such ties in one direction and the error
grows step by step.  The update is therefore pinned to its sequence of FP32
operations: the weight last, on a (+-) c.
"""
import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
              (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
F = np.float32
K = F(1024)


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()
    return torch


def fma(a, b, c):
    """a b + c rounded once to FP32 (the product of two FP32 values is exact in FP64)."""
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(F)


def step(h, tau):
    """One step of stored values h[19][z][y][x] (FP16, 1024 times the deviations)."""
    f = np.stack([np.roll(h[b], E[b][::-1], (0, 1, 2)) for b in range(19)]).astype(F)
    omega = 1.0 / tau
    om1 = F(1.0 - omega)
    s, j = f[0], [None, None, None]
    for p in range(9):
        b = 2 * p + 1
        s = s + (f[b] + f[b + 1])
        d = f[b] - f[b + 1]
        for a in range(3):
            if E[b][a]:
                j[a] = d if j[a] is None else (j[a] + d if E[b][a] > 0 else j[a] - d)
    rho = s / K + F(1)
    inv = (F(1) / rho) / K
    u = [x * inv for x in j]
    usq = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]))
    kr = rho * K
    base = fma(F(-1.5) * kr, usq, s)
    out = [fma(f[0], om1, base * F(omega * W[0]))]
    for p in range(9):
        b = 2 * p + 1
        eu = None
        for a in range(3):
            if E[b][a]:
                eu = u[a] if eu is None else (eu + u[a] if E[b][a] > 0 else eu - u[a])
        a_ = fma(F(4.5) * kr, eu * eu, base)
        c = (F(3) * kr) * eu
        ow = F(omega * W[b])
        out += [fma(f[b], om1, (a_ + c) * ow), fma(f[b + 1], om1, (a_ - c) * ow)]
    return np.stack(out).astype(np.float16)


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("nx", [40, 36, 34])            # 8, 4 and 2 cells a thread
def test_fp16_bulk_step_is_its_fp32_sequence(gpu, nx, tau):
    nz, ny = 12, 10
    lat = lbm.from_scenario(wl.Scenario("slow flow", nx, ny, nz, tau), precision="f16")
    if nx % 8 == 0:
        lat.tune(8)
    rest = lat.pop()                                        # zero deviations
    rng = np.random.default_rng(7)
    h = (W[:, None, None, None] * 5e-3 * rng.standard_normal((19, nz, ny, nx))).astype(np.float16)
    # rest + deviation in FP64: the upload takes rest off again, to 1e-17 of a 1e-6 deviation
    lat.set_pop(rest + (h.astype(np.float64) / 1024).reshape(rest.shape))
    for _ in range(4):
        lat.step(1)
        h = step(h, tau)
    got = ((lat.pop() - rest) * 1024).reshape(h.shape).astype(np.float16)
    lat.close()
    assert np.array_equal(got, h)
