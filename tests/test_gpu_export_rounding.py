"""FP32 output of FP32 and FP16 storage is no further from the exact value than FP64
sums rounded once are: populations, density and velocity of 200,000 cells near
equilibrium whose momenta are down to 10^-6 of the density's deviation.

The exact value comes from extended precision (a mantissa of 64 bits or more); it and numpy's own
roundings are allowed 2^-20 of an ulp."""
import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
L = np.longdouble


@pytest.fixture(scope="module")
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()
    return torch


def cells_near_equilibrium(n, seed):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((3, n)) * 10.0 ** rng.uniform(-10, -2, (3, n))
    drho = rng.standard_normal(n) * 1e-4
    eu = E @ u
    return W[:, None] * (drho + (1 + drho) * (3 * eu + 4.5 * eu ** 2 - 1.5 * (u ** 2).sum(0)))


def stored(delta, precision):
    """The FP64 input and the deviations storage makes of it."""
    pop = W[:, None] + delta
    d = (pop - W[:, None]).astype(np.float32)
    if precision == "f16":
        d = (d * np.float32(1024)).astype(np.float16).astype(np.float32) / np.float32(1024)
    return pop, d


def exact_and_fp64(d, g):
    x = d.astype(L)
    rho = 1 + x.sum(0)
    u = np.array([((E[:, i:i + 1] * x).sum(0) - L(0.5) * L(g[i])) / rho for i in range(3)])
    r64, j64 = np.zeros(d.shape[1]), np.zeros((3, d.shape[1]))
    for a in range(19):
        r64 = r64 + d[a]
        j64 = j64 + E[a][:, None] * d[a].astype(np.float64)
    u64 = (j64 - 0.5 * np.array(g)[:, None]) / (1.0 + r64)
    pop64 = W[:, None] + d.astype(np.float64)
    return ({"rho": rho[None], "u": u, "pop": W[:, None].astype(L) + x},
            {"rho": (1.0 + r64)[None].astype(np.float32), "u": u64.astype(np.float32), "pop": pop64.astype(np.float32)})


def beyond(got, exact, fp64):
    ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(L)
    mine, theirs = np.abs(got.astype(L) - exact), np.abs(fp64.astype(L) - exact)
    return (mine > np.maximum(theirs, ulp / 2) + ulp * L(2.0) ** -20).sum()


@pytest.mark.parametrize("g", [(0.0, 0.0, 0.0), (1e-6, -2e-6, 0.0)])
@pytest.mark.parametrize("precision", ["f32", "f16"])
def test_fp32_fields_as_from_fp64_sums(cuda, precision, g):
    torch = cuda
    assert np.finfo(L).nmant >= 63
    n = (500, 400, 1)
    pop, d = stored(cells_near_equilibrium(200000, 3), precision)
    exact, fp64 = exact_and_fp64(d, g)
    lat = lbm.Lattice(*n, 0.9, precision=precision, g=g)
    lat.set_pop(pop)
    for name, what, lead in (("pop", lbm.FIELD_POP, 19), ("rho", lbm.FIELD_RHO, 1), ("u", lbm.FIELD_U, 3)):
        t = torch.empty((lead, 200000), dtype=torch.float32, device="cuda")
        lat.field_device(what, t, lbm.DTYPE_F32)
        lat.sync()
        assert beyond(t.cpu().numpy(), exact[name], fp64[name]) == 0, name
    lat.close()
