"""The field export (lbm_get_fields_device) of every storage type at sizes where
its vector width, its tails and its output alignment change, against the same
field formed by numpy in FP64 from the FP64 populations.

Bounds: an FP32 output is the FP64 value rounded once, but for ties (one ulp,
2^-23 relative); numpy's own moments of w + delta lose up to 19 roundings of
populations of at most 2/3 (about 2e-15)."""
import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.fixture(scope="module")
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()
    return torch


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [(1, 1, 1), (7, 3, 1), (16, 5, 3), (33, 31, 9)])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
def test_export_matches_fp64_moments(cuda, precision, n, shift):
    torch = cuda
    nx, ny, nz = n
    cells = nx * ny * nz
    rng = np.random.default_rng(17)
    g = (3e-4, -1e-4, 2e-5)
    lat = lbm.Lattice(nx, ny, nz, 0.9, precision=precision, g=g)
    lat.set_pop((W[:, None] * (1 + 0.05 * rng.standard_normal((19, cells)))))
    pop = lat.pop().reshape(19, cells)
    rho = pop.sum(0)
    u = ((E.T @ pop) - 0.5 * np.array(g)[:, None]) / rho
    for name, what, ref in (("pop", lbm.FIELD_POP, pop), ("rho", lbm.FIELD_RHO, rho[None]), ("u", lbm.FIELD_U, u)):
        for dtype, code in ((torch.float32, lbm.DTYPE_F32), (torch.float64, lbm.DTYPE_F64)):
            buf = torch.full((shift + ref.size + 1,), -7.0, dtype=dtype, device="cuda")
            out = buf[shift:shift + ref.size]
            lat.field_device(what, out, code)
            lat.sync()
            got = out.cpu().double().numpy().reshape(ref.shape)
            ulp = 2.0 ** -23 * np.abs(ref) if dtype == torch.float32 else 0.0
            assert (np.abs(got - ref) <= ulp + 2e-15).all(), (name, dtype)
            assert (buf[:shift] == -7.0).all() and buf[-1] == -7.0     # nothing beside the field
    lat.close()


@pytest.mark.parametrize("precision", ["f32", "f16"])
def test_export_keeps_infinities_and_nan(cuda, precision):
    """Non-finite populations come out as the FP64 sums give them."""
    torch = cuda
    lat = lbm.Lattice(4, 3, 2, 0.9, precision=precision)
    pop = np.repeat(W[:, None], 24, axis=1)
    pop[3, 5], pop[4, 6], pop[7, 9] = np.inf, -np.inf, np.nan
    lat.set_pop(pop)
    for what, lead in ((lbm.FIELD_POP, 19), (lbm.FIELD_RHO, 1), (lbm.FIELD_U, 3)):
        a = torch.empty((lead, 24), dtype=torch.float32, device="cuda")
        b = torch.empty((lead, 24), dtype=torch.float64, device="cuda")
        lat.field_device(what, a, lbm.DTYPE_F32)
        lat.field_device(what, b, lbm.DTYPE_F64)
        torch.cuda.synchronize()
        a, b = a.cpu().double().numpy(), b.cpu().numpy()
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
        assert np.array_equal(a[np.isinf(a)], b[np.isinf(b)])
    lat.close()
