"""BF16 storage keeps the momentum of a uniform flow: the rounding is stochastic
(zero mean), and no factor's own rounding repeats in every cell and step.

Bound for n steps on N cells: a unit roundoff of the FP32 arithmetic, 2^-24, a step,
and five standard deviations of the storage's rounding.  A population 3 w e.u is
rounded to 8 bits, a variance of at most (2^-7 3 w e.u)^2 / 6, so with u = (v, v, v)
the momentum's error along an axis has a standard deviation of at most
2^-7 3 v sqrt((2 / 18^2 + 4 (2 / 36)^2) / 6) < 1.4e-3 v a cell and step, and
sqrt(n / N) of that after n steps."""
import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.mark.parametrize("shape", [(8, 2), (1, 1)])
def test_uniform_flow_keeps_its_momentum(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    n, steps, u = (128, 128, 128), 100000, np.full(3, 1.1e-3)
    cells = int(np.prod(n))
    eu = E @ u
    f = W * (1 + 3 * eu + 4.5 * eu ** 2 - 1.5 * (u ** 2).sum())
    lat = lbm.Lattice(*n, 1.0, precision="bf16")
    lat.tune(*shape)
    lat.set_pop(np.repeat(f[:, None], cells, axis=1))
    t = torch.empty((19, cells), dtype=torch.float64, device="cuda")

    def momentum():
        lat.field_device(lbm.FIELD_POP, t, lbm.DTYPE_F64)
        lat.sync()
        return (torch.from_numpy(E.T.astype(np.float64)).cuda() @ t.mean(1)).cpu().numpy()

    lat.step(1)                     # past the rounding of the start to nearest
    j0 = momentum()
    lat.step(steps)
    j1 = momentum()
    lat.close()
    drift = np.abs(j1 / j0 - 1)
    assert drift.max() < steps * 2.0 ** -24 + 5 * 1.4e-3 * np.sqrt(steps / cells), drift
