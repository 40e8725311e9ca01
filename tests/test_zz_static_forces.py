"""lbm_momentum_exchange_static against the link sum written out in numpy, where
the minimum image is decided: a periodic axis of one or two cells, a centre past
half a cell, links half a period away from the centre; and with non-finite inputs.

Bound: the same FP64 terms summed in another order, at most a few hundred links
of magnitude about 0.3 (1e-12)."""
import ctypes

import numpy as np
import pytest

from paper_1108_0786_gb300 import lbm

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def link_sum(pop, flags, bodies, n, bc):
    """Force and torque of each body: every link once (all cells scanned)."""
    per = np.array([bc >> a & 1 for a in range(3)], bool)
    n = np.array(n)
    pop = pop.reshape(19, n[2], n[1], n[0])
    flags = flags.reshape(n[2], n[1], n[0])
    rho = pop.sum(0)
    out = np.zeros((len(bodies), 6))
    image = lambda d: np.where(per, d - n * np.floor(d / n + 0.5), d)
    with np.errstate(invalid="ignore"):
        for z, y, x in np.argwhere(flags == 0):
            at = np.array((x, y, z))
            for a in range(1, 19):
                end = at + E[a]
                if ((~per) & ((end < 0) | (end >= n))).any():
                    continue
                b = int(flags[tuple((end % n)[::-1])]) - 1
                if b < 0:
                    continue
                X, V, O = bodies[b, :3], bodies[b, 7:10], bodies[b, 10:13]
                u = V + np.cross(O, image(end - X))
                mag = 2 * pop[a, z, y, x] - 6 * W[a] * rho[z, y, x] * (E[a] * u).sum()
                f = E[a] * mag
                out[b, :3] += f
                out[b, 3:] += np.cross(image(at + 0.5 * E[a] - X), f)
    return out


@pytest.fixture(scope="module")
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1108_0786_gb300 import _build
    _build.build()
    return torch


def static(torch, pop, flags, bodies, n, bc, hw):
    p, f, b = (torch.from_numpy(v).cuda() for v in (pop, flags, bodies))
    out = torch.zeros(len(bodies), 6, dtype=torch.float64, device="cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (p, f, b)]
    rc = lbm.load_library().lbm_momentum_exchange_static(*ptr, len(bodies), *n, bc, hw, ctypes.c_void_p(out.data_ptr()),
                                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == lbm.OK
    return out.cpu().numpy()


def inputs(n, centre, radius, bc):
    """A ball of cells around the centre (periodic axes wrap) and noise around rest."""
    rng = np.random.default_rng(int(sum(n)))
    d2 = np.zeros((n[2], n[1], n[0]))
    for a, ax in ((0, 2), (1, 1), (2, 0)):
        d = np.arange(n[a]) - centre[a]
        if bc >> a & 1:
            d = d - n[a] * np.floor(d / n[a] + 0.5)
        d2 = d2 + (d ** 2).reshape([-1 if k == ax else 1 for k in range(3)])
    flags = (d2 <= radius ** 2).astype(np.uint8)
    pop = W[:, None] * (1 + 0.01 * rng.standard_normal((19, int(np.prod(n)))))
    body = np.zeros((1, 13))
    body[0, :3], body[0, 3] = centre, 1.0
    body[0, 7:13] = rng.uniform(-1e-2, 1e-2, 6)
    return pop, flags.reshape(-1), body


@pytest.mark.parametrize("n,centre,radius,bc", [
    ((1, 15, 15), (0.7, 7.2, 7.6), 3.2, 7),         # one cell: the centre past its half
    ((1, 15, 15), (0.5, 7.2, 7.6), 3.2, 7),
    ((1, 15, 15), (-0.2, 7.2, 7.6), 3.2, 1),
    ((2, 13, 1), (1.8, 6.1, 0.6), 2.3, 7),
    ((14, 3, 1), (6.9, 1.6, 0.9), 2.1, 7),
    ((10, 11, 9), (4.5, 5.25, 3.0), 4.9, 7),        # links half a period from the centre
    ((10, 10, 10), (4.5 + 1e-10, 5.5 - 1e-10, 24.0), 5.0, 7),
    ((12, 11, 13), (6.0, 5.0, 6.0), 3.0, 0),
])
def test_minimum_image(cuda, n, centre, radius, bc):
    pop, flags, body = inputs(n, np.array(centre), radius, bc)
    want = link_sum(pop, flags, body, n, bc)
    got = static(cuda, pop, flags, body, n, bc, 8)
    assert np.abs(want[:, :3]).max() > 1e-4
    assert np.abs(got - want).max() < 1e-12


@pytest.mark.parametrize("where", ["population", "density", "velocity", "turn"])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_inputs_show_in_every_component_they_reach(cuda, where, value):
    n, bc = (11, 12, 10), 7
    pop, flags, body = inputs(n, np.array((5.2, 5.7, 4.6)), 2.4, bc)
    p = pop.reshape(19, n[2], n[1], n[0])
    if where == "population":
        p[2, 5, 6, 8] = value                      # the link of one cell towards -x
    elif where == "density":
        p[0, 5, 6, 8] = value
    elif where == "velocity":
        body[0, 7] = value
    else:
        body[0, 11] = value
    want = link_sum(pop, flags, body, n, bc)
    got = static(cuda, pop, flags, body, n, bc, 5)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.abs(got[ok] - want[ok]).max(initial=0.0) < 1e-12
