"""Total momentum of periodic FP64 flows over many steps.

Collisions and streaming conserve it; what remains is rounding.  A step's rounding
errors differ from cell to cell (each below 2^-55 for values of 0.05; some 30 per cell),
so over N cells and n steps they add up to about sqrt(30 N n) 2^-55 beside a total of
0.05 N: below 1e-15 here.  A collision whose constants do not sum to 1 instead multiplies
the momentum by 1 - 2^-53 at every step.  The bound, n 2^-56, lies between."""
import math

import numpy as np
import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import Case

pytestmark = pytest.mark.gpu

STEPS = 1000


def _momentum(lat, q, c):
    f = lat.get_populations().cpu().numpy().reshape(q, -1)
    return math.fsum(math.fsum((c[i] * f[i]).tolist()) for i in range(q) if c[i])


@pytest.mark.parametrize("d,collision,tau", [(0, "bgk", 0.8), (0, "trt", 0.75), (1, "bgk", 0.7), (1, "trt", 1.3)])
def test_total_momentum_does_not_drift(d, collision, tau):
    from oracle import oracle as orc

    nx, ny, nz = (64, 62, 1) if d == 0 else (31, 32, 30)
    m = I.periodic_box(nx, ny, nz)
    y, x = np.meshgrid(2 * np.pi * np.arange(ny) / ny, 2 * np.pi * np.arange(nx) / nx, indexing="ij")
    u = np.zeros((3,) + m.shape)
    u[0] = 0.05 + 0.02 * np.sin(x) * np.cos(y)
    u[1] = 0.03 - 0.02 * np.cos(x) * np.sin(y)
    rho = 1.0 + 1e-3 * np.cos(x + y) * np.ones(m.shape)
    case = Case(d, m, 7 if d else 3, tau, rho=rho, u=u, collision=collision, magic=3.0 / 16.0)
    lat = case.gpu("f64", "pull")
    c = orc.descriptor(d)[2]
    for axis in (0, 1):
        assert abs(_momentum(lat, case.q, c[:, axis])) > 0.02 * m.size  # not a vanishing total
    before = [_momentum(lat, case.q, c[:, a]) for a in (0, 1)]
    lat.step(STEPS)
    after = [_momentum(lat, case.q, c[:, a]) for a in (0, 1)]
    lat.close()
    for b, a in zip(before, after):
        assert abs(a - b) <= STEPS * 2.0 ** -56 * abs(b), (b, a, (a - b) / b)
