"""A gradient run on a slab (a lattice with halo planes): the handle ends in the state that
as many steps leave, halo planes as the steps read them, whatever device memory held
before (no tolerance)."""
import numpy as np
import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import Case

pytestmark = pytest.mark.gpu


def _slab(dtype):
    nx, ny, nz = 20, 14, 9
    m = I.periodic_box(nx, ny, nz)
    m[:, 0, :] = I.WALL
    m[:, -1, :] = I.WALL
    rho = 1.0 + 0.01 * (I.uniform(5, m.shape) - 0.5)
    u = 0.04 * (I.uniform(6, (3,) + m.shape) - 0.5)
    lat = Case(1, m, 1, 0.7, force=(1e-5, 0.0, 0.0), rho=rho, u=u).gpu(dtype, "pull")
    lat.set_active_planes(1, nz - 2)
    return lat


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("before", [0, 3])
@pytest.mark.parametrize("every", [6, 4, 1])
def test_state_after_a_gradient_run_is_the_one_after_its_steps(dtype, before, every):
    import torch

    a = _slab(dtype)
    a.step(before + 6)
    want = a.get_populations()
    b = _slab(dtype)
    b.step(before)
    # what the next buffers of the state's size find in their memory
    state = 19 * ((20 * 14 * 9 + 63) // 64 * 64 + 256) * (4 if dtype == "f32" else 8)
    held = [torch.full((state // 8,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(12)]
    torch.cuda.synchronize()
    del held
    b.adjoint_run(6, every, (0, 3, 0))
    got = b.get_populations()
    assert bool(torch.isfinite(want).all())
    assert torch.equal(got[:, 1:-1], want[:, 1:-1])
    for lat in (a, b):
        lat.close()
