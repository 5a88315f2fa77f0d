"""A fluid's velocity handed to a scalar lattice in the scalar's storage type, and the
adjoint's segments: both must not depend on how the work is cut (no tolerance)."""
import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import porous_channel_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scalar", ["f32", "f64"])
@pytest.mark.parametrize("fluid", ["f32", "f16", "f64"])
@pytest.mark.parametrize("shape", [(45, 13, 1), (33, 12, 10)])
def test_velocity_from_fluid_equals_its_moments(shape, fluid, scalar):
    import torch

    from paper_2307_11752_gb300 import olb

    nx, ny, nz = shape
    g = porous_channel_case(nx, ny, nz, d=1 if nz > 1 else 0).gpu(fluid, "pull")
    C = torch.from_numpy(I.uniform(3, (nz, ny, nx))).cuda()
    a, b = [olb.AdeLattice(olb.D3Q7 if nz > 1 else olb.D2Q5, shape, scalar) for _ in range(2)]
    for lat in (a, b):
        lat.set_tau(0.7)
    for k in range(4):
        a.set_velocity_from(g)
        b.set_velocity(field=g.moments()[1])
        if k == 0:
            a.init(C)
            b.init(C)
        a.step(2)
        b.step(2)
        g.step(1)
    assert torch.equal(a.density(), b.density())


@pytest.mark.parametrize("dtype", ["f32", "f16", "f64"])
@pytest.mark.parametrize("before", [0, 2])
def test_adjoint_does_not_depend_on_the_segments(dtype, before):
    """7 steps in segments of 1, 3 (the last one shorter), 7 and 50 (one segment), from
    the state after initialisation and from the one after steps."""
    import torch

    case = porous_channel_case(36, 14, 11, moving=True)
    got = []
    for every in (1, 3, 7, 50):
        g = case.gpu(dtype, "pull")
        g.step(before)
        loss, dg, dtau = g.adjoint_run(7, every, (0, 35, 0))
        got.append((loss, dg.clone(), dtau, g.get_populations(), g.counters()[0]))
        g.close()
    ref = case.gpu(dtype, "pull")
    ref.step(before + 7)
    for loss, dg, dtau, f, t in got:
        assert loss == got[0][0] and dtau == got[0][2] and t == before + 7
        assert torch.equal(dg, got[0][1])
        assert torch.equal(f, ref.get_populations())
    ref.close()
