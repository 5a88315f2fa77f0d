"""The velocity handover between a fluid and a scalar lattice on different streams: the
scalar's stream is kept busy, so that the handover runs long after the host has queued
the fluid's next steps, and still it has to read the state at the time of the call.  The
reference is the same loop on one stream (no tolerance)."""
import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import porous_channel_case

pytestmark = pytest.mark.gpu


def _run(scheme, shape, fluid_stream, scalar_stream, between):
    import torch

    from paper_2307_11752_gb300 import olb

    nx, ny, nz = shape
    g = porous_channel_case(nx, ny, nz, d=1 if nz > 1 else 0).gpu("f32", scheme)
    torch.cuda.synchronize()
    lib = olb.load()
    a = olb.AdeLattice(olb.D3Q7 if nz > 1 else olb.D2Q5, shape, "f32", stream=scalar_stream)
    busy = olb.AdeLattice(olb.D3Q7, (96, 96, 96), "f32", stream=scalar_stream)
    C = torch.from_numpy(I.uniform(3, (nz, ny, nx))).cuda()
    Cb = torch.full((96, 96, 96), 0.5, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.olb_set_stream(g.handle, fluid_stream.cuda_stream) == 0
    a.set_tau(0.7)
    a.set_velocity((0.0, 0.0, 0.0))
    a.init(C)
    busy.set_velocity((0.01, 0.0, 0.0))
    busy.init(Cb)
    for _ in range(4):
        busy.step(200)
        a.set_velocity_from(g)
        g.step(between)
        a.step(1)
    torch.cuda.synchronize()
    C_out, f_out = a.density(), g.get_populations()
    torch.cuda.synchronize()
    for lat in (a, busy, g):
        lat.close()
    return C_out, f_out


@pytest.mark.parametrize("between", [1, 2, 3])
@pytest.mark.parametrize("scheme", ["aa", "pull"])
@pytest.mark.parametrize("shape", [(46, 13, 1), (33, 12, 10)])
def test_handover_between_streams(shape, scheme, between):
    import torch

    one = torch.cuda.Stream()
    want = _run(scheme, shape, one, one, between)
    got = _run(scheme, shape, torch.cuda.Stream(), torch.cuda.Stream(), between)
    assert torch.equal(want[0], got[0])
    assert torch.equal(want[1], got[1])
