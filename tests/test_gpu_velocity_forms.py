"""One scalar lattice whose velocity comes in turn from a fluid lattice, from a field and
uniform: each form takes effect at once, changing the form needs no device memory after
the first field, and a first field that finds none leaves the velocity as it was."""
import ctypes

import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import porous_channel_case

pytestmark = pytest.mark.gpu

SHAPE = (33, 12, 10)


class _NoMemory:
    """Within it the library's allocator has no memory to give (buffers held stay valid)."""

    def __enter__(self):
        from paper_2307_11752_gb300 import olb

        self.asked = []

        def refuse(size, ctx):
            self.asked.append(size)
            return None

        self.keep = (olb._ALLOC_T(refuse), olb._FREE_T(lambda ptr, ctx: None))
        assert olb.load().olb_set_allocator(ctypes.cast(self.keep[0], ctypes.c_void_p),
                                            ctypes.cast(self.keep[1], ctypes.c_void_p), None) == 0
        return self

    def __exit__(self, *exc):
        from paper_2307_11752_gb300 import olb

        alloc, free = olb._callbacks  # torch's, as before (its buffers are still held)
        assert olb.load().olb_set_allocator(ctypes.cast(alloc, ctypes.c_void_p),
                                            ctypes.cast(free, ctypes.c_void_p), None) == 0


def _scalar(olb, dtype, C):
    lat = olb.AdeLattice(olb.D3Q7, SHAPE, dtype)
    lat.set_tau(0.7)
    lat.set_velocity((0.02, -0.01, 0.03))
    lat.init(C)
    return lat


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_velocity_forms_in_turn(dtype):
    import torch

    from paper_2307_11752_gb300 import olb

    nx, ny, nz = SHAPE
    g = porous_channel_case(nx, ny, nz).gpu("f32", "pull")
    g.step(5)
    u = g.moments()[1]
    other = (0.5 * u).contiguous()
    C = torch.from_numpy(I.uniform(3, (nz, ny, nx))).cuda()
    a, b = _scalar(olb, dtype, C), _scalar(olb, dtype, C)

    a.set_velocity_from(g)
    b.set_velocity(field=u)
    for form in ("field", "fluid", "uniform", "fluid", "field"):
        a.step(3)
        b.step(3)
        with _NoMemory() as none:
            if form == "field":
                a.set_velocity(field=other)
            elif form == "fluid":
                a.set_velocity_from(g)
            else:
                a.set_velocity((0.01, 0.0, 0.02))
        assert none.asked == []
        if form == "uniform":
            b.set_velocity((0.01, 0.0, 0.02))
        else:
            b.set_velocity(field=other if form == "field" else u)
    a.step(3)
    b.step(3)
    assert torch.equal(a.density(), b.density())


@pytest.mark.parametrize("form", ["field", "fluid"])
def test_a_field_without_memory_leaves_the_velocity(form):
    import torch

    from paper_2307_11752_gb300 import olb

    nx, ny, nz = SHAPE
    g = porous_channel_case(nx, ny, nz).gpu("f32", "pull")
    u = g.moments()[1]
    C = torch.from_numpy(I.uniform(3, (nz, ny, nx))).cuda()
    a, b = _scalar(olb, "f32", C), _scalar(olb, "f32", C)
    with _NoMemory():
        with pytest.raises(olb.OlbError) as e:
            if form == "field":
                a.set_velocity(field=u)
            else:
                a.set_velocity_from(g)
    assert e.value.status == -3
    a.step(3)
    b.step(3)
    assert torch.equal(a.density(), b.density())
