"""FP32 values are widened to FP64 on readout by integer instructions; here over every
exponent.  A lattice at rest with a force field F reads back u = F/2 (rho = 1, j = 0),
with nothing added that would absorb a small value, so the field carries the patterns
in: both signs, subnormals, the smallest and largest normals, infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _patterns():
    mantissas = np.array([0, 1, 2, 0x155555, 0x2aaaab, 0x400000, 0x7ffffe, 0x7fffff], np.uint32)
    exponents = np.arange(256, dtype=np.uint32)
    bits = (exponents[:, None] << 23 | mantissas).reshape(-1)
    subnormal = np.concatenate([np.uint32(1) << np.arange(23, dtype=np.uint32), np.uint32(0x7fffff) >> np.arange(23, dtype=np.uint32)])
    bits = np.concatenate([bits, subnormal])
    return np.concatenate([bits, bits | np.uint32(0x80000000)]).view(np.float32)


@pytest.mark.parametrize("descriptor", ["D2Q9", "D3Q19"])
def test_readout_widens_every_float_exactly(descriptor):
    import torch

    from paper_2307_11752_gb300 import olb

    F = _patterns()
    n = len(F)
    three = descriptor == "D3Q19"
    lat = olb.Lattice(getattr(olb, descriptor), (n, 1, 1), dtype="f32")
    field = np.zeros((3, n))
    with np.errstate(invalid="ignore"):
        for a in range(3 if three else 2):
            field[a] = np.roll(F, 7 * a).astype(np.float64)
    lat.set_force_field(torch.from_numpy(field).cuda())
    lat.init_equilibrium()
    rho, u = lat.moments()
    u = u.reshape(3, n).cpu().numpy()
    assert bool((rho == 1.0).all())
    with np.errstate(invalid="ignore", over="ignore"):
        for a in range(3 if three else 2):
            half = np.float32(0.0) + np.float32(0.5) * np.roll(F, 7 * a)  # what the kernel holds in FP32
            want = half.astype(np.float64)
            assert (np.abs(want[np.isfinite(want) & (want != 0)]) < 2.0 ** -126).sum() > 50  # subnormals are among them
            nan = np.isnan(want)
            assert np.array_equal(np.isnan(u[a]), nan)
            zero = want == 0  # of either sign: that of j at rest, a sum of zeros, is not specified
            assert np.array_equal(u[a] == 0, zero)
            other = ~(nan | zero)
            assert np.array_equal(u[a][other].view(np.uint64), want[other].view(np.uint64))
    lat.close()
