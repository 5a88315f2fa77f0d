"""Steps that run several to a kernel against the same steps one to a kernel.

``step(n)`` may advance the lattice by several steps in one pass; n calls of ``step(1)``
never do.  Both round to the storage type after every step and use the same arithmetic,
so the populations must agree bit for bit (no tolerance)."""
import numpy as np
import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import Case, cavity_case, porous_channel_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def olb():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11752_gb300 import build, olb as _olb
    build.build()
    _olb.load()
    return _olb


def periodic_case(nx, ny, nz, seed=5, tau=0.6, force=(0.0, 0.0, 0.0)):
    d = 1 if nz > 1 else 0
    m = I.periodic_box(nx, ny, nz)
    rho = 1.0 + 0.01 * (I.uniform(seed, m.shape) - 0.5)
    u = 0.04 * (I.uniform(seed + 1, (3,) + m.shape) - 0.5)
    if not d:
        u[2] = 0.0
    return Case(d, m, 7 if d else 3, tau, force=force, rho=rho, u=u)


def scattered_case(nx, ny, nz, seed=7):
    """Obstacles at random (15 %), walls on both y faces (one moving), periodic elsewhere."""
    d = 1 if nz > 1 else 0
    m = np.full((nz, ny, nx), I.FLUID, np.uint8)
    m[I.uniform(seed, m.shape) < 0.15] = I.WALL
    m[:, 0, :] = I.WALL
    m[:, -1, :] = I.LID
    return Case(d, m, 5 if d else 1, 0.62, walls={I.LID: (0.04, 0.0, 0.01 if d else 0.0)},
                noise=I.population_noise(seed + 1, 19 if d else 9, m, 1e-3))


def moving_case(nx, ny, nz):
    """Two moving walls that meet (links the link word holds in plane form and others)."""
    m = I.cavity_box(nx, ny, nz)
    m[1:-1, -1, :] = I.LID
    m[:, :, -1] = 4
    return Case(1, m, 0, 0.58, walls={I.LID: (0.04, 0.0, 0.01), 4: (0.0, -0.02, 0.015)},
                noise=I.population_noise(9, 19, m, 1e-3))


def porous_box(nx, ny, nz):
    case = periodic_case(nx, ny, nz)
    case.gamma = I.smoothed_porosity(3, case.material)
    return case


def with_trt(case):
    case.collision, case.magic = "trt", 3.0 / 16.0
    return case


# Two D3Q19 steps per pass over memory: FP32 beyond L2, and 16-bit storage without
# walls from four times L2.  Sizes at the edges of a tile (64 x 14), of the blocks' planes and of the
# lattice; every kind of link the pass tells apart.
CASES_3D = {
    "box128x112x72": (lambda: periodic_case(128, 112, 72), ("f32",)),
    "box126x112x96_porous": (lambda: porous_box(126, 112, 96), ("f32",)),
    "box128x299x51": (lambda: periodic_case(128, 299, 51), ("f32",)),
    "box190x280x150": (lambda: periodic_case(190, 280, 150), ("f16", "bf16")),
    "box_trt": (lambda: with_trt(periodic_case(128, 126, 72)), ("f32",)),
    "cavity": (lambda: cavity_case(128, 128, 114, lid=0.08), ("f32",)),
    "cavity126x127x120": (lambda: cavity_case(126, 127, 120, lid=0.08), ("f32",)),
    "scattered": (lambda: scattered_case(128, 114, 130), ("f32",)),
    "moving": (lambda: with_trt(moving_case(192, 100, 96)), ("f32",)),
}


@pytest.mark.parametrize("name,dtype", [(n, t) for n, (_, ts) in sorted(CASES_3D.items()) for t in ts])
def test_two_steps_per_pass_d3q19(olb, name, dtype):
    _compare(CASES_3D[name][0](), dtype, (1, 2, 7), fused=True)


# Several D2Q9 steps per launch (tiles of 64 x 32 cells with a halo of 8 or, on the
# large lattices, 4): lattices below, at and just over a tile's part, smaller than a halo,
# with force, porosity and TRT.
CASES_2D = {
    "box2x1": lambda: periodic_case(2, 1, 1, force=(1e-4, -2e-4, 0.0)),
    "box2x3": lambda: periodic_case(2, 3, 1),
    "box48x16": lambda: periodic_case(48, 16, 1),
    "box50x17": lambda: periodic_case(50, 17, 1, force=(1e-4, -2e-4, 0.0)),
    "box112x120": lambda: porous_box(112, 120, 1),
    "trt": lambda: with_trt(periodic_case(96, 43, 1, force=(1e-4, -2e-4, 0.0))),
}


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("name", sorted(CASES_2D))
def test_several_steps_per_launch_d2q9(olb, name, dtype):
    _compare(CASES_2D[name](), dtype, (1, 2, 5, 19), fused=True)


@pytest.mark.parametrize("dtype,nx,ny", [("f32", 1100, 291), ("f16", 2002, 1990)])
def test_several_steps_per_launch_d2q9_large(olb, dtype, nx, ny):
    _compare(periodic_case(nx, ny, 1), dtype, (1, 2, 5, 19), fused=True)


def test_populations_read_back_exactly(olb):
    """Populations come back as (double)f + w for every FP32 pattern: zeros of both signs,
    subnormals, the largest and smallest normals, infinities and NaN (D2Q9, whose
    weights are added in FP64; stored values f - w are read through the rest weight)."""
    import torch

    bits = np.array([0, 0x80000000, 1, 0x80000001, 0x007fffff, 0x00800000, 0x80800000, 0x33d6bf95, 0x3f800000,
                     0xbf7fffff, 0x7f7fffff, 0x7f800000, 0xff800000, 0x7fc00000], np.uint32)
    v = bits.view(np.float32).astype(np.float64)
    lat = olb.Lattice(olb.D2Q9, (len(v), 1, 1), dtype="f32")
    lat.set_material(np.ones(len(v), np.uint8), 3)
    w = 4.0 / 9.0
    f = np.zeros((9, 1, 1, len(v)))
    f[0, 0, 0] = v + w
    lat.set_populations(torch.from_numpy(f).cuda())
    got = lat.get_populations()[0, 0, 0].cpu().numpy()
    with np.errstate(over="ignore"):
        want = (f[0, 0, 0] - w).astype(np.float32).astype(np.float64) + w  # as stored, then widened
    assert np.array_equal(got, want, equal_nan=True)
    lat.close()


def _compare(case, dtype, counts, fused):
    import torch

    a, b = case.gpu(dtype, "pull"), case.gpu(dtype, "pull")
    k0 = a.counters()[1], b.counters()[1]
    for n in counts:
        a.step(n)
        for _ in range(n):
            b.step(1)
    ka, kb = a.counters()[1] - k0[0], b.counters()[1] - k0[1]
    assert ka < kb if fused else ka == kb  # the path under test is the one that ran
    assert torch.equal(a.get_populations(), b.get_populations())
    assert a.counters()[0] == b.counters()[0] == sum(counts)
    sa, sb = a.step_stats(4), [b.step(1), b.step(1), b.step(1), b.step_stats(1)][-1]
    assert np.array_equal(sa, sb)
    a.close()
    b.close()
