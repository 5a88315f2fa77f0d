"""Several steps per launch in the combinations that the kernels' own tests leave out:
walls with porosity, TRT in 16-bit storage, and the forward segments of a gradient run.
Bit for bit against steps one by one."""
import pytest

from paper_2307_11752_gb300 import inputs as I

from test_gpu_fused_steps import _compare, moving_case, olb, periodic_case, porous_box, scattered_case, with_trt  # noqa: F401

pytestmark = pytest.mark.gpu


def _porous(case):
    case.gamma = I.smoothed_porosity(4, case.material)
    return case


CASES = {
    "scattered_porous": (lambda: _porous(scattered_case(128, 114, 130)), "f32"),
    "moving_porous_trt": (lambda: _porous(with_trt(moving_case(192, 100, 96))), "f32"),
    "box_trt_f16": (lambda: with_trt(periodic_case(192, 280, 150)), "f16"),
    "box_porous_trt_bf16": (lambda: with_trt(porous_box(190, 280, 150)), "bf16"),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_two_steps_per_pass_combined(olb, name):  # noqa: F811
    make, dtype = CASES[name]
    _compare(make(), dtype, (1, 2, 7), fused=True)


@pytest.mark.parametrize("make,n,every", [
    (lambda: porous_box(96, 64, 1), 20, 7),          # several 2D steps per launch
    (lambda: porous_box(128, 112, 72), 9, 4),        # two 3D steps per pass
    (lambda: scattered_case(128, 114, 130), 9, 4),
])
def test_forward_segments_of_a_gradient(olb, make, n, every):  # noqa: F811
    import torch

    case = make()
    got = []
    for k in (every, 1):  # segments of one step never hold several to a launch
        lat = case.gpu("f32", "pull")
        lat.step(2)
        launches = lat.counters()[1]
        loss, dg, dtau = lat.adjoint_run(n, k, (0, 5, 0))
        launches = lat.counters()[1] - launches
        got.append((loss, dg.clone(), dtau, lat.get_populations(), launches))
        lat.close()
    (la, ga, ta, fa, ka), (lb, gb, tb, fb, kb) = got
    assert la == lb and ta == tb
    assert torch.equal(ga, gb) and torch.equal(fa, fb)
    # without fusion: n forward, n adjoint, 3 others; recomputed: (segments - 1)(K - 1)
    segments = (n + every - 1) // every
    assert kb == 2 * n + 3
    assert ka < 2 * n + 3 + (segments - 1) * (every - 1)
