"""FP64 steps of lattices whose cells do not fill the warps or the blocks evenly,
against the FP64 oracle (relative bound 1e-12: some 50 steps of about 200 operations at
2^-53 each), with BGK and TRT, force, porosity and walls, and statistics."""
import numpy as np
import pytest

from paper_2307_11752_gb300 import inputs as I

from _cases import cavity_case, porous_channel_case, rel_err, tgv2d_case

pytestmark = pytest.mark.gpu


def _trt(case):
    case.collision, case.magic = "trt", 3.0 / 16.0
    return case


CASES = {
    "d2q9_1024": lambda: tgv2d_case(32),                                  # 32 blocks of 32 threads
    "d2q9_odd": lambda: porous_channel_case(nx=77, ny=43, d=0, moving=True),
    "d3q19_rows75": lambda: porous_channel_case(nx=75, ny=31, nz=17),     # rows span warps unevenly
    "d3q19_one_over": lambda: cavity_case(nx=33, ny=35, nz=33),
    "d3q19_trt": lambda: _trt(porous_channel_case(nx=41, ny=30, nz=33, moving=True)),
}


@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_steps_against_the_oracle(oracle, name, scheme):
    case = CASES[name]()
    ref = case.oracle(oracle)
    f = case.oracle_state(ref)
    ref.step(f, 50)
    want = ref.diagnostics(f)
    ref.step(f, 1)
    g = case.gpu("f64", scheme)
    stats = g.step_stats(51)
    assert rel_err(g.get_populations().cpu().numpy(), f, case.material == I.FLUID) <= 1e-12
    assert abs(stats[0] - want[0]) <= 1e-12 * want[0] and stats[6] == 0
    assert np.allclose(stats[4:6], want[4:6], rtol=1e-9)
    g.close()
