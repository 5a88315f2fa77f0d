"""Gradients of lattices just below and just above three blocks of the adjoint kernel per
SM, where it changes from the instance with more registers to the one with more blocks
resident, in FP32 and 16-bit storage against the FP64 gradient of the same run.  Bounds
per cell as in the comparison with the oracle (relative to the cell, and to the largest
cell): FP32 1e-4 and 1e-6, FP16 2e-2 and 5e-4."""
import pytest

from _cases import assert_cells_close, porous_channel_case

pytestmark = pytest.mark.gpu

BOUNDS = {"f32": (1e-4, 1e-6), "f16": (2e-2, 5e-4)}


@pytest.mark.parametrize("dtype", sorted(BOUNDS))
@pytest.mark.parametrize("over", [-1, 0, 1])
def test_gradient_at_three_blocks_per_sm(dtype, over):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # 64 x 12 cells a plane: 3 blocks of 64 x 4
    case = porous_channel_case(nx=64, ny=12, nz=sms + over)
    got = {}
    for t in ("f64", dtype):
        lat = case.gpu(t, "pull")
        loss, dg, dtau = lat.adjoint_run(7, 3, (0, 63, 0))
        got[t] = loss, dg.cpu().numpy(), dtau
        lat.close()
    rtol, floor = BOUNDS[dtype]
    assert_cells_close(got[dtype][1], got["f64"][1], rtol, floor)
    assert abs(got[dtype][2] - got["f64"][2]) <= rtol * abs(got["f64"][2])
