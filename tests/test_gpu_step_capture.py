"""Steps captured into a CUDA graph: every replay of an even number of steps goes on from
the state that the one before left, for lattices whose uncaptured steps run several to a
launch too (no tolerance)."""
import pytest

from test_gpu_fused_steps import periodic_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,dtype,scheme,n", [
    ((96, 64, 1), "f32", "pull", 8),      # several 2D steps per launch
    ((96, 64, 1), "f16", "pull", 2),
    ((128, 112, 72), "f32", "pull", 2),   # two 3D steps per pass
    ((128, 112, 72), "f32", "pull", 6),
    ((40, 21, 11), "f32", "aa", 4),
    ((33, 20, 9), "f64", "pull", 2),
])
def test_replayed_steps_go_on(shape, dtype, scheme, n):
    import torch

    from paper_2307_11752_gb300 import olb

    case = periodic_case(*shape)
    a, b = case.gpu(dtype, scheme), case.gpu(dtype, scheme)
    b.step(4 + 3 * n)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    assert olb.load().olb_set_stream(a.handle, s.cuda_stream) == 0
    a.step(4)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.step(n)
    torch.cuda.synchronize()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    got, want = a.get_populations(), b.get_populations()
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    for lat in (a, b):
        lat.close()
