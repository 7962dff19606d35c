"""The projection of one channel has a form of its own, or the several-channel
form, by the rows' width and size: on every width, on both sides of its limit
where a small dictionary reaches it, and on a grid of CTAs set by hand, the
scores are those of a two-channel call bit for bit."""
import pytest
import torch

from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu
Axis = synth.Axis


# rows of 128, 256, 384, 512, 1,024 and 2,048 floats; the last two grids are past the 160 MiB of their widths
@pytest.mark.parametrize("n,fc", [(100, 9), (200, 9), (300, 7), (500, 5), (900, 5), (2000, 3), (120, 420), (1000, 53)])
def test_one_channel_equals_two(n, fc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    grid = synth.Grid(n, 256.0, Axis(0.3, 2.5, 33), Axis.linspace(0.5, 32.0, fc), Axis.linspace(-3.0, -0.5, 5),
                      Axis.linspace(-20.0, 20.0, 5))
    x = torch.randn((2, n), dtype=torch.float32, device="cuda")
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_FP32)
        two = torch.full((2, grid.n_atoms), 7.0, device="cuda")
        act.act_project(h, x, 2, two)
        for grid_ctas in (0, 152, 37):
            act.act_set_tuning(h, grid_ctas)
            for c in range(2):
                one = torch.full((1, grid.n_atoms), 9.0, device="cuda")
                act.act_project(h, x[c:c + 1], 1, one)
                torch.cuda.synchronize()
                assert act.act_grid_status(h) == act.ACT_OK
                assert torch.equal(one[0], two[c])
    finally:
        act.act_destroy(h)
