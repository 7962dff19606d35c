"""The projection of one channel has a form of its own, or the several-channel
form, by the rows' width and size: on every width, on both sides of its limit
where a small dictionary reaches it, and on a grid of CTAs set by hand, the
scores are those of a two-channel call bit for bit.  Few long rows are passed
over channel by channel where a last pass would hold one or two of them: the
scores and selections are those of single calls."""
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


@pytest.mark.parametrize("channels", [2, 3, 5, 6, 9])
@pytest.mark.parametrize("fc", [2, 27])  # 13 and 179 MiB of rows of 2,048 floats
def test_few_long_rows(fc, channels):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    grid = synth.Grid(1900, 1000.0, Axis(0.3, 55.0, 34), Axis.linspace(0.5, 32.0, fc), Axis.linspace(-3.0, -0.5, 5),
                      Axis.linspace(-20.0, 20.0, 5))
    K, stride = grid.n_atoms, 2048
    x = torch.randn((channels, grid.n_samples), dtype=torch.float32, device="cuda")
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_FP32)
        got = torch.full((channels, K), 7.0, device="cuda")
        act.act_project(h, x, channels, got)
        one = torch.empty((1, K), device="cuda")
        for c in range(channels):
            act.act_project(h, x[c:c + 1], 1, one)
            torch.cuda.synchronize()
            assert torch.equal(got[c], one[0])
        rows = torch.zeros((K, stride), device="cuda")
        flat = torch.empty((K, grid.n_samples), device="cuda")
        act.act_dictionary_rows(h, 0, K, flat)
        rows[:, :grid.n_samples] = flat
        r = torch.zeros((channels, stride), device="cuda")
        r[:, :grid.n_samples] = x
        index = torch.empty(channels, dtype=torch.int64, device="cuda")
        score = torch.empty(channels, device="cuda")
        act.act_search_noalloc(rows, K, stride, r, channels, index, score)
        torch.cuda.synchronize()
        want = got.abs()
        assert torch.equal(score, want.max(1).values)
        for c in range(channels):  # the lowest of equal scores
            assert int(index[c]) == int((want[c] == score[c]).nonzero()[0])
    finally:
        act.act_destroy(h)


@pytest.mark.parametrize("stride", [128, 512])
@pytest.mark.parametrize("rows", [1, 7, 8, 1216, 1217, 2432, 2433, 5000, 8400, 9728, 9729])
def test_chunks_of_few_tiles(stride, rows):
    """Row counts on both sides of one, two and the most tiles of 8 rows a
    chunk with a chunk for every SM (152 of them), of five and seven, and a
    last tile of less than 8 rows: three channels at once equal one at a
    time."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gen = torch.Generator(device="cuda").manual_seed(rows)
    d = torch.randn((rows, stride), generator=gen, device="cuda")
    r = torch.randn((3, stride), generator=gen, device="cuda")
    index, score = torch.empty(3, dtype=torch.int64, device="cuda"), torch.empty(3, device="cuda")
    act.act_search_noalloc(d, rows, stride, r, 3, index, score)
    for c in range(3):
        i, s = torch.empty(1, dtype=torch.int64, device="cuda"), torch.empty(1, device="cuda")
        act.act_search_noalloc(d, rows, stride, r[c:c + 1], 1, i, s)
        torch.cuda.synchronize()
        assert int(i[0]) == int(index[c]) and torch.equal(s[0], score[c])
