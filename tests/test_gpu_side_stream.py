"""A dictionary built and first used on a stream that is not ordered behind the
legacy one: the BF16 rows, the cleared work buffers and the template scratch
are whole, and the searches equal the FP32 search bit for bit."""
import pytest
import torch

from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu
Axis = synth.Axis


@pytest.mark.parametrize("tc,build,search", [
    (Axis(0.25, 5.0, 101), act.ACT_DICT_BF16, act.ACT_SEARCH_BF16),           # the GEMM over the rows
    (Axis(0.0, 5.0, 101), act.ACT_DICT_BF16, act.ACT_SEARCH_BF16),            # templates screen
    (Axis(0.0, 5.0, 101), act.ACT_DICT_RECOMPUTE, act.ACT_SEARCH_SHIFT_BF16),
])
def test_first_calls_on_a_side_stream(tc, build, search):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    grid = synth.Grid(512, 256.0, tc, Axis.linspace(0.5, 60.0, 41), Axis.linspace(-4.0, -0.5, 4),
                      Axis.linspace(-20.0, 20.0, 9))
    sig = torch.tensor(synth.random_signals(51, 40, grid.n_samples), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    h = act.act_grid_create(grid, 0)
    try:
        with torch.cuda.stream(side):
            act.act_dictionary_build(h, build, side)
            act.act_set_search(h, search)
            got = act.decompose(h, sig, 3, side)
            side.synchronize()
            assert act.act_grid_status(h, side) == act.ACT_OK
            act.act_set_search(h, act.ACT_SEARCH_SHIFT if build == act.ACT_DICT_RECOMPUTE else act.ACT_SEARCH_FP32)
            want = act.decompose(h, sig, 3, side)
            side.synchronize()
        for x, y in zip(got, want):
            assert torch.equal(x, y)
    finally:
        act.act_destroy(h)
