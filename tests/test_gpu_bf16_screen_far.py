"""Atoms centred more than 2^24 samples outside the window, wide enough to be
seen in it: their sample offsets are no whole FP32 numbers any more, and the
templates that screen a BF16 build's rows have to hold the rows' samples all
the same.  The search equals the FP32 search over the rows bit for bit."""
import pytest
import torch

from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu
Axis = synth.Axis


@pytest.mark.parametrize("first", [-float(2 ** 25), float(2 ** 25 + 3)])
def test_far_wide_atoms(first):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    grid = synth.Grid(200, 256.0, Axis(first, 1.0, 70), Axis.linspace(0.5, 60.0, 83), Axis.linspace(11.0, 13.0, 8),
                      Axis.linspace(-1e-5, 1e-5, 8))
    assert grid.n_atoms * 256 * 2 >= 128 << 20
    sig = torch.tensor(synth.random_signals(41, 5, grid.n_samples), dtype=torch.float32, device="cuda")
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_BF16)
        out = []
        for search in (act.ACT_SEARCH_BF16, act.ACT_SEARCH_FP32):
            act.act_set_search(h, search)
            out.append(act.decompose(h, sig, 4))
            torch.cuda.synchronize()
            assert act.act_grid_status(h) == act.ACT_OK
        for x, y in zip(*out):
            assert torch.equal(x, y)
    finally:
        act.act_destroy(h)
