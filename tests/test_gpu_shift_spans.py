"""The tensor-core template search multiplies only the lags where a template
tile does not vanish; its templates are ordered by duration.  Where that cut
and that order could go wrong (very short atoms, durations mixed within a
32-template block, durations falling along the axis, time centres outside the
window, a step longer than the window, template counts around the tile
widths), the whole decomposition still equals the FP32 template search's bit
for bit, by the search's own error bound."""
import numpy as np
import pytest
import torch

from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu
Axis = synth.Axis


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    act.load_library()


GRIDS = {
    # 9 to 111 samples of 2,048; 24 chirp rates: a block holds two durations
    "emg_long": synth.Grid(2048, 500.0, Axis(0.0, 8.0, 256), Axis.linspace(20.0, 200.0, 9),
                           Axis.linspace(-4.0, -1.5, 8), Axis.linspace(-100.0, 100.0, 24)),
    # 5 chirp rates: every block holds all durations; 325 templates (256 + 69)
    "mixed_blocks": synth.Grid(777, 500.0, Axis(2.0, 7.0, 111), Axis.linspace(20.0, 200.0, 13),
                               Axis.linspace(-6.0, -1.0, 5), Axis.linspace(-100.0, 100.0, 5)),
    # durations falling along the axis; atoms from under a sample to the whole window
    "falling": synth.Grid(400, 256.0, Axis(0.0, 3.0, 133), Axis.linspace(0.5, 32.0, 8),
                          Axis(-0.5, -0.9, 8), Axis.linspace(-20.0, 20.0, 32)),
    # centres before, in and after the window: tails are all that some atoms have
    "outside": synth.Grid(203, 500.0, Axis(-160.0, 5.0, 101), Axis.linspace(20.0, 180.0, 6),
                          Axis.linspace(-4.5, -2.0, 6), Axis.linspace(-60.0, 60.0, 32)),
    # a step longer than the window: lags no window sees
    "long_step": synth.Grid(96, 256.0, Axis(-250.0, 130.0, 5), Axis.linspace(2.0, 60.0, 16),
                            Axis.linspace(-4.0, -0.5, 8), Axis.linspace(-20.0, 20.0, 3)),
}


@pytest.mark.parametrize("channels", [1, 3, 40])
@pytest.mark.parametrize("name", sorted(GRIDS))
def test_equals_fp32_template_search(name, channels):
    g = GRIDS[name]
    sig = torch.tensor(synth.random_signals(123, channels, g.n_samples), dtype=torch.float32, device="cuda")
    for b in range(0, channels, 2):  # chirps in every other channel, white noise in the others
        sig[b] = torch.tensor(synth.chirp_burst(g.n_samples, g.fs, g.n_samples / (2.0 + b), 40.0, -3.0, 10.0, 2.0))
    h = act.act_grid_create(g, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_RECOMPUTE)
        got = []
        for search in (act.ACT_SEARCH_SHIFT, act.ACT_SEARCH_SHIFT_BF16):
            act.act_set_search(h, search)
            got.append(act.decompose(h, sig, 5))
            torch.cuda.synchronize()
            assert act.act_grid_status(h) == act.ACT_OK
    finally:
        act.act_destroy(h)
    for x, y in zip(*got):
        assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
