"""An autotune with several channels times the one FP32 form they have; the
form that one channel takes, the default or one set by hand, stays in use."""
import pytest
import torch

from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("build", [act.ACT_DICT_FP32, act.ACT_DICT_BF16])
@pytest.mark.parametrize("set_by_hand", [0, -1, 152])
def test_several_channels_leave_the_one_channel_form(build, set_by_hand):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    grid = synth.scaled_grid(synth.grid_eeg(), tc_count=64, fc_count=32)  # 1,074 MB of FP32 rows
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, build)
        if set_by_hand:
            act.act_set_tuning(h, set_by_hand)
        in_use = act.act_get_tuning(h)[0]
        assert in_use == (set_by_hand or -1)  # from 64 MiB on the bulk-copy stream is the default
        assert act.act_autotune(h, torch.randn(3, grid.n_samples, device="cuda"), 3) > 0.0
        if set_by_hand or build == act.ACT_DICT_FP32:
            assert act.act_get_tuning(h)[0] == in_use
        else:  # names the grid of the tensor-core search's queued full searches
            assert act.act_get_tuning(h)[0] > 0
        act.act_set_tuning(h, 0)  # keeps the form, which is its caller's own from here on
        assert act.act_get_tuning(h)[0] == in_use
    finally:
        act.act_destroy(h)
