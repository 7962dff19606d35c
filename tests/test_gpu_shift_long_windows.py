"""The longest windows that the tensor-core template search serves where the
time centres lie one and two samples apart: its rescore keeps two buffers of
P = ceil(L / step) (a multiple of 16) rows of 128 bytes and a residual beside
them, and the windows here fill that exactly (864 samples at step 1, 1,696 at
step 2: 225,280 bytes) or up to the last sixteenth of a phase.  The search is
named, so a build that no longer offers it fails, and must equal the FP32
template search bit for bit, with few channels and with many."""
import numpy as np
import pytest
import torch

from paper_2607_16629_gb300 import act, synth
from parity_helpers import gpu_decompose

pytestmark = pytest.mark.gpu
Axis = synth.Axis


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    act.load_library()


@pytest.mark.parametrize("channels", [2, 20])
@pytest.mark.parametrize("step,n", [(1, 849), (1, 864), (2, 1665), (2, 1696)])
def test_equals_fp32_template_search(step, n, channels):
    grid = synth.Grid(n, 500.0, Axis(3.0, float(step), 70), Axis(20.0, 30.0, 5), Axis(-4.0, 0.7, 5), Axis(-60.0, 40.0, 4))
    sig = synth.random_signals(23, channels, n)
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_RECOMPUTE)
        act.act_set_search(h, act.ACT_SEARCH_SHIFT)
        want = gpu_decompose(h, sig, 4)
        act.act_set_search(h, act.ACT_SEARCH_SHIFT_BF16)
        for x, y in zip(gpu_decompose(h, sig, 4), want):
            assert np.array_equal(x, y)
    finally:
        act.act_destroy(h)


@pytest.mark.parametrize("channels", [3, 5])
@pytest.mark.parametrize("step,n", [(4, 832), (4, 833), (8, 1696), (9, 1700)])
def test_few_channels_phases_in_flight(step, n, channels):
    """Rescores with every phase in flight up to the last window that leaves
    room for it (832 samples at step 4) and to eight phases, and past them
    with the buffers there is room for (4 channels and fewer) or with two."""
    grid = synth.Grid(n, 500.0, Axis(3.0, float(step), 70), Axis(20.0, 30.0, 5), Axis(-4.0, 0.7, 5), Axis(-60.0, 40.0, 4))
    sig = synth.random_signals(29, channels, n)
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_RECOMPUTE)
        act.act_set_search(h, act.ACT_SEARCH_SHIFT)
        want = gpu_decompose(h, sig, 4)
        act.act_set_search(h, act.ACT_SEARCH_SHIFT_BF16)
        for x, y in zip(gpu_decompose(h, sig, 4), want):
            assert np.array_equal(x, y)
    finally:
        act.act_destroy(h)
