"""Channels past whole blocks of 32 have row tiles of their own in the
tensor-core template search (8 or 16 channels x 16 or 8 time centres): around
the counts where that changes, with time centres that no tile divides, on one
SM per MMA and on pairs, the decomposition equals the FP32 template search's
bit for bit, and calls of different counts alternate on one grid."""
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


def grid(n, tc, T=40):
    return synth.Grid(n, 256.0, tc, Axis.linspace(1.0, 60.0, 10), Axis.linspace(-4.0, -1.0, 5),
                      Axis.linspace(-20.0, 20.0, T))


GRIDS = {
    "pairs": grid(400, Axis(0.0, 3.0, 101)),          # 2,000 templates; a last tile of five centres
    "step_at_limit": grid(300, Axis(-4.0, 5.0, 61)),  # 15 steps of 5 are a quarter of the window: 16 centres a tile
    "step_past_limit": grid(296, Axis(0.0, 5.0, 60)), # only 8 centres a tile
    "few_centres": grid(256, Axis(3.0, 9.0, 7), 7),   # fewer centres than a tile has
}


@pytest.mark.parametrize("name", sorted(GRIDS))
def test_equals_fp32_template_search(name):
    g = GRIDS[name]
    sig = torch.tensor(synth.random_signals(77, 113, g.n_samples), dtype=torch.float32, device="cuda")
    sig[33] = 0.0
    h = act.act_grid_create(g, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_RECOMPUTE)

        def run(search, B):
            act.act_set_search(h, search)
            out = act.decompose(h, sig[:B].contiguous(), 3)
            torch.cuda.synchronize()
            assert act.act_grid_status(h) == act.ACT_OK
            return out

        want = run(act.ACT_SEARCH_SHIFT, 113)
        for pairs in (True, False):
            act.act_set_cta_pairs(h, pairs)
            for B in (33, 113, 40, 41, 48, 49, 64, 65, 73, 80, 81, 32, 17, 24, 25):
                for x, y in zip(run(act.ACT_SEARCH_SHIFT_BF16, B), want):
                    assert torch.equal(x, y[:B]), (pairs, B)
    finally:
        act.act_destroy(h)
