"""A BF16 build that screens through templates, when the scratch of a larger
call cannot be had: that call takes the dense GEMM and the FP32 search's
answer, and smaller calls screen through the templates again."""
import pytest
import torch

from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu
Axis = synth.Axis
P = 2
TEMPLATES, DENSE = 1 + P * 6, 1 + P * 5  # kernels of a call: the initialisation, and per order the search and the update


@pytest.fixture(autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    act.load_library()
    yield
    act.act_inject_alloc_failure(0)


def test_a_larger_call_without_memory_leaves_the_smaller_ones_their_templates():
    grid = synth.Grid(512, 256.0, Axis(0.0, 5.0, 101), Axis.linspace(0.5, 60.0, 41), Axis.linspace(-4.0, -0.5, 4),
                      Axis.linspace(-20.0, 20.0, 9))  # 153 MB of BF16 rows
    sig = torch.tensor(synth.random_signals(31, 70, grid.n_samples), dtype=torch.float32, device="cuda")
    h = act.act_grid_create(grid, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_BF16)
        act.act_set_search(h, act.ACT_SEARCH_FP32)
        want = act.decompose(h, sig, P)
    finally:
        act.act_destroy(h)

    def run(h, B):
        out = act.decompose(h, sig[:B], P)
        torch.cuda.synchronize()
        assert act.act_grid_status(h) == act.ACT_OK
        for x, y in zip(out, want):
            assert torch.equal(x, y[:B])
        return act.act_profile_read(h)[3]

    dense = 0
    for nth in range(1, 40):
        h = act.act_grid_create(grid, 0)
        try:
            act.act_dictionary_build(h, act.ACT_DICT_BF16)
            act.act_set_profiling(h, True)
            assert run(h, 20) == TEMPLATES
            act.act_inject_alloc_failure(nth)
            try:
                form = run(h, 70)
            except act.ActError as e:  # a buffer that every search needs
                assert e.status == act.ACT_ERR_OOM
                form = None
            act.act_inject_alloc_failure(0)
            if form == DENSE:
                dense += 1
                assert run(h, 70) == DENSE and run(h, 69) == TEMPLATES
            assert run(h, 20) == TEMPLATES
        finally:
            act.act_destroy(h)
        if form == TEMPLATES:  # the call has no nth allocation
            break
    assert form == TEMPLATES and dense == 7  # each of the screening's buffers failed once
