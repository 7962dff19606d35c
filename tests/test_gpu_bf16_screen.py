"""A BF16 build whose time centres are whole samples screens its atoms with
the template GEMM and scores the flagged rows with the FP32 GEMV's
arithmetic.  On grids just above the size from which it does (time centres
that are no multiple of a tile, template counts that are no multiple of a
block or a tile, centres outside the window, steps of 1 and 9), with many and
few channels, silent ones, refinement and in an uneven batch, everything
equals the FP32 search bit for bit; a grid with centres between samples (the
dense GEMM) does too."""
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


def grid(n, tc, fc, logdt, c):
    return synth.Grid(n, 256.0, tc, Axis.linspace(0.5, 60.0, fc), Axis.linspace(-4.0, -0.5, logdt),
                      Axis.linspace(-20.0, 20.0, c))


GRIDS = {
    "step1_ragged": grid(200, Axis(0.0, 1.0, 200), 59, 5, 7),       # 2,065 templates
    "step9_outside": grid(301, Axis(-45.0, 9.0, 43), 71, 7, 13),    # 6,461 templates
    "mid": grid(512, Axis(0.0, 5.0, 101), 41, 4, 9),                # 1,476 templates
    "between": grid(512, Axis(0.25, 5.0, 101), 41, 4, 9),           # no templates: the dense GEMM
}


def run(h, search, sig, P):
    act.act_set_search(h, search)
    out = act.decompose(h, sig, P)
    torch.cuda.synchronize()
    assert act.act_grid_status(h) == act.ACT_OK
    return out


@pytest.mark.parametrize("channels,refine", [(1, 0), (5, 4), (33, 0), (140, 0)])
@pytest.mark.parametrize("name", sorted(GRIDS))
def test_equals_fp32_search(name, channels, refine):
    g = GRIDS[name]
    assert g.n_atoms * ((g.n_samples + 63) // 64 * 64) * 2 >= 128 << 20
    sig = np.stack([synth.eeg_like_signal(3, 500 + b, n_samples=g.n_samples)[0] for b in range(channels)])
    if channels > 4:
        sig[2] = 0.0
        sig[4] = synth.random_signals(7, 1, g.n_samples)[0]
    sig = torch.tensor(sig, dtype=torch.float32, device="cuda")
    h = act.act_grid_create(g, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_BF16)
        act.act_set_refinement(h, refine)
        for x, y in zip(run(h, act.ACT_SEARCH_BF16, sig, 4), run(h, act.ACT_SEARCH_FP32, sig, 4)):
            assert torch.equal(x, y)
        with pytest.raises(act.ActError):  # a build of rows has no template search
            act.act_set_search(h, act.ACT_SEARCH_SHIFT_BF16)
            act.decompose(h, sig, 1)
    finally:
        act.act_destroy(h)


def test_uneven_batch_and_a_later_larger_call():
    """The plan owns its screening scratch: a larger call on one of its grids
    between two runs changes nothing."""
    gs = [GRIDS["step1_ragged"], GRIDS["step9_outside"]]
    lengths = [gs[i % 2].n_samples for i in range(7)]
    sig = [synth.eeg_like_signal(3, 700 + i, n_samples=n)[0].astype(np.float32) for i, n in enumerate(lengths)]
    flat = torch.tensor(np.concatenate(sig), device="cuda")
    off = np.concatenate([[0], np.cumsum(lengths)])
    hs = [act.act_grid_create(g, 0) for g in gs]
    plan = None
    try:
        for h in hs:
            act.act_dictionary_build(h, act.ACT_DICT_BF16)
        plan = act.act_ragged_plan_create(hs, off, 3)

        def once():
            atoms = torch.empty((7, 3, act.ATOM_BYTES), dtype=torch.uint8, device="cuda")
            coef = torch.empty((7, 3), device="cuda")
            act.act_ragged_decompose(plan, flat, atoms, coef)
            torch.cuda.synchronize()
            return atoms, coef

        a0, c0 = once()
        run(hs[0], act.ACT_SEARCH_AUTO, torch.randn(50, gs[0].n_samples, device="cuda"), 2)
        a1, c1 = once()
        assert torch.equal(a0, a1) and torch.equal(c0, c1)
        for i in range(7):
            x = torch.tensor(sig[i][None], device="cuda")
            atoms, coef, _, _ = run(hs[i % 2], act.ACT_SEARCH_FP32, x, 3)
            assert torch.equal(atoms[0], a0[i]) and torch.equal(coef[0], c0[i])
    finally:
        act.act_ragged_plan_destroy(plan)
        for h in hs:
            act.act_destroy(h)


def test_more_channels_than_the_templates_screen():
    """Past the channel count whose screening scratch would outgrow the rows
    (1,980 on this grid) the dense GEMM screens; calls on either side of it
    alternate on one grid."""
    g = GRIDS["mid"]
    sig = torch.tensor(synth.random_signals(11, 2100, g.n_samples), dtype=torch.float32, device="cuda")
    h = act.act_grid_create(g, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_BF16)
        want = run(h, act.ACT_SEARCH_FP32, sig, 2)
        for B in (3, 2100, 1900, 2100, 3):
            for x, y in zip(run(h, act.ACT_SEARCH_BF16, sig[:B], 2), want):
                assert torch.equal(x, y[:B])
    finally:
        act.act_destroy(h)
