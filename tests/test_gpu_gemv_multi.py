"""Several channels share passes over the stored FP32 dictionary, in tiles of
8 rows and groups of 4 and 8 channels: at every group boundary, row width and
remainder of rows, each channel's decomposition equals its own one-channel
run bit for bit (scores, selections, ties), and act_project's scores equal
the dictionary rows times the signals within FP32 rounding."""
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


def grid(n, tc, fc, c):
    return synth.Grid(n, 500.0, Axis(0.0, n / tc, tc), Axis.linspace(20.0, 200.0, fc), Axis.linspace(-4.0, -2.0, 3),
                      Axis.linspace(-50.0, 50.0, c))


# row widths 128 .. 2048 floats; atoms: fewer than a tile, one more than a
# chunk, more chunks than SMs, none a multiple of the tile
GRIDS = {"n37": grid(37, 1, 2, 1), "n100": grid(100, 11, 37, 5), "n256": grid(256, 13, 41, 7),
         "n300": grid(300, 9, 33, 5), "n512": grid(512, 17, 29, 7), "n1024": grid(1024, 5, 23, 3),
         "n2048": grid(2048, 7, 31, 3)}


@pytest.mark.parametrize("channels", [2, 3, 4, 5, 8, 9, 12, 13, 16, 17, 29])
@pytest.mark.parametrize("name", sorted(GRIDS))
def test_equals_one_channel_runs(name, channels):
    g = GRIDS[name]
    sig = torch.tensor(synth.random_signals(31, channels, g.n_samples), dtype=torch.float32, device="cuda")
    sig[1] = 0.0  # every score ties
    h = act.act_grid_create(g, 0)
    try:
        act.act_dictionary_build(h, act.ACT_DICT_FP32)
        act.act_set_fused(h, 0)
        many = act.decompose(h, sig, 3)
        scores = torch.full((channels + 1, g.n_atoms), -7.0, device="cuda")
        act.act_project(h, sig, channels, scores)
        for b in range(channels):
            for x, y in zip(many, act.decompose(h, sig[b:b + 1], 3)):
                assert torch.equal(x[b], y[0]), b
        rows = torch.empty((g.n_atoms, g.n_samples), device="cuda")
        act.act_dictionary_rows(h, 0, g.n_atoms, rows)
        torch.cuda.synchronize()
        assert act.act_grid_status(h) == act.ACT_OK
    finally:
        act.act_destroy(h)
    ref = sig.double() @ rows.double().T
    # a score sums at most n products of |g| = 1 and the signal in FP32
    bound = (g.n_samples / 32 + 8) * 2.0**-24 * sig.double().norm(dim=1, keepdim=True)
    assert bool(((scores[:channels].double() - ref).abs() <= bound).all())
    assert bool((scores[channels] == -7.0).all())  # nothing past the last channel
