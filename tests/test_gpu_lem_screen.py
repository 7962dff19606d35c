"""The hierarchical search screens its candidates in FP32 and projects again
those that the screening's error bound leaves in reach.  Against the FP64
oracle where that could pick wrongly: coarse samples of one, a few, a number
that is no power of two, and the most allowed (the ranking's buckets); all 16
kept; windows of part of a row, odd lengths and the longest; atoms shorter
than a sample and centres far outside the window (which the bound does not
cover); and a zero residual."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_16629_gb300 import act, synth

pytestmark = pytest.mark.gpu
Axis = synth.Axis


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    act.load_library()


def grid(n, fs, tc=None, logdt=(-3.0, -0.5)):
    lo, hi = tc or (0.0, n - 1.0)
    return synth.Grid(n, fs, Axis.linspace(lo, hi, 9), Axis.linspace(0.5, fs / 8.0, 9), Axis.linspace(*logdt, 5),
                      Axis.linspace(-20.0, 20.0, 5))


CASES = {
    "one": (grid(37, 256.0), 1, 1, 0),
    "few": (grid(129, 256.0), 5, 4, 1),
    "odd_count": (grid(512, 256.0), 777, 4, 2),
    "most": (grid(512, 256.0), 16384, 16, 1),
    "longest": (grid(2048, 500.0), 2048, 16, 2),
    "tiny_atoms": (grid(200, 256.0, logdt=(-9.0, -5.0)), 600, 4, 2),
    "outside": (grid(300, 256.0, tc=(-900.0, 1200.0)), 1500, 4, 2),
}
STEPS = ((64, 2, 2, 5), (32, 1, 1, 2.5), (16, 0.5, 0.5, 0.5))
RADIUS = (2, 2, 1, 2)


@pytest.mark.parametrize("name", sorted(CASES))
def test_screened_selection_is_the_oracles(name):
    g, n_coarse, top_k, levels = CASES[name]
    axes = [g.tc, g.fc, g.logdt, g.c]
    lo, hi = (np.array([f(a.lo, a.lo + (a.count - 1) * a.step) for a in axes]) for f in (min, max))
    params = oracle.lem_params(n_coarse, top_k, levels, STEPS, RADIUS)
    B, seed = 3, 99
    sig = np.stack([synth.eeg_like_signal(2, 200 + b, n_samples=g.n_samples, fs=g.fs)[0] for b in range(B)])
    sig = sig.astype(np.float32)
    sig[1] = 0.0
    h = act.act_grid_create(g, 0)
    try:
        act.act_set_search(h, act.ACT_SEARCH_LEM)
        act.act_set_lem(h, n_coarse, top_k, levels, STEPS, RADIUS, seed)
        atoms, coef, resid, energy = act.decompose(h, torch.tensor(sig, device="cuda"), 1)
        torch.cuda.synchronize()
        assert act.act_grid_status(h) == act.ACT_OK
        th = act.atom_params(atoms).cpu().numpy()[:, 0]
    finally:
        act.act_destroy(h)
    assert np.all(coef.cpu().numpy()[1] == 0.0)
    for b in (0, 2):
        th_o, s_o = oracle.lem_select(params, lo, hi, g.fs, sig[b].astype(np.float64), seed, b, 0)
        if not np.array_equal(th[b], th_o):  # a near-tie: scores within 1e-5 relative, as elsewhere
            atom, _ = oracle.atom(*th[b], g.fs, g.n_samples)
            assert abs(abs(atom @ sig[b].astype(np.float64)) - abs(s_o)) <= 1e-5 * abs(s_o), (th[b], th_o)
