"""The calls whose speed this repository is judged by, through its Python binding.

A case is one call that a user's program makes again and again on a grid it set up once: a matching-pursuit
decomposition (`act.decompose`) of one or several signals over a stored or a template dictionary, the same with
off-grid refinement, the hierarchical search, an uneven batch, a projection on all atoms, or the differentiable
chirplet score. Launch configurations are the library's defaults.

Grids are those of `synth` (the 16,384-atom check, EEG-, EMG- and radar-like) and of the paper's Table 2; signals
are seeded Gaussian-windowed chirps plus noise at the recipes' counts, ranges and noise levels.
"""
import math

import numpy as np
import torch

from paper_2607_16629_gb300 import act, synth
from paper_2607_16629_gb300.autograd import chirplet_score

DICT = {"fp32": act.ACT_DICT_FP32, "bf16": act.ACT_DICT_BF16, "template": act.ACT_DICT_RECOMPUTE}

# family: sample rate, the axes' first and last values (fc in Hz, logDt, c in Hz/s), chirps per signal, noise
FAMILIES = {
    "check": dict(fs=128.0, fc=(1.0, 31.0), logdt=(-3.0, -1.5), c=(-8.0, 6.0), bursts=(3, 3), snr_db=16.0, pink=False),
    "eeg": dict(fs=256.0, fc=(0.5, 32.0), logdt=(-3.0, -0.5), c=(-20.0, 20.0), bursts=(5, 5), snr_db=10.0, pink=True),
    "emg": dict(fs=500.0, fc=(20.0, 200.0), logdt=(-4.0, -1.5), c=(-100.0, 100.0), bursts=(8, 15), snr_db=5.0, pink=False),
    "radar": dict(fs=1000.0, fc=(50.0, 400.0), logdt=(-3.0, -0.7), c=(-300.0, 300.0), bursts=(4, 4), snr_db=15.0, pink=False),
    "table2_eeg": dict(fs=256.0, fc=(0.5, 14.5), logdt=(-4.0, 0.5), c=(-10.0, 9.5), bursts=(5, 5), snr_db=10.0, pink=True),
    "table2_emg": dict(fs=2000.0, fc=(20.0, 440.0), logdt=(-4.0, -0.1), c=(-10.0, 9.5), bursts=(8, 15), snr_db=5.0, pink=False),
}


def _case(kind, family, n, counts, tc_step, channels, **more):
    tc, fc, logdt, c = counts
    return dict(kind=kind, family=family, n=n, tc=tc, fc=fc, logdt=logdt, c=c, tc_step=float(tc_step), channels=channels, **more)


EEG, EMG, RADAR = (128, 64, 8, 32), (256, 96, 8, 24), (256, 128, 8, 32)
LENGTHS = (256, 512, 1024, 2048)  # windows of the uneven EMG-like batch


def listed():
    return [
        # one short window in a loop that waits for each answer: 16,384 atoms that stay in the cache
        dict(_case("mp", "check", 256, (32, 16, 4, 8), 8, 1, dict="fp32", orders=5, refine=0, host=False), name="check_fp32_1ch"),
        # the paper's 1-s EEG epoch (Table 2's ranges, 92,800 atoms, order 10) with BFGS, from and to host memory
        dict(_case("mp", "table2_eeg", 256, (8, 29, 10, 40), 32, 1, dict="fp32", orders=10, refine=20, host=True), name="epoch_fp32_bfgs_host"),
        # the paper's EMG window (Table 2: 200 samples, 113,778 atoms), 12 electrodes at once
        dict(_case("mp", "table2_emg", 200, (7, 43, 14, 27), 32, 12, dict="fp32", orders=10, refine=0, host=False), name="emg_fp32_12ch"),
        # a 2-s EEG-like channel over 2,097,152 stored atoms
        dict(_case("mp", "eeg", 512, EEG, 4, 1, dict="fp32", orders=20, refine=0, host=False), name="eeg_fp32_1ch"),
        # the same channel over the template dictionary
        dict(_case("mp", "eeg", 512, EEG, 4, 1, dict="template", orders=20, refine=0, host=False), name="eeg_template_1ch"),
        # a 64-electrode recording over the template dictionary
        dict(_case("mp", "eeg", 512, EEG, 4, 64, dict="template", orders=20, refine=0, host=False), name="eeg_template_64ch"),
        # the same recording over stored BF16 atoms
        dict(_case("mp", "eeg", 512, EEG, 4, 64, dict="bf16", orders=20, refine=0, host=False), name="eeg_bf16_64ch"),
        # 32 radar-like windows over 8.4 M template atoms, every order refined off the grid
        dict(_case("mp", "radar", 1024, RADAR, 4, 32, dict="template", orders=10, refine=20, host=False), name="radar_template_32ch_bfgs"),
        # an archive of 256 EMG-like signals of uneven length in one plan
        dict(_case("ragged", "emg", 2048, EMG, 1, 256, orders=30), name="emg_ragged_256ch"),
        # the 64-electrode recording with no dictionary in memory: hierarchical search and BFGS
        dict(_case("hier", "eeg", 512, EEG, 4, 64, orders=20, refine=20), name="eeg_hier_64ch_bfgs"),
        # all scores of four channels, for a program that does its own selection
        dict(_case("project", "eeg", 512, EEG, 4, 4, dict="fp32"), name="eeg_project_4ch"),
        # score and gradients of 64 chirplets: one step of a training loop
        dict(_case("score", "eeg", 512, (1, 1, 1, 1), 1, 64), name="score_grad_64ch"),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["mp_small", "mp_fp32", "mp_template", "mp_template", "mp_bf16", "mp_refined", "ragged", "hier", "project", "score"])
    odd = rng.choice([193, 200, 256, 300, 384, 512, 512])
    if kind == "mp_small":
        n = rng.choice([100, 128, 200, 256, 301])
        tc = rng.randint(7, 40)
        return _case("mp", "check", n, (tc, rng.randint(10, 32), rng.randint(3, 9), rng.randint(5, 30)), max(1, n // tc), rng.choice([1, 1, 2, 3]),
                     dict="fp32", orders=rng.randint(3, 15), refine=0, host=rng.random() < 0.3)
    if kind == "mp_fp32":  # time centres between samples too
        tc = rng.randint(16, 100)
        return _case("mp", rng.choice(["eeg", "table2_emg"]), odd, (tc, rng.randint(20, 64), rng.randint(4, 10), rng.randint(11, 33)),
                     rng.choice([odd / tc, float(max(1, odd // tc))]), log(1, 24), dict="fp32", orders=rng.randint(3, 20), refine=0, host=False)
    if kind == "mp_template":
        family = rng.choice(["eeg", "emg", "radar"])
        n = rng.choice([203, 256, 400, 512, 777, 1024, 1500, 2048])
        tc = rng.randint(48, 256)
        return _case("mp", family, n, (tc, rng.randint(24, 128), rng.randint(5, 9), rng.randint(15, 33)), max(1, n // tc), log(1, 200),
                     dict="template", orders=rng.randint(3, 20), refine=0, host=False)
    if kind == "mp_bf16":
        n = rng.choice([200, 256, 400, 512])
        tc = rng.randint(48, 128)
        return _case("mp", "eeg", n, (tc, rng.randint(24, 64), rng.randint(5, 8), rng.randint(15, 32)), max(1, n // tc), log(4, 160),
                     dict="bf16", orders=rng.randint(3, 20), refine=0, host=False)
    if kind == "mp_refined":
        n = rng.choice([256, 500, 1024])
        tc = rng.randint(32, 128)
        return _case("mp", rng.choice(["eeg", "radar"]), n, (tc, rng.randint(24, 64), rng.randint(5, 8), rng.randint(15, 32)), max(1, n // tc), log(1, 64),
                     dict=rng.choice(["fp32", "template"]) if n <= 512 else "template", orders=rng.randint(2, 10), refine=rng.choice([5, 10, 20]), host=False)
    if kind == "ragged":
        return _case("ragged", "emg", 2048, (256, rng.randint(24, 96), rng.randint(5, 8), rng.randint(11, 24)), 1, log(8, 256), orders=rng.randint(3, 30))
    if kind == "hier":
        return _case("hier", "eeg", odd, (max(2, odd // 4), 64, 8, 32), 4, log(1, 64), orders=rng.randint(2, 20), refine=rng.choice([0, 20]))
    if kind == "project":
        tc = rng.randint(24, 128)
        return _case("project", "eeg", odd, (tc, rng.randint(20, 64), rng.randint(4, 8), rng.randint(11, 32)), max(1, odd // tc), log(1, 12),
                     dict=rng.choice(["fp32", "template"]))
    return _case("score", rng.choice(["eeg", "radar"]), rng.choice([129, 256, 512, 1000, 2048]), (1, 1, 1, 1), 1, log(1, 512))


def _grid(case, n=None):
    f = FAMILIES[case["family"]]
    n = n or case["n"]
    step = float(n // case["tc"]) if case["kind"] == "ragged" else case["tc_step"]
    return synth.Grid(n, f["fs"], synth.Axis(0.0, step, case["tc"]), synth.Axis.linspace(*f["fc"], case["fc"]),
                      synth.Axis.linspace(*f["logdt"], case["logdt"]), synth.Axis.linspace(*f["c"], case["c"]))


def _signal(case, n, rng):
    """One window: chirps off the grid, the recipe's noise, float32."""
    f = FAMILIES[case["family"]]
    count = int(rng.integers(f["bursts"][0], f["bursts"][1] + 1))
    low = max(f["logdt"][0], -4.0)
    tc, fc, w, c = (rng.uniform(a, b, (count, 1)) for a, b in ((0, n), f["fc"], (low, min(f["logdt"][1], -0.5)), f["c"]))
    tau = (np.arange(n) - tc) / f["fs"]
    u = np.exp(-0.5 * (tau / np.exp(w)) ** 2) * np.cos(2 * np.pi * (c * tau * tau + fc * tau))
    norm = np.sqrt((u * u).sum(1, keepdims=True))
    amp = rng.uniform(0.5, 2.0, (count, 1)) * rng.choice([-1.0, 1.0], (count, 1))
    clean = (u / np.where(norm > 1e-12, norm, 1.0) * amp).sum(0)
    noise = rng.standard_normal(n)
    if f["pink"]:
        spec = np.fft.rfft(noise)
        spec[0] = 0.0
        spec[1:] /= np.sqrt(np.arange(1, spec.size))
        noise = np.fft.irfft(spec, n=n)
    noise *= math.sqrt((clean @ clean) / (noise @ noise) / 10.0 ** (f["snr_db"] / 10.0))
    return (clean + noise).astype(np.float32)


def _inputs(case, seed):
    """The signals of a case: a list of float32 windows, and the generator for what else it draws."""
    rng = np.random.default_rng([seed, 20])
    # an archive's lengths are its own: the same for every seed
    lengths = np.random.default_rng([case["channels"], 4]).choice(LENGTHS, case["channels"]) if case["kind"] == "ragged" else [case["n"]] * case["channels"]
    return [_signal(case, int(n), rng) for n in lengths], rng


class _Handles:
    """The grids (and plan) a program keeps; given back with the state."""

    def __init__(self):
        self.grids, self.plan = [], None

    def grid(self, g, mode, refine=0):
        h = act.act_grid_create(g, 0)
        self.grids.append(h)
        if mode is not None:
            act.act_dictionary_build(h, mode)
        if refine:
            act.act_set_refinement(h, refine)
        return h

    def __del__(self):
        act.act_ragged_plan_destroy(self.plan)
        for h in self.grids:
            act.act_destroy(h)


def _score_inputs(case, seed):
    windows, rng = _inputs(case, seed)
    f = FAMILIES[case["family"]]
    B, n = case["channels"], case["n"]
    theta = np.stack([rng.uniform(a, b, B) for a, b in ((0, n), f["fc"], (max(f["logdt"][0], -3.0), f["logdt"][1]), f["c"])], 1)
    return theta, np.stack(windows), rng.standard_normal(B)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "score":
        theta, r, up = _score_inputs(case, seed)
        s["theta"] = torch.tensor(theta, device="cuda", requires_grad=True)
        s["r"] = torch.tensor(r, device="cuda", requires_grad=True)
        s["up"] = torch.tensor(up, device="cuda")
        return s
    windows, _ = _inputs(case, seed)
    h = s["handles"] = _Handles()
    if kind == "ragged":
        lengths = sorted({w.size for w in windows})
        grids = [h.grid(_grid(case, n), act.ACT_DICT_RECOMPUTE) for n in lengths]
        offsets = np.concatenate([[0], np.cumsum([w.size for w in windows])])
        h.plan = act.act_ragged_plan_create(grids, offsets, case["orders"])
        s["signals"] = torch.tensor(np.concatenate(windows), device="cuda")
        return s
    s["grid"] = h.grid(_grid(case), None if kind == "hier" else DICT[case["dict"]], case.get("refine", 0))
    if kind == "hier":
        act.act_set_search(s["grid"], act.ACT_SEARCH_LEM)
    s["signals"] = torch.tensor(np.stack(windows), device="cpu" if case.get("host") else "cuda")
    return s


def _answer(atoms, coeffs, residuals, energy):
    # an act_atom is four doubles (tc, fc, logDt, c) and the int64 flat index
    return {"params": atoms.view(torch.float64)[..., :4], "index": atoms.view(torch.int64)[..., 4], "coeffs": coeffs, "residuals": residuals, "energy": energy}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "score":
        f = FAMILIES[case["family"]]
        score = chirplet_score(state["theta"], state["r"], f["fs"])
        g_theta, g_r = torch.autograd.grad(score, (state["theta"], state["r"]), state["up"])
        return {"score": score, "g_theta": g_theta, "g_r": g_r}
    x = state["signals"]
    if kind == "project":
        scores = torch.empty((case["channels"], case["tc"] * case["fc"] * case["logdt"] * case["c"]), dtype=torch.float32, device=x.device)
        act.act_project(state["grid"], x, case["channels"], scores)
        return scores
    if kind == "ragged":
        C, P = case["channels"], case["orders"]
        atoms = torch.empty((C, P, act.ATOM_BYTES), dtype=torch.uint8, device=x.device)
        coeffs = torch.empty((C, P), dtype=torch.float32, device=x.device)
        residuals = torch.empty_like(x)
        energy = torch.empty((C, P + 1), dtype=torch.float64, device=x.device)
        act.act_ragged_decompose(state["handles"].plan, x, atoms, coeffs, residuals, energy)
        return _answer(atoms, coeffs, residuals, energy)
    return _answer(*act.decompose(state["grid"], x, case["orders"]))


def _samples(case):
    """Samples of all channels together (a ragged batch: the mean of its lengths)."""
    return case["channels"] * (sum(LENGTHS) / len(LENGTHS) if case["kind"] == "ragged" else case["n"])


def work(case):
    atoms = case["tc"] * case["fc"] * case["logdt"] * case["c"]
    n, B, kind = case["n"], case["channels"], case["kind"]
    if kind == "score":  # reads r, writes the atom and g_r = upstream x atom; about 30 operations a sample
        return {"bytes": 4 * B * n * 3 + B * 9 * 8, "flops": 30 * B * n}
    if kind == "project":
        rows = atoms * n * 4 if case["dict"] == "fp32" else (atoms // case["tc"]) * (n + case["tc"] * case["tc_step"]) * 4
        return {"bytes": rows + 4 * B * (atoms + n), "flops": 2 * atoms * n * B}
    P = case["orders"]
    out = 8 * _samples(case) + B * P * 52
    refine = 40 * case.get("refine", 0) * _samples(case) * P  # one evaluation of the objective an iteration
    if kind == "hier":  # 2,048 coarse candidates and two pools of 4 x 375, each generated and scored: about 12 operations a sample
        return {"bytes": out, "flops": 12 * (2048 + 2 * 1500) * n * B * P + refine}
    flops = 2 * atoms * _samples(case) * P + refine
    if kind == "ragged":  # BF16 templates over the lags of each window
        return {"bytes": out + sum((atoms // case["tc"]) * 2 * m * 2 for m in LENGTHS), "flops": flops}
    if case["dict"] == "template":
        return {"bytes": out + (atoms // case["tc"]) * (n + case["tc"] * case["tc_step"]) * 2, "flops": flops}
    return {"bytes": out + atoms * n * (2 if case["dict"] == "bf16" else 4), "flops": flops}


# ---- in 64 bits, with plain torch ---------------------------------------------------------------------------------


def _atoms64(g, dev):
    """Every unit-norm atom of the grid, [K][n] float64, in flat-index order."""
    tc, fc, ld, c = (torch.tensor(a.values(), device=dev) for a in (g.tc, g.fc, g.logdt, g.c))
    per = fc.numel() * ld.numel() * c.numel()
    D = torch.empty((tc.numel() * per, g.n_samples), dtype=torch.float64, device=dev)
    t = torch.arange(g.n_samples, dtype=torch.float64, device=dev)
    for i in range(tc.numel()):
        tau = (t - tc[i]) / g.fs
        env = torch.exp(-0.5 * (tau / torch.exp(ld)[:, None]) ** 2)
        phase = fc[:, None, None] * tau + c[None, :, None] * (tau * tau)
        phase = torch.cos(2 * math.pi * (phase - torch.round(phase)))
        u = (phase[:, None] * env[None, :, None]).reshape(per, -1)
        norm = u.square().sum(1, keepdim=True).sqrt()
        D[i * per:(i + 1) * per] = torch.where(norm > 1e-150, u / norm, torch.zeros_like(u))
    return D


def _mp64(g, x, P):
    """Residual-projection matching pursuit of x [B][n] float64: what `run` returns."""
    D = _atoms64(g, x.device)
    r, coeffs, energy, index = x.clone(), [], [x.square().sum(1)], []
    for _ in range(P):
        best, at = torch.full((x.shape[0],), -1.0, dtype=torch.float64, device=x.device), torch.zeros(x.shape[0], dtype=torch.int64, device=x.device)
        for k in range(0, D.shape[0], 1 << 19):
            v, i = (r @ D[k:k + (1 << 19)].T).abs().max(1)
            at, best = torch.where(v > best, i + k, at), torch.maximum(best, v)
        d = D[at]
        a = (d * r).sum(1)
        r = r - a[:, None] * d
        index.append(at)
        coeffs.append(a)
        energy.append(r.square().sum(1))
    index = torch.stack(index, 1)
    axes, params, rest = (g.tc, g.fc, g.logdt, g.c), [], index
    for a in reversed(axes):
        params.append(torch.tensor(a.values(), device=x.device)[rest % a.count])
        rest = rest // a.count
    return {"params": torch.stack(params[::-1], -1), "index": None, "coeffs": torch.stack(coeffs, 1), "residuals": r, "energy": torch.stack(energy, 1)}


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "score":
        theta, r, up = _score_inputs(case, seed)
        theta = torch.tensor(theta, device=dev, requires_grad=True)
        r = torch.tensor(r.astype(np.float64), device=dev, requires_grad=True)
        tau = (torch.arange(case["n"], dtype=torch.float64, device=dev) - theta[:, :1]) / FAMILIES[case["family"]]["fs"]
        u = torch.exp(-0.5 * (tau / torch.exp(theta[:, 2:3])) ** 2) * torch.cos(2 * math.pi * (theta[:, 1:2] * tau + theta[:, 3:] * tau * tau))
        score = (r * u).sum(1) / u.square().sum(1).sqrt()
        g_theta, g_r = torch.autograd.grad(score, (theta, r), torch.tensor(up, device=dev))
        return {"score": score.detach(), "g_theta": g_theta, "g_r": g_r}
    if kind == "hier" or case.get("refine"):  # the trajectories of a random search and of a line search: no value to hold them to
        return None
    windows, _ = _inputs(case, seed)
    atoms = case["tc"] * case["fc"] * case["logdt"] * case["c"]
    lengths = sorted({w.size for w in windows})
    if max(lengths) * atoms * 8 > 40e9 or atoms * (4e-10 * sum(lengths) + 3e-12 * case.get("orders", 1) * sum(w.size for w in windows)) > 15:
        return None
    if kind == "project":
        x = torch.tensor(np.stack(windows), dtype=torch.float64, device=dev)
        return x @ _atoms64(_grid(case), dev).T
    if kind == "mp":
        return _mp64(_grid(case), torch.tensor(np.stack(windows), dtype=torch.float64, device=dev), case["orders"])
    parts = {}
    for n in lengths:
        of = [i for i, w in enumerate(windows) if w.size == n]
        got = _mp64(_grid(case, n), torch.tensor(np.stack([windows[i] for i in of]), dtype=torch.float64, device=dev), case["orders"])
        parts.update({i: (got, j) for j, i in enumerate(of)})
    pick = lambda key: [parts[i][0][key][parts[i][1]] for i in range(len(windows))]  # noqa: E731
    return {"params": torch.stack(pick("params")), "index": None, "coeffs": torch.stack(pick("coeffs")), "residuals": torch.cat(pick("residuals")),
            "energy": torch.stack(pick("energy"))}
