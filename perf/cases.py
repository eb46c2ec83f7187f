"""Performance cases: the work a user of the library has it do, through its
public entry points.

Every case is one call sequence of a user's program: single chambers stepped
or run to completion, many chambers in one batch, and the surrogate network.
`listed()` holds the named cases, `draw(rng)` one more from the same ranges,
`prepare(case, seed)` what the program has in hand before the call, `run` the
call, `work` the bytes and operations it cannot do without and `exact` the
result in 64 bits by plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import surrogate, synth

MU, DIFF, ALPHA, W_EV = (1.73, 1.87), (0.037, 0.037), 1.6e-6, 34.0
Q_OVER_EPS0 = 1.602176634e-19 / 8.8541878128e-14     # V cm
LR = 1e-3


def _grid(name, nx, ny, nz, dx_um, volts, **kw):
    """A single chamber.  steps = 0: run to completion (tol 1e-6, checked
    every 64 steps); let = 0: log-uniform 1-1000 keV/um per track; theta < 0:
    tracks parallel to the field; rate > 0: a continuous beam (Poisson
    arrivals per cm^2 and s) instead of one pulse; tune: the launch-shape
    autotuner is run once before the call, as a long run does."""
    c = {"name": name, "kind": "grid", "nx": nx, "ny": ny, "nz": nz, "dx_um": dx_um, "volts": volts, "fp64": False,
         "absorbing": False, "upwind": False, "space_charge": False, "ladder": False, "kappa": 0.5, "tracks": 1,
         "let": 0.0, "b_um": 10.0, "theta": -1.0, "rate": 0.0, "steps": 0, "tune": False}
    c.update(kw)
    return c


def listed():
    return [
        # a service that must not allocate takes single steps on its own buffers: one small chamber, one step
        {"name": "noalloc_step_64x32x40", "kind": "noalloc", "nx": 64, "ny": 32, "nz": 40, "dx_um": 5.0,
         "volts": 200.0, "absorbing": False, "tracks": 40},
        # the paper's main experiment: one ion track in double precision until its charge has left the gap
        _grid("track_fp64_48x48x100", 48, 48, 100, 2.0, 200.0, fp64=True, absorbing=True, let=100.0),
        # one iron track at an angle on the paper's resolution rule (dx = b/20, a box of 10 b, 2 mm gap)
        _grid("track_angled_200x200x800", 200, 200, 800, 2.5, 200.0, absorbing=True, let=1.02, b_um=50.0, theta=0.4,
              steps=64),
        # a pulsed beam on the benchmark's chamber: one pulse of 2000 tracks, 200 steps of the paper's scheme
        _grid("pulse_256x256x400", 256, 256, 400, 5.0, 200.0, tracks=2000, steps=200, tune=True),
        # the collection efficiency of a mid-sized chamber: run to completion with the time-step ladder
        _grid("completion_128x128x200", 128, 128, 200, 5.0, 200.0, tracks=500, absorbing=True, upwind=True,
              ladder=True, kappa=0.0625),
        # a continuous beam on a wide section: scheduled Poisson arrivals between the steps
        _grid("continuous_512x512x256", 512, 512, 256, 8.0, 300.0, upwind=True, let=-1.0, rate=1e7, steps=128,
              tune=True),
        # a section whose sides are whatever the chamber's are: odd sizes on every axis
        _grid("ragged_301x173x97", 301, 173, 97, 5.0, 200.0, absorbing=True, tracks=300, steps=64),
        # a wide section that is no multiple of 256 cells, with the space-charge term, no autotuner
        _grid("space_charge_384x320x128", 384, 320, 128, 5.0, 300.0, upwind=True, space_charge=True, tracks=600,
              steps=64),
        # a parameter study: 256 uneven chambers to completion in one batch, as the benchmark runs it
        {"name": "batch_256_ladder", "kind": "batch", "sims": 256, "tune": True},
        # training data for the surrogate: many small single-pulse chambers to completion
        {"name": "solves_256_single_pulse", "kind": "solves", "configs": 256},
        # training the surrogate's ensemble of networks: two epochs of Adam in mini-batches
        {"name": "train_5x4096", "kind": "train", "members": 5, "samples": 4096, "batch": 256, "epochs": 2},
        # answers from the trained ensemble for a set of configurations
        {"name": "predict_5x2000", "kind": "predict", "members": 5, "samples": 2000, "max_batch": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "track", "angled", "pulse", "pulse", "completion", "continuous", "space_charge",
                       "batch", "solves", "train", "predict"])
    absorbing = rng.random() < 0.5
    if kind == "noalloc":
        return {"kind": "noalloc", "nx": _log(rng, 16, 160), "ny": _log(rng, 16, 160), "nz": _log(rng, 16, 160),
                "dx_um": rng.uniform(2.0, 8.0), "volts": rng.uniform(50.0, 400.0), "absorbing": absorbing,
                "tracks": _log(rng, 1, 100)}
    volts, dx = rng.uniform(100.0, 400.0), rng.uniform(2.0, 8.0)
    c = None
    if kind == "track":
        n = rng.randint(32, 72)
        c = _grid("", n, n, rng.randint(60, 150), 2.0, rng.uniform(100.0, 300.0), fp64=True, absorbing=True,
                  let=rng.uniform(20.0, 200.0))
    elif kind == "angled":
        n = rng.randint(100, 200)
        c = _grid("", n, n, rng.randint(200, 800), 2.5, volts, absorbing=absorbing, let=1.02, b_um=n / 4.0,
                  theta=rng.uniform(0.0, 1.2), steps=rng.randint(16, 64))
    elif kind == "pulse":
        # any sides: a third of them multiples of 4, the rest as they come
        step = 4 if rng.random() < 0.34 else 1
        nx, ny = step * (_log(rng, 48, 400) // step), _log(rng, 32, 300)
        c = _grid("", nx, ny, _log(rng, 24, 300), dx, volts, absorbing=absorbing, tracks=1 + nx * ny // 64,
                  upwind=rng.random() < 0.5, steps=rng.randint(32, 100), tune=rng.random() < 0.3)
    elif kind == "completion":
        c = _grid("", 4 * rng.randint(12, 40), rng.randint(32, 160), rng.randint(40, 200), 5.0, volts,
                  absorbing=absorbing, tracks=rng.randint(20, 500), upwind=True, ladder=True, kappa=0.0625)
    elif kind == "continuous":
        c = _grid("", 64 * rng.randint(2, 8), 8 * rng.randint(12, 64), rng.randint(64, 256), 8.0, volts, upwind=True,
                  let=-1.0, rate=1e7, steps=rng.randint(64, 128), tune=rng.random() < 0.5)
    elif kind == "space_charge":
        c = _grid("", 4 * rng.randint(16, 96), rng.randint(40, 320), rng.randint(32, 128), 5.0, volts, upwind=True,
                  absorbing=absorbing, space_charge=True, tracks=rng.randint(20, 600), steps=rng.randint(32, 64))
    if c is not None:
        c.pop("name")
        return c
    if kind == "batch":
        return {"kind": "batch", "sims": _log(rng, 8, 200), "tune": rng.random() < 0.5}
    if kind == "solves":
        return {"kind": "solves", "configs": _log(rng, 16, 240)}
    if kind == "train":
        return {"kind": "train", "members": rng.randint(1, 5), "samples": _log(rng, 512, 4096),
                "batch": rng.choice([64, 100, 128, 256, 384]), "epochs": rng.randint(1, 2)}
    return {"kind": "predict", "members": rng.randint(1, 5), "samples": _log(rng, 1, 20000),
            "max_batch": rng.choice([256, 1024, 4096])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _pulse(c, seed):
    """Tracks of one pulse: uniform positions over the section; a single
    track stands near the centre."""
    Lx, Ly = c["nx"] * c["dx_um"] * 1e-4, c["ny"] * c["dx_um"] * 1e-4
    let = c.get("let", 0.0)
    tr = synth.uniform_tracks(seed, c["tracks"], Lx, Ly, c.get("b_um", 10.0) * 1e-4, let=let if let > 0 else "loguniform")
    if c["tracks"] == 1:
        tr.x_cm[:] = 0.5 * Lx + 0.05 * (tr.x_cm - 0.5 * Lx)
        tr.y_cm[:] = 0.5 * Ly + 0.05 * (tr.y_cm - 0.5 * Ly)
    return tr


def _dt_bound(c):
    """The largest stable step of the scheme (either species, field along z)."""
    dx = c["dx_um"] * 1e-4
    E, best = c["volts"] / (c["nz"] * dx), math.inf
    for mu, D in zip(MU, DIFF):
        q, v = 6.0 * D / dx ** 2, mu * E / dx
        best = min(best, 1.0 / (q + v) if c.get("upwind") else (-q + math.sqrt(q * q + 4 * v * v)) / (2 * v * v))
    return best


def _params(c, n_peak):
    return B.it_params_default(
        gap_cm=c["nz"] * (c["dx_um"] * 1e-4), voltage_V=c["volts"], n_peak_cm3=n_peak,
        precision=B.IT_FP64 if c.get("fp64") else B.IT_FP32,
        lateral_bc=B.IT_ABSORBING if c["absorbing"] else B.IT_PERIODIC,
        scheme=B.IT_UPWIND if c.get("upwind") else B.IT_LAX_WENDROFF, react_kappa=c.get("kappa", 0.5),
        space_charge=int(c.get("space_charge", False)), dt_ladder=int(c.get("ladder", False)))


def _chamber_tracks(c, seed):
    """(tracks, peak density, time step) of a single-chamber case."""
    if c["rate"] > 0:
        npk = B.it_peak_density([200.0], [c["b_um"] * 1e-4])
        dt = B.it_auto_dt(_params(c, npk), c["dx_um"] * 1e-4)
        tr = synth.poisson_tracks(seed, c["rate"], c["nx"] * c["dx_um"] * 1e-4, c["ny"] * c["dx_um"] * 1e-4, dt,
                                  c["steps"], c["b_um"] * 1e-4, synth.CONTINUOUS_LET)
        if len(tr) == 0:       # a weak beam on a small section: one arrival at the start
            tr = synth.uniform_tracks(seed, 1, c["nx"] * c["dx_um"] * 1e-4, c["ny"] * c["dx_um"] * 1e-4,
                                      c["b_um"] * 1e-4, let=200.0)
        return tr, npk, dt
    tr = _pulse(c, seed)
    npk = B.it_peak_density(tr.let_keV_um, tr.b_cm)
    return tr, npk, B.it_auto_dt(_params(c, npk), c["dx_um"] * 1e-4)


def _study(c, seed):
    """The simulations of a batch and their tracks (the batched workload's
    generator, another seed)."""
    descs = synth.batch_descriptors(1000 + seed, c["sims"])
    tracks = [synth.batch_tracks(d) for d in descs]
    sims = [dict(nx=d["nx"], ny=d["ny"], nz=d["nz"], dx_cm=d["dx_cm"], voltage_V=d["voltage_V"],
                 n_peak_cm3=B.it_peak_density(t.let_keV_um, t.b_cm)) for d, t in zip(descs, tracks)]
    return sims, tracks


def _single_pulses(c, seed):
    cfgs = [x for x in synth.surrogate_configs(2000 + seed, 4 * c["configs"] + 64) if x["pulses"] == 1]
    return cfgs[:c["configs"]]


def _samples(n, seed):
    """Network inputs of n surrogate configurations and smooth targets in (0, 1)."""
    cfgs = synth.surrogate_configs(3000 + seed, n)
    X = np.stack([synth.surrogate_features(x, x["period_s"]) for x in cfgs])
    w = np.array([-0.9, 0.8, -0.6, 0.5, -0.7, 0.1])
    y = 1.0 / (1.0 + np.exp(-(X - X.mean(0) if n > 1 else X) @ w))
    return X, y


def prepare(case, seed):
    c = case
    if c["kind"] == "grid":
        tr, npk, dt = _chamber_tracks(c, seed)
        prec = B.IT_FP64 if c["fp64"] else B.IT_FP32
        nbytes = B.it_state_bytes(c["nx"], c["ny"], c["nz"], prec)
        buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        stream = torch.cuda.Stream()
        h = B.it_create_ex(c["nx"], c["ny"], c["nz"], c["dx_um"] * 1e-4, 0.0, _params(c, npk), buf.data_ptr(), nbytes,
                           stream.cuda_stream)
        s = {"case": c, "h": h, "buf": buf, "stream": stream, "tr": tr, "xy": np.stack([tr.x_cm, tr.y_cm], axis=1)}
        if c["tune"]:
            B.it_autotune(h)
        return _Owner(s, B.it_destroy)
    if c["kind"] == "noalloc":
        tr = _pulse(c, seed)
        npk = B.it_peak_density(tr.let_keV_um, tr.b_cm)
        p = _params(c, npk)
        dt = B.it_auto_dt(p, c["dx_um"] * 1e-4)
        n = _deposit64(c, tr).float().expand(c["nz"], -1, -1).contiguous()
        return _Owner({"case": c, "p": p, "dt": dt, "plus": n, "minus": n.clone(), "op": torch.zeros_like(n),
                       "om": torch.zeros_like(n), "tal": torch.zeros(7, dtype=torch.float64, device="cuda")})
    if c["kind"] == "batch":
        sims, tracks = _study(c, seed)
        return _Owner({"case": c, "sims": sims, "tracks": tracks})
    if c["kind"] == "solves":
        return _Owner({"case": c, "cfgs": _single_pulses(c, seed)})
    X, y = _samples(c["samples"], seed)
    theta = synth.mlp_init(4000 + seed, c["members"]).astype(np.float32)
    h = B.it_mlp_create(c["members"], c["batch"] if c["kind"] == "train" else c["max_batch"])
    if c["kind"] == "predict":
        for m in range(c["members"]):
            B.it_mlp_set_params(h, m, theta[m])
        mean, std = _norm(c, X)
        B.it_mlp_set_normalization(h, mean, std)
    return _Owner({"case": c, "h": h, "theta": theta, "X": X, "y": y}, B.it_mlp_destroy)


def _norm(c, X):
    """The normalisation a trained ensemble carries (its training set's)."""
    T, _ = _samples(256, 5)
    return T.mean(0), T.std(0, ddof=1)


class _Owner(dict):
    """A state that frees its handle when it goes out of use."""

    def __init__(self, d, free=None):
        super().__init__(d)
        self._free = free

    def __del__(self):
        h = self.pop("h", None)
        if self._free is not None and h is not None:
            torch.cuda.synchronize()
            self._free(h)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _numbers(t):
    """The tallies of a simulation, as the library's numbers."""
    return {"steps": int(t.steps), "f": t.f, "recombined": t.recombined, "t_s": t.t_s, "dt_s": t.dt_s,
            "released": [t.released[0], t.released[1]], "in_domain": [t.in_domain[0], t.in_domain[1]],
            "anode": [t.collected_anode[0], t.collected_anode[1]],
            "cathode": [t.collected_cathode[0], t.collected_cathode[1]],
            "lateral": [t.lost_lateral[0], t.lost_lateral[1]],
            "space_charge": [t.space_charge[0], t.space_charge[1]], "n_max": [t.n_max[0], t.n_max[1]]}


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "grid":
        h, tr = s["h"], s["tr"]
        B.it_reset(h)
        if c["rate"] > 0:
            B.it_schedule_tracks(h, s["xy"], tr.let_keV_um, tr.b_cm, tr.step)
        elif c["theta"] >= 0:
            B.it_deposit_tracks_angled(h, s["xy"], tr.let_keV_um, tr.b_cm, np.full(len(tr), c["theta"]))
        else:
            B.it_deposit_tracks(h, s["xy"], tr.let_keV_um, tr.b_cm)
        if c["steps"]:
            B.it_step(h, c["steps"])
        else:
            if c["ladder"]:
                B.it_retime(h)      # from the deposited peak; the last pass left a later rung
            B.it_run_to_completion(h, tol=1e-6, max_steps=200_000, check_every=64)
        t = B.it_tallies(h)
        out = _numbers(t)
        p, m, _ = B.it_device_state(h)
        cells, dt = c["nx"] * c["ny"] * c["nz"], torch.float64 if c["fp64"] else torch.float32
        base, size = s["buf"].data_ptr(), (8 if c["fp64"] else 4) * cells
        out["plus"] = s["buf"][p - base:p - base + size].view(dt)
        out["minus"] = s["buf"][m - base:m - base + size].view(dt)
        return out
    if c["kind"] == "noalloc":
        B.it_step_noalloc(c["nx"], c["ny"], c["nz"], c["dx_um"] * 1e-4, s["dt"], s["p"], s["plus"].data_ptr(),
                          s["minus"].data_ptr(), s["op"].data_ptr(), s["om"].data_ptr(), s["tal"].data_ptr(),
                          torch.cuda.current_stream().cuda_stream)
        return {"plus": s["op"], "minus": s["om"], "tallies": s["tal"]}
    if c["kind"] == "batch":
        with B.Batch(s["sims"], scheme=B.IT_UPWIND, dt_ladder=True, react_kappa=0.0625) as bt:
            for k, tr in enumerate(s["tracks"]):
                bt.deposit(k, tr.x_cm, tr.y_cm, tr.let_keV_um, tr.b_cm)
            bt.retime()
            if c["tune"]:
                bt.autotune(trial_steps=8)
            launches = bt.run(tol=1e-6, check_every=64)
            rows = [B.it_batch_tallies(bt.h, k) for k in range(len(s["sims"]))]
        return {"launches": int(launches), "steps": np.array([t.steps for t in rows]), **_columns(rows)}
    if c["kind"] == "solves":
        f, dt, per = surrogate.solve_batch(s["cfgs"])
        return {"f": f.astype(np.float32), "dt": dt, "period": per}     # f of FP32 simulations
    if c["kind"] == "train":
        h = s["h"]
        for m in range(c["members"]):
            B.it_mlp_set_params(h, m, s["theta"][m])
        B.it_mlp_fit_normalization(h, s["X"])
        B.it_mlp_set_data(h, s["X"], s["y"])
        loss = B.it_mlp_train(h, c["epochs"], c["batch"], LR, 11)
        return {"loss": loss.tolist(), "params": [B.it_mlp_get_params(h, m) for m in range(c["members"])]}
    mean, spread, per = B.it_mlp_predict(s["h"], c["members"], s["X"])
    return {"mean": mean, "spread": spread, "members": per}


def _columns(rows):
    """Per-simulation results of a batch: its densities and the partial sums of
    its tallies are FP32, so are the columns (time steps are FP64)."""
    a = lambda get: np.array([get(t) for t in rows], dtype=np.float32)  # noqa: E731
    return {"f": a(lambda t: t.f), "recombined": a(lambda t: t.recombined),
            "anode": a(lambda t: t.collected_anode[1]), "cathode": a(lambda t: t.collected_cathode[0]),
            "released": a(lambda t: t.released[0]), "in_domain": a(lambda t: t.in_domain[0] + t.in_domain[1]),
            "n_max": a(lambda t: t.n_max[0]), "dt": np.array([t.dt_s for t in rows])}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """A chamber's state is larger than the chip's registers and shared
    memory, so each explicit step reads and writes both species once (16
    bytes per cell in FP32); about 20 operations per cell and species.  A run
    to completion takes at least one transit of the gap at the largest
    stable step."""
    c = case
    if c["kind"] in ("grid", "noalloc"):
        cells, es = c["nx"] * c["ny"] * c["nz"], 8 if c.get("fp64") else 4
        steps = 1 if c["kind"] == "noalloc" else c["steps"] or _transit(c)
        return {"bytes": 4.0 * es * cells * steps, "flops": 40.0 * cells * steps}
    if c["kind"] == "batch":
        # the generator's mean grid (80 x 80 x 132 cells) and transit (~ 300 stable steps)
        return {"bytes": 16.0 * 80 * 80 * 132 * 300 * c["sims"], "flops": 40.0 * 80 * 80 * 132 * 300 * c["sims"]}
    if c["kind"] == "solves":
        return {"bytes": 16.0 * 48 * 48 * 60 * 120 * c["configs"], "flops": 40.0 * 48 * 48 * 60 * 120 * c["configs"]}
    P, n, M = B.IT_MLP_PARAMS, c["samples"], c["members"]
    if c["kind"] == "predict":
        return {"bytes": 56.0 * n + 8.0 * n * (2 + M) + 4.0 * P * M, "flops": 2.0 * P * n * M}
    steps = c["epochs"] * max(1, n // c["batch"])
    # Adam reads the gradient, the weights and two moments and writes three of them, every mini-batch
    return {"bytes": 28.0 * P * M * steps, "flops": 6.0 * P * M * steps * min(n, c["batch"])}


def _transit(c):
    E = c["volts"] / (c["nz"] * c["dx_um"] * 1e-4)
    return max(1.0, c["nz"] * c["dx_um"] * 1e-4 / (min(MU) * E * _dt_bound(c)))


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    c = case
    if c["kind"] == "grid":
        return _exact_grid(c, seed)
    if c["kind"] == "noalloc":
        tr = _pulse(c, seed)
        dt = B.it_auto_dt(_params(c, B.it_peak_density(tr.let_keV_um, tr.b_cm)), c["dx_um"] * 1e-4)
        n = _deposit64(c, tr).float().double().expand(c["nz"], -1, -1).contiguous()
        sim = _Sim64(c, dt)
        sim.n = [n, n.clone()]
        sim.step()
        return {"plus": sim.n[0], "minus": sim.n[1],
                "tallies": torch.stack([sim.rec, *sim.anode, *sim.cathode, *sim.lateral])}
    if c["kind"] in ("batch", "solves"):
        return None             # hundreds of chambers, hundreds of steps each: minutes in plain torch
    X, y = _samples(c["samples"], seed)
    theta = torch.tensor(synth.mlp_init(4000 + seed, c["members"]).astype(np.float32).astype(np.float64), device="cuda")
    if c["kind"] == "predict":
        mean, std = _norm(c, X)
        x = torch.tensor((X - mean) / std, device="cuda").expand(c["members"], -1, -1)
        f = _net64(theta, x)
        return {"mean": f.mean(0), "spread": f.max(0).values - f.min(0).values, "members": f.T}
    return _exact_train(c, X, y, theta)


def _erf_weights(n, dx, ctr, b, periodic):
    """Fraction of each track's 1-D profile in each cell, within 6 b of the
    track's cell; images added when the faces are periodic.  [tracks, n]"""
    w, ic = torch.ceil(6.0 * b / dx), torch.floor(ctr / dx)
    lo, hi = ic - w, ic + w
    out = torch.zeros(ctr.numel(), n, dtype=torch.float64, device=ctr.device)
    i = torch.arange(n, dtype=torch.float64, device=ctr.device)
    reach = int(max(-float(lo.min()), float(hi.max()) - n) // n) + 2 if periodic else 0
    for k in range(-reach, reach + 1):
        q = i + k * n
        v = 0.5 * (torch.erf(((q + 1) * dx - ctr[:, None]) / b[:, None]) - torch.erf((q * dx - ctr[:, None]) / b[:, None]))
        out += torch.where((q >= lo[:, None]) & (q <= hi[:, None]), v, torch.zeros((), dtype=torch.float64, device=ctr.device))
    return out


def _deposit64(c, tr, sel=slice(None)):
    """Density added by tracks parallel to the field, [ny][nx]."""
    dx = c["dx_um"] * 1e-4
    t = lambda a: torch.tensor(np.asarray(a[sel]), dtype=torch.float64, device="cuda")  # noqa: E731
    x, y, let, b = t(tr.x_cm), t(tr.y_cm), t(tr.let_keV_um), t(tr.b_cm)
    wx = _erf_weights(c["nx"], dx, x, b, not c["absorbing"])
    wy = _erf_weights(c["ny"], dx, y, b, not c["absorbing"])
    return (wy * (let * 1e7 / W_EV)[:, None]).T @ wx / dx ** 2


def _deposit_tilted64(c, tr):
    """Density added by one tilted track, [nz][ny][nx]."""
    dx, th = c["dx_um"] * 1e-4, c["theta"]
    per = not c["absorbing"]
    one = lambda v: torch.tensor([float(v)], dtype=torch.float64, device="cuda")  # noqa: E731
    b, N0 = float(tr.b_cm[0]), float(tr.let_keV_um[0]) * 1e7 / W_EV
    wy = _erf_weights(c["ny"], dx, one(tr.y_cm[0]), one(b), per)[0]
    z = (torch.arange(c["nz"], dtype=torch.float64, device="cuda") + 0.5) * dx
    xc = float(tr.x_cm[0]) + (z - 0.5 * c["nz"] * dx) * math.sin(th) / math.cos(th)
    wx = _erf_weights(c["nx"], dx, xc, torch.full_like(xc, b / math.cos(th)), per)
    return (N0 / math.cos(th) / dx ** 2) * wy[None, :, None] * wx[:, None, :]


class _Sim64:
    """The explicit scheme in FP64 on [nz][ny][nx], with its tallies."""

    def __init__(self, c, dt):
        self.c, self.dx = c, c["dx_um"] * 1e-4
        self.vol = self.dx ** 3
        z = torch.zeros((), dtype=torch.float64, device="cuda")
        self.n = [torch.zeros(c["nz"], c["ny"], c["nx"], dtype=torch.float64, device="cuda") for _ in range(2)]
        self.rec, self.t = z.clone(), 0.0
        self.anode, self.cathode, self.lateral, self.sc = ([z.clone(), z.clone()] for _ in range(4))
        self.set_dt(dt)

    def set_dt(self, dt):
        c, self.dt = self.c, dt
        E = c["volts"] / (c["nz"] * self.dx)
        self.w = []
        for s, (mu, D) in enumerate(zip(MU, DIFF)):
            cc, sd, sg = mu * E * dt / self.dx, D * dt / self.dx ** 2, 1.0 if s == 0 else -1.0
            if c.get("upwind"):
                down, up = sd + (cc if sg > 0 else 0.0), sd + (0.0 if sg > 0 else cc)
            else:
                down, up = sd + 0.5 * cc * cc + 0.5 * sg * cc, sd + 0.5 * cc * cc - 0.5 * sg * cc
            self.w.append((sd, down, up))

    def _side(self, n, dim, shift):
        if not self.c["absorbing"]:
            return torch.roll(n, shift, dim)
        out = torch.zeros_like(n)
        k = n.shape[dim]
        out.narrow(dim, 1 if shift > 0 else 0, k - 1).copy_(n.narrow(dim, 0 if shift > 0 else 1, k - 1))
        return out

    def step(self):
        c, dt = self.c, self.dt
        P, M = self.n
        rr = P * M
        new = []
        for s in range(2):
            n, (sd, down, up) = self.n[s], self.w[s]
            v = self._side(n, 2, 1) + self._side(n, 2, -1)
            v += self._side(n, 1, 1)
            v += self._side(n, 1, -1)
            v -= 4.0 * n
            v *= sd
            v[1:] += down * n[:-1]
            v[:-1] += up * n[1:]
            v -= (down + up) * n
            v -= ALPHA * dt * rr
            v += n
            if c.get("space_charge"):
                k = (-1.0 if s == 0 else 1.0) * dt * MU[s] * Q_OVER_EPS0
                d = n * (P - M)
                v += k * d
                self.sc[s] += k * self.vol * d.sum()
            self.anode[s] += up * self.vol * n[0].sum()
            self.cathode[s] += down * self.vol * n[-1].sum()
            if c["absorbing"]:
                self.lateral[s] += sd * self.vol * (n[:, :, 0].sum() + n[:, :, -1].sum() + n[:, 0].sum() + n[:, -1].sum())
            new.append(v)
        self.rec += ALPHA * dt * self.vol * rr.sum()
        self.n = new
        self.t += dt


def _exact_grid(c, seed):
    tr, _, dt = _chamber_tracks(c, seed)
    sim = _Sim64(c, dt)
    rel, steps = 0.0, 0

    def add(d):
        nonlocal rel
        sim.n = [n + d for n in sim.n]
        rel += float(d.sum()) * sim.vol * (1 if d.dim() == 3 else c["nz"])

    if c["rate"] <= 0:
        add(_deposit_tilted64(c, tr) if c["theta"] >= 0 else _deposit64(c, tr))
    if c["steps"]:
        for k in range(c["steps"]):
            if c["rate"] > 0 and (tr.step == k).any():
                add(_deposit64(c, tr, tr.step == k))
            sim.step()
        steps = c["steps"]
    else:
        cap, nmax = _dt_bound(c), max(float(n.max()) for n in sim.n)
        if c["ladder"]:
            sim.set_dt(min(cap, c["kappa"] / (ALPHA * nmax)))
        while float(sim.n[0].sum() + sim.n[1].sum()) * sim.vol >= 1e-6 * 2 * rel and steps < 200_000:
            if c["ladder"]:
                nmax, r = max(float(n.max()) for n in sim.n), sim.dt
                while r < cap and ALPHA * 2.0 * r * nmax <= c["kappa"]:
                    r *= 2.0
                sim.set_dt(max(sim.dt, min(r, cap)))
            for _ in range(64):
                sim.step()
            steps += 64
    two = lambda v: [float(v[0]), float(v[1])]  # noqa: E731
    got = sum(float(x) for x in sim.anode + sim.cathode)
    return {"steps": None, "f": got / (2 * rel), "recombined": float(sim.rec), "t_s": sim.t, "dt_s": sim.dt,
            "released": [rel, rel], "in_domain": [float(n.sum()) * sim.vol for n in sim.n], "anode": two(sim.anode),
            "cathode": two(sim.cathode), "lateral": two(sim.lateral), "space_charge": two(sim.sc),
            "n_max": [float(n.max()) for n in sim.n], "plus": sim.n[0].reshape(-1), "minus": sim.n[1].reshape(-1)}


_SHAPES = [(256, 6), (256,), (256, 256), (256,), (256, 256), (256,), (256, 256), (256,), (1, 256), (1,)]


def _net64(theta, x):
    """The ensemble's outputs, [members][samples]: weights in bf16 as the
    network stores them for its products, everything else in FP64."""
    o, a = 0, x
    for q in range(0, 10, 2):
        sh = _SHAPES[q]
        k = sh[0] * sh[1]
        W = theta[:, o:o + k].reshape(-1, *sh)
        W = W + (W.detach().float().bfloat16().double() - W.detach())
        b = theta[:, o + k:o + k + sh[0]]
        o += k + sh[0]
        a = torch.baddbmm(b[:, None, :], a, W.transpose(1, 2))
        a = torch.nn.functional.silu(a) if q < 8 else torch.sigmoid(a)
    return a[:, :, 0]


def _orders(members, n, seed):
    """SplitMix64 Fisher-Yates order of one epoch for every member (a generator over epochs)."""
    mask = (1 << 64) - 1
    st = [(seed + 0x9E3779B97F4A7C15 * (z + 1)) & mask for z in range(members)]
    while True:
        out = []
        for z in range(members):
            p = list(range(n))
            for i in range(n - 1, 0, -1):
                st[z] = (st[z] + 0x9E3779B97F4A7C15) & mask
                v = st[z]
                v = ((v ^ (v >> 30)) * 0xBF58476D1CE4E5B9) & mask
                v = ((v ^ (v >> 27)) * 0x94D049BB133111EB) & mask
                j = (v ^ (v >> 31)) % (i + 1)
                p[i], p[j] = p[j], p[i]
            out.append(p)
        yield torch.tensor(out, device="cuda")


def _exact_train(c, X, y, theta):
    x = torch.tensor((X - X.mean(0)) / X.std(0, ddof=1), device="cuda")
    t = torch.tensor(y, device="cuda")
    theta = theta.clone().requires_grad_(True)
    opt = torch.optim.Adam([theta], lr=LR)
    orders, losses = _orders(c["members"], c["samples"], 11), []
    for _ in range(c["epochs"]):
        order, batches = next(orders), []
        for b0 in range(0, max(1, c["samples"] - c["batch"] + 1), c["batch"]):
            idx = order[:, b0:b0 + c["batch"]]
            per = ((_net64(theta, x[idx]) - t[idx]) ** 2).mean(1)
            opt.zero_grad()
            per.sum().backward()
            opt.step()
            batches.append(float(per.detach().mean()))
        losses.append(sum(batches) / len(batches))
    return {"loss": losses, "params": list(theta.detach())}
