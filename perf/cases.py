"""The work a user of lbmrare has it do, as cases that can be timed and compared.

Kinds of cases (each goes through the binding's public calls only):

  step      advance an ensemble, read its drag history and its network input:
            direct sampling, the initial ensemble of AMS, the periods of GKTL
  gktl      lbm_gktl_run: periods, weights, resampling, perturbed cloning
  resample  one cloning step of a GKTL loop driven by hand: refill the App. D
            bank, clone, check the conserved moments, read the network input
  ams       one iteration of an AMS loop driven by hand: crossing, bank from a
            checkpoint, branch, re-simulation, scores
  score     the learned score of every trajectory (block means + network)
  train     one training step of the network; gradient and updated parameters
  stats     the direct-sampling statistics of recorded drag series

Sizes are those of bench.py's workloads and of the tests, and generic ones
between them.  No case calls lbm_ensemble_autotune: it picks by timing, so two
runs of one program may group the drag's partial sums differently.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2005_09323_gb300 import lbmrare as L

EPS, N_SNAP = 0.002, 10          # App. D perturbation
RHO_SCALE, U_SCALE = 1000.0, 50.0  # network input scales
OPEN_UC = 0.05
OPEN_TAU = 0.5 + 3.0 * OPEN_UC * 8 / 1200
ITEM = {"fp32": 4, "fp16": 2, "bf16": 2}
DEV = "cuda"


def _periodic(kind, nx, ny, clones, side, storage, collision="bgk", tau=0.505, gx=1e-6, **more):
    return dict(kind=kind, nx=nx, ny=ny, clones=clones, side=side, storage=storage, collision=collision, tau=tau,
                gx=gx, open=False, **more)


def _open(kind, nx, ny, clones, side, storage, tau=OPEN_TAU, **more):
    return dict(kind=kind, nx=nx, ny=ny, clones=clones, side=side, storage=storage, collision="cm", tau=tau,
                gx=0.0, open=True, **more)


def listed():
    return [
        # a single trajectory by the plain method: the smallest calls, one clone that fits on chip
        _periodic("step", 256, 64, 1, 8, "fp32", tau=0.52, steps=200, factor=4, obs=False, name="single-256x64"),
        # the GKTL ensemble between two cloning steps: the main workload
        _periodic("step", 1024, 256, 64, 32, "fp32", steps=100, factor=4, obs=False, name="ensemble-64x1024x256"),
        # the precision sweep's ensemble in shifted FP16
        _periodic("step", 2048, 512, 16, 64, "fp16", steps=100, factor=4, obs=False, name="ensemble-16x2048x512-fp16"),
        # the paper's open channel (odd sizes, grid, sponge, central moments): direct sampling
        _open("step", 513, 129, 64, 16, "fp32", steps=200, factor=2, obs=False, name="open-64x513x129"),
        # the same with 16-bit populations, as the return-time runs use
        _open("step", 513, 129, 64, 16, "fp16", steps=200, factor=2, obs=False, name="open-64x513x129-fp16"),
        # the perturbation check: the square's observables recorded after every step
        _open("step", 513, 129, 64, 16, "fp32", steps=100, factor=2, obs=True, name="open-64x513x129-obs"),
        # a whole GKTL run of two periods, resampling every 500 steps
        _periodic("gktl", 1024, 256, 64, 32, "fp32", period=500, periods=2, name="gktl-run-64x1024x256"),
        # the cloning step alone, with the bank refilled and the moments checked
        _periodic("resample", 1024, 256, 64, 32, "fp32", name="resample-64x1024x256"),
        # one AMS iteration on trajectories of 1000 steps, checkpoints every 250
        _periodic("ams", 512, 128, 32, 16, "fp32", horizon=1000, ckpt=250, window=200, branch_at=390,
                  name="ams-iteration-512x128"),
        # the learned score of the GKTL ensemble at a cloning time
        _periodic("score", 1024, 256, 64, 32, "fp32", factor=4, name="score-64x1024x256"),
        # a training step of the learned score: 256 inputs of 64 x 256
        dict(kind="train", height=64, width=256, batch=256, name="train-256x64x256"),
        # statistics of the open-channel workload's drag: 64 series, steps 500 to 7000
        dict(kind="stats", clones=64, t0=500, t1=7000, lags=2000, levels=3, window=1000, name="statistics-64x6500"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _channel(rng, most_sites):
    """an ensemble of periodic or open channels with at most most_sites nodes"""
    while True:
        is_open = rng.random() < 0.4
        nx = int(_log(rng, 64, 2048))
        ny = max(24, int(nx * rng.choice([0.25, 0.25, 0.25, 0.37, 0.5])) + rng.choice([0, 0, 1, -1]))
        nx = nx + rng.choice([0, 1, 3]) if is_open else (nx + 7) // 8 * 8
        if is_open and nx < 192:
            continue
        clones = max(1, int(_log(rng, 1, 256)))
        if nx * ny * clones <= most_sites:
            side = max(4, ny // 8)
            storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
            return is_open, nx, ny, clones, side, storage


def draw(rng):
    kind = rng.choice(["step"] * 8 + ["gktl", "resample", "ams", "score", "train", "train", "stats", "stats"])
    if kind == "train":
        height, width = rng.choice([(64, 256), (64, 256), (32, 256), (16, 64), (8, 32), (24, 80), (32, 128)])
        return dict(kind=kind, height=height, width=width,
                    batch=int(_log(rng, 2, min(256, 256 * 64 * 256 // (height * width)))))
    if kind == "stats":
        clones, n = int(_log(rng, 8, 128)), int(_log(rng, 1000, 20000))
        t0 = rng.randrange(0, 500)
        return dict(kind=kind, clones=clones, t0=t0, t1=t0 + n, lags=int(_log(rng, 100, min(2000, n // 2))),
                    levels=rng.randrange(1, 9), window=rng.randrange(50, 800))
    is_open, nx, ny, clones, side, storage = _channel(rng, 1 << 24)
    # a force whose terminal velocity stays below 0.08: the flow of a long run stays laminar enough to be finite
    tau = rng.choice([0.505, 0.51, 0.52, 0.55])
    gx = min(1e-6, 0.64 * (tau - 0.5) / 3.0 / ny ** 2)
    coll = rng.choice(["bgk", "bgk", "cm"])
    if kind in ("step", "gktl", "resample"):
        if kind == "step":
            more = dict(steps=int(_log(rng, 4, 150)), factor=rng.choice([1, 2, 4]), obs=rng.random() < 0.2)
        else:
            clones = max(2, clones)
            more = dict(period=int(_log(rng, 20, 250)), periods=rng.randrange(1, 4)) if kind == "gktl" else {}
        if is_open:
            return _open(kind, nx, ny, clones, side, storage, rng.choice([OPEN_TAU, 0.51, 0.53]), **more)
        return _periodic(kind, nx, ny, clones, side, storage, coll, tau, gx, **more)
    if kind == "ams":
        nx, ny = rng.choice([(512, 128), (256, 64), (264, 70), (384, 96)])
        horizon, ckpt = 50 * rng.randrange(6, 21), rng.choice([50, 100, 250])
        return _periodic(kind, nx, ny, rng.randrange(4, 33), ny // 8, storage, coll, tau, gx, horizon=horizon,
                         ckpt=ckpt, window=rng.randrange(1, 200), branch_at=rng.randrange(horizon // 4, horizon // 2))
    # the learned score takes whole blocks of 8 x 16 inputs
    nx, ny, factor = rng.choice([(1024, 256, 4), (512, 128, 2), (256, 64, 4), (256, 64, 2)])
    return _periodic("score", nx, ny, rng.randrange(2, 65), ny // 8, storage, coll, tau, gx, factor=factor)


# ---------------------------------------------------------------- geometry and configuration
def _square(case):
    s = case["side"]
    x0 = case["nx"] // 2 if case["open"] else case["nx"] // 4
    return (x0 - s // 2, case["ny"] // 2 - s // 2, s, s)


def _grid(case):
    """entrance grid of the open channel: x0, width, bar rows, gap rows"""
    s = case["side"]
    return (s, max(1, s // 2), max(1, s // 2), max(1, s // 2))


def _sponge(case):
    return case["nx"] // 4


def _config(case, max_steps, **more):
    kw = dict(obstacle=_square(case), tau=case["tau"], gx=case["gx"], storage=case["storage"], max_steps=max_steps,
              init_amp=0.01, collision=case["collision"], **more)
    if case["open"]:
        kw.update(open_x=1, u_in=OPEN_UC, grid=_grid(case), sponge_len=_sponge(case), sponge_tau=1.0)
    return L.config(case["nx"], case["ny"], **kw)


def _history(case):
    """drag history of an ensemble that is stepped for about three seconds"""
    sites = case["nx"] * case["ny"] * case["clones"]
    return int(3.0 / max(0.5e-6 if sites <= 1 << 18 else 1.5e-6, sites * 9 * ITEM[case["storage"]] / 2 / 7e12)) + 4096


class _Ensemble:
    """an ensemble handle that is destroyed with its last reference"""

    def __init__(self, cfg, n, seed):
        self.h, self.n, self.cfg = None, n, cfg
        self.h = L.lbm_ensemble_create(cfg, n, seed, torch.cuda.current_stream())
        self.t = 0

    def __del__(self):
        if self.h is not None:
            L.lbm_ensemble_destroy(self.h)
            self.h = None


class _Network:
    def __init__(self, height, width, batch, params):
        self.h = None
        self.h = L.cnn_create(height, width, batch, 1)
        L.cnn_set_params(self.h, params)

    def __del__(self):
        if self.h is not None:
            L.cnn_destroy(self.h)
            self.h = None


def _params(seed):
    """network parameters in the documented flat layout: He-uniform taps, small biases, uniform head"""
    g = np.random.default_rng([seed, 77])
    out = []
    for cin, real, pad in ((8, 3, 80), (32, 32, 304), (32, 32, 304), (32, 32, 304)):
        block = np.zeros((32, pad), np.float32)
        a = math.sqrt(6.0 / (9 * real))
        taps = g.uniform(-a, a, (32, 9, cin)).astype(np.float32)
        taps[:, :, real:] = 0
        block[:, :9 * cin] = taps.reshape(32, 9 * cin)
        block[:, 9 * cin] = g.uniform(-0.1, 0.1, 32)
        out.append(block.ravel())
    out.append(np.append(g.uniform(-1, 1, 32) / math.sqrt(32), 0.0).astype(np.float32))
    return np.concatenate(out).astype(np.float32)


def _inputs(case, seed):
    """network inputs: smooth fields of order one with small-scale fluctuations, and labels of unit variance"""
    B, H, W = case["batch"], case["height"], case["width"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    yy = torch.arange(H, device=DEV, dtype=torch.float32).view(1, H, 1, 1) / H
    xx = torch.arange(W, device=DEV, dtype=torch.float32).view(1, 1, W, 1) / W
    ph = torch.rand((B, 1, 1, 3), generator=g, device=DEV) * 2 * math.pi
    x = torch.zeros((B, H, W, 8), device=DEV)
    x[..., :3] = torch.sin(2 * math.pi * (3 * xx + 2 * yy) + ph) + 0.3 * torch.randn((B, H, W, 3), generator=g,
                                                                                      device=DEV)
    y = torch.randn(B, generator=g, device=DEV)
    return x.to(torch.bfloat16).contiguous(), y


def _series(case, seed):
    """drag series of correlated fluctuations around a mean, [clones][t1]"""
    g = torch.Generator(device="cpu").manual_seed(seed)
    n, t = case["clones"], case["t1"]
    a = math.exp(-1.0 / 300.0)
    noise = torch.randn((n, t), generator=g, dtype=torch.float64)
    # AR(1) by blocks: x_t = a x_{t-1} + noise, each block from the state before it
    block = 128
    k = torch.arange(block, dtype=torch.float64)
    lower = torch.tril(a ** (k.view(-1, 1) - k.view(1, -1)).clamp(min=0))
    out = torch.empty_like(noise)
    last = noise[:, 0] / math.sqrt(1 - a * a)
    for s in range(0, t, block):
        m = min(block, t - s)
        out[:, s:s + m] = noise[:, s:s + m] @ lower[:m, :m].T + last.view(-1, 1) * a ** (k[:m] + 1)
        last = out[:, s + m - 1].clone()
    return (0.028 + 0.03 * math.sqrt(1 - a * a) * out).numpy()


def _weights(n, seed):
    s = np.random.default_rng([seed, 5]).normal(0.0, 1.0, n)
    w = np.exp(s - s.max())
    return n * w / w.sum()


def _field_buffer(case, n):
    """the network input of n states (block means over factor x factor nodes)"""
    f = case.get("factor", 4)
    return torch.zeros((n, case["ny"] // f, case["nx"] // f, 8), dtype=torch.bfloat16, device=DEV)


def _read_fields(st, clones):
    case = st["case"]
    L.lbm_ensemble_fields(st["e"].h, clones, case.get("factor", 4), RHO_SCALE, U_SCALE, st["fields"], case["nx"],
                          case["ny"])
    return st["fields"]


def _bank(n):
    k = min(N_SNAP, n)
    return [i * n // k for i in range(k)]


# ---------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind == "train":
        st["net"] = _Network(case["height"], case["width"], case["batch"], _params(seed))
        st["x"], st["y"] = _inputs(case, seed)
        st["loss"] = torch.zeros(1, device=DEV)
        return st
    if kind == "stats":
        # a short channel whose clones have reached t1; the statistics read the recorded series only
        cfg = L.config(64, 16, tau=0.6, max_steps=case["t1"])
        e = st["e"] = _Ensemble(cfg, case["clones"], seed)
        L.lbm_ensemble_step(e.h, case["t1"])
        series = _series(case, seed)
        L.lbm_ensemble_set_drag(e.h, 0, case["t1"], series)
        mu, sd = series.mean(), series.std()
        st["levels"] = torch.tensor([mu + (1 + 0.5 * k) * sd for k in range(case["levels"])], dtype=torch.float64,
                                    device=DEV)
        st["c"] = torch.zeros(case["lags"] + 1, dtype=torch.float64, device=DEV)
        st["maxima"] = torch.zeros(case["clones"], dtype=torch.float64, device=DEV)
        st["sums"] = torch.zeros_like(st["maxima"])
        return st
    n, nx, ny = case["clones"], case["nx"], case["ny"]
    f64 = dict(dtype=torch.float64, device=DEV)
    if kind == "step":
        e = st["e"] = _Ensemble(_config(case, _history(case)), n, seed)
        if case["obs"]:
            L.lbm_ensemble_set_observables(e.h, True)
            st["obs"] = torch.zeros((n, case["steps"], 4), **f64)
        st["drag"] = torch.zeros((n, case["steps"]), **f64)
        st["fields"] = _field_buffer(case, n)
    elif kind == "gktl":
        st["fields"] = _field_buffer(case, n)
        e = st["e"] = _Ensemble(_config(case, _history(case), n_snapshots=N_SNAP), n, seed)
        L.lbm_ensemble_set_snapshots(e.h, _bank(n))
        st["logR"] = torch.zeros(case["periods"], **f64)
        st["parent"] = torch.zeros((case["periods"], n), dtype=torch.int32, device=DEV)
        st["integral"], st["maxima"] = torch.zeros(n, **f64), torch.zeros(n, **f64)
    elif kind == "resample":
        st["fields"] = _field_buffer(case, n)
        e = st["e"] = _Ensemble(_config(case, 64, n_snapshots=N_SNAP), n, seed)
        st["parent"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        L.gktl_select(torch.tensor(_weights(n, seed), device=DEV), seed, 0, st["parent"])
    elif kind == "ams":
        st["fields"] = _field_buffer(case, 1)
        e = st["e"] = _Ensemble(_config(case, case["horizon"], n_snapshots=N_SNAP, ckpt_stride=case["ckpt"]), n, seed)
        L.lbm_ensemble_step(e.h, case["horizon"])
        st["Q"] = torch.zeros(n, **f64)
        st["drag"] = torch.zeros((n, case["horizon"]), **f64)
        L.lbm_ensemble_scores(e.h, case["window"], 0, case["horizon"], st["Q"])
        st["level"] = float(st["Q"].min())
    elif kind == "score":
        f = case["factor"]
        e = st["e"] = _Ensemble(_config(case, 64), n, seed)
        L.lbm_ensemble_step(e.h, 20)
        st["net"] = _Network(ny // f, nx // f, min(n, 64), _params(seed))
        L.lbm_ensemble_attach_score(e.h, st["net"].h, f, RHO_SCALE, U_SCALE)
        st["out"] = torch.zeros(n, **f64)
    else:
        raise ValueError(kind)
    return st


# ---------------------------------------------------------------- run
def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "train":
        m = st["net"].h
        L.cnn_train_step(m, st["x"], st["y"], 1e-4, st["loss"], torch.cuda.current_stream())
        return {"loss": st["loss"], "gradient": L.cnn_get_gradient(m), "params": L.cnn_get_params(m)}
    e = st["e"]
    if kind == "step":
        t0, t1 = e.t, e.t + case["steps"]
        L.lbm_ensemble_step(e.h, case["steps"])
        e.t = t1
        L.lbm_ensemble_drag(e.h, t0, t1, st["drag"])
        out = {"drag": st["drag"]}
        if case["obs"]:
            L.lbm_ensemble_observables(e.h, t0, t1, st["obs"])
            out["obs"] = st["obs"]
        out["fields"] = _read_fields(st, range(e.n))
        return out
    if kind == "gktl":
        steps = case["period"] * case["periods"]
        L.lbm_gktl_run(e.h, case["period"], case["periods"], 1.0 / (1e-3 * case["period"]), EPS, st["seed"],
                       min(steps, case["period"]), st["logR"], st["parent"], st["integral"], st["maxima"],
                       refresh_snapshots=True)
        return {"logR": st["logR"], "parent": st["parent"], "integral": st["integral"], "maxima": st["maxima"],
                "fields": _read_fields(st, range(e.n))}
    if kind == "resample":
        L.lbm_ensemble_set_snapshots(e.h, _bank(e.n))
        L.lbm_ensemble_clone(e.h, st["parent"], EPS, st["seed"], 0)
        mass, px, py = L.lbm_ensemble_moments(e.h, e.n)
        return {"mass": mass, "px": px, "py": py, "fields": _read_fields(st, range(e.n))}
    if kind == "ams":
        T, w = case["horizon"], case["window"]
        dst, src, tb = 0, e.n - 1, case["branch_at"]
        # (the branching time is the case's, so that every pass replays the same length)
        crossing = L.lbm_ensemble_first_crossing(e.h, src, st["level"])
        L.lbm_ensemble_set_snapshots_from_checkpoint(e.h, _bank(e.n), tb // case["ckpt"])
        L.lbm_ensemble_branch(e.h, dst, src, tb, EPS, st["seed"], 1)
        L.lbm_ensemble_step_clones(e.h, T - tb, [dst])
        L.lbm_ensemble_scores(e.h, w, 0, T, st["Q"])
        L.lbm_ensemble_drag(e.h, 0, T, st["drag"])
        return {"crossing": crossing, "Q": st["Q"], "drag": st["drag"], "fields": _read_fields(st, [dst])}
    if kind == "score":
        L.lbm_ensemble_evaluate_score(e.h, st["out"])
        return {"score": st["out"]}
    t0, t1 = case["t0"], case["t1"]
    tau_c = L.lbm_drag_autocorrelation(e.h, t0, t1, case["lags"], st["c"])
    events, r = L.lbm_drag_return_times(e.h, t0, t1, st["levels"], max(tau_c, 1))
    L.lbm_ensemble_scores(e.h, case["window"], t0, t1, st["maxima"])
    L.lbm_ensemble_window_sum(e.h, t0, t1, 1.0, st["sums"])
    return {"c": st["c"], "tau_c": tau_c, "events": events, "r": r, "maxima": st["maxima"], "sums": st["sums"]}


# ---------------------------------------------------------------- work
def _cnn_flops(H, W, backward):
    taps = 2.0 * H * W * 9 * 32
    fwd = taps * (3 + 3 * 32)
    return fwd + (taps * (3 + 3 * 32) + taps * 3 * 32 if backward else 0.0)


def work(case):
    kind = case["kind"]
    if kind == "train":
        px = case["batch"] * case["height"] * case["width"]
        # the input once; each hidden activation and its gradient written once and read once
        return {"bytes": px * 16.0 + 2.0 * (4 + 4) * px * 64.0,
                "flops": case["batch"] * _cnn_flops(case["height"], case["width"], True)}
    if kind == "stats":
        n, t = case["clones"], case["t1"] - case["t0"]
        return {"bytes": 8.0 * n * t, "flops": 2.0 * n * (case["lags"] + 1) * (t - 0.5 * case["lags"])}
    sites = float(case["nx"]) * case["ny"]
    state = 9.0 * ITEM[case["storage"]] * sites  # one trajectory
    per_site = 250.0 if case["collision"] == "cm" else 130.0
    n = case["clones"]
    if kind == "step":
        # the state read once and written once over the whole call, the histories, the network input
        hist = 8.0 * n * case["steps"] * (5 if case["obs"] else 1)
        return {"bytes": 2 * n * state + hist + 16.0 * n * sites / case["factor"] ** 2,
                "flops": per_site * sites * n * case["steps"]}
    if kind == "gktl":
        steps = case["period"] * case["periods"]
        return {"bytes": 2 * n * state * case["periods"] + 8.0 * n * steps + n * sites, "flops": per_site * sites * n * steps}
    if kind == "resample":
        # the bank copied, about 3/8 of the slots replaced, every state read for its moments
        return {"bytes": (2 * min(N_SNAP, n) + 0.75 * n + n) * state + n * sites, "flops": n * sites * (27 + 0.375 * 30 * N_SNAP)}
    if kind == "ams":
        steps = case["horizon"] - case["branch_at"] + case["branch_at"] % case["ckpt"]
        return {"bytes": state * (2 * min(N_SNAP, n) + 2 * (case["branch_at"] // case["ckpt"] + 1) + 4) +
                16.0 * n * case["horizon"], "flops": per_site * sites * steps}
    f = case["factor"]
    return {"bytes": n * (state + 16.0 * sites / f ** 2),
            "flops": n * (30 * sites + _cnn_flops(case["ny"] // f, case["nx"] // f, False))}


# ---------------------------------------------------------------- 64-bit reference
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WQ = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
M64 = (1 << 64) - 1
M32 = 0xFFFFFFFF


def _signed(v):
    v &= M64
    return v - (1 << 64) if v >> 63 else v


def _mulhi(a, b):
    """high word of the unsigned 64 x 64 product; a an int64 tensor of bits, b a number"""
    al, ah, bl, bh = a & M32, (a >> 32) & M32, b & M32, b >> 32
    p0, p1, p2, p3 = al * bl, ah * bl, al * bh, ah * bh
    mid = ((p0 >> 32) & M32) + (p1 & M32) + (p2 & M32)
    return p3 + ((p1 >> 32) & M32) + ((p2 >> 32) & M32) + ((mid >> 32) & M32)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x64-10, key (seed, 0): the first two output words, for int64 tensors of counter bits"""
    k0, k1 = seed & M64, 0
    for _ in range(10):
        h0, l0 = _mulhi(c0, 0xD2E7470EE14C6C93), c0 * _signed(0xD2E7470EE14C6C93)
        h1, l1 = _mulhi(c2, 0xCA5A826395121157), c2 * _signed(0xCA5A826395121157)
        c0, c1, c2, c3 = h1 ^ c1 ^ _signed(k0), l1, h0 ^ c3 ^ _signed(k1), l0
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & M64, (k1 + 0xBB67AE8584CAA73B) & M64
    return c0, c1


def _unit(x):
    return ((x >> 11) & ((1 << 53) - 1)).double() * 2.0 ** -53


def _feq(rho, ux, uy):
    usq = ux * ux + uy * uy
    return [WQ[q] * rho * (1 + 3 * (CX[q] * ux + CY[q] * uy) + 4.5 * (CX[q] * ux + CY[q] * uy) ** 2 - 1.5 * usq)
            for q in range(9)]


class _Flow:
    """plain FP64 simulation of every trajectory of a case, f [9][n][ny][nx]"""

    def __init__(self, case, seed):
        self.case, self.n = case, case["clones"]
        nx, ny = self.nx, self.ny = case["nx"], case["ny"]
        y = torch.arange(ny, device=DEV).view(ny, 1)
        x = torch.arange(nx, device=DEV).view(1, nx)
        x0, y0, w, h = self.square = _square(case)
        sq = (x >= x0) & (x < x0 + w) & (y >= y0) & (y < y0 + h)
        solid = sq.clone()
        self.om = torch.full((1, nx), 1.0 / case["tau"], dtype=torch.float64, device=DEV)
        if case["open"]:
            gx0, gw, bar, gap = _grid(case)
            solid |= (x >= gx0) & (x < gx0 + gw) & (y % (bar + gap) >= gap)
            ln = _sponge(case)
            s = (x - (nx - ln) + 1).double() / ln
            tau = torch.where(x >= nx - ln, case["tau"] + (1.0 - case["tau"]) * s * s, torch.full_like(s, case["tau"]))
            self.om = 1.0 / tau
            self.tau_out = float(tau[0, -1])
            yy = y.double() + 0.5
            self.u_in = OPEN_UC * 4 * yy * (ny - yy) / (ny * ny)
        self.sq, self.solid = sq, solid
        pad = torch.zeros((ny + 2, nx), dtype=torch.bool, device=DEV)
        pad[1:-1] = solid
        self.back = [torch.roll(pad, CX[q], 1)[1 - CY[q]:ny + 1 - CY[q]] for q in range(9)]  # upstream node solid
        psq = torch.zeros_like(pad)
        psq[1:-1] = sq
        self.link = [~sq & torch.roll(psq, -CX[q], 1)[1 + CY[q]:ny + 1 + CY[q]] for q in range(9)]  # into the square
        clone = torch.arange(self.n, device=DEV).view(-1, 1, 1).expand(self.n, ny, nx)
        site = (y * nx + x).expand(self.n, ny, nx)
        r0, r1 = _philox(torch.full_like(site, 5), clone.contiguous(), site.contiguous(), torch.zeros_like(site), seed)
        ux, uy = 0.01 * (2 * _unit(r0) - 1), 0.01 * (2 * _unit(r1) - 1)
        if case["open"]:
            ux = ux + self.u_in
        ux, uy = ux * ~solid, uy * ~solid
        self.f = torch.stack(_feq(torch.ones_like(ux), ux, uy))

    def step(self):
        f, ny, case = self.f, self.ny, self.case
        g = torch.empty_like(f)
        for q in range(9):
            s = torch.roll(f[q], CX[q], 2) if CX[q] else f[q]
            if CY[q] == 1:
                g[q, :, 1:], g[q, :, 0] = s[:, :-1], f[OPP[q], :, 0]
            elif CY[q] == -1:
                g[q, :, :-1], g[q, :, -1] = s[:, 1:], f[OPP[q], :, -1]
            else:
                g[q] = s
            if q:
                g[q] = torch.where(self.back[q], f[OPP[q]], g[q])
        fx = case["gx"]
        rho = g.sum(0)
        ux = (g[1] - g[3] + g[5] - g[6] - g[7] + g[8] + 0.5 * fx) / rho
        uy = (g[2] - g[4] + g[5] + g[6] - g[7] - g[8]) / rho
        eq = _feq(rho, ux, uy)
        src = [WQ[q] * (3 * (CX[q] - ux) + 9 * (CX[q] * ux + CY[q] * uy) * CX[q]) * fx for q in range(9)]
        if case["collision"] == "bgk":
            for q in range(9):
                g[q] += self.om * (eq[q] - g[q]) + (1 - 0.5 * self.om) * src[q]
        else:
            h = [g[q] - eq[q] + 0.5 * src[q] for q in range(9)]
            for q, d in enumerate(self._relaxed(h, ux, uy)):
                g[q] += src[q] - d
        for q in range(9):
            g[q] = torch.where(self.solid, torch.full_like(rho, WQ[q]), g[q])
        if case["open"]:
            self._boundaries(g)
        self.f = g
        return sum(2 * CX[q] * (g[q] * self.link[q]).sum((1, 2)) for q in range(1, 9) if CX[q])

    def _relaxed(self, h, u, v):
        """T^-1 Omega T h: central moments at rates 1 (bulk, third, fourth order) and omega (shear)"""
        raw = [[sum(float(CX[q] ** a * CY[q] ** b) * h[q] for q in range(9) if CX[q] ** a * CY[q] ** b)
                for b in range(3)] for a in range(3)]

        def shift(m, du, dv):
            rows = [[m[0][b], m[1][b] + du * m[0][b], m[2][b] + 2 * du * m[1][b] + du * du * m[0][b]]
                    for b in range(3)]
            m = [[rows[b][a] for b in range(3)] for a in range(3)]
            return [[m[a][0], m[a][1] + dv * m[a][0], m[a][2] + 2 * dv * m[a][1] + dv * dv * m[a][0]]
                    for a in range(3)]

        k = shift(raw, -u, -v)
        zero = torch.zeros_like(u)
        s, d = k[2][0] + k[0][2], self.om * (k[2][0] - k[0][2])
        k = [[zero, zero, 0.5 * (s - d)], [zero, self.om * k[1][1], k[1][2]], [0.5 * (s + d), k[2][1], k[2][2]]]
        m = shift(k, u, v)
        by_x = {0: [m[0][b] - m[2][b] for b in range(3)], 1: [0.5 * (m[2][b] + m[1][b]) for b in range(3)],
                -1: [0.5 * (m[2][b] - m[1][b]) for b in range(3)]}
        out = []
        for q in range(9):
            p = by_x[CX[q]]
            out.append(p[0] - p[2] if CY[q] == 0 else 0.5 * (p[2] + CY[q] * p[1]))
        return out

    def _boundaries(self, g):
        one = torch.ones((self.n, self.ny), dtype=torch.float64, device=DEV)
        for q, e in enumerate(_feq(one, self.u_in.view(1, -1) * one, 0 * one)):
            g[q, :, :, 0] = e
        c = g[:, :, :, -3:-1]
        rho = c.sum(0)
        ux = (c[1] - c[3] + c[5] - c[6] - c[7] + c[8]) / rho
        uy = (c[2] - c[4] + c[5] + c[6] - c[7] - c[8]) / rho
        u, v = 2 * ux[..., 1] - ux[..., 0], 2 * uy[..., 1] - uy[..., 0]

        def dy(a):
            d = torch.empty_like(a)
            d[:, 1:-1] = 0.5 * (a[:, 2:] - a[:, :-2])
            d[:, 0], d[:, -1] = a[:, 1] - a[:, 0], a[:, -1] - a[:, -2]
            return d

        pre = -2.0 / 3.0 * (self.tau_out - 1.0)
        pxx, pyy = pre * (ux[..., 1] - ux[..., 0]), pre * dy(v)
        pxy = 0.5 * pre * (dy(u) + uy[..., 1] - uy[..., 0])
        for q, e in enumerate(_feq(one, u, v)):
            qp = (CX[q] ** 2 - 1 / 3) * pxx + 2 * CX[q] * CY[q] * pxy + (CY[q] ** 2 - 1 / 3) * pyy
            g[q, :, :, -1] = e + 4.5 * WQ[q] * qp

    def velocity(self):
        f = self.f
        rho = f.sum(0)
        ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8] - 0.5 * self.case["gx"]) / rho
        uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
        return rho, ux, uy

    def fields(self, k):
        rho, ux, uy = self.velocity()
        H, W = self.ny // k, self.nx // k
        out = torch.zeros((self.n, H, W, 8), dtype=torch.float64, device=DEV)
        for i, a in enumerate(((rho - 1) * RHO_SCALE, ux * U_SCALE, uy * U_SCALE)):
            out[..., i] = a[:, :H * k, :W * k].reshape(self.n, H, k, W, k).mean((2, 4))
        return out

    def observables(self):
        rho, ux, _ = self.velocity()
        x0, y0, w, h = self.square
        rows, cols = slice(y0, y0 + h), slice(x0, x0 + w)
        slope = lambda a, b: ((9 * ux[:, a, cols] - ux[:, b, cols]) / 3).mean(1)  # noqa: E731
        return torch.stack([rho[:, rows, x0 - 1].sum(1) / 3, rho[:, rows, x0 + w].sum(1) / 3,
                            slope(y0 + h, y0 + h + 1), -slope(y0 - 1, y0 - 2)], 1)

    def masses(self, f):
        return (f * ~self.solid).sum((0, 2, 3))

    def perturbed(self, f, snaps, slots, seed, it):
        """App. D: states f [9][m][ny][nx] of the listed slots, moved along the snapshots [9][k][ny][nx]"""
        k = snaps.shape[1]
        full = lambda v: torch.tensor(v, device=DEV)  # noqa: E731
        s = full([[i] * k for i in slots])
        j = full([list(range(k)) for _ in slots])
        a = EPS * _unit(_philox(torch.full_like(s, 4), torch.full_like(s, it), s, j, seed)[0])
        mass, add = self.masses(f), self.masses(snaps)
        out = f + torch.einsum("mk,qkyx->qmyx", a, snaps)
        out = out * (mass / (mass + a @ add)).view(1, -1, 1, 1)
        return torch.where(self.solid, f, out)


def _network(params, x, need_grad):
    """the learned score in FP64, weights as the BF16 copies the kernels multiply by"""
    p, o = torch.tensor(params, device=DEV), 0
    leaves = []
    a = x.permute(0, 3, 1, 2)
    for cin, pad in ((8, 80), (32, 304), (32, 304), (32, 304)):
        blk = p[o:o + 32 * pad].view(32, pad).to(torch.bfloat16).double()
        o += 32 * pad
        w = blk[:, :9 * cin].reshape(32, 3, 3, cin).permute(0, 3, 1, 2).contiguous().requires_grad_(need_grad)
        b = blk[:, 9 * cin].clone().requires_grad_(need_grad)
        leaves.append((w, b, pad, cin))
        a = torch.relu(torch.nn.functional.conv2d(a, w, b, padding=1))
    v = p[o:].double().clone().requires_grad_(need_grad)
    return (a.mean((2, 3)) * v[:32]).sum(1) + v[32], leaves, v


def _exact_train(case, seed):
    x, y = _inputs(case, seed)
    params, B = _params(seed), case["batch"]
    parts, loss = None, 0.0
    step = max(1, (1 << 19) // (case["height"] * case["width"]))
    for s in range(0, B, step):
        with torch.enable_grad():
            pred, leaves, v = _network(params, x[s:s + step].double(), True)
            part = ((pred - y[s:s + step].double()) ** 2).sum() / B
            g = torch.autograd.grad(part, [t for w, b, _, _ in leaves for t in (w, b)] + [v])
        loss += float(part)
        parts = list(g) if parts is None else [a + b for a, b in zip(parts, g)]
    out = []
    for i, (_, _, pad, cin) in enumerate(leaves):
        blk = torch.zeros((32, pad), dtype=torch.float64, device=DEV)
        blk[:, :9 * cin] = parts[2 * i].permute(0, 2, 3, 1).reshape(32, 9 * cin)
        blk[:, 9 * cin] = parts[2 * i + 1]
        out.append(blk.reshape(-1))
    out.append(parts[-1])
    return {"loss": torch.tensor([loss], dtype=torch.float64), "gradient": torch.cat(out).cpu().numpy(),
            "params": None}


def _trailing(d, window):
    """trailing means F(t) of the series [n][T], t = window .. T"""
    c = np.concatenate([np.zeros((d.shape[0], 1), np.longdouble), np.cumsum(d.astype(np.longdouble), 1)], 1)
    return ((c[:, window:] - c[:, :-window]) / window).astype(np.float64)


def _exact_stats(case, seed):
    d = _series(case, seed)[:, case["t0"]:case["t1"]]
    n, t = d.shape
    x = torch.tensor((d.astype(np.longdouble) - d.astype(np.longdouble).mean()).astype(np.float64), device=DEV)
    var = float((x * x).mean())
    c = torch.stack([(x[:, :t - k] * x[:, k:]).sum() / (n * (t - k)) / var for k in range(case["lags"] + 1)])
    return {"c": c, "tau_c": None, "events": None, "r": None, "maxima": _trailing(d, case["window"]).max(1),
            "sums": d.astype(np.longdouble).sum(1).astype(np.float64)}


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "stats":
        return _exact_stats(case, seed)
    if kind == "gktl":
        return None  # thousands of steps of the whole ensemble
    flow = _Flow(case, seed)
    if kind == "step":
        drag, obs = [], []
        for _ in range(case["steps"]):
            drag.append(flow.step())
            if case["obs"]:
                obs.append(flow.observables())
        out = {"drag": torch.stack(drag, 1), "fields": flow.fields(case["factor"])}
        if case["obs"]:
            out["obs"] = torch.stack(obs, 1)
        return out
    if kind == "resample":
        parent = _select(_weights(case["clones"], seed), seed)
        slots = [s for s, p in enumerate(parent) if p != s]
        if slots:
            snaps = flow.f[:, _bank(flow.n)].clone()
            flow.f[:, slots] = flow.perturbed(flow.f[:, [parent[s] for s in slots]], snaps, slots, seed, 0)
        f = flow.f * ~flow.solid
        m = f.sum((2, 3))
        return {"mass": m.sum(0).cpu().numpy(),
                "px": sum(CX[q] * m[q] for q in range(9)).cpu().numpy(),
                "py": sum(CY[q] * m[q] for q in range(9)).cpu().numpy(), "fields": flow.fields(4)}
    if kind == "score":
        for _ in range(20):
            flow.step()
        pred, _, _ = _network(_params(seed), flow.fields(case["factor"]), False)
        return {"score": pred}
    # one AMS iteration
    T, tb, w = case["horizon"], case["branch_at"], case["window"]
    drag, src = [], flow.n - 1
    for t in range(T):
        if t == tb // case["ckpt"] * case["ckpt"]:
            snaps = flow.f[:, _bank(flow.n)].clone()
        if t == tb:
            branch = flow.f[:, src:src + 1].clone()
        drag.append(flow.step())
    drag = torch.stack(drag, 1)
    flow.f, flow.n = flow.perturbed(branch, snaps, [0], seed, 1), 1
    drag[0, :tb] = drag[src, :tb]
    for t in range(tb, T):
        drag[0, t] = flow.step()[0]
    d = drag.cpu().numpy()
    return {"crossing": None, "Q": _trailing(d, w).max(1), "drag": drag, "fields": flow.fields(4)}


def _select(W, seed):
    """residual resampling with a systematic draw of the residuals, iteration 0"""
    n = len(W)
    fl = np.floor(W)
    cnt, res = fl.astype(int), W - fl
    R = n - int(cnt.sum())
    if R > 0:
        z = torch.zeros(1, dtype=torch.int64)
        u = float(_unit(_philox(z + 1, z, z, z, seed)[0]))
        spacing, i, edge = float(np.add.accumulate(res)[-1]) / R, 0, res[0]
        for k in range(R):
            while (u + k) * spacing >= edge and i < n - 1:
                i += 1
                edge += res[i]
            cnt[i] += 1
    parent = [i if cnt[i] else -1 for i in range(n)]
    extra = [i for i in range(n) for _ in range(cnt[i] - 1)]
    for s in range(n):
        if parent[s] < 0:
            parent[s] = extra.pop(0)
    return parent
