"""The work a user of this library has it do, as timed cases.

Every case is one pass through the public entry points of
`paper_2509_25110_gb300.gcamb`, on inputs of the repository's own seeded
generator (`synth`), at the sizes of its named workloads and at odd sizes in
between.  What each listed case stands for:

  plain64_l500      one model's temperature transfer and C_l in FP64 at
                    l <= 500: the smallest single call
  plain64_l5000     the same at the paper's high-accuracy size (3000 k, 2000
                    tau, l <= 5000): the largest single-model call
  emode32_odd       E-mode transfer functions of a few models in FP32 (a
                    finite-difference set), at sizes that fill no tile
  tensor64_l1500    the second projection of a CAMB run, tensor modes: three
                    transfers and TT, EE, BB, TE of one model in FP64
  camb_run_l2500    one default CAMB run (sampled multipoles, FP64): Bessel
                    functions, transfer, C_l at the samples, spline to every l
  batch_f16_l2500   the headline: 256 models on one grid, F16X3 tensor cores
  batch_bf16_odd    a small odd batch (37 models, 998 tau), BF16X3
  te_bf16_l2500     TT, EE and TE of 256 models
  uneven_f16_l6000  1000 models with their own l_max <= 6000 and k range, as a
                    plan replayed from its graph
  features_f32      sources of 256 models splined from 1000 onto 8000 k
                    (primordial features)
  emu_train         training the emulator: 16 Adam steps of 4096 spectra, then
                    the parameters are read (a checkpoint)
  emu_serve         4096 emulator requests in trusted cells
"""
import math

import numpy as np
import torch

from paper_2509_25110_gb300 import gcamb, synth

TAU0 = 14000.0
TAU_MIN = 200.0
MODES = {"plain64": gcamb.PLAIN64, "plain32": gcamb.PLAIN32, "bf16x3": gcamb.BF16X3, "f16x3": gcamb.F16X3}


def listed():
    return [
        {"name": "plain64_l500", "kind": "plain", "nk": 300, "ntau": 400, "lmax": 500, "kmin": 1e-4, "kmax": 0.3,
         "dense": False, "M": 1},
        {"name": "plain64_l5000", "kind": "plain", "nk": 3000, "ntau": 2000, "lmax": 5000, "kmin": 1e-5, "kmax": 1.0,
         "dense": True, "M": 1},
        {"name": "emode32_odd", "kind": "emode", "nk": 1001, "ntau": 1003, "lmax": 2001, "kmin": 1e-4, "kmax": 0.3,
         "M": 5},
        {"name": "tensor64_l1500", "kind": "tensor", "nk": 1000, "ntau": 1000, "lmax": 1500, "kmin": 1e-4,
         "kmax": 3000.0 / TAU0, "M": 1},
        {"name": "camb_run_l2500", "kind": "run", "nk": 2000, "ntau": 1000, "lmax": 2500, "kmin": 1e-4, "kmax": 0.3,
         "boost": 1.0, "M": 1},
        {"name": "batch_f16_l2500", "kind": "batch", "mode": "f16x3", "nk": 2000, "ntau": 1000, "lmax": 2500,
         "kmin": 1e-4, "kmax": 0.3, "M": 256},
        {"name": "batch_bf16_odd", "kind": "batch", "mode": "bf16x3", "nk": 701, "ntau": 998, "lmax": 1237,
         "kmin": 1e-4, "kmax": 0.3, "M": 37},
        {"name": "te_bf16_l2500", "kind": "te", "nk": 2000, "ntau": 1000, "lmax": 2500, "kmin": 1e-4, "kmax": 0.3,
         "M": 256},
        {"name": "uneven_f16_l6000", "kind": "uneven", "nk": 3000, "ntau": 1000, "lmax": 6000, "kmax": 0.5, "M": 1000},
        {"name": "features_f32", "kind": "interp", "nk": 8000, "nk_in": 1000, "ntau": 1000, "kmin": 1e-4, "kmax": 0.3,
         "M": 256},
        {"name": "emu_train", "kind": "train", "lmax": 2500, "width": 512, "depth": 3, "B": 4096, "steps": 16},
        {"name": "emu_serve", "kind": "serve", "lmax": 2500, "width": 512, "depth": 3, "B": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "emode", "tensor", "run", "batch", "batch", "te", "uneven", "interp", "train", "serve"])
    c = {"kind": kind}
    if kind in ("train", "serve"):
        c.update(lmax=_log(rng, 300, 2500), width=rng.choice([128, 200, 256, 384, 512]), depth=rng.randint(2, 3))
        c.update(B=_log(rng, 256, 4096) if kind == "train" else _log(rng, 1, 4096))
        if kind == "train":
            c["steps"] = 16
        return c
    c.update(nk=_log(rng, 200, 2000), ntau=_log(rng, 300, 1000), kmin=1e-4, kmax=rng.uniform(0.1, 0.3))
    if kind == "plain":
        c.update(lmax=_log(rng, 300, 3000), dense=False, M=rng.randint(1, 4))
    elif kind == "emode":
        c.update(lmax=_log(rng, 300, 2500), M=rng.randint(1, 8))
    elif kind == "tensor":
        c.update(lmax=_log(rng, 200, 1500), nk=_log(rng, 200, 1000), kmax=3000.0 / TAU0, M=rng.randint(1, 4))
    elif kind == "run":
        c.update(lmax=_log(rng, 500, 2500), boost=rng.choice([1.0, 2.0, 3.0]), M=rng.randint(1, 2))
    elif kind == "batch":
        c.update(lmax=_log(rng, 300, 2500), mode=rng.choice(["f16x3", "f16x3", "bf16x3"]), M=_log(rng, 8, 256))
        if rng.random() < 0.6:
            c["ntau"] -= c["ntau"] % 4
    elif kind == "te":
        c.update(lmax=_log(rng, 300, 2500), M=_log(rng, 8, 256))
        c["ntau"] -= c["ntau"] % 4
    elif kind == "uneven":
        c.update(nk=_log(rng, 1000, 3000), lmax=_log(rng, 2000, 6000), kmax=rng.uniform(0.2, 0.5), M=_log(rng, 50, 500))
        del c["kmin"]
    else:
        c.update(nk=_log(rng, 1000, 8000), nk_in=_log(rng, 200, 1000), M=_log(rng, 8, 256))
    return c


# ------------------------------------------------------------------ inputs

def _grids(c):
    if c["kind"] == "uneven":
        k = synth.master_linear_k(c["nk"], c["kmax"])
    else:
        k = synth.log_grid(c["kmin"], c["kmax"], c["nk"])
    if c.get("dense"):
        return k, synth.dense_tau_grid(c["ntau"] // 2, c["ntau"] - c["ntau"] // 2)
    return k, synth.uniform_grid(TAU_MIN, TAU0, c["ntau"])


def _lrows(c):
    """The multipoles of the outputs: every l, or CAMB's sampled list (steps of round(l / (20 boost)), at most
    ceil(50 / boost), l_max always listed)."""
    if c["kind"] != "run":
        return np.arange(2, c["lmax"] + 1)
    rows, cap = [2], max(1, math.ceil(50.0 / c["boost"]))
    while rows[-1] < c["lmax"]:
        step = int(math.floor(rows[-1] / (20.0 * c["boost"]) + 0.5))
        rows.append(min(c["lmax"], rows[-1] + max(1, min(cap, step))))
    return np.asarray(rows, dtype=np.int64)


def _sources(c, seed):
    """The models' sources and primordial spectra, in the types the calls take."""
    k, tau = _grids(c)
    kind = c["kind"]
    if kind == "uneven":  # l_max per model, and the k prefix that goes with it
        p = synth.model_params(c["M"], seed=seed, lmax_range=(c["lmax"] // 4, c["lmax"]))
        nk_m = np.maximum(1, np.rint(c["nk"] * (1.0 + 2.0 * p.lmax / c["lmax"]) / 3.0)).astype(np.int64)
        S = [synth.sources_torch(k, tau, p, "cuda", torch.float32, nk_per_model=nk_m)]
        return S, torch.as_tensor(synth.primordial(k, p), device="cuda"), p.lmax, nk_m
    p = synth.model_params(c["M"], seed=seed)
    dt = torch.float64 if kind in ("plain", "tensor", "run") else torch.float32
    if kind == "tensor":
        S = [torch.as_tensor(a, device="cuda") for a in synth.sources_tensor(k, tau, p)]
        return S, torch.as_tensor(synth.primordial_tensor(k, p), device="cuda"), None, None
    if kind == "interp":
        k_in = synth.log_grid(c["kmin"], c["kmax"], c["nk_in"])
        k_in[0], k_in[-1] = min(k_in[0], k[0]), max(k_in[-1], k[-1])
        return [synth.sources_torch(k_in, tau, p, "cuda", dt)], k_in, None, None
    if kind == "emode":
        S = [synth.sources_pol_torch(k, tau, p, "cuda", dt)]
    else:
        S = [synth.sources_torch(k, tau, p, "cuda", dt)]
    if kind == "te":
        S.append(synth.sources_pol_torch(k, tau, p, "cuda", dt))
    return S, torch.as_tensor(synth.primordial(k, p), device="cuda"), None, None


def _features(n, seed):
    return synth.emulator_features(synth.model_params(n, seed=seed))


def _smooth_log_cl(X, lmax):
    """log C_l targets with the shape of acoustic spectra, smooth in the features."""
    x = torch.as_tensor(np.asarray(X, dtype=np.float64), device="cuda")
    l = torch.arange(2, lmax + 1, dtype=torch.float64, device="cuda")[None, :]
    c = [x[:, j:j + 1] for j in range(9)]
    u = l / 14000.0
    env = c[8] - 2.0 * torch.log(l) - 20.0 + (c[7] - 1.0) * torch.log(u / 0.05)
    osc = torch.cos(u * c[2] + torch.atan2(c[4], c[3]))
    damp = torch.exp(-((u / c[5]) ** 2) - (u * c[1]) ** 2)
    return env + torch.log(0.3 * damp + damp * osc ** 2 + 0.02 + c[6] * torch.exp(-u / 0.01))


def _network(c, seed):
    """Parameters of a network (a checkpoint the program starts from), flat as gcamb.emu_params takes them."""
    r = np.random.default_rng(seed + 101)
    sizes = [9] + [c["width"]] * c["depth"] + [c["lmax"] - 1]
    Ws = [r.uniform(-1, 1, (b, a)) / math.sqrt(a) for a, b in zip(sizes[:-1], sizes[1:])]
    bs = [r.uniform(-1, 1, b) / math.sqrt(a) for a, b in zip(sizes[:-1], sizes[1:])]
    return gcamb.flatten(Ws, bs), sizes


def _emu_grid(c):
    return gcamb.grid_create(synth.log_grid(1e-4, 0.3, 64), synth.uniform_grid(TAU_MIN, TAU0, 64), TAU0, 2, c["lmax"])


N_TRAIN = 8192


def _train_set(c, seed):
    X = _features(N_TRAIN, seed)
    idx = np.random.default_rng(seed + 7).integers(0, N_TRAIN, (c["steps"], c["B"])).astype(np.int32)
    return X, torch.exp(_smooth_log_cl(X, c["lmax"])), idx


LR = 1e-3


def _norms(c, X):
    """Normalisation arrays of a served network: features to zero mean and unit deviation, outputs about log C_l."""
    sd_x = X.std(0).astype(np.float32)
    sd_x[sd_x < 1e-6] = 0.0
    l = np.arange(2, c["lmax"] + 1)
    return (X.mean(0).astype(np.float32), sd_x, (-20.0 - 2.0 * np.log(l)).astype(np.float32),
            np.full(l.size, 0.2, dtype=np.float32))


# ------------------------------------------------------------------ the cases' protocol

def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"c": c}
    if kind in ("train", "serve"):
        g = _emu_grid(c)
        e = gcamb.emu_create(g, width=c["width"], depth=c["depth"], max_batch=4096, seed=1)
        params, _ = _network(c, seed)
        gcamb.emu_params(e, params)
        s.update(g=g, e=e)
        if kind == "train":
            X, C, idx = _train_set(c, seed)
            s["X"] = torch.as_tensor(X, device="cuda")
            s["Y"] = gcamb.emu_fit_norm(e, s["X"], C)
            s["idx"] = torch.as_tensor(idx, device="cuda")
            s["loss"] = torch.zeros(1, dtype=torch.float32, device="cuda")
            return s
        Xc = _features(2048, seed + 1)
        norms = _norms(c, Xc)
        gcamb.emu_norm(e, *norms)
        # the held-out check: every cell trusted (the reference spectra are the network's)
        Xd = torch.as_tensor(Xc, device="cuda")
        Y = gcamb.emu_forward(e, Xd).double()
        shift = (Xd[:, 8:9] - float(norms[0][8])).double()
        ref = torch.exp(Y * torch.as_tensor(norms[3], device="cuda").double()
                        + torch.as_tensor(norms[2], device="cuda").double() + shift)
        gcamb.emu_check(e, Xd, ref.contiguous(), tol=1e-2, min_count=1)
        s["X"] = torch.as_tensor(_features(c["B"], seed), device="cuda")
        s["Cl"] = torch.empty((c["B"], g.nl), dtype=torch.float64, device="cuda")
        s["fb"] = torch.empty(c["B"], dtype=torch.int32, device="cuda")
        return s

    k, tau = _grids(c)
    S, P, lmax_m, nk_m = _sources(c, seed)
    s.update(S=S, P=P)
    M = c["M"]
    if kind == "run":
        g = gcamb.grid_create_lsampled(k, tau, TAU0, gcamb.l_sampling(2, c["lmax"], c["boost"]))
    else:
        g = gcamb.grid_create(k, tau, TAU0, 2, c.get("lmax", 2))
    s["g"] = g
    f64 = {"dtype": torch.float64, "device": "cuda"}
    if kind in ("plain", "tensor"):
        gcamb.bessel_table(g, gcamb.PLAIN64)
        n = 3 if kind == "tensor" else 1
        s["D"] = tuple(torch.empty((M, g.nk, g.nl), **f64) for _ in range(n))
        s["Cl"] = tuple(torch.empty((M, g.nl), **f64) for _ in range(n + 1 if n > 1 else 1))
    elif kind == "emode":
        gcamb.bessel_table(g, gcamb.PLAIN32)
        s["D"] = torch.empty((M, g.nk, g.nl), dtype=torch.float32, device="cuda")
    elif kind == "run":
        gcamb.bessel_table(g, gcamb.PLAIN64)
        s["D"] = torch.empty((M, g.nk, g.nl), **f64)
    elif kind == "batch":
        s["mode"] = MODES[c["mode"]]
        gcamb.bessel_table(g, s["mode"])
        s["ws"] = torch.empty(gcamb.los_cl_workspace(g, M, s["mode"]), dtype=torch.uint8, device="cuda")
        s["Cl"] = torch.empty((M, g.nl), **f64)
    elif kind == "te":
        gcamb.bessel_table(g, gcamb.BF16X3)
        s["ws"] = torch.empty(gcamb.los_cl_te_workspace(g, M), dtype=torch.uint8, device="cuda")
        s["Cl"] = tuple(torch.empty((M, g.nl), **f64) for _ in range(3))
    elif kind == "uneven":
        gcamb.bessel_table(g, gcamb.F16X3)
        s["plan"] = gcamb.plan_create(g, M, lmax_m, nk_m, gcamb.F16X3)
        s["ws"] = torch.empty(gcamb.plan_workspace(s["plan"]), dtype=torch.uint8, device="cuda")
        s["Cl"] = torch.empty((M, g.nl), **f64)
    else:
        s["out"] = torch.empty((M, g.nk, g.ntau), dtype=torch.float32, device="cuda")
    return s


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "plain":
        gcamb.los_transfer(s["g"], s["S"][0], gcamb.PLAIN64, s["D"][0])
        return s["D"][0], gcamb.cl(s["g"], s["D"][0], s["P"], s["Cl"][0])
    if kind == "emode":
        return gcamb.los_transfer_e(s["g"], s["S"][0], gcamb.PLAIN32, s["D"])
    if kind == "tensor":
        g, P, (tt, ee, bb, te) = s["g"], s["P"], s["Cl"]
        DT, DE, DB = gcamb.los_transfer_tensor(g, s["S"][0], s["S"][1], gcamb.PLAIN64, out=s["D"])
        gcamb.cl(g, DT, P, tt)
        gcamb.cl(g, DE, P, ee)
        gcamb.cl(g, DB, P, bb)
        gcamb.cl_cross(g, DT, DE, P, te)
        return DT, DE, DB, tt, ee, bb, te
    if kind == "run":
        g = s["g"]
        gcamb.bessel_table(g, gcamb.PLAIN64)
        gcamb.los_transfer(g, s["S"][0], gcamb.PLAIN64, s["D"])
        Cs = gcamb.cl(g, s["D"], s["P"])
        return s["D"], Cs, gcamb.cl_interp(g, Cs)
    if kind == "batch":
        return gcamb.los_cl(s["g"], s["S"][0], s["P"], s["mode"], s["Cl"], s["ws"])
    if kind == "te":
        return gcamb.los_cl_te(s["g"], s["S"][0], s["S"][1], s["P"], out=s["Cl"], ws=s["ws"])
    if kind == "uneven":
        return gcamb.plan_launch(s["plan"], s["S"][0], s["P"], s["Cl"], s["ws"])
    if kind == "interp":
        return gcamb.interp_sources(s["g"], s["P"], s["S"][0], s["out"])
    if kind == "train":
        for i in range(c["steps"]):
            gcamb.emu_train_step(s["e"], s["X"], s["Y"], s["idx"][i], c["B"], LR, s["loss"])
        return gcamb.emu_params(s["e"]), s["loss"]
    return gcamb.emulate(s["e"], s["X"], s["Cl"], s["fb"])


# ------------------------------------------------------------------ what a pass cannot do without

def _active(k, tau, lrows):
    """(l, k, tau) entries whose Bessel function is not negligible: l up to a little past x = k (tau0 - tau)."""
    x = k[:, None] * (TAU0 - tau)[None, :]
    return int(np.searchsorted(lrows, x + 4.0 * np.cbrt(x) + 1.0).sum())


def work(case):
    c, kind = case, case["kind"]
    if kind in ("train", "serve"):
        sizes = [9] + [c["width"]] * c["depth"] + [c["lmax"] - 1]
        n = sum(a * b + b for a, b in zip(sizes[:-1], sizes[1:]))
        B = c["B"]
        if kind == "serve":
            return {"bytes": 4 * n + 36 * B + 8 * B * (c["lmax"] - 1) + 4 * B, "flops": 2 * B * n}
        # per step: the batch's targets and features, parameters and both moments read and written
        return {"bytes": c["steps"] * (B * (c["lmax"] - 1 + 9) * 4 + 24 * n) + 4 * n, "flops": c["steps"] * 6 * B * n}
    k, tau = _grids(c)
    M, nk, nt = c["M"], k.size, tau.size
    if kind == "interp":
        return {"bytes": 4 * M * nt * (c["nk_in"] + nk), "flops": M * nt * (12 * c["nk_in"] + 10 * nk)}
    rows = _lrows(c)
    nl = rows.size
    if kind == "uneven":
        p = synth.model_params(M, seed=0, lmax_range=(c["lmax"] // 4, c["lmax"]))
        nk_m = np.maximum(1, np.rint(nk * (1.0 + 2.0 * p.lmax / c["lmax"]) / 3.0)).astype(np.int64)
        flops = 0
        for b in range(8):  # models by l_max, in eight bins
            lo, hi = c["lmax"] * (2 + b * 0.75) / 8, c["lmax"] * (2 + (b + 1) * 0.75) / 8
            sel = (p.lmax >= lo) & (p.lmax < hi + (b == 7))
            if sel.any():
                a = _active(k[:int(nk_m[sel].mean())], tau, np.arange(2, int(p.lmax[sel].mean()) + 1))
                flops += 6 * int(sel.sum()) * a
        return {"bytes": 4 * _active(k, tau, rows) + 4 * int(nk_m.sum()) * nt + 8 * M * (nk + nl), "flops": flops}
    a = _active(k, tau, rows)
    if kind == "plain":
        return {"bytes": 8 * (a + M * nk * (nt + nl + 1) + M * nl), "flops": 2 * a * M + 3 * M * nk * nl}
    if kind == "emode":
        return {"bytes": 4 * (a + M * nk * (nt + nl)), "flops": 2 * a * M}
    if kind == "tensor":
        return {"bytes": 8 * (a + M * nk * (2 * nt + 3 * nl + 1) + 4 * M * nl), "flops": 8 * a * M + 12 * M * nk * nl}
    if kind == "run":  # the recurrence runs through every l; the table is written, then read
        full = _active(k, tau, np.arange(2, c["lmax"] + 1))
        return {"bytes": 8 * (2 * a + M * nk * (nt + nl) + M * (nl + c["lmax"])), "flops": 2 * full + 2 * a * M}
    f = 2 if kind == "te" else 1
    return {"bytes": 4 * a + 4 * f * M * nk * nt + 8 * M * nk + 8 * M * nl * (3 if f == 2 else 1),
            "flops": 6 * a * f * M}


# ------------------------------------------------------------------ 64-bit references, plain torch

def _bessel_rows(x, lmax):
    """j_0..j_lmax at x (1-D, > 0) -> [lmax + 1][n] in FP64.  Downward recurrence from an order where j_l is
    negligible, scaled to j_0 or j_1, where that order is at hand; forward recurrence for the larger x."""
    n = x.numel()
    J = torch.zeros((lmax + 1, n), dtype=torch.float64, device=x.device)
    top = (x + 25.0 * x.pow(1.0 / 3.0) + 45.0).ceil().long()
    H = int(lmax + 25.0 * lmax ** (1.0 / 3.0) + 60.0)
    down = top < H
    di, ui = down.nonzero()[:, 0], (~down).nonzero()[:, 0]
    if di.numel():
        xd = x[di]
        h = int(top[di].max()) + 1
        F = torch.zeros((h + 1, di.numel()), dtype=torch.float64, device=x.device)
        F.scatter_(0, top[di][None, :], 1e-120)
        inv = 1.0 / xd
        # f_(l-1) = (2l+1)/x f_l - f_(l+1); signs chosen so that each step is one add and one multiply-add:
        # f_l = sgn_l F_l with sgn_(l-1) = -sgn_(l+1)
        sgn = [1.0, 1.0, -1.0, -1.0]
        F *= torch.tensor([sgn[l % 4] for l in range(h + 1)], dtype=torch.float64, device=x.device)[:, None]
        for l in range(h - 1, 0, -1):
            F[l - 1].add_(F[l + 1])
            F[l - 1].addcmul_(inv, F[l], value=sgn[(l - 1) % 4] * sgn[l % 4] * (2 * l + 1))
        F *= torch.tensor([sgn[l % 4] for l in range(h + 1)], dtype=torch.float64, device=x.device)[:, None]
        j0 = torch.where(xd < 1e-3, 1.0 - xd * xd / 6.0, torch.sin(xd) / xd)
        j1 = torch.where(xd < 1e-2, xd / 3.0 * (1.0 - xd * xd / 10.0 * (1.0 - xd * xd / 28.0)),
                         (torch.sin(xd) / xd - torch.cos(xd)) / xd)
        scale = torch.where(j0.abs() >= j1.abs(), j0 / F[0], j1 / F[1])
        m = min(h, lmax)
        F[:m + 1] *= scale
        J[:m + 1].index_copy_(1, di, F[:m + 1])
        del F
    if ui.numel():
        xu = x[ui]
        U = torch.empty((lmax + 1, ui.numel()), dtype=torch.float64, device=x.device)
        inv = 1.0 / xu
        U[0] = torch.sin(xu) * inv
        U[1] = (U[0] - torch.cos(xu)) * inv
        for l in range(1, lmax):
            torch.mul(U[l], inv, out=U[l + 1])
            U[l + 1].mul_(2 * l + 1).sub_(U[l - 1])
        J.index_copy_(1, ui, U)
    return J


def _trapezoid(x):
    w = torch.zeros_like(x)
    w[1:] += 0.5 * (x[1:] - x[:-1])
    w[:-1] += 0.5 * (x[1:] - x[:-1])
    return w


def _project(k, tau, lrows, sources, kernels, chunk_gb=8.0):
    """For each (source, kernel) pair the sum over tau of w S kernel_l(x): [M][nk][rows] in FP64.  kernels: "j",
    "eps" (c_l j_l/x^2), "e", "b" (the tensor E and B kernels)."""
    kt = torch.as_tensor(k, device="cuda")
    w = _trapezoid(torch.as_tensor(tau, device="cuda"))
    dt = (TAU0 - torch.as_tensor(tau, device="cuda"))
    lr = torch.as_tensor(np.asarray(lrows), device="cuda")
    lmax = int(lrows[-1])
    l = lr.double()[:, None]
    cl = torch.sqrt((l + 2) * (l + 1) * l * (l - 1))
    outs = [torch.empty((S.shape[0], kt.numel(), lr.numel()), dtype=torch.float64, device="cuda") for S in sources]
    step = max(1, int(chunk_gb * 2 ** 30 / (8.0 * (lmax + 400) * dt.numel())))
    for a in range(0, kt.numel(), step):
        kk = kt[a:a + step]
        x = (kk[:, None] * dt[None, :]).clamp_min(1e-7).reshape(-1)
        J = _bessel_rows(x, lmax)
        full = lr.numel() == lmax - 1
        Jl = J[2:] if full else J[lr]
        Jm = (J[1:-1] if full else J[lr - 1]) if ("e" in kernels or "b" in kernels) else None
        for S, kern, D in zip(sources, kernels, outs):
            if kern == "j":
                K = Jl
            elif kern == "eps":
                K = cl * Jl / (x * x)
            elif kern == "e":
                K = (l * (l - 1) / (x * x) - 2.0) * Jl + 2.0 * Jm / x
            else:
                K = 2.0 * Jm - 2.0 * (l - 1) * Jl / x
            K = K.reshape(lr.numel(), kk.numel(), dt.numel()).permute(1, 2, 0)        # [k][tau][rows]
            A = (S[:, a:a + step].double() * w).permute(1, 0, 2)                      # [k][M][tau]
            D[:, a:a + step] = torch.bmm(A, K).permute(1, 0, 2)
        del J, Jl, Jm, K
    return outs


def _cl(k, DX, DY, P):
    wk = _trapezoid(torch.log(torch.as_tensor(k, device="cuda")))
    out = torch.zeros((DX.shape[0], DX.shape[2]), dtype=torch.float64, device="cuda")
    for m in range(DX.shape[0]):
        out[m] = 4.0 * math.pi * ((wk * P[m])[:, None] * DX[m] * DY[m]).sum(0)
    return out


def _spline(xs, ys, xq):
    """Natural cubic spline along the first axis of ys (FP64) at xq, by the tridiagonal system of its second
    derivatives."""
    n = xs.size
    h = np.diff(xs)
    m = torch.zeros((n,) + tuple(ys.shape[1:]), dtype=torch.float64, device=ys.device)
    if n > 2:
        cp = np.zeros(n)
        for j in range(1, n - 1):
            den = 2.0 * (h[j - 1] + h[j]) - h[j - 1] * cp[j - 1]
            cp[j] = h[j] / den
            r = 6.0 * ((ys[j + 1] - ys[j]) / h[j] - (ys[j] - ys[j - 1]) / h[j - 1])
            m[j] = (r - h[j - 1] * m[j - 1]) / den
        for j in range(n - 2, 0, -1):
            m[j] -= cp[j] * m[j + 1]
    j = np.clip(np.searchsorted(xs, xq, side="right") - 1, 0, n - 2)
    shape = (-1,) + (1,) * (ys.dim() - 1)
    hh = torch.as_tensor(h[j], device=ys.device).reshape(shape)
    t = torch.as_tensor((xq - xs[j]) / h[j], device=ys.device).reshape(shape)
    j = torch.as_tensor(j, device=ys.device)
    u = 1.0 - t
    return u * ys[j] + t * ys[j + 1] + hh * hh / 6.0 * ((u ** 3 - u) * m[j] + (t ** 3 - t) * m[j + 1])


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _gelu_grad(z):
    return 0.5 * (1.0 + torch.erf(z / math.sqrt(2.0))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)


def _unpack(flat, sizes):
    flat = torch.as_tensor(np.asarray(flat, dtype=np.float64), device="cuda")
    W, b, o = [], [], 0
    for i, j in zip(sizes[:-1], sizes[1:]):
        W.append(flat[o:o + i * j].reshape(j, i).clone())
        o += i * j
        b.append(flat[o:o + j].clone())
        o += j
    return W, b


def _exact_emu(c, seed):
    params, sizes = _network(c, seed)
    W, b = _unpack(params, sizes)
    n = len(W)

    def forward(x):
        Z, H = [], [x]
        for i in range(n):
            Z.append(H[-1] @ W[i].T + b[i])
            H.append(_gelu(Z[-1]) if i < n - 1 else Z[-1])
        return Z, H

    if c["kind"] == "serve":
        mu_x, sd_x, mu_y, sd_y = (torch.as_tensor(a, device="cuda").double()
                                  for a in _norms(c, _features(2048, seed + 1)))
        X = torch.as_tensor(_features(c["B"], seed), device="cuda").double()
        isd = torch.where(sd_x > 0, 1.0 / sd_x, torch.zeros_like(sd_x))
        _, H = forward((X - mu_x) * isd)
        return torch.exp(H[-1] * sd_y + mu_y + (X[:, 8:9] - mu_x[8])), None
    X, C, idx = _train_set(c, seed)
    X = torch.as_tensor(X, device="cuda").double()
    mu_x, sd_x = X.mean(0), X.std(0, unbiased=False)
    isd = torch.where(sd_x > 1e-12, 1.0 / sd_x, torch.zeros_like(sd_x))
    Y = torch.log(C) - (X[:, 8:9] - mu_x[8])
    mu_y, sd_y = Y.mean(0), Y.std(0, unbiased=False)
    Y = (Y - mu_y) / torch.sqrt((sd_y ** 2).mean())
    xs = (X - mu_x) * isd
    par = W + b
    mom, vel = [torch.zeros_like(t) for t in par], [torch.zeros_like(t) for t in par]
    loss = None
    for s in range(c["steps"]):
        i = torch.as_tensor(idx[s].astype(np.int64), device="cuda")
        Z, H = forward(xs[i])
        d = H[-1] - Y[i]
        loss = (d * d).mean().reshape(1)
        d = 2.0 * d / d.numel()
        gW, gb = [None] * n, [None] * n
        for layer in range(n - 1, -1, -1):
            gW[layer], gb[layer] = d.T @ H[layer], d.sum(0)
            if layer:
                d = (d @ W[layer]) * _gelu_grad(Z[layer - 1])
        for p, g, m, v in zip(par, gW + gb, mom, vel):
            m.mul_(0.9).add_(g, alpha=0.1)
            v.mul_(0.999).addcmul_(g, g, value=0.001)
            p.sub_(LR * (m / (1.0 - 0.9 ** (s + 1))) / (torch.sqrt(v / (1.0 - 0.999 ** (s + 1))) + 1e-8))
    return torch.cat([t.reshape(-1) for layer in range(n) for t in (W[layer], b[layer])]).cpu().numpy(), loss


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "uneven":
        return None  # about 2e13 FP64 operations
    if kind in ("train", "serve"):
        return _exact_emu(c, seed)
    k, tau = _grids(c)
    S, P, _, _ = _sources(c, seed)
    if kind == "interp":
        y = S[0]
        out = torch.empty((c["M"], k.size, tau.size), dtype=torch.float64, device="cuda")
        for m in range(0, c["M"], 64):  # in slices: [n][models][tau]
            out[m:m + 64] = _spline(P, y[m:m + 64].double().permute(1, 0, 2).contiguous(), k).permute(1, 0, 2)
        return out
    rows = _lrows(c)
    if kind == "plain":
        D, = _project(k, tau, rows, S, ["j"])
        return D, _cl(k, D, D, P)
    if kind == "emode":
        return _project(k, tau, rows, S, ["eps"])[0]
    if kind == "tensor":
        T, E, B = _project(k, tau, rows, [S[0], S[1], S[1]], ["eps", "e", "b"])
        return T, E, B, _cl(k, T, T, P), _cl(k, E, E, P), _cl(k, B, B, P), _cl(k, T, E, P)
    if kind == "run":
        D, = _project(k, tau, rows, S, ["j"])
        Cs = _cl(k, D, D, P)
        l = np.arange(2, c["lmax"] + 1).astype(np.float64)
        f = rows.astype(np.float64)
        y = (torch.as_tensor(f * (f + 1.0), device="cuda") * Cs).T.contiguous()
        full = _spline(f, y, l).T / torch.as_tensor(l * (l + 1.0), device="cuda")
        full[:, torch.as_tensor(rows - 2, device="cuda")] = Cs
        return D, Cs, full.contiguous()
    if kind == "te":
        T, E = _project(k, tau, rows, S, ["j", "eps"])
        return _cl(k, T, T, P), _cl(k, E, E, P), _cl(k, T, E, P)
    D, = _project(k, tau, rows, S, ["j"])
    return _cl(k, D, D, P)
