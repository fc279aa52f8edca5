"""What the framework is used for, as cases that can be timed: the transport of photon
packages through one model (two or four dust species, with the path-length estimator,
with images), through a batch of models and through a model set up from host arrays; the
emission of transiently heated PAHs (exact, and by the network with exact fallback); the
network's forward pass and its training; the temperature distribution of single PAHs.

The transport cases run the frozen-temperature mode (the mode of the Lucy iteration and
of the replays): its histories do not depend on the order in which packages arrive, so
the same seed gives the same counts. The Bjorkman-Wood mode runs through the same
kernels. Every case goes through the public binding (``rt``, ``surrogate``)."""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1201_3588_gb300 import rt, surrogate, workloads as w

EV = 1.602176634e-12       # erg
H = 6.62607015e-27         # erg s
KB = 1.380649e-16          # erg / K
C = 2.99792458e10          # cm / s


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest model: a sphere that is a few cubes wide, where the launches and
        # the longest histories count
        {"name": "sphere", "kind": "transport", "model": "sphere", "n_base": 16, "levels": 0,
         "bins": 64, "tau": 1.0, "packages": 100_000, "dirs": 1},
        # the flared disk of two dust species, refined twice towards the midplane
        {"name": "disk", "kind": "transport", "model": "disk", "n_base": 64, "levels": 2,
         "bins": 200, "tau": 1e3, "packages": 5_000_000, "dirs": 1},
        # the disk with gap and spiral, four species and 400 bins: the grid exceeds L2
        {"name": "disk_four_species", "kind": "transport", "model": "disk4", "n_base": 96,
         "levels": 2, "bins": 400, "tau": 1e3, "packages": 10_000_000, "dirs": 1},
        # one step of the Lucy iteration: path lengths tallied in every cell crossed
        {"name": "lucy_step", "kind": "lucy", "model": "disk", "n_base": 48, "levels": 2,
         "bins": 100, "tau": 100.0, "packages": 2_000_000, "dirs": 1},
        # peel-off images of an inclined disk at two wavelengths
        {"name": "disk_images", "kind": "images", "model": "disk", "n_base": 64, "levels": 1,
         "bins": 200, "tau": 1e3, "packages": 2_000_000, "dirs": 1, "pixels": 256,
         "incline": 60.0},
        # uneven spheres and disks in one launch
        {"name": "batch", "kind": "batch", "models": 24, "bins": 100, "share": 0.1},
        # exact emission of the PAHs in every cell that absorbed
        {"name": "pah_exact", "kind": "pah", "n_base": 96, "levels": 1, "bins": 200,
         "tau": 1e3, "packages": 30_000_000, "surrogate": False},
        # the same by the network, the cells outside its range solved exactly
        {"name": "pah_auto", "kind": "pah", "n_base": 64, "levels": 1, "bins": 200,
         "tau": 300.0, "packages": 30_000_000, "surrogate": True},
        # the network alone over the cells of a large disk
        {"name": "surrogate_forward", "kind": "forward", "rows": 400_000, "inputs": 66,
         "hidden": 256, "layers": 3, "outputs": 200},
        # one epoch of the network's training in minibatches
        {"name": "surrogate_train", "kind": "train", "rows": 16 * 1024 + 77, "batch": 1024,
         "inputs": 66, "hidden": 256, "layers": 3, "outputs": 200},
        # temperature distributions of PAHs heated by single photons of 3.8 eV to 1 keV
        {"name": "pah_distribution", "kind": "pt", "cases": 12, "levels": 400, "bins": 200},
        # one model of a series: set up from host arrays, transported, read back, closed
        {"name": "model_series", "kind": "series", "model": "disk", "n_base": 48, "levels": 1,
         "bins": 100, "tau": 30.0, "packages": 1_000_000, "dirs": 4},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["transport", "transport", "lucy", "images", "batch", "pah", "pah",
                       "forward", "train", "pt", "series"])
    if kind in ("transport", "lucy", "images", "series"):
        model = rng.choice(["sphere", "disk", "disk4"] if kind == "transport" else
                           ["sphere", "disk"])
        c = {"kind": kind, "model": model,
             "n_base": 2 * round(_log(rng, 6, 28)) if model == "sphere" else
             round(_log(rng, 20, 56)),
             "levels": 0 if model == "sphere" else rng.choice([1, 2]),
             "bins": rng.choice([47, 64, 100, 129, 200, 333]),
             "tau": round(_log(rng, 0.3, 3.0 if model == "sphere" else 1e3), 3),
             "packages": round(_log(rng, 2e4, 3e6)), "dirs": rng.choice([1, 1, 3, 8])}
        if kind == "images":
            c.update(pixels=round(_log(rng, 33, 300)), incline=round(rng.uniform(0, 90), 1))
        return c
    if kind == "batch":
        return {"kind": kind, "models": rng.randint(3, 20), "bins": rng.choice([48, 75, 100]),
                "share": round(_log(rng, 0.01, 0.08), 4)}
    if kind == "pah":
        return {"kind": kind, "n_base": round(_log(rng, 24, 60)), "levels": 1,
                "bins": rng.choice([96, 131, 200, 257]), "tau": round(_log(rng, 30, 1e3), 2),
                "packages": round(_log(rng, 1e5, 3e6)),
                "surrogate": rng.choice([False, True])}
    if kind == "forward":
        return {"kind": kind, "rows": round(_log(rng, 200, 3.5e5)),
                "inputs": rng.choice([34, 49, 66]), "hidden": rng.choice([64, 100, 128, 256]),
                "layers": rng.choice([2, 3]), "outputs": rng.choice([99, 131, 200, 400])}
    if kind == "train":
        batch = rng.choice([256, 500, 1024, 2048])
        return {"kind": kind, "rows": batch * rng.randint(3, 12) + rng.randint(0, batch - 1),
                "batch": batch, "inputs": rng.choice([49, 66]),
                "hidden": rng.choice([128, 200, 256]), "layers": rng.choice([2, 3]),
                "outputs": rng.choice([131, 200])}
    return {"kind": kind, "cases": rng.randint(1, 10), "levels": round(_log(rng, 100, 500)),
            "bins": rng.choice([48, 77, 100, 200])}


# ------------------------------------------------------------------ models

@functools.lru_cache(maxsize=8)
def _model(model, n_base, levels, bins, dirs=1):
    """The unit-depth model and a smooth temperature field on its cells."""
    if model == "sphere":
        m = w.sphere_model(n_base=n_base, n_bins=bins, n_sed_dirs=dirs)
    elif model == "disk":
        m = w.disk_model(n_base=n_base, max_level=levels, n_bins=bins, tau_v_mid=1.0,
                         n_sed_dirs=dirs)
    elif model == "disk4":
        m = w.disk4_model(n_base=n_base, max_level=levels, n_bins=bins)
        m = dataclasses.replace(m, rho=m.rho * 1e-3, n_sed_dirs=dirs)
    else:
        m = w.disk_pah_model(n_base=n_base, max_level=levels, n_bins=bins, tau_v_mid=1.0)
    lo, hi = w.leaf_bounds_cm(m.tree, m.half_size)
    r = np.sqrt((((lo + hi) * 0.5) ** 2).sum(axis=1)) / (0.1 * m.half_size)
    T = np.clip(40.0 * np.maximum(r, 1e-3) ** -0.4, 5.0, 800.0).astype(np.float32)
    return m, np.ascontiguousarray(np.repeat(T[None], m.n_species, axis=0))


def _scaled(case, model, seed):
    """The case's model at an optical depth a few percent around the case's."""
    m, T = _model(model, case["n_base"], case["levels"], case["bins"], case.get("dirs", 1))
    rng = np.random.default_rng(seed)
    tau = case["tau"] * 10.0 ** rng.uniform(-0.02, 0.02)
    return dataclasses.replace(m, rho=m.rho * tau), T


@functools.lru_cache(maxsize=4)
def _batch(models, bins):
    got = w.batch_models(models, seed=0, n_bins=bins, sizes=(32, 48, 64))
    fields = {}
    for m, _ in got:
        key = id(m.tree)
        if key not in fields:
            lo, hi = w.leaf_bounds_cm(m.tree, m.half_size)
            r = np.sqrt((((lo + hi) * 0.5) ** 2).sum(axis=1)) / (0.1 * m.half_size)
            T = np.clip(40.0 * np.maximum(r, 1e-3) ** -0.4, 5.0, 800.0).astype(np.float32)
            fields[key] = np.repeat(T[None], m.n_species, axis=0)
    return [(m, n, fields[id(m.tree)]) for m, n in got]


def _grid(model, n_total, T):
    g = rt.Grid(model)
    g.emit_star(n_total)
    g.set_frozen_temperatures(T)
    return g


def _seed64(seed):
    return int(np.random.default_rng(seed + 77).integers(1, 1 << 60))


def _net_params(n_in, n_hidden, n_layers, n_out, rng, out_bias=None, out_scale=1.0):
    """Weights in the exchange layout: per layer W [out][in], then b [out]."""
    parts = []
    for l in range(n_layers + 1):
        a, b = (n_in if l == 0 else n_hidden), (n_out if l == n_layers else n_hidden)
        lim = math.sqrt(6.0 / a) * (out_scale if l == n_layers else 1.0)
        parts.append(rng.uniform(-lim, lim, size=a * b))
        bias = rng.uniform(-0.1, 0.1, size=b)
        parts.append(out_bias if l == n_layers and out_bias is not None else bias)
    return np.concatenate(parts).astype(np.float32)


def _net_rows(case, seed, rows):
    """Feature rows as the PAH cells give them, and targets of a smooth function."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    F = case["inputs"]
    X = torch.empty((rows, F), device="cuda").uniform_(-1.0, 1.0, generator=gen)
    X[:, F - 2].uniform_(0.2, 1.2, generator=gen)
    X[:, F - 1] = torch.where(torch.rand(rows, device="cuda", generator=gen) < 0.5,
                              math.log10(30) - 2, math.log10(200) - 2)
    return X


# ------------------------------------------------------------------ prepare

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("transport", "lucy", "images"):
        m, T = _scaled(case, case["model"], seed)
        n = case["packages"]
        g = _grid(m, n, T)
        s = {"kind": kind, "grid": g, "n": n, "seed": _seed64(seed),
             "counts": torch.zeros((g.S, g.N), dtype=torch.int64, device="cuda"),
             "T": torch.zeros((g.S, g.N), dtype=torch.float32, device="cuda"),
             "sed": torch.zeros((2, g.n_dir, g.B), dtype=torch.int64, device="cuda")}
        if kind == "lucy":
            s["tallies"] = torch.zeros((g.S, g.N), dtype=torch.float32, device="cuda")
        if kind == "images":
            lam = w.bin_centre_wavelength(m.nu_edges) / w.MICRON
            pob = np.full(g.B, -1, np.int32)
            for plane, um in enumerate((11.3, 10.0)):
                pob[int(np.argmin(np.abs(lam - um)))] = plane
            a = math.radians(case["incline"])
            g.set_images((0.0, math.sin(a), math.cos(a)), pob, case["pixels"], case["pixels"],
                         1.05 * m.half_size)
            s["images"] = torch.zeros(g.image_shape, dtype=torch.float64, device="cuda")
        return s
    if kind == "series":
        m, T = _scaled(case, case["model"], seed)
        return {"kind": kind, "model": m, "T": T, "n": case["packages"], "seed": _seed64(seed)}
    if kind == "batch":
        rng = np.random.default_rng(seed)
        grids, npk = [], []
        for m, n, T in _batch(case["models"], case["bins"]):
            n = max(1000, int(n * case["share"]))
            grids.append(_grid(dataclasses.replace(m, rho=m.rho * 10.0 ** rng.uniform(-.02, .02)),
                               n, T))
            npk.append(n)
        return {"kind": kind, "grids": grids,
                "batch": rt.Batch(grids, npk, seed=_seed64(seed), mode=rt.REEMIT_FROZEN),
                "T": [torch.zeros((g.S, g.N), dtype=torch.float32, device="cuda")
                      for g in grids],
                "counts": [torch.zeros((g.S, g.N), dtype=torch.int64, device="cuda")
                           for g in grids]}
    if kind == "pah":
        m, T = _scaled(case, "pah", seed)
        g = _grid(m, case["packages"], T)
        g.transport(case["packages"], seed=_seed64(seed), mode=rt.REEMIT_FROZEN)
        s = {"kind": kind, "grid": g, "net": None,
             "out": torch.zeros((g.N, g.B), dtype=torch.float32, device="cuda")}
        if case["surrogate"]:
            s["params"] = _pah_net(m, g.n_coarse, np.random.default_rng(seed))
            s["net"] = rt.MLP(g.n_coarse + 2, surrogate.N_HIDDEN, surrogate.N_LAYERS, g.B)
            s["net"].set_params(s["params"])
            # the range of absorbed powers it was trained on: all but the brightest and
            # the faintest hundredth of these cells
            x = np.concatenate([f["power"][f["power"] > -1e3] for f in _features(m, g)])
            s["range"] = tuple(float(np.float32(v)) for v in np.quantile(x, (0.01, 0.99)))
            s["net"].set_range(*s["range"])
        return s
    if kind == "forward":
        rng = np.random.default_rng(seed)
        net = rt.MLP(case["inputs"], case["hidden"], case["layers"], case["outputs"])
        p = _net_params(case["inputs"], case["hidden"], case["layers"], case["outputs"], rng)
        net.set_params(p)
        return {"kind": kind, "net": net, "params": p, "x": _net_rows(case, seed, case["rows"]),
                "y": torch.zeros((case["rows"], case["outputs"]), device="cuda")}
    if kind == "train":
        rng = np.random.default_rng(seed)
        net = rt.MLP(case["inputs"], case["hidden"], case["layers"], case["outputs"])
        p = _net_params(case["inputs"], case["hidden"], case["layers"], case["outputs"], rng)
        net.set_params(p)
        X = _net_rows(case, seed, case["rows"])
        A = torch.from_numpy(rng.normal(0, 0.3, (case["inputs"], case["outputs"])
                                        ).astype(np.float32)).cuda()
        return {"kind": kind, "net": net, "params": p, "X": X, "Y": torch.tanh(X @ A),
                "batch": case["batch"], "seed": seed & 0xffff}
    rng = np.random.default_rng(seed)
    nu = w.frequency_edges(case["bins"])
    cases, sig = [], []
    for i in range(case["cases"]):
        nc = int(rng.integers(30, 201))
        sp = w.pah_species(nu, nc)
        # the hardest photons always among them: they alone reach sublimation
        e = (1000.0 if i == 0 else 10.0 ** rng.uniform(math.log10(3.8), 3.0)) * EV
        flux = 10.0 ** rng.uniform(2.0, 6.0)
        cases.append({"modes": sp.modes, "h_nu": e, "rate": 2e-18 * nc * flux / e,
                      "t_top": 4000.0})
        sig.append(sp.kabs * sp.mol_mass)
    return {"kind": kind, "cases": cases, "nu": nu, "sigma": np.array(sig),
            "levels": case["levels"]}


# ------------------------------------------------------------------ run

def run(s):
    kind = s["kind"]
    if kind in ("transport", "lucy", "images"):
        g = s["grid"]
        g.reset()
        g.transport(s["n"], seed=s["seed"], mode=rt.REEMIT_FROZEN,
                    estimators=rt.EST_PATHLENGTH if kind == "lucy" else 0)
        g.counts(out=s["counts"])
        g.sed(out=s["sed"])
        out = {"counts": s["counts"], "sed": s["sed"]}
        if kind == "lucy":
            g.pathlength(out=s["tallies"])
            out["tallies"] = s["tallies"]
            out["T"] = g.temperatures_pathlength(out=s["T"])
        else:
            out["T"] = g.temperatures(out=s["T"])
        if kind == "images":
            out["images"] = g.images(out=s["images"])
        return out
    if kind == "series":
        with rt.Grid(s["model"]) as g:
            g.emit_star(s["n"])
            g.set_frozen_temperatures(s["T"])
            g.transport(s["n"], seed=s["seed"], mode=rt.REEMIT_FROZEN)
            return {"T": g.temperatures(), "counts": g.counts().view(np.int64),
                    "sed": g.sed()[0].view(np.int64)}
    if kind == "batch":
        s["batch"].run_graph()
        for i, g in enumerate(s["grids"]):
            s["batch"].temperatures(i, out=s["T"][i])
            g.counts(out=s["counts"][i])
        return {"T": s["T"], "counts": s["counts"]}
    if kind == "pah":
        if s["net"] is None:
            out, n = s["grid"].pah_emission(mode=rt.PAH_EXACT, out=s["out"])
        else:
            out, n = s["grid"].pah_emission(mode=rt.PAH_AUTO, surrogate=s["net"], tol=0.25,
                                            out=s["out"])
        return {"emission": out, "fallback": n}
    if kind == "forward":
        return s["net"].forward(s["x"], s["y"])
    if kind == "train":
        surrogate.train(s["net"], s["X"], s["Y"], epochs=1, batch=s["batch"], seed=s["seed"])
        return {"params": s["net"].get_params()}
    P, T, above, em = rt.pah_temperature_distribution(s["cases"], s["nu"], s["sigma"],
                                                      n_levels=s["levels"])
    return {"P": P, "T": T, "above": above, "emission": em}


# ------------------------------------------------------------------ work

def work(case):
    """Inputs read once and outputs written once. The operations of a transport are
    those of crossing cells: a package crosses about twice as many as lie along an edge,
    some forty operations each."""
    kind = case["kind"]
    if kind in ("transport", "lucy", "images", "series"):
        m, _ = _model(case["model"], case["n_base"], case["levels"], case["bins"],
                      case.get("dirs", 1))
        return _transport_work(m, case["packages"])
    if kind == "batch":
        each = [_transport_work(m, max(1000, int(n * case["share"])))
                for m, n, _ in _batch(case["models"], case["bins"])]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    if kind == "pah":
        m, _ = _model("pah", case["n_base"], case["levels"], case["bins"])
        N, B, M = m.tree.n_leaves, case["bins"], 400
        active = 0.045 * N   # the lit surface of the disk
        flops = active * 2 * ((2 * (66 * 256 + 2 * 256 * 256 + 256 * B)) if case["surrogate"]
                              else (M * M + 2 * M * B))
        return {"bytes": 4.0 * N * (1 + B) + active * 2 * 64 * 4, "flops": float(flops)}
    if kind in ("forward", "train"):
        per = case["inputs"] * case["hidden"] + (case["layers"] - 1) * case["hidden"] ** 2 + \
            case["hidden"] * case["outputs"]
        io = 4.0 * case["rows"] * (case["inputs"] + case["outputs"])
        if kind == "forward":
            return {"bytes": io + 2.0 * per, "flops": 2.0 * per * case["rows"]}
        steps = case["rows"] // case["batch"]
        return {"bytes": io + steps * 32.0 * per, "flops": 6.0 * per * steps * case["batch"]}
    n, M, B = case["cases"], case["levels"], case["bins"]
    return {"bytes": 8.0 * n * (2 * M + 2 * B), "flops": n * M * B * 60.0}


def _transport_work(m, packages):
    t, S = m.tree, m.n_species
    grid = 4.0 * (t.n_base ** 3 + 8 * t.n_blocks) + 8.0 * S * t.n_leaves
    return {"bytes": grid + 12.0 * S * t.n_leaves,
            "flops": packages * 2.0 * t.n_base * 40.0}


# ------------------------------------------------------------------ exact values

def exact(case, seed):
    """FP64 values of the PAH emission (from the absorbed spectra that prepare() leaves
    in the grid), the network, its training and the temperature distributions. The
    transports have none: their counts are whole numbers, and the sums and temperatures
    that go with them belong to those histories."""
    kind = case["kind"]
    if kind == "pah":
        s = prepare(case, seed)
        m, _ = _scaled(case, "pah", seed)
        with s["grid"] as g:
            out, n = _exact_emission(m, g, s.get("params"), s.get("range"))
        return {"emission": out, "fallback": None}
    if kind == "forward":
        s = prepare(case, seed)
        p = _layers(case, torch.from_numpy(s["params"]).cuda().double())
        return torch.cat([_net(p, x.double()) for x in s["x"].split(65536)])
    if kind == "train":
        return _exact_train(case, prepare(case, seed))
    if kind == "pt":
        s = prepare(case, seed)
        got = [_distribution(c, s["nu"], s["sigma"][i], s["levels"], 2500.0)
               for i, c in enumerate(s["cases"])]
        return {k: np.array([g[k] for g in got]) for k in ("P", "T", "above", "emission")}
    return None


def _layers(case, p):
    dims = [case["inputs"]] + [case["hidden"]] * case["layers"] + [case["outputs"]]
    out, o = [], 0
    for a, b in zip(dims[:-1], dims[1:]):
        out.append((p[o:o + a * b].view(b, a), p[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _net(layers, x):
    for i, (W, b) in enumerate(layers):
        x = x @ W.T + b
        if i + 1 < len(layers):
            x = torch.nn.functional.silu(x)
    return x


def _exact_train(case, s):
    p = torch.from_numpy(s["params"]).cuda().double().requires_grad_(True)
    X, Y, batch = s["X"].double(), s["Y"].double(), case["batch"]
    n = X.shape[0]
    gen = torch.Generator(device="cuda").manual_seed(s["seed"])
    perm = torch.randperm(n, generator=gen, device="cuda")
    steps, lr = max(1, n // batch), 2e-3
    decay = (2e-5 / lr) ** (1.0 / max(1, steps - 1))
    m1, m2 = torch.zeros_like(p), torch.zeros_like(p)
    for k in range(n // batch):
        idx = perm[k * batch:(k + 1) * batch]
        value = ((_net(_layers(case, p), X[idx]) - Y[idx]) ** 2).mean()
        g, = torch.autograd.grad(value, p)
        m1 = 0.9 * m1 + 0.1 * g
        m2 = 0.999 * m2 + 0.001 * g * g
        step = lr * decay ** k * (m1 / (1 - 0.9 ** (k + 1))) / \
            (torch.sqrt(m2 / (1 - 0.999 ** (k + 1))) + 1e-8)
        p = (p.detach() - step).requires_grad_(True)
    return {"params": p.detach().cpu().numpy()}


# integral of t^3 / (e^t - 1) from x to infinity: the exponential series where x is not
# small, else pi^4/15 less the integral from 0, by Gauss-Legendre (a smooth integrand)
def _planck_tail(x):
    x = np.asarray(x, dtype=np.float64)
    out = np.empty_like(x)
    big = x >= 0.5
    xb = x[big]
    acc = np.zeros_like(xb)
    for k in range(1, 91):
        acc += np.exp(-k * xb) * (xb ** 3 / k + 3 * xb ** 2 / k ** 2 + 6 * xb / k ** 3 +
                                  6.0 / k ** 4)
    out[big] = acc
    xs = x[~big]
    t, wt = np.polynomial.legendre.leggauss(20)
    u = 0.5 * xs[..., None] * (t + 1)
    out[~big] = math.pi ** 4 / 15 - (0.5 * xs[..., None] * wt * u ** 3 / np.expm1(u)).sum(-1)
    return out


def _planck_bins(nu, T):
    """Integral of B_nu over each bin, [len(T)][bins] (T > 0)."""
    x = H * nu[None, :] / (KB * T[:, None])
    G = _planck_tail(x)
    # bins below x = 1/2: the difference of the integrals from 0, without cancellation
    t, wt = np.polynomial.legendre.leggauss(12)
    a, b = x[:, :-1], x[:, 1:]
    u = 0.5 * (b - a)[..., None] * t + 0.5 * (a + b)[..., None]
    low = (0.5 * (b - a)[..., None] * wt * u ** 3 / np.expm1(np.minimum(u, 600.0))).sum(-1)
    d = np.where(b < 0.5, low, np.maximum(G[:, :-1] - G[:, 1:], 0.0))
    return 2 * (KB * T[:, None]) ** 4 / (H ** 3 * C ** 2) * d


def _heat(T, modes):
    e = np.zeros_like(T)
    for n, th in modes:
        x = th / T
        e += np.where(x < 700.0, n * KB * th / np.expm1(np.minimum(x, 700.0)), 0.0)
    return e


def _temperature_of(E, modes):
    lo, hi = np.full_like(E, 1e-3), np.full_like(E, 1e9)
    for _ in range(140):
        mid = np.sqrt(lo * hi)
        low = _heat(mid, modes) < E
        lo, hi = np.where(low, mid, lo), np.where(low, hi, mid)
    return np.sqrt(lo * hi)


def _levels(modes, nu, sigma, M, e_max):
    """Level spacing, temperatures, emission per bin and cooling rate per second."""
    dE = e_max / (M - 1)
    T = np.zeros(M)
    T[1:] = _temperature_of(np.arange(1, M) * dE, modes)
    s = np.zeros((M, nu.size - 1))
    s[1:] = 4 * math.pi * sigma[None, :] * _planck_bins(nu, T[1:])
    return dE, T, s, s.sum(axis=1) / dE


def _distribution(case, nu, sigma, M, t_sub):
    top = _heat(np.array([case["t_top"]]), case["modes"])[0]
    dE, T, s, cool = _levels(case["modes"], nu, sigma, M, top + case["h_nu"])
    x = case["h_nu"] / dE
    q, frac = int(math.floor(x)), x - math.floor(x)
    # rate of landing d or more levels up
    G = np.zeros(M + 1)
    G[1:min(q, M) + 1] += case["rate"] * (1 - frac)
    G[1:min(q + 1, M) + 1] += case["rate"] * frac
    P = np.zeros(M)
    P[0] = 1.0
    for f in range(1, M):
        P[f] = np.dot(G[1:f + 1], P[f - 1::-1]) / cool[f] if cool[f] > 0 else 0.0
        if P[f] > 1e200:
            P[:f + 1] *= 1e-200
    P /= P.sum()
    return {"P": P, "T": T, "above": P[T > t_sub].sum(), "emission": P @ s}


def _features(m, g):
    """Per PAH: absorbed spectra, molecules per cell, absorbed power and its feature."""
    K = g.n_coarse
    cnt = g.pah_absorbed(out=torch.zeros((g.n_pah, g.N, K), dtype=torch.int32, device="cuda"))
    eps = g.sed(out=torch.zeros((2, g.n_dir, g.B), dtype=torch.int64, device="cuda"))[1]
    size = m.cell_size_cm() * np.ldexp(1.0, -m.tree.leaf_level.astype(np.int64))
    out = []
    pahs = [i for i, sp in enumerate(m.species) if sp.is_pah]
    for p, i in enumerate(pahs):
        n_mol = m.rho[i] * size ** 3 / m.species[i].mol_mass
        tot = cnt[p].sum(dim=1).cpu().numpy().astype(np.float64)
        with np.errstate(divide="ignore", invalid="ignore"):
            power = np.where((tot > 0) & (n_mol > 0),
                             (np.log10(tot * eps / n_mol) + 12.0) / 4.0, -1e9)
        out.append({"species": m.species[i], "cnt": cnt[p], "n_mol": n_mol, "tot": tot,
                    "power": power, "eps": eps})
    return out


def _pah_net(m, K, rng):
    """A network whose prediction is near the emission of a PAH at some hundred kelvin."""
    sp = next(s for s in m.species if s.is_pah)
    q = sp.kabs * _planck_bins(m.nu_edges, np.array([500.0]))[0]
    bias = np.log(q / q.sum() + 1e-6) / 7.0 + 1.0
    return _net_params(K + 2, surrogate.N_HIDDEN, surrogate.N_LAYERS, m.n_bins, rng,
                       out_bias=bias, out_scale=0.01)


def _exact_emission(m, g, params, power_range):
    K, B, N, M = g.n_coarse, g.B, g.N, 400
    nu = m.nu_edges
    edge = [(k * B + K - 1) // K for k in range(K + 1)]
    e_k = np.array([H * math.sqrt(nu[edge[k]] * nu[edge[k + 1]]) for k in range(K)])
    feats = _features(m, g)
    present = [(f["tot"] > 0) & (f["n_mol"] > 0) for f in feats]
    solve = present[0] | present[1]
    out = torch.zeros((N, B), dtype=torch.float64, device="cuda")
    if params is not None:
        lo, hi = power_range
        fall = np.zeros(N, dtype=bool)
        q_of = []
        case = {"inputs": K + 2, "hidden": surrogate.N_HIDDEN, "layers": surrogate.N_LAYERS,
                "outputs": B}
        layers = _layers(case, torch.from_numpy(params).cuda().double())
        for f, here in zip(feats, present):
            rows = torch.from_numpy(np.flatnonzero(here)).cuda()
            a = f["cnt"][rows].double()
            a /= a.sum(dim=1, keepdim=True)
            x = torch.cat([torch.log(a + 1e-4) / 4.6 + 1.0,
                           torch.from_numpy(f["power"][here]).cuda()[:, None],
                           torch.full((rows.numel(), 1), math.log10(f["species"].n_carbon) - 2.0,
                                      dtype=torch.float64, device="cuda")], dim=1)
            q = torch.clamp(torch.exp(7.0 * (_net(layers, x) - 1.0)) - 1e-6, min=0.0)
            tot = q.sum(dim=1)
            pw = f["power"][here].astype(np.float32)
            fall[here] |= (np.abs(tot.cpu().numpy() - 1.0) > 0.25) | (pw < np.float32(lo)) | \
                (pw > np.float32(hi))
            q_of.append((rows, q / tot[:, None] *
                         torch.from_numpy(f["tot"][here] * f["eps"]).cuda()[:, None]))
        keep = torch.from_numpy(~fall).cuda()
        for rows, j in q_of:
            out[rows] += j * keep[rows][:, None]
        solve &= fall
    for f, here in zip(feats, present):
        sp = f["species"]
        dE, _, s, cool = _levels(sp.modes, nu, sp.kabs * sp.mol_mass, M,
                                 _heat(np.array([2500.0]), sp.modes)[0] + H * nu[-1])
        s = torch.from_numpy(s).cuda()
        x = e_k / dE
        q, frac = np.floor(x), x - np.floor(x)
        d = np.arange(1, M)
        land = torch.from_numpy((1 - frac)[:, None] * (q[:, None] >= d) +
                                frac[:, None] * (q[:, None] + 1 >= d)).cuda()   # [K][M-1]
        e = torch.from_numpy(e_k).cuda()
        cells = np.flatnonzero(solve & here)
        for c0 in range(0, cells.size, 32768):
            cc = cells[c0:c0 + 32768]
            n_mol = torch.from_numpy(f["n_mol"][cc]).cuda()
            rows = torch.from_numpy(cc).cuda()
            G = (f["cnt"][rows].double() * f["eps"] / n_mol[:, None] / e) @ land
            P = torch.zeros((cc.size, M), dtype=torch.float64, device="cuda")  # P[M-1-f]
            P[:, M - 1] = 1.0
            for lev in range(1, M):
                v = (G[:, :lev] * P[:, M - lev:]).sum(dim=1) / float(cool[lev]) \
                    if cool[lev] > 0 else torch.zeros_like(n_mol)
                P[:, M - 1 - lev] = v
                if lev % 8 == 0:
                    P *= torch.where(v > 1e100, 1e-100, 1.0)[:, None]
            P = P.flip(1)
            out[rows] += (n_mol / P.sum(dim=1))[:, None] * (P @ s)
    return out, int(solve.sum())
