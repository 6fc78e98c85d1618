"""Performance cases: what a program of this library has it do.

An opacity program uploads a line list, asks for the opacity at one or many
(T, P) conditions on a wavenumber grid, reduces each spectrum to
k-distribution tables and takes band transmissions from them; now and then it
trains the Voigt surrogate.  The sizes are those of the workloads in
``synth.py``, of the tests and of ``bench.py``.  Spectra and tables of the
FP64 form are returned as they are; those of the FP32 form, whose values
carry FP32 accuracy, are kept the way opacity tables are stored, in float32.
"""
import math

import numpy as np
import torch

from paper_1503_03806_gb300 import helk

BAR = 1.0 / 1.01325  # atm


def listed():
    full = dict(kind="opacity", nu_min=0.0, T=1500.0, P=1.0, strengths="loguniform", elower=False, species=1)
    cut100 = dict(cut="abs", cut_value=100.0, cut_cap=0.0)
    cut500 = dict(cut="lorentz", cut_value=500.0, cut_cap=100.0)
    logn = dict(strengths="lognormal", elower=True)
    return [
        # the smallest call: a few hundred lines on one short band, FP64, then its
        # tables; latency and launches count (the size of the smoke run)
        dict({**full, "T": 1800.0, "P": 0.5, "elower": True, "kind": "spectrum"}, name="band_f64_300",
             precision="f64", nlines=300, ngrid=10_000, dnu=0.01, cut="lorentz", cut_value=500.0, cut_cap=20.0,
             nbins=10, ncheb=20),
        # a molecule's band, FP64: the "small" workload
        dict(**full, name="small_f64", precision="f64", nlines=10_000, ngrid=300_000, dnu=0.01, cut="abs",
             cut_value=25.0, cut_cap=0.0),
        # a whole spectrum in the reference form: the "medium" workload
        dict({**full, **cut100}, name="medium_f64", precision="f64", nlines=100_000, ngrid=3_000_000, dnu=0.01),
        # one step of a retrieval or an atmosphere: spectrum and k-tables of one
        # layer, FP32 form: the "medium" workload
        dict({**full, **cut100, "kind": "spectrum"}, name="medium_step_f32", precision="f32", nlines=100_000,
             ngrid=3_000_000, dnu=0.01, nbins=300, ncheb=20),
        # an opacity table over temperatures and pressures: 1e6 lines, 3 x 4 of the
        # "tp_grid" workload's range, one batch call
        dict({**full, **cut500, **logn, "kind": "batch"}, name="tp_batch_f32", precision="f32", nlines=1_000_000,
             ngrid=3_000_000, dnu=0.01, nT=3, nP=4),
        # the longest list of one molecule on the whole range: the "surrogate"
        # workload's 1e7 lines, FP32 form
        dict({**full, **cut500, **logn}, name="dense_f32_1e7", precision="f32", nlines=10_000_000, ngrid=3_000_000,
             dnu=0.01),
        # four species on the fine grid of the "mixed" workload, a tenth of its range
        # and a hundredth of its lines, hot upper layer
        dict({**full, **cut500, **logn, "nu_min": 12_000.0, "T": 2200.0, "P": 0.1 * BAR, "species": 4},
             name="mixed_fine_f32", precision="f32", nlines=1_000_000, ngrid=2_999_999, dnu=0.001),
        # a new list read from disk (host arrays, several species one after the
        # other) through to tables on the host: upload, opacity, k-tables
        dict({**full, **logn, "species": 4, "kind": "whole"}, name="new_list_f32", precision="f32", nlines=200_000,
             ngrid=300_000, dnu=0.01, cut="lorentz", cut_value=500.0, cut_cap=25.0, nbins=30, ncheb=20),
        # k-tables of several spectra at once: bins of 10000 points (eight layers of
        # the "medium" workload)
        dict(name="ktables_2400x10000", kind="ktables", nbins=2400, nb=10_000, ncheb=20, gaps=0.0, kg=False),
        # k-tables of the fine grid: bins of 30000 points, the sorted k(g) kept
        dict(name="ktables_1000x30000", kind="ktables", nbins=1000, nb=30_000, ncheb=20, gaps=0.1, kg=True),
        # the transmission stage: every bin of the "medium" workload, 1000 column
        # masses, from k(g) and from the fit
        dict(name="transmission_300x1000", kind="transmission", nbins=300, nb=10_000, ncheb=20, nm=1000, ng=1000),
        # surrogate training: one pass over fresh samples
        dict(name="surrogate_epoch", kind="train", samples=262_144, batch=4096),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["opacity", "opacity", "opacity", "spectrum", "batch", "whole", "ktables", "transmission",
                       "train"])
    if kind == "ktables":
        nb = int(_log(rng, 300, 40_000))
        return dict(kind=kind, nb=nb, nbins=max(1, int(_log(rng, 3e4, 2.4e7) / nb)),
                    ncheb=rng.choice([5, 12, 20, 24]), gaps=rng.choice([0.0, 0.0, 0.3]), kg=rng.random() < 0.5)
    if kind == "transmission":
        return dict(kind=kind, nbins=int(_log(rng, 10, 300)), nb=int(_log(rng, 500, 10_000)),
                    ncheb=rng.choice([12, 20]), nm=int(_log(rng, 30, 1000)), ng=rng.choice([333, 1000]))
    if kind == "train":
        return dict(kind=kind, samples=int(_log(rng, 33_000, 262_000)), batch=rng.choice([1024, 4096]))
    c = dict(kind=kind, nu_min=rng.choice([0.0, 500.0, 8000.0]), T=rng.uniform(300.0, 3000.0), P=_log(rng, 1e-5, 100.0),
             species=rng.choice([1, 1, 4]), precision=rng.choice(["f64", "f32"]), dnu=rng.choice([0.001, 0.01, 0.01]),
             nlines=int(_log(rng, 300, 1e6)), ngrid=int(_log(rng, 1e4, 3e6)),
             **rng.choice([dict(strengths="loguniform", elower=False), dict(strengths="lognormal", elower=True)]),
             **rng.choice([dict(cut="abs", cut_value=25.0, cut_cap=0.0), dict(cut="abs", cut_value=100.0, cut_cap=0.0),
                           dict(cut="lorentz", cut_value=500.0, cut_cap=100.0),
                           dict(cut="none", cut_value=0.0, cut_cap=0.0)]))
    if kind == "batch":
        c.update(nT=rng.choice([1, 2, 4]), nP=rng.choice([2, 3]))
    if kind == "spectrum" or kind == "whole":
        c.update(nbins=max(1, c["ngrid"] // rng.choice([1000, 5000, 10_000, 30_000])), ncheb=20)
        c["ngrid"] -= c["ngrid"] % c["nbins"]
    most = 1.5e9 if c["precision"] == "f64" else 2.0e10
    while _pairs(c) > most:  # no more work than the largest listed case of the form
        c["nlines"] = max(300, c["nlines"] // 2)
        if c["nlines"] == 300:
            c["cut"], c["cut_value"] = "abs", 25.0
    return c


# ------------------------------------------------------------- the sizes --
def _conditions(c):
    if c["kind"] != "batch":
        return [(c["T"], c["P"])]
    T = np.linspace(500.0, 3000.0, c["nT"])
    P = np.logspace(-5.0, 2.0, c["nP"]) * BAR
    return [(float(t), float(p)) for t in T for p in P]


def _mean_window(c, T, P):
    if c["cut"] == "none":
        return float(c["ngrid"])
    half = c["cut_value"]
    if c["cut"] == "lorentz":
        half = min(c["cut_value"] * 0.06 * P * math.sqrt(296.0 / T), c["cut_cap"])
    return min(float(c["ngrid"]), 2.0 * half / c["dnu"] + 1.0)


def _pairs(c):
    return sum(c["nlines"] * _mean_window(c, T, P) for T, P in _conditions(c))


def work(case):
    c = case
    if c["kind"] == "ktables":
        n = c["nbins"] * c["nb"]
        return {"bytes": n * (16.0 if c["kg"] else 8.0) + c["nbins"] * (c["ncheb"] + 1) * 8.0,
                "flops": n * (2.0 * c["ncheb"] + 20.0)}
    if c["kind"] == "transmission":
        # the terms within e^-87 of a bin's largest: about half of them over these
        # column masses
        terms = c["nbins"] * c["nm"] * (0.5 * c["nb"] + c["ng"])
        return {"bytes": c["nbins"] * 8.0 * (c["nb"] + c["ncheb"] + 2 * c["nm"]), "flops": terms}
    if c["kind"] == "train":
        # forward and backward multiply-adds of the 2-64-64-64-1 network
        return {"bytes": 8577 * 8.0, "flops": c["samples"] * 3 * 2 * 8384.0}
    # Opacity: the line fields read and the spectrum written once.  Arithmetic:
    # the parameters of each line, its core points (a^2 + u^2 < 100, one
    # evaluation of the profile there) and the sum at each point; the wings are
    # smooth and have no such count of their own.
    fields = 3 + (1 if c["elower"] else 0) + (2 if c["species"] > 1 else 0)
    conds = _conditions(c)
    core = 0.0
    for T, P in conds:
        mid = c["nu_min"] + 0.5 * c["ngrid"] * c["dnu"]
        core += c["nlines"] * min(_mean_window(c, T, P), 24.0 * mid * 3.27e-6 * math.sqrt(T / 1500.0) / c["dnu"])
    out = 8.0 if c["precision"] == "f64" else 4.0
    return {"bytes": fields * 8.0 * c["nlines"] + out * c["ngrid"] * len(conds),
            "flops": len(conds) * (100.0 * c["nlines"] + 2.0 * c["ngrid"]) + 60.0 * core}


# ------------------------------------------------------------- the inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _lines(c, seed):
    """A line list as synth.py draws them (uniform centres, log-uniform or
    log-normal strengths, gamma in [0.02, 0.1]), on the device; several species
    one after the other, each ordered by wavenumber."""
    g, out = _gen(seed), {}

    def uni(n, lo, hi):
        return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo

    # centres over the grid's range, kept off zero where ranges start there
    lo, hi = max(c["nu_min"], 0.05), c["nu_min"] + c["ngrid"] * c["dnu"]
    parts = []
    for s in range(c["species"]):
        n = c["nlines"] // c["species"] + (1 if s < c["nlines"] % c["species"] else 0)
        d = {"nu0": torch.sort(uni(n, lo, hi)).values}
        if c["strengths"] == "lognormal":
            x = torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * 3.0 - 24.0
            d["S0"] = torch.where((x < -30.0) | (x > -18.0), uni(n, -28.0, -20.0), x)
        else:
            d["S0"] = uni(n, -26.0, -19.0)
        d["S0"] = 10.0 ** d["S0"]
        d["gamma_air"] = uni(n, 0.02, 0.1)
        if c["elower"]:
            d["E_lower"] = uni(n, 0.0, 1.0e4)
        if c["species"] > 1:
            d["mass"] = torch.full((n,), (18.0, 16.0, 44.0, 17.0)[s], dtype=torch.float64, device="cuda")
            d["weight"] = torch.full((n,), 0.25, dtype=torch.float64, device="cuda")
        parts.append(d)
    for k in parts[0]:
        out[k] = torch.cat([p[k] for p in parts]).contiguous()
    return out


def _spectrum(nbins, nb, gaps, seed):
    """An opacity-like spectrum: one line in 30 points, strengths over seven
    decades, Lorentz widths of 2-10 points, each point the sum of the 24 lines
    about it on either side; `gaps`: the share of the range without opacity."""
    g, n = _gen(seed), nbins * nb
    m = n // 30 + 64
    x = torch.sort(torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * n).values
    S = 10.0 ** (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * 7.0 - 26.0)
    w = torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * 8.0 + 2.0
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    at = torch.searchsorted(x, i)
    k = torch.zeros(n, device="cuda", dtype=torch.float64)
    for o in range(-24, 24):
        j = (at + o).clamp_(0, m - 1)
        k += S[j] * w[j] / ((i - x[j]) ** 2 + w[j] ** 2)
    if gaps > 0.0:  # stretches of 700 points
        dark = torch.rand(n // 700 + 1, generator=g, device="cuda") < gaps
        k = torch.where(dark.repeat_interleave(700)[:n], torch.zeros_like(k), k)
    return k


def _chebyshev(nb, ncheb):
    t = (2.0 * torch.arange(nb, dtype=torch.float64, device="cuda") + 1.0) / nb - 1.0
    cols = [torch.ones_like(t), t]
    while len(cols) < ncheb:
        cols.append(2.0 * t * cols[-1] - cols[-2])
    return torch.stack(cols[:ncheb], dim=1)


def _fit(k_sorted, ncheb, floor=1e-250):
    """Least-squares Chebyshev coefficients of ln k(g), [nbins, ncheb]."""
    L = torch.log(torch.clamp(k_sorted, min=floor))
    Q, R = torch.linalg.qr(_chebyshev(L.shape[1], ncheb))
    return torch.linalg.solve_triangular(R, Q.T @ L.T, upper=True).T.contiguous()


def _masses(c):
    return np.logspace(14.0, 30.0, c["nm"])


def prepare(case, seed):
    c, s = case, {"case": case}
    s["ctx"] = ctx = helk.Context(0)
    if c["kind"] == "ktables":
        s["kappa"] = _spectrum(c["nbins"], c["nb"], c["gaps"], seed)
    elif c["kind"] == "transmission":
        k = _spectrum(c["nbins"], c["nb"], 0.0, seed).view(c["nbins"], c["nb"])
        s["sorted"] = torch.sort(k, dim=1).values.contiguous()
        s["coef"] = _fit(s["sorted"], c["ncheb"])
        s["m"] = _masses(c)
    elif c["kind"] == "train":
        ctx.surrogate_init(seed)
        s["params"], s["seed"] = ctx.surrogate_params(), int(seed) + 1
    else:
        lines = _lines(c, seed)
        s["prec"] = helk.HELK_PREC_F64 if c["precision"] == "f64" else helk.HELK_PREC_F32_KAHAN
        s["grid"] = (c["nu_min"], c["dnu"], c["ngrid"])
        s["cut"] = {"abs": ("abs", c["cut_value"]), "lorentz": ("lorentz", c["cut_value"], c["cut_cap"]),
                    "none": ("none",)}[c["cut"]]
        conds = _conditions(c)
        s["T"], s["P"] = np.array([t for t, _ in conds]), np.array([p for _, p in conds])
        s["q"] = (296.0 / s["T"]) ** 1.5
        if c["kind"] == "whole":
            s["lines"] = {k: v.cpu().numpy() for k, v in lines.items()}
        else:
            ctx.upload(lines)
        shape = (len(conds), c["ngrid"]) if c["kind"] == "batch" else (c["ngrid"],)
        s["out"] = torch.empty(shape, dtype=torch.float64, device="cuda")
    return s


# --------------------------------------------------------------- one pass --
def run(state):
    s = state
    c, ctx = s["case"], s["ctx"]
    if c["kind"] == "ktables":
        coef, mean, kg = ctx.kdist(s["kappa"], c["nbins"], c["ncheb"], want_sorted=c["kg"])
        return {"coef": coef, "mean": mean, "sorted": kg}
    if c["kind"] == "transmission":
        direct, fit = ctx.transmission(c["nbins"], s["m"], sorted_k=s["sorted"], coeffs=s["coef"], ng=c["ng"])
        return {"direct": direct, "fit": fit}
    if c["kind"] == "train":
        ctx.surrogate_params(new=s["params"])
        loss = ctx.surrogate_train(c["samples"], s["seed"], 1, c["batch"], 2e-3)
        return {"params": ctx.surrogate_params(), "loss": np.float32(loss)}
    if c["kind"] == "batch":
        k = ctx.opacity_batch(s["T"], s["P"], 18.0, s["cut"], s["grid"], out=s["out"], precision=s["prec"],
                              q_ratio=s["q"])
        return {"kappa": list((k if c["precision"] == "f64" else k.float()).unbind(0))}
    if c["kind"] == "whole":
        ctx.upload(s["lines"])
    k = ctx.opacity(c["T"], c["P"], 18.0, s["cut"], s["grid"], out=s["out"], precision=s["prec"],
                    q_ratio=float(s["q"][0]))
    out = {"kappa": k if c["precision"] == "f64" else k.float()}
    if c["kind"] != "opacity":
        coef, mean, _ = ctx.kdist(k, c["nbins"], c["ncheb"], on_host=c["kind"] == "whole")
        if c["precision"] == "f32":
            coef, mean = ((coef.astype(np.float32), mean.astype(np.float32)) if c["kind"] == "whole"
                          else (coef.float(), mean.float()))
        out.update(coef=coef, mean=mean)
    return out


# ------------------------------------------------- the same in 64 bits --
EXACT_PAIRS = 3.0e10  # (line, point) pairs that take about twenty seconds


def _voigt(x, y):
    """K(x, y) by the trapezoidal rule with the pole's residue, h = 1/2."""
    h, x = 0.5, x.abs()
    ex2 = torch.exp(-x * x)
    s, co = torch.sin(x * y), torch.cos(2.0 * x * y)
    sinc = torch.where(x * y == 0.0, torch.ones_like(x), s / (x * y))
    S1, S23 = torch.zeros_like(x), torch.zeros_like(x)
    for n in range(1, 34):
        d = (n * h) ** 2 + y * y
        S1 += math.exp(-((n * h) ** 2)) / d
        S23 += (torch.exp(-((n * h + x) ** 2)) + torch.exp(-((n * h - x) ** 2))) / d
    K = ex2 * torch.special.erfcx(y) * co + (2.0 * h / math.pi) * x * ex2 * s * sinc
    return K + (2.0 * h / math.pi) * (0.5 * y * S23 - y * co * ex2 * S1)


def _exact_kappa(c, L, T, P, q):
    """The opacity of lines L (tensors) at (T, P), or None when it would take long."""
    ln2, kb, amu, cl, c2 = math.log(2.0), 1.380649e-16, 1.66053906660e-24, 2.99792458e10, 1.4387768775039338
    nu0, S, g = L["nu0"], L["S0"], L["gamma_air"]
    if c["elower"]:
        S = S * q * torch.exp(-c2 * L["E_lower"] / T + c2 * L["E_lower"] / 296.0)
        S = S * (torch.expm1(-c2 * nu0 / T) / torch.expm1(-c2 * nu0 / 296.0))
    mass = torch.full_like(nu0, 18.0)
    if c["species"] > 1:
        S, mass = S * L["weight"], L["mass"]
    gL = math.sqrt(296.0 / T) * (g * (P - 0.5 * P) + g * (0.5 * P))
    gD = nu0 * (torch.sqrt(2.0 * ln2 * kb * T / (mass * amu)) / cl)
    a, ku, Sp = math.sqrt(ln2) * gL / gD, math.sqrt(ln2) / gD, S * math.sqrt(ln2 / math.pi) / gD
    n, dnu, nu_min = c["ngrid"], c["dnu"], c["nu_min"]
    if c["cut"] == "none":
        lo, hi = torch.zeros_like(nu0), torch.full_like(nu0, n - 1.0)
    else:
        C = torch.full_like(nu0, c["cut_value"])
        if c["cut"] == "lorentz":
            C = torch.clamp(c["cut_value"] * gL, max=c["cut_cap"])
        lo = torch.ceil((nu0 - C - nu_min) / dnu).clamp(0.0, float(n))
        hi = torch.floor((nu0 + C - nu_min) / dnu).clamp(-1.0, n - 1.0)
    lo, cnt = lo.long(), (hi.long() - lo.long() + 1).clamp(min=0)
    if int(cnt.sum()) > EXACT_PAIRS:
        return None
    kappa = torch.zeros(n, dtype=torch.float64, device=nu0.device)
    ends = torch.cumsum(cnt, 0)
    l0, done, total = 0, 0, int(cnt.sum())
    while done < total:
        l1 = int(torch.searchsorted(ends, torch.tensor(done + (1 << 25), device=ends.device), right=True))
        l1 = max(l1, l0 + 1)
        l = torch.repeat_interleave(torch.arange(l0, l1, device=nu0.device), cnt[l0:l1])
        start = ends[l0:l1] - cnt[l0:l1] - done
        i = lo[l] + torch.arange(l.numel(), device=nu0.device) - start[l - l0]
        u = ((nu_min + i.double() * dnu) - nu0[l]) * ku[l]
        al = a[l]
        r2 = u * u + al * al
        t = math.sqrt(1.5)
        gh3 = 4.0 / r2 + 1.0 / ((u - t) ** 2 + al * al) + 1.0 / ((u + t) ** 2 + al * al)
        H = torch.where(r2 >= 1.0e6, al / (math.sqrt(math.pi) * r2), gh3 * (al * (math.sqrt(math.pi) / 6.0) / math.pi))
        core = torch.nonzero(r2 < 100.0).squeeze(1)
        for part in core.split(1 << 23):
            H[part] = _voigt(u[part], al[part])
        kappa.index_add_(0, i, Sp[l] * H)
        done = int(ends[l1 - 1])
        l0 = l1
    return kappa


def _exact_tables(k, nbins, ncheb):
    k_sorted = torch.sort(k.view(nbins, -1), dim=1).values
    return _fit(k_sorted, ncheb), k_sorted.mean(dim=1), k_sorted


def exact(case, seed):
    c = case
    if c["kind"] == "train":
        return None
    if c["kind"] == "ktables":
        coef, mean, k = _exact_tables(_spectrum(c["nbins"], c["nb"], c["gaps"], seed), c["nbins"], c["ncheb"])
        return {"coef": coef, "mean": mean, "sorted": k.view(-1) if c["kg"] else None}
    if c["kind"] == "transmission":
        k = torch.sort(_spectrum(c["nbins"], c["nb"], 0.0, seed).view(c["nbins"], c["nb"]), dim=1).values
        m = torch.from_numpy(_masses(c)).cuda()
        kf = torch.exp(_fit(k, c["ncheb"]) @ _chebyshev(c["ng"], c["ncheb"]).T)
        return {w: torch.stack([torch.exp(-v[b][None, :] * m[:, None]).mean(dim=1) for b in range(c["nbins"])])
                for w, v in (("direct", k), ("fit", kf))}
    L = _lines(c, seed)
    if c["kind"] == "batch":
        left, rows = EXACT_PAIRS, []
        for T, P in _conditions(c):  # the conditions with the shorter windows
            cost = c["nlines"] * _mean_window(c, T, P)
            rows.append(_exact_kappa(c, L, T, P, (296.0 / T) ** 1.5) if cost <= left else None)
            left -= cost if rows[-1] is not None else 0.0
        return {"kappa": rows}
    k = _exact_kappa(c, L, c["T"], c["P"], (296.0 / c["T"]) ** 1.5)
    if k is None or c["kind"] == "opacity":
        return None if k is None else {"kappa": k}
    coef, mean, _ = _exact_tables(k, c["nbins"], c["ncheb"])
    return {"kappa": k, "coef": coef, "mean": mean}
