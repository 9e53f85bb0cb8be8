"""The performance cases: what a user of the library has it compute.

Every case goes through the public binding (``paper_1708_01608_gb300.lbm``)
and stands for one of seven uses:

``foam``    a foam run: time steps in diagnostic intervals (totals, labels,
            merge bookkeeping, film test, bubble census), then a dump of the
            density field in the precision the lattice stores;
``disks``   the two-disk run: steps, then density, pressure, the pressure
            Laplacian along the gap and the gas labels;
``rupture`` a seeded pair of bubbles advanced under the film probe;
``sweep``   a batched ensemble of two-bubble domains run to its end;
``multi``   the multi-lattice model under the film probe;
``static``  the allocation-free step on the caller's own device buffers;
``survey``  the analysis of a foam state: labels, census, film pairs, fields.

Lattices run on the plan the library picks by itself: a program that calls
``lbm_autotune`` first pays seconds for it, which only the longest runs
repay.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1708_01608_gb300 import lbm
from paper_1708_01608_gb300 import workloads as W

BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
# a field dump keeps the precision the lattice stores
DUMP = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16,
        "bf16": torch.bfloat16}
H_MAX, EPS_ARM, FIRED_CAP, BINS = 12, 1e-3, 4096, 32


# ---- the cases ---------------------------------------------------------------

def _foam(name, lattice, nx, ny, nz, storage, tau, *, residual=False, rho_l=1.8, sites=0,
          r_min=4.0, r_max=12.0, spacing=0.0, gap=4.0, rate=0.0, budget=0.0, intervals=1,
          steps=100, dump=True):
    case = dict(kind="foam", lattice=lattice, nx=nx, ny=ny, nz=nz, storage=storage, tau=tau,
                residual=residual, rho_l=rho_l, sites=sites, r_min=r_min, r_max=r_max,
                spacing=spacing, gap=gap, rate=rate, budget=budget, intervals=intervals,
                steps=steps, dump=dump)
    return dict(case, name=name) if name else case


def listed():
    f128, f512, f768 = W.FOAM_128, W.FOAM_512, W.FOAM_768
    nuclei = dict(rho_l=f128["rho_l"], sites=f128["sites"]["n"], r_min=3.0, r_max=3.0,
                  spacing=12.0, gap=0.0, rate=f128["rate"], budget=f128["budget"])
    bubbles = dict(rho_l=f512["rho_l"], sites=f512["sites"]["n"], r_min=4.0, r_max=12.0,
                   spacing=0.0, gap=4.0)
    full = dict(rho_l=f768["rho_l"], sites=f768["sites"]["n"], r_min=3.0, r_max=3.0,
                spacing=12.0, gap=0.0, rate=f768["rate"], budget=50.0)
    return [
        # 128^3 foam of injecting nuclei: five diagnostic intervals and a dump
        _foam("foam128_f32", "D3Q19", 128, 128, 128, "f32", f128["tau"], intervals=5, **nuclei),
        # the same foam in FP64, the reference precision: one interval
        _foam("foam128_f64", "D3Q19", 128, 128, 128, "f64", f128["tau"], **nuclei),
        # the benchmark foam: one interval of 512^3, its labels to the host
        _foam("foam512_f32", "D3Q19", 512, 512, 512, "f32", f512["tau"], dump=False, **bubbles),
        # the same foam in 16-bit offset storage
        _foam("foam512_f16", "D3Q19", 512, 512, 512, "f16", f512["tau"], dump=False, **bubbles),
        # the full foam: 4096 injecting nuclei, 16-bit storage that keeps mass
        _foam("foam768_f16r", "D3Q19", 768, 768, 768, "f16", f768["tau"], residual=True,
              dump=False, **full),
        # a box cut to a sample's own size: no extent a multiple of anything
        _foam("foam_ragged_f32", "D3Q19", 201, 150, 99, "f32", 0.8, sites=22, intervals=2),
        # two disks at a 4-cell gap, FP64 (the paper's Fig. 2): small and
        # latency-bound, fields and labels read every 100 steps
        dict(name="two_disks_128_f64", kind="disks", side=128, radius=20.0, gap=4.0, tau=1.0,
             storage="f64", steps=100),
        # one domain of the bubble-size sweep by itself, probed every 20 steps
        dict(name="rupture_200_f32", kind="rupture", side=200, radius=40.0, gap=6.0, tau=0.8,
             storage="f32", every=20, steps=1000),
        # the 256-domain sweep (Fig. 3) run to completion
        dict(name="sweep_256", kind="sweep", n=256, side_min=64, side_max=512, steps=20000),
        # the multi-lattice model at a middle bubble size (R_b = 20, L = 104)
        dict(name="multi_104_f64", kind="multi", lattice="D2Q9", side=104, depth=1, radius=20.0,
             gap=4.0, nl=3, storage="f64", every=20, steps=600),
        # the allocation-free step on a caller's own FP32 buffers
        dict(name="static_f32", kind="static", lattice="D3Q19", nx=127, ny=101, nz=90, tau=0.9,
             steps=10),
        # what a foam run reports at one state of 256^3
        dict(name="survey_256_f32", kind="survey", nx=256, ny=256, nz=256, storage="f32",
             tau=0.8, sites=125),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extent(rng, base):
    """An extent near base: a multiple of 8 in half of the draws, else any."""
    n = max(16, int(base * rng.uniform(0.6, 1.5)))
    return (n + 7) // 8 * 8 if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["foam", "foam", "foam", "disks", "rupture", "sweep", "multi", "static",
                       "survey"])
    tau = rng.choice([0.8, 0.9, 1.0, round(rng.uniform(0.7, 1.0), 3)])
    if kind == "foam":
        storage = rng.choice(["f64", "f32", "f32", "f16", "f16", "bf16"])
        residual = storage in ("f16", "bf16") and rng.random() < 0.4
        if rng.random() < 0.25:  # plane foams
            base = _log(rng, 64, 512 if storage == "f64" else 2500)
            nx, ny = _extent(rng, base), _extent(rng, base)
            return _foam(None, "D2Q9", nx, ny, 1, storage, tau, residual=residual, rho_l=2.0,
                         sites=max(1, nx * ny // 6000), r_min=8.0, r_max=16.0, gap=3.0,
                         intervals=rng.choice([1, 2]))
        base = _log(rng, 32, 96 if storage == "f64" else 340)
        nx, ny, nz = (_extent(rng, base) for _ in range(3))
        cells = nx * ny * nz
        inject = rng.random() < 0.5
        return _foam(None, "D3Q19", nx, ny, nz, storage, tau, residual=residual,
                     sites=max(1, cells // 130000), r_max=rng.choice([6.0, 9.0, 12.0]),
                     rate=1e-4 if inject else 0.0, budget=50.0 if inject else 0.0,
                     intervals=1 if cells > 4000000 else rng.choice([1, 2]),
                     steps=rng.choice([50, 100]))
    if kind == "disks":
        side = int(_log(rng, 64, 320))
        gap = rng.uniform(3.0, 8.0)
        return dict(kind="disks", side=side, radius=round((side - 2 * gap) / 4 - 2, 2),
                    gap=round(gap, 2), tau=tau, storage=rng.choice(["f64", "f64", "f32"]),
                    steps=rng.choice([50, 100, 200]))
    if kind == "rupture":
        side = int(_log(rng, 64, 512))
        gap = rng.uniform(5.0, 10.0)
        return dict(kind="rupture", side=side,
                    radius=round(min(60.0, (side - 2 * gap) / 4 - 2), 2), gap=round(gap, 2),
                    tau=tau, storage=rng.choice(["f32", "f32", "f64"]) if side < 300 else "f32",
                    every=rng.choice([10, 20, 50]), steps=rng.choice([200, 400, 1000]))
    if kind == "sweep":
        n = int(_log(rng, 8, 256))
        lo = rng.choice([64, 96])
        return dict(kind="sweep", n=n, side_min=lo, side_max=rng.choice([128, 256, 512]),
                    steps=rng.choice([1000, 4000, 20000]))
    if kind == "multi":
        if rng.random() < 0.3:
            side = rng.choice([32, 40, 47, 64])
            return dict(kind="multi", lattice="D3Q19", side=side, depth=rng.choice([24, 33, 48]),
                        radius=round(side / 4 - 2.0, 2), gap=4.0, nl=3,
                        storage=rng.choice(["f64", "f32"]), every=20, steps=100)
        radius = round(rng.uniform(8.0, 38.0), 1)
        return dict(kind="multi", lattice="D2Q9", side=int(4 * radius + 24) + rng.randrange(8),
                    depth=1, radius=radius, gap=4.0, nl=3, storage=rng.choice(["f64", "f64", "f32"]),
                    every=rng.choice([10, 20]), steps=rng.choice([200, 400, 600]))
    if kind == "static":
        if rng.random() < 0.4:
            return dict(kind="static", lattice="D2Q9", nx=int(_log(rng, 48, 1400)),
                        ny=int(_log(rng, 48, 1400)), nz=1, tau=tau, steps=rng.choice([1, 10]))
        base = _log(rng, 24, 100)
        return dict(kind="static", lattice="D3Q19", nx=min(127, _extent(rng, base)),
                    ny=min(127, _extent(rng, base)), nz=min(127, _extent(rng, base)), tau=tau,
                    steps=rng.choice([1, 10]))
    base = _log(rng, 64, 220)
    nx, ny, nz = (_extent(rng, base) for _ in range(3))
    return dict(kind="survey", nx=nx, ny=ny, nz=nz, storage=rng.choice(["f32", "f32", "f16"]),
                tau=tau, sites=max(2, nx * ny * nz // 130000))


# ---- inputs --------------------------------------------------------------------

def _pair(case):
    """Two disks (spheres) on the middle line at a surface distance gap, and
    the probe line from centre to centre."""
    n, r, gap = case["side"], case["radius"], case["gap"]
    depth = case.get("depth", 1)
    c1, c2 = n / 2 - r - gap / 2, n / 2 + r + gap / 2
    zc = float(depth // 2) if depth > 1 else 0.0
    bub = np.array([[c1, float(n // 2), zc, r], [c2, float(n // 2), zc, r]])
    x0 = int(math.floor(c1))
    return bub, (x0, n // 2, int(zc), 0, int(math.ceil(c2)) - x0 + 1)


def _sites(case, seed):
    nz = case.get("nz", 1)
    return lbm.sample_sites(case["nx"], case["ny"], nz, case["sites"], case.get("r_min", 4.0),
                            case.get("r_max", 12.0), case.get("spacing", 0.0),
                            case.get("gap", 4.0), seed)


def _static_rho(case, seed):
    """A noisy liquid with one gas ball, as FP32 densities on the GPU."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ax = [torch.arange(n, dtype=torch.float64) - n / 2 for n in (nx, ny, nz)]
    d = torch.sqrt(ax[0][None, None, :] ** 2 + ax[1][None, :, None] ** 2
                   + (ax[2][:, None, None] ** 2 if nz > 1 else 0.0))
    rho = 0.15 + 0.5 * 1.65 * (1.0 + torch.tanh(d - min(nx, ny) / 5))
    return rho + 1e-3 * (2.0 * torch.rand(rho.shape, generator=g, dtype=torch.float64) - 1.0)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "foam":
        L = lbm.Lattice(case["lattice"], case["nx"], case["ny"], case["nz"], tau=case["tau"],
                        storage=case["storage"], rho_ref=case["rho_l"],
                        mass_residual=case["residual"])
        bub = _sites(case, seed)
        L.seed_bubbles(bub, case["rho_l"], 0.15, 2.0, 1e-3, seed)
        if case["rate"] > 0:
            L.inject(np.full(len(bub), case["rate"]), np.full(len(bub), case["budget"]))
        return dict(case=case, L=L)
    if kind == "survey":
        L = lbm.Lattice("D3Q19", case["nx"], case["ny"], case["nz"], tau=case["tau"],
                        storage=case["storage"], rho_ref=1.8)
        L.seed_bubbles(_sites(case, seed), 1.8, 0.15, 2.0, 1e-3, seed)
        return dict(case=case, L=L)
    if kind in ("disks", "rupture"):
        bub, line = _pair(case)
        n = case["side"]
        L = lbm.Lattice("D2Q9", n, n, 1, tau=case["tau"], storage=case["storage"], rho_ref=2.0)
        if kind == "disks":
            L.seed_bubbles(bub, 2.0, 0.15, 2.0, 1e-3, seed)
        return dict(case=case, L=L, bub=bub, line=line, seed=seed)
    if kind == "multi":
        bub, line = _pair(case)
        n, s = case["side"], W.ML_SWEEP_9
        M = lbm.MultiLattice(case["lattice"], n, n, case["depth"], nl=case["nl"], tau=s["tau"],
                             G=s["G"], G_x=s["G_x"], G_b=s["G_b"], storage=case["storage"])
        return dict(case=case, M=M, bub=bub, line=line, seed=seed)
    if kind == "sweep":
        return dict(case=case, domains=W.ensemble_domains(
            dict(W.ENSEMBLE_256, seed=seed % 100003), n=case["n"],
            side=(case["side_min"], case["side_max"])))
    rho = _static_rho(case, seed).cuda()
    w = torch.tensor(_WEIGHTS[case["lattice"]], dtype=torch.float64, device="cuda")
    f = (w.view(-1, 1, 1, 1) * rho).float().contiguous()
    return dict(case=case, f=f, g=torch.empty_like(f))


# ---- one pass ------------------------------------------------------------------

def _table(a, rows=4096):
    """A list of a length that depends on the state, as a table of a fixed one."""
    out = np.zeros(rows, dtype=a.dtype)
    out[:min(rows, len(a))] = a[:rows]
    return out


def _interval_outputs(d):
    fired = d["fired"]
    return dict(totals=d["totals"], ncomp=d["ncomp"], merges=d["merge_events"], film=d["film"],
                fired_cell=_table(fired["cell"]), fired_axis=_table(fired["axis"]),
                fired_d2p=_table(fired["d2p"]), roots=_table(d["roots"]),
                sizes=_table(d["sizes"]), hist=d["hist"], labels=d["labels"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "foam":
        L = state["L"]
        for k in range(case["intervals"]):
            L.step(case["steps"])
            d = L.diagnostic_interval(H_MAX, EPS_ARM, FIRED_CAP, BINS,
                                      want_labels=k + 1 == case["intervals"])
        out = _interval_outputs(d)
        if case["dump"]:
            out["rho"] = torch.from_numpy(L.read("rho")).to(DUMP[case["storage"]])
        return out
    if kind == "survey":
        L = state["L"]
        L.step(1)
        labels, ncomp = L.label_gas()
        roots, sizes, hist = L.bubble_sizes(BINS)
        census, pairs = L.film_pairs(H_MAX, EPS_ARM)
        return dict(labels=labels, ncomp=ncomp, roots=_table(roots), sizes=_table(sizes),
                    hist=hist, census=census, pair_a=_table(pairs["label_a"]),
                    pair_b=_table(pairs["label_b"]), pair_lines=_table(pairs["lines"]),
                    pair_r_d=_table(pairs["r_d"]), p=L.read("p"),
                    laplacian=L.pressure_laplacian())
    if kind == "disks":
        L = state["L"]
        L.step(case["steps"])
        dump = DUMP[case["storage"]]
        labels, ncomp = L.label_gas()
        return dict(rho=torch.from_numpy(L.read("rho")).to(dump),
                    p=torch.from_numpy(L.read("p")).to(dump),
                    line=torch.from_numpy(L.pressure_laplacian(state["line"])).to(dump),
                    labels=labels, ncomp=ncomp)
    if kind == "rupture":
        L = state["L"]
        L.seed_bubbles(state["bub"], 2.0, 0.15, 2.0, 1e-3, state["seed"])
        r = L.run_until_rupture(state["line"], 1.075, EPS_ARM, case["every"], case["steps"])
        return dict(fired=r["fired"], merged=r["merged"], steps=r["steps"], h_c=r["h_c"],
                    r_d=r["r_d"], f=torch.from_numpy(L.read("f")).to(DUMP[case["storage"]]))
    if kind == "multi":
        M, s = state["M"], W.ML_SWEEP_9
        M.seed(state["bub"], s["rho_l"], s["rho_v"], s["rho_gas"], s["width"], s["noise"],
               state["seed"])
        r = M.run_until_rupture(state["line"], 0.5 * (s["rho_l"] + s["rho_v"]), s["eps_arm"],
                                case["every"], case["steps"], s["h_max"])
        rho, p = M.fields()
        dump = DUMP[case["storage"]]
        return dict(fired=r["fired"], merged=r["merged"], steps=r["steps"], h_c=r["h_c"],
                    r_d=r["r_d"], rho=torch.from_numpy(rho).to(dump),
                    p=torch.from_numpy(p).to(dump))
    if kind == "sweep":
        s = W.ENSEMBLE_256
        E = lbm.Ensemble(state["domains"], eps_arm=s["eps_arm"], diag_every=s["diag_every"],
                         h_max=s["h_max"])
        E.run(case["steps"])
        res = E.results()
        E.close()
        return {k: np.array([r[k] for r in res]) for k in ("fired", "merged", "steps", "h_c",
                                                           "h_probe", "r_d")}
    stream = torch.cuda.current_stream().cuda_stream
    for _ in range(case["steps"]):
        lbm.step_static_f32(case["lattice"], case["nx"], case["ny"], case["nz"], case["tau"], -5.0,
                            1.0, state["f"].data_ptr(), state["g"].data_ptr(), stream)
        state["f"], state["g"] = state["g"], state["f"]
    return state["f"]


# ---- the work a pass cannot do without --------------------------------------------

def work(case):
    """Bytes: every population of a step read once and written once, every
    output written once.  Operations: about 270 (D3Q19) or 120 (D2Q9) per
    lattice update."""
    kind = case["kind"]
    if kind == "sweep":
        # the domains of the recipe's own seed; a cell of a whole sweep is
        # updated about 1000 times before its domain's film is gone
        doms = W.ensemble_domains(W.ENSEMBLE_256, n=case["n"],
                                  side=(case["side_min"], case["side_max"]))
        updates = sum(d["nx"] * d["ny"] for d in doms) * min(case["steps"], 1000)
        return dict(bytes=updates * 72, flops=updates * 120)
    if kind in ("disks", "rupture"):
        n = case["side"] ** 2
        S = BYTES[case["storage"]]
        out = 9 * S * n if kind == "rupture" else (2 * S + 4) * n
        return dict(bytes=case["steps"] * n * 18 * S + out, flops=case["steps"] * n * 120)
    if kind == "multi":
        n = case["side"] ** 2 * case["depth"]
        S, Q = BYTES[case["storage"]], 19 if case["lattice"] == "D3Q19" else 9
        return dict(bytes=case["steps"] * n * case["nl"] * 2 * Q * S + (case["nl"] + 1) * n * S,
                    flops=case["steps"] * n * case["nl"] * (300 if Q == 19 else 140))
    n = case["nx"] * case["ny"] * case["nz"]
    Q = 19 if case.get("lattice", "D3Q19") == "D3Q19" else 9
    ops = 270 if Q == 19 else 120
    if kind == "static":
        return dict(bytes=case["steps"] * n * 2 * Q * 4, flops=case["steps"] * n * ops)
    S = BYTES[case["storage"]]
    if kind == "survey":
        # one step, the populations read for labels and for the pressure
        return dict(bytes=n * (4 * Q * S + 4 + 16), flops=n * (ops + 60))
    per_step = 2 * Q * S + (8 if case["residual"] else 0)
    steps = case["intervals"] * case["steps"]
    out = n * (4 + (S if case["dump"] else 0))
    return dict(bytes=n * (steps * per_step + case["intervals"] * Q * S) + out,
                flops=n * steps * ops)


# ---- the same in 64 bits ------------------------------------------------------------

_C2 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0),
       (-1, -1, 0), (1, -1, 0)]
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
       (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_VELOCITIES = {"D2Q9": _C2, "D3Q19": _C3}
_WEIGHTS = {"D2Q9": [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4,
            "D3Q19": [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12}


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _noise(n, seed):
    """u in [0, 1): outputs 0 .. n-1 of SplitMix64 on the noise stream (the
    seed with the text "noise" in its upper bytes)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed ^ 0x6E6F697365000000) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _seeded_rho(lattice, nx, ny, nz, bub, rho_l, rho_g, width, amp, seed):
    """rho_g + (rho_l - rho_g)/2 (1 + tanh(2 s / width)) with s the least
    periodic distance to a bubble's surface, plus uniform noise."""
    dev = _device()
    s = torch.full((nz, ny, nx), 1e30, dtype=torch.float64, device=dev)
    for x, y, z, r in np.asarray(bub):
        box, dist = [], []
        for n, c in zip((nz, ny, nx), (z, y, x)):
            half = int(r + 12 * width) + 2  # tanh is 1 in 64 bits beyond this
            at = (torch.arange(n) if 2 * half + 1 >= n else
                  torch.remainder(torch.arange(-half, half + 1) + int(round(c)), n)).to(dev)
            d = torch.remainder(at.double() - c, n)
            box.append(at)
            dist.append(torch.where(d > 0.5 * n, d - n, d))
        d = torch.sqrt(dist[2][None, None, :] ** 2 + dist[1][None, :, None] ** 2
                       + dist[0][:, None, None] ** 2) - r
        at = (box[0][:, None, None], box[1][None, :, None], box[2][None, None, :])
        s[at] = torch.minimum(s[at], d)
    rho = rho_g + 0.5 * (rho_l - rho_g) * (1.0 + torch.tanh(2.0 * s / width))
    if amp:
        u = torch.from_numpy(_noise(nx * ny * nz, seed)).to(dev)
        rho += amp * (2.0 * u - 1.0).view(nz, ny, nx)
    return rho


def _roll(a, c, sign=1):
    shift = [(sign * v, d) for v, d in zip(c, (2, 1, 0)) if v]
    return torch.roll(a, [v for v, _ in shift], [d for _, d in shift]) if shift else a


def _psi(rho):
    return 1.0 - torch.exp(-rho)


def _sum_c(terms, C, axis):
    out = None
    for t, c in zip(terms, C):
        if c[axis]:
            out = (t * c[axis] if out is None else out.add_(t, alpha=c[axis]))
    return out


def _step64(lattice, f, tau, G, deposit=None):
    """One step: moments, Shan-Chen force as a velocity shift, BGK, blowing
    agent into the collided populations, streaming."""
    C, w = _VELOCITIES[lattice], _WEIGHTS[lattice]
    rho = f.sum(0)
    psi = _psi(rho)
    u = []
    for axis in range(3 if lattice == "D3Q19" else 2):
        j = _sum_c(f, C, axis)
        F = None
        for c, wi in zip(C, w):
            if c[axis]:
                t = _roll(psi, c, -1) * (wi * c[axis])
                F = t if F is None else F.add_(t)
        u.append((j - tau * G * psi * F) / rho)
    uu = 1.5 * sum(v * v for v in u)
    g = torch.empty_like(f)
    for i, (c, wi) in enumerate(zip(C, w)):
        cu = sum(v * k for v, k in zip(u, c) if k) if any(c) else 0.0
        feq = wi * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - uu)
        fs = f[i] - (f[i] - feq) / tau
        if deposit is not None:
            fs.view(-1).index_add_(0, deposit[0], wi * deposit[1])
        g[i] = _roll(fs, c)
    return g


def _rest(lattice, rho):
    w = torch.tensor(_WEIGHTS[lattice], dtype=torch.float64, device=rho.device)
    return w.view(-1, 1, 1, 1) * rho


def _totals64(lattice, f):
    C = _VELOCITIES[lattice]
    j = [sum(float(f[i].sum()) * c[a] for i, c in enumerate(C) if c[a]) for a in range(3)]
    return np.array([float(f.sum())] + j)


def _pressure64(rho, G=-5.0):
    return rho / 3.0 + G / 6.0 * _psi(rho) ** 2


def _laplacian64(p):
    s = -6.0 * p
    for c in ((1, 0, 0), (0, 1, 0), (0, 0, 1)):
        s += _roll(p, c) + _roll(p, c, -1)
    return s


def _numpy(t):
    return t.cpu().numpy()


class _Probe:
    """The film probe's state machine: whether a run under it goes on."""

    def __init__(self, line, h_max):
        self.line, self.h_max, self.armed = line, h_max, False

    def goes_on(self, rho, p):
        x, y, z, _, length = self.line
        at = torch.arange(x - 1, x + length + 1, device=rho.device) % rho.shape[2]
        r, q = rho[z, y, at].tolist(), p[z, y, at].tolist()
        cross = []
        for m in range(1, length):
            lo, hi = r[m], r[m + 1]
            if (lo < 1.075 <= hi) if len(cross) == 0 else (hi < 1.075 <= lo):
                cross.append(m - 1 + (1.075 - lo) / (hi - lo))
                if len(cross) == 2:
                    break
        if len(cross) < 2:
            return False  # no film: the run ends as merged
        m = 1 + int(math.floor(0.5 * (cross[0] + cross[1]) + 0.5))
        d2 = q[m - 1] - 2.0 * q[m] + q[m + 1]
        if cross[1] - cross[0] > self.h_max:
            self.armed = False
        elif d2 < -EPS_ARM:
            self.armed = True
        elif self.armed and d2 >= 0.0:
            return False  # the criterion fires
        return True


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return None  # up to 20000 steps of every domain
    if kind in ("foam", "survey"):
        lattice = case.get("lattice", "D3Q19")
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        n = nx * ny * nz
        steps = case["intervals"] * case["steps"] if kind == "foam" else 1
        if n * steps > 3_000_000_000:
            return None
        rho_l = case.get("rho_l", 1.8)
        bub = _sites(case, seed)
        f = _rest(lattice, _seeded_rho(lattice, nx, ny, nz, bub, rho_l, 0.15, 2.0, 1e-3, seed))
        if kind == "survey":
            p = _pressure64(_step64(lattice, f, case["tau"], -5.0).sum(0))
            return dict(p=_numpy(p), laplacian=_numpy(_laplacian64(p)))
        deposit = budget = None
        if case["rate"] > 0:
            at = np.floor(bub[:, :3] + 0.5).astype(np.int64) % np.array([nx, ny, nz])
            cells = torch.from_numpy(at[:, 0] + nx * (at[:, 1] + ny * at[:, 2])).to(f.device)
            budget = torch.full((len(bub),), case["budget"], dtype=torch.float64, device=f.device)
        for _ in range(steps):
            if budget is not None:
                dm = torch.clamp(budget, max=case["rate"])
                budget = budget - dm
                deposit = (cells, dm)
            f = _step64(lattice, f, case["tau"], -5.0, deposit)
        out = dict(totals=_totals64(lattice, f))
        if case["dump"]:
            out["rho"] = _numpy(f.sum(0))
        return out
    if kind in ("disks", "rupture"):
        bub, line = _pair(case)
        n = case["side"]
        f = _rest("D2Q9", _seeded_rho("D2Q9", n, n, 1, bub, 2.0, 0.15, 2.0, 1e-3, seed))
        probe = _Probe(line, 8.0)
        for k in range(case["steps"]):
            f = _step64("D2Q9", f, case["tau"], -5.0)
            if kind == "rupture" and (k + 1) % case["every"] == 0:
                rho = f.sum(0)
                if not probe.goes_on(rho, _pressure64(rho)):
                    return None
        if kind == "rupture":
            return dict(f=_numpy(f))
        rho = f.sum(0)
        p = _pressure64(rho)
        row = p[0, line[1]]
        at = torch.arange(line[0], line[0] + line[4], device=row.device) % n
        d2 = torch.roll(row, -1) - 2.0 * row + torch.roll(row, 1)
        return dict(rho=_numpy(rho), p=_numpy(p), line=_numpy(d2[at]))
    if kind == "multi":
        return _multi64(case, seed)
    f = (torch.tensor(_WEIGHTS[case["lattice"]], dtype=torch.float64).view(-1, 1, 1, 1)
         * _static_rho(case, seed)).float().double().to(_device())
    for _ in range(case["steps"]):
        f = _step64(case["lattice"], f, case["tau"], -5.0)
    return f


def _multi64(case, seed):
    """The coupled lattices: common velocity sum j / sum rho, force
    -psi_s sum_t Gm[s][t] sum_i w_i psi_t(x + c_i) c_i, one relaxation time."""
    s = W.ML_SWEEP_9
    lattice, nl = case["lattice"], case["nl"]
    n, depth = case["side"], case["depth"]
    bub, line = _pair(case)
    C, w, dims = _VELOCITIES[lattice], _WEIGHTS[lattice], 3 if lattice == "D3Q19" else 2
    Gm = np.full((nl, nl), s["G_b"])
    np.fill_diagonal(Gm, 0.0)
    Gm[0, :] = Gm[:, 0] = s["G_x"]
    Gm[0, 0] = s["G"]
    rho = [_seeded_rho(lattice, n, n, depth, bub, s["rho_l"], s["rho_v"], s["width"], s["noise"],
                       seed)]
    for b in bub:
        rho.append(_seeded_rho(lattice, n, n, depth, [b], 0.0, s["rho_gas"], s["width"], 0.0, 0))
    f = [_rest(lattice, r) for r in rho]
    probe = _Probe(line, s["h_max"])

    def pressure(rho, psi):
        return sum(rho) / 3.0 + sum(float(Gm[a, b]) * psi[a] * psi[b] for a in range(nl)
                                    for b in range(nl)) / 6.0

    for k in range(case["steps"]):
        rho = [g.sum(0) for g in f]
        psi = [_psi(r) for r in rho]
        if k and k % case["every"] == 0 and not probe.goes_on(rho[0], pressure(rho, psi)):
            return None
        total = sum(rho)
        S = [[sum(_roll(q, c, -1) * (wi * c[a]) for c, wi in zip(C, w) if c[a])
              for a in range(dims)] for q in psi]
        up = [sum(_sum_c(g, C, a) for g in f) / total for a in range(dims)]
        new = []
        for m in range(nl):
            r = rho[m]
            safe = torch.where(r != 0, r, torch.ones_like(r))
            u = [up[a] + torch.where(r != 0, -s["tau"] * psi[m]
                                     * sum(float(Gm[m, t]) * S[t][a] for t in range(nl)) / safe,
                                     torch.zeros_like(r)) for a in range(dims)]
            uu = 1.5 * sum(v * v for v in u)
            g = torch.empty_like(f[m])
            for i, (c, wi) in enumerate(zip(C, w)):
                cu = sum(v * q for v, q in zip(u, c) if q) if any(c) else 0.0
                feq = wi * r * (1.0 + 3.0 * cu + 4.5 * cu * cu - uu)
                g[i] = _roll(f[m][i] - (f[m][i] - feq) / s["tau"], c)
            new.append(g)
        f = new
    rho = [g.sum(0) for g in f]
    p = pressure(rho, [_psi(r) for r in rho])
    return dict(rho=np.stack([_numpy(r) for r in rho]), p=_numpy(p))
