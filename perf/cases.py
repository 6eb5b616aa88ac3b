"""What this framework is used for, as cases that can be timed and checked.

Each case is one call, or the short sequence of calls, that a program makes
through the public entry points of ``paper_1911_01353_gb300``, on inputs made
from a seed: noise spectra with a few injected chirps, in raw (unnormalised)
units.  Listed cases:

search_small      one spectrum of 2^16 bins against the 147-template bank, the
                  smallest configuration of the tests: latency and launches
search_mid        an odd-length spectrum against a 3131-template bank with
                  harmonic stages 1-2-4: an ordinary search
search_paper      2^21 bins against the paper-scale bank (zmax 200, wmax 600,
                  12 261 templates), stages 1-2-4-8: the headline search, at
                  half its length so that several states fit the card
search_fp16       the paper-scale bank on the FP16 tensor-core filter
search_bf16       an odd length on the BF16 tensor-core filter, stages 1-2
batch_short       24 short uneven spectra in one batch call: launches count
batch_dm          DM-trial spectra of uneven length, zmax 200, wmax 300,
                  stages 1-2-4-8, replayed as a CUDA graph
serve_mix         requests with ranges of their own on one resident bank
                  (zmax 300, wmax 900), stage 1: one batch of the server
plane_rows        power rows of some templates around a candidate (jerk_plane)
subharmonic       the search with the sum indexed by the highest harmonic
refine            candidates refined off the grid
bank              building a template bank (every new configuration pays it),
                  and FP64 taps read back

The max-projections are returned as their powers, for every stage and cell;
template indices come with the candidates.
"""
import math

import numpy as np
import torch

from paper_1911_01353_gb300 import jerk

# threshold in sigmas per stage H of a search: a few false candidates per search
_SIGMAS = {1: 19.0, 2: 17.0, 3: 16.0, 4: 15.0, 8: 14.0}
# grids of the tests, the benchmark and the server's requests: zmax, dz, wmax, dw
_GRIDS = ((20, 2, 60, 20), (50, 2, 0, 20), (50, 2, 300, 20), (100, 2, 300, 20), (200, 2, 300, 20),
          (200, 2, 600, 20))
_LARGEST = 2 * (1 << 21) * 12261          # cells x templates of the largest listed search


def _templates(zmax, dz, wmax, dw):
    return (2 * zmax // dz + 1) * (2 * wmax // dw + 1)


def listed():
    def search(name, n, zmax, wmax, stages, precision=0, mode="sigma"):
        return {"name": name, "kind": "search", "n": n, "zmax": zmax, "dz": 2, "wmax": wmax, "dw": 20,
                "stages": stages, "precision": precision, "mode": mode}
    return [
        search("search_small", 1 << 16, 20, 60, "1-2", mode="abs"),
        search("search_mid", 700001, 100, 300, "1-2-4"),
        search("search_paper", 1 << 21, 200, 600, "1-2-4-8"),
        search("search_fp16", 1 << 20, 200, 600, "1-2-4-8", precision=2),
        search("search_bf16", 300007, 100, 300, "1-2", precision=1),
        {"name": "batch_short", "kind": "batch", "count": 24, "lo": 13.0, "hi": 16.0, "lengths": 5, "zmax": 20,
         "dz": 2, "wmax": 60, "dw": 20, "stages": "1-2", "precision": 0, "mode": "sigma", "graph": False},
        {"name": "batch_dm", "kind": "batch", "count": 6, "lo": 17.0, "hi": 19.0, "lengths": 3, "zmax": 200,
         "dz": 2, "wmax": 300, "dw": 20, "stages": "1-2-4-8", "precision": 0, "mode": "sigma", "graph": True},
        {"name": "serve_mix", "kind": "serve", "count": 6, "lo": 16.0, "hi": 20.0, "lengths": 9, "zmax": 300,
         "dz": 2, "wmax": 900, "dw": 20, "stages": "1", "precision": 0, "mode": "sigma"},
        {"name": "plane_rows", "kind": "plane", "n": 1 << 18, "zmax": 200, "dz": 2, "wmax": 600, "dw": 20,
         "t0": 6000, "nt": 64, "precision": 0},
        {"name": "subharmonic", "kind": "subharmonic", "n": 1 << 16, "zmax": 20, "dz": 2, "wmax": 60, "dw": 20,
         "stages": "1-2-3-4", "mode": "sigma"},
        {"name": "refine", "kind": "refine", "n": 1 << 18, "zmax": 200, "dz": 2, "wmax": 600, "dw": 20,
         "count": 40, "hr": 3, "hz": 2, "hw": 2},
        {"name": "bank", "kind": "bank", "zmax": 200, "dz": 2, "wmax": 600, "dw": 20, "precision": 0},
    ]


def draw(rng):
    kind = rng.choice(("search", "search", "search", "search", "batch", "batch", "serve", "plane", "subharmonic",
                       "refine", "bank"))

    def grid(at_most=len(_GRIDS)):
        zmax, dz, wmax, dw = _GRIDS[rng.randrange(at_most)]
        return {"zmax": zmax, "dz": dz, "wmax": wmax, "dw": dw}

    def length(lo, hi):
        return int(2.0 ** rng.uniform(lo, hi))

    stages = rng.choice(("1", "1-2", "1-3", "1-2-4", "1-2-4-8"))
    precision = rng.choice((0, 0, 0, 1, 2))
    mode = rng.choice(("sigma", "sigma", "abs"))
    if kind == "search":
        c = {"kind": kind, "n": 0, **grid(), "stages": stages, "precision": precision, "mode": mode}
        T = _templates(c["zmax"], c["dz"], c["wmax"], c["dw"])
        c["n"] = length(13.0, math.log2(min(1 << 22, _LARGEST // (2 * T))))
        return c
    if kind == "batch":
        short = rng.random() < 0.5
        lo = rng.uniform(12.0, 14.0) if short else rng.uniform(15.0, 17.5)
        return {"kind": kind, "count": rng.randrange(8, 25) if short else rng.randrange(2, 7), "lo": round(lo, 2),
                "hi": round(lo + rng.uniform(0.5, 1.5), 2), "lengths": rng.randrange(1 << 20),
                **grid(3 if short else 5), "stages": rng.choice(("1", "1-2")) if short else stages,
                "precision": precision, "mode": mode, "graph": rng.random() < 0.5}
    if kind == "serve":
        return {"kind": kind, "count": rng.randrange(1, 7), "lo": 15.0, "hi": round(rng.uniform(16.0, 17.5), 2),
                "lengths": rng.randrange(1 << 20), "zmax": 300, "dz": 2, "wmax": rng.choice((300, 600, 900)),
                "dw": 20, "stages": "1", "precision": precision, "mode": "sigma"}
    if kind == "plane":
        c = {"kind": kind, "n": length(14.0, 18.0), **grid(), "t0": 0, "nt": 0, "precision": precision}
        T = _templates(c["zmax"], c["dz"], c["wmax"], c["dw"])
        c["nt"] = min(int(2.0 ** rng.uniform(0.0, 8.0)), T)
        c["t0"] = rng.randrange(T - c["nt"] + 1)
        return c
    if kind == "subharmonic":
        return {"kind": kind, "n": length(13.0, 17.0), **grid(2),
                "stages": rng.choice(("1-2", "1-3", "1-2-4", "1-2-3-4", "1-2-4-8")), "mode": mode}
    if kind == "refine":
        return {"kind": kind, "n": length(14.0, 20.0), **grid(), "count": rng.randrange(1, 41),
                "hr": rng.randrange(1, 4), "hz": rng.randrange(1, 3), "hw": rng.randrange(1, 3)}
    return {"kind": "bank", **grid(), "precision": precision}


# ---- inputs ------------------------------------------------------------------

def _thresh(case):
    H = [int(s) for s in case.get("stages", "1").split("-")]
    if case.get("mode") == "abs":
        # powers that unit noise over the bank exceeds rarely
        return H, [h + 15.0 * math.sqrt(h) for h in H], jerk.THRESH_ABS
    return H, [_SIGMAS[h] for h in H], jerk.THRESH_SIGMA


def _params(case, max_bins, max_batch=1):
    H, thresh, mode = _thresh(case)
    return jerk.make_params(case["zmax"], case["dz"], case["wmax"], case["dw"], stages=tuple(H),
                            thresh=tuple(thresh), thresh_mode=mode, max_bins=max_bins, max_candidates=1 << 16,
                            precision=case.get("precision", 0), max_batch=max_batch)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _signals(rs, n, zmax, wmax, count):
    """(r, z, w, power SNR, phase) of injected chirps."""
    return [(rs.uniform(0.02 * n, 0.98 * n), rs.uniform(-zmax, zmax), rs.uniform(-wmax, wmax),
             rs.uniform(25.0, 50.0), rs.uniform(0.0, 2.0 * math.pi)) for _ in range(count)]


def _spectrum(n, seed, signals=(), harmonics=1):
    """complex64[n] on the GPU: complex Gaussian noise plus chirps, times a slowly
    varying gain (the units and the red slope of a raw spectrum)."""
    g = _generator(seed)
    f = torch.view_as_complex(torch.randn(n, 2, generator=g, device="cuda", dtype=torch.float64)) / math.sqrt(2.0)
    if signals:
        u = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n - 0.5
        x = torch.zeros(n, device="cuda", dtype=torch.complex128)
        for r, z, w, snr, phase in signals:
            for h in range(1, harmonics + 1):
                cyc = (h * r) * u + (h * z) * u * u / 2.0 + (h * w) * u ** 3 / 6.0
                x += torch.polar(torch.full_like(u, math.sqrt(snr)), 2.0 * math.pi * (cyc - cyc.floor()) + h * phase)
        k = torch.arange(n, device="cuda", dtype=torch.float64)
        # time origin at mid-observation: exp(-2 pi i k (1/(2n) - 1/2))
        turn = torch.remainder(k * 0.5 - k / (2 * n), 1.0)
        f = f + torch.fft.fft(x) / n * torch.polar(torch.ones_like(u), 2.0 * math.pi * turn)
    gain = 50.0 * (1.0 + 3.0 * torch.exp(-torch.arange(n, device="cuda", dtype=torch.float64) / (0.1 * n)))
    return (f * gain).to(torch.complex64).contiguous()


def _one(case, seed, count=8, harmonics=1):
    rs = np.random.RandomState(seed % (1 << 31))
    return _spectrum(case["n"], seed, _signals(rs, case["n"], case["zmax"] / harmonics, case["wmax"] / harmonics,
                                               count), harmonics)


def _lengths(case):
    rs = np.random.RandomState(case["lengths"])
    return [int(2.0 ** rs.uniform(case["lo"], case["hi"])) for _ in range(case["count"])]


def _ranges(case):
    """(zmax, wmax) of each request of a served batch."""
    rs = np.random.RandomState(case["lengths"] + 1)
    zs = [z for z in (50, 100, 200, 300) if z <= case["zmax"]]
    ws = [w for w in (0, 300, 600, 900) if w <= case["wmax"]]
    return [(int(rs.choice(zs)), int(rs.choice(ws))) for _ in range(case["count"])]


def _several(case, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    return [_spectrum(n, seed * 64 + i, _signals(rs, n, case["zmax"], case["wmax"], int(rs.randint(0, 4))))
            for i, n in enumerate(_lengths(case))]


def _points(case, seed):
    """Candidates to refine: chirps of the spectrum, moved to the nearest grid point."""
    rs = np.random.RandomState(seed % (1 << 31))
    sig = _signals(rs, case["n"], case["zmax"], case["wmax"], 8)
    out = []
    for i in range(case["count"]):
        r, z, w = sig[i % 8][:3]
        c = jerk.Candidate()
        c.p = int(round(2 * r)) + int(rs.randint(-1, 2))
        c.r = c.p / 2.0
        c.z = float(case["dz"] * round(z / case["dz"]))
        c.w = float(case["dw"] * round(w / case["dw"]))
        c.stage = 1
        out.append(c)
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind in ("search", "plane", "refine", "subharmonic"):
        s["plan"] = jerk.Plan(_params(case, case["n"]))
        s["x"] = _one(case, seed, harmonics=4 if kind == "subharmonic" else 1)
        if kind == "plane":
            s["out"] = torch.empty(case["nt"], 2 * case["n"], dtype=torch.float32, device="cuda")
        if kind == "refine":
            s["cands"] = _points(case, seed)
    elif kind in ("batch", "serve"):
        s["x"] = _several(case, seed)
        s["plan"] = jerk.Plan(_params(case, sum(_lengths(case)), max_batch=case["count"]))
        if kind == "serve":
            s["zmax"], s["wmax"] = (list(v) for v in zip(*_ranges(case)))
    else:
        s["plan"] = jerk.Plan(_params(case, 1 << 16), build_templates=False)
        info = s["plan"].info
        # templates whose taps are read back: of the seed's choosing
        s["nt"] = min(32, info.n_templates)
        s["t0"] = int(np.random.RandomState(seed % (1 << 31)).randint(0, info.n_templates - s["nt"] + 1))
        s["taps"] = torch.empty(s["nt"], info.taps, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    return s


# ---- one pass ------------------------------------------------------------------

class _Device:
    """Device memory of a plan as something torch can view; holds the plan, whose memory ends with it."""

    def __init__(self, plan, ptr, n, typestr):
        self.plan = plan
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": typestr, "data": (ptr, False), "version": 3}


def _powers(plan, si, item=0):
    """The powers of a stage's packed max-projection: a view of its upper halves."""
    ptr, n = plan.maxproj_ptr(si, item)
    return _upper(torch.as_tensor(_Device(plan, ptr, n, "<i8"), device="cuda:%d" % plan.device))


def _upper(packed):
    return packed.view(torch.int32)[1::2].view(torch.float32)


_RECORDS = 1024                           # rows of the candidate table; unused ones are 0


def _records(cands, fields=(("item", np.int32), ("stage", np.int32), ("p", np.int64), ("t", np.int32),
                            ("power", np.float32))):
    """The candidates, in the order they come in, as a table of a fixed length."""
    table = {}
    for name, kind in fields:
        table[name] = np.zeros(_RECORDS, dtype=kind)
        table[name][:len(cands)] = [getattr(c, name) for c in cands[:_RECORDS]]
    return table


def run(state):
    kind, plan = state["kind"], state["plan"]
    case = state["case"]
    if kind == "search":
        plan.search(state["x"])
        found = plan.candidates()
        return {"M": [_powers(plan, si) for si in range(case["stages"].count("-") + 1)],
                "found": _records(found), "stats": plan.stats()}
    if kind in ("batch", "serve"):
        if kind == "serve":
            plan.search_batch(state["x"], zmax=state["zmax"], wmax=state["wmax"], transient=True)
        else:
            plan.search_batch(state["x"], graph=case["graph"])
        found = plan.candidates()
        items = range(case["count"])
        mean, std, theta = (np.array(v, dtype=np.float32) for v in zip(*[plan.stats(i) for i in items]))
        return {"M": [[_powers(plan, si, i) for si in range(case["stages"].count("-") + 1)]
                      for i in items], "found": _records(found), "mean": mean, "std": std, "theta": theta}
    if kind == "plane":
        plan.plane(state["x"], case["t0"], case["nt"], state["out"])
        return state["out"]
    if kind == "subharmonic":
        found, stats, M = plan.search_subharmonic(state["x"])
        p, t = np.zeros(_RECORDS, dtype=np.int64), np.zeros(_RECORDS, dtype=np.int32)
        p[:len(found)], t[:len(found)] = [c[0] for c in found[:_RECORDS]], [c[2] for c in found[:_RECORDS]]
        return {"M": [_upper(m) for m in M], "stats": [list(s) for s in stats], "p": p, "t": t}
    if kind == "refine":
        out = plan.refine(state["x"], state["cands"], (0.125, case["dz"] / 4.0, case["dw"] / 4.0),
                          (case["hr"], case["hz"], case["hw"]))
        return {"power": np.array([c.power for c in out], dtype=np.float32),
                "power_in": np.array([c.power_in for c in out], dtype=np.float32),
                "rzw": np.array([(c.r, c.z, c.w) for c in out], dtype=np.float32)}
    plan.templates()
    plan.taps(state["t0"], state["nt"], state["taps"])
    info = plan.info
    bank = torch.as_tensor(_Device(plan, info.d_bank, info.n_templates * info.seg_len, "<c8"),
                           device="cuda:%d" % plan.device)
    return {"bank": bank, "taps": state["taps"]}


# ---- what a pass cannot do without ------------------------------------------------

def _halfwidth(z, w):
    return math.ceil(abs(z) / 2.0 + abs(w) / 8.0) + 16


def _rows(case, H, zmax=None, wmax=None):
    """Harmonic rows as (h, floats per cell) summed: cells that the stages above the first add up per output cell."""
    zmax, wmax = case["zmax"] if zmax is None else zmax, case["wmax"] if wmax is None else wmax
    total = 0.0
    for a, b in zip(H[:-1], H[1:]):
        zs, ws = 2 * (zmax // b // case["dz"]) + 1, 2 * (wmax // b // case["dw"]) + 1
        total += zs * ws * (b - a) / b
    return total


def _search_work(case, n, zmax=None, wmax=None):
    """One spectrum: FFT filtering (5 log2 L + product 6 + power 3 flops per cell and template at L = 4096, no
    overlap), the harmonic sums' additions; the spectrum read once, the max-projections written once."""
    zmax, wmax = case["zmax"] if zmax is None else zmax, case["wmax"] if wmax is None else wmax
    H = [int(h) for h in case["stages"].split("-")]
    T = _templates(zmax, case["dz"], wmax, case["dw"])
    return {"bytes": 8 * n + sum(8 * 2 * n // h for h in H),
            "flops": 2.0 * n * (T * (5 * 12 + 6 + 3) + _rows(case, H, zmax, wmax))}


def work(case):
    kind = case["kind"]
    T = _templates(case["zmax"], case["dz"], case["wmax"], case["dw"])
    bank = 8 * 4096 * T
    if kind in ("search", "subharmonic"):
        w = _search_work(case, case["n"])
        return {"bytes": w["bytes"] + bank, "flops": w["flops"]}
    if kind == "batch":
        parts = [_search_work(case, n) for n in _lengths(case)]
    elif kind == "serve":
        parts = [_search_work(case, n, z, w) for n, (z, w) in zip(_lengths(case), _ranges(case))]
    elif kind == "plane":
        n, nt = case["n"], case["nt"]
        return {"bytes": 8 * n + 8 * 4096 * nt + 8 * n * nt, "flops": 2.0 * n * nt * (5 * 12 + 6 + 3)}
    elif kind == "refine":
        points = case["count"] * (2 * case["hr"] + 1) * (2 * case["hz"] + 1) * (2 * case["hw"] + 1)
        nk = 2 * _halfwidth(case["zmax"] / 2, case["wmax"] / 2)
        # one response value per bin of the window and its product: nodes as for one sample per half cycle
        return {"bytes": 8 * case["n"], "flops": points * 8.0 * nk * nk}
    else:
        taps = sum(4 * _halfwidth(z, w) + 1 for z in range(-case["zmax"], case["zmax"] + 1, case["dz"])
                   for w in range(-case["wmax"], case["wmax"] + 1, case["dw"]))
        # each tap an integral over about two nodes per cycle, each template one FP64 transform of 4096 points
        return {"bytes": bank, "flops": 8.0 * taps * 2 * _halfwidth(case["zmax"] / 2, case["wmax"] / 2)
                + T * 5.0 * 4096 * 12}
    return {"bytes": bank + sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


# ---- the same in 64 bits ------------------------------------------------------------

_MAX_POINTS = 2.0e10                       # transform points that stay well below 20 seconds


def _exact_normalised(x):
    """complex128 spectrum, each block of 1024 bins scaled to unit median noise power."""
    f = x.to(torch.complex128)
    p = f.real.square() + f.imag.square()
    out = torch.empty_like(f)
    for b in range(0, f.numel(), 1024 * 1024):
        q, g = p[b:b + 1024 * 1024], f[b:b + 1024 * 1024]
        whole = q.numel() // 1024 * 1024
        for lo, hi in ((0, whole), (whole, q.numel())):
            if lo == hi:
                continue
            nb = 1024 if lo == 0 and whole else hi - lo
            med = q[lo:hi].reshape(-1, nb).sort(dim=1).values[:, (nb - 1) // 2]
            scale = torch.where(med > 0, (med / math.log(2.0)).rsqrt(), torch.ones_like(med))
            out[b + lo:b + hi] = (g[lo:hi].reshape(-1, nb) * scale[:, None]).reshape(-1)
    return out


def _exact_response(q, z, w):
    """rho(q; z, w) for FP64 tensors q [..., K], z, w [...] (panelled Gauss-Legendre quadrature)."""
    cycles = float(q.abs().max()) + float(z.abs().max()) / 2.0 + float(w.abs().max()) / 8.0
    panels = int(math.ceil(cycles / 6.0)) + 1
    x, g = np.polynomial.legendre.leggauss(40)
    u = -0.5 + (np.arange(panels)[:, None] + 0.5 * (x[None, :] + 1.0)) / panels
    u = torch.from_numpy(u.reshape(-1)).cuda()
    g = torch.from_numpy(np.tile(g * 0.5 / panels, panels)).cuda()
    ph = z[:, None] * u.square() / 2.0 + w[:, None] * u ** 3 / 6.0
    chirp = torch.polar(g.expand_as(ph).contiguous(), 2.0 * math.pi * (ph - ph.round()))        # [T, nodes]
    turn = q[:, None] * u[None, :]
    kernel = torch.polar(torch.ones_like(turn), -2.0 * math.pi * (turn - turn.round()))          # [K, nodes]
    return chirp @ kernel.T                                                                      # [T, K]


def _exact_taps(case, zs, ws, M):
    """complex128 [T, 4 M + 1]: conj(rho(d / 2; z, w)), zero outside each template's own half-width."""
    d = torch.arange(-2 * M, 2 * M + 1, device="cuda")
    z = torch.tensor(zs, dtype=torch.float64, device="cuda")
    w = torch.tensor(ws, dtype=torch.float64, device="cuda")
    m = torch.tensor([_halfwidth(a, b) for a, b in zip(zs, ws)], device="cuda")
    c = _exact_response(d.double() / 2.0, z, w).conj()
    return c * (d[None, :].abs() <= 2 * m[:, None])


def _grid(case):
    zs = list(range(-case["zmax"], case["zmax"] + 1, case["dz"]))
    ws = list(range(-case["wmax"], case["wmax"] + 1, case["dw"]))
    return [(z, w) for w in ws for z in zs]


class _ExactPlane:
    """Power rows of one spectrum, by whole-spectrum FP64 transforms."""

    def __init__(self, case, x):
        f = _exact_normalised(x)
        self.case, self.bN = case, 2 * f.numel()
        self.M = _halfwidth(case["zmax"], case["wmax"])
        need, size = self.bN + 4 * self.M + 1, 1
        while size < need:
            size *= 2
        for odd in (9, 5, 3, 15):                        # a smaller smooth length, where there is one
            t = odd
            while t < need:
                t *= 2
            size = min(size, t)
        self.size = size
        spread = torch.zeros(size, dtype=torch.complex128, device="cuda")
        spread[0:self.bN:2] = f
        self.S = torch.fft.fft(spread)
        grid = _grid(case)
        self.at = {zw: i for i, zw in enumerate(grid)}
        self.taps = torch.cat([_exact_taps(case, [z for z, _ in grid[k:k + 512]], [w for _, w in grid[k:k + 512]],
                                           self.M) for k in range(0, len(grid), 512)])

    def rows(self, zw):
        """[len(zw), bN]: |sum_d s[p + d] c_d|^2."""
        c = self.taps[[self.at[v] for v in zw]]
        g = torch.zeros(len(zw), self.size, dtype=torch.complex128, device="cuda")
        g[:, :2 * self.M + 1] = c[:, :2 * self.M + 1].flip(1)          # d = 0, -1, .. at 0, 1, ..
        g[:, self.size - 2 * self.M:] = c[:, 2 * self.M + 1:].flip(1)   # d = 2 M .. 1 at the end
        y = torch.fft.ifft(torch.fft.fft(g, dim=1) * self.S, dim=1)[:, :self.bN]
        return y.real.square() + y.imag.square()


def _exact_maxima(case, x, zmax=None, wmax=None):
    """(M_H for every stage, mean and standard deviation per stage) of one spectrum in 64 bits."""
    H = [int(h) for h in case["stages"].split("-")]
    zmax, wmax = case["zmax"] if zmax is None else zmax, case["wmax"] if wmax is None else wmax
    plane = _ExactPlane(case, x)
    bN = plane.bN
    M = [torch.full(((bN - 1) // h + 1,), -1.0, dtype=torch.float64, device="cuda") for h in H]
    sums = torch.zeros(len(H), 3, dtype=torch.float64, device="cuda")
    todo = []
    for z, w in _grid(case):
        if abs(z) <= zmax and abs(w) <= wmax:
            top = max(i for i, h in enumerate(H) if i == 0 or (h * abs(z) <= zmax and h * abs(w) <= wmax))
            todo.append((z, w, top))
    chunk = max(1, min(64, (1 << 27) // plane.size))
    for k in range(0, len(todo), chunk):
        part = todo[k:k + chunk]
        first = plane.rows([(z, w) for z, w, _ in part])
        for i, (z, w, top) in enumerate(part):
            acc = first[i]
            for si, h in enumerate(H):
                if si > top:
                    break
                n = M[si].numel()
                if si > 0:
                    hs = list(range(H[si - 1] + 1, h + 1))
                    more = plane.rows([(a * z, a * w) for a in hs])
                    acc = acc[:n].clone()
                    for a, row in zip(hs, more):
                        acc += row[::a][:n]
                torch.maximum(M[si], acc[:n], out=M[si])
                sums[si] += torch.stack((acc[:n].sum(), acc[:n].square().sum(), acc.new_tensor(float(n))))
    mean = sums[:, 0] / sums[:, 2]
    return M, mean, (sums[:, 1] / sums[:, 2] - mean.square()).clamp(min=0).sqrt()


def _points_of(case, n, zmax, wmax):
    H = [int(h) for h in case["stages"].split("-")]
    rows = _templates(zmax, case["dz"], wmax, case["dw"])
    for a, b in zip(H[:-1], H[1:]):
        rows += (2 * (zmax // b // case["dz"]) + 1) * (2 * (wmax // b // case["dw"]) + 1) * (b - a)
    return 2.0 * rows * 2.5 * n


def _exact_powers(f, r, zw):
    """P(r, z, w) at r and every (z, w) of zw: direct sums over the window's bins."""
    z = torch.tensor([a for a, _ in zw], dtype=torch.float64, device="cuda")
    w = torch.tensor([b for _, b in zw], dtype=torch.float64, device="cuda")
    m = torch.tensor([float(_halfwidth(a, b)) for a, b in zw], dtype=torch.float64, device="cuda")
    top = float(m.max())
    k0, k1 = max(0, math.ceil(r - top)), min(f.numel() - 1, math.floor(r + top))
    q = torch.arange(k0, k1 + 1, device="cuda", dtype=torch.float64) - r
    rho = _exact_response(q, z, w).conj() * (q[None, :].abs() <= m[:, None])
    v = rho @ f[k0:k1 + 1]
    return v.real.square() + v.imag.square()


def exact(case, seed):
    kind = case["kind"]
    if kind == "search":
        if _points_of(case, case["n"], case["zmax"], case["wmax"]) > _MAX_POINTS:
            return None
        H = case["stages"].count("-") + 1
        M, mean, std = _exact_maxima(case, _one(case, seed))
        sigma = case["mode"] == "sigma"
        return {"M": M, "found": None,
                "stats": [[float(v) for v in mean], [float(v) for v in std], [None] * H] if sigma else None}
    if kind in ("batch", "serve"):
        n = _lengths(case)
        sub = _ranges(case) if kind == "serve" else [(case["zmax"], case["wmax"])] * len(n)
        if sum(_points_of(case, k, *zw) for k, zw in zip(n, sub)) > _MAX_POINTS:
            return None
        found = [_exact_maxima(case, x, *zw) for x, zw in zip(_several(case, seed), sub)]
        sigma = case["mode"] == "sigma"
        return {"M": [m for m, _, _ in found], "found": None, "theta": None,
                "mean": torch.stack([mean for _, mean, _ in found]) if sigma else None,
                "std": torch.stack([std for _, _, std in found]) if sigma else None}
    if kind == "plane":
        plane = _ExactPlane(case, _one(case, seed))
        zw = _grid(case)[case["t0"]:case["t0"] + case["nt"]]
        return torch.cat([plane.rows(zw[k:k + 16]) for k in range(0, len(zw), 16)])
    if kind == "subharmonic":
        x = _one(case, seed, harmonics=4)
        plane = _ExactPlane(case, x)
        grid = _grid(case)
        rows = torch.cat([plane.rows(grid[k:k + 16]) for k in range(0, len(grid), 16)])
        nz, zc, wc = 2 * case["zmax"] // case["dz"] + 1, case["zmax"] // case["dz"], case["wmax"] // case["dw"]

        def near(a, h, H):                                # h a / H to the nearest, halves away from zero
            q = (2 * abs(a) * h + H) // (2 * H)
            return q if a >= 0 else -q

        out, stats = [], []
        for H in (int(h) for h in case["stages"].split("-")):
            q = torch.arange(plane.bN, device="cuda")
            best = torch.full((plane.bN,), -1.0, dtype=torch.float64, device="cuda")
            s1 = s2 = 0.0
            at = [(2 * q * h + H) // (2 * H) for h in range(1, H + 1)]
            for t in range(len(grid)):
                zi, wi = t % nz - zc, t // nz - wc
                S = sum(rows[(near(wi, h, H) + wc) * nz + near(zi, h, H) + zc][at[h - 1]] for h in range(1, H + 1))
                best = torch.maximum(best, S)
                s1, s2 = s1 + S.sum(), s2 + S.square().sum()
            n = float(len(grid) * plane.bN)
            out.append(best)
            stats.append([float(s1 / n), float((s2 / n - (s1 / n) ** 2).clamp(min=0).sqrt()), None])
        return {"M": out, "stats": stats, "p": None, "t": None}
    if kind == "refine":
        f = _exact_normalised(_one(case, seed))
        power, inside = [], []
        for c in _points(case, seed):
            zw = [(c.z + j * case["dz"] / 4.0, c.w + k * case["dw"] / 4.0)
                  for j in range(-case["hz"], case["hz"] + 1) for k in range(-case["hw"], case["hw"] + 1)]
            grid = [_exact_powers(f, c.r + 0.125 * i, zw) for i in range(-case["hr"], case["hr"] + 1)]
            power.append(torch.stack(grid).max())
            inside.append(grid[case["hr"]][len(zw) // 2])
        return {"power": torch.stack(power), "power_in": torch.stack(inside), "rzw": None}
    zw = _grid(case)
    nt = min(32, len(zw))
    t0 = int(np.random.RandomState(seed % (1 << 31)).randint(0, len(zw) - nt + 1))
    part = zw[t0:t0 + nt]
    return {"bank": None, "taps": _exact_taps(case, [z for z, _ in part], [w for _, w in part],
                                              _halfwidth(case["zmax"], case["wmax"]))}
