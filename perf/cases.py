"""Timing cases of the cross-section library: what a user of the package has it do.

A case is a call (or the short sequence of calls) that a program makes through the package's
public functions, on synthetic line lists with the distributions of the repository's workloads
(rox_synth/workloads.py): the plain HITRAN list, the ExoMol list, the (P,T) table, the large list
streamed in chunks, the resident lists of the request server, user-provided nodes, line selection,
broadening mixtures, CIA restructuring, loading a list, and the line tables alone.

Inputs are drawn on the GPU from the seed. exact() restates the definitions of include/rox.h in
64-bit torch arithmetic, with a Faddeeva function of its own (Matta and Reichel 1971: trapezoidal
or midpoint rule with the pole correction).
"""
import math

import numpy as np
import torch

import paper_2510_20870_gb300 as rox

DEV = "cuda"
HITRAN, EXOMOL = 0, 1
C_CM, C_M, KB, HPL, AMU = 2.99792458e10, 2.99792458e8, 1.380649e-23, 6.62607015e-34, 1.66053906660e-27
C2 = HPL * C_CM / KB
T_REF, P_REF = 296.0, 1.01325
Q_A = 0.05                     # Q(T) = Q_A T^1.5
FLOPS_PAIR = 11                # FP32 operations of one far-wing profile value added to a point
FLOPS_LINE = 60                # strength, widths and profile constants of one line at one (P,T) point
NEAR = 64                      # points of a line's window that lie near its centre (the rest is a smooth wing)


def listed():
    return [
        # one pass over a small HITRAN list: the smallest call, launches and latency
        {"name": "plain_1e4", "kind": "xsec", "conv": HITRAN, "lines": 10_000, "lo": 2000.0, "hi": 2500.0, "dnu": 0.01,
         "points": 50_001, "cutoff": 25.0, "mass": 18.0, "el": 3000.0, "half": False, "bands": 0,
         "p": 1.0, "t": 1000.0},
        # a laboratory window at room temperature and low pressure, finer grid, odd sizes
        {"name": "window_2e5", "kind": "xsec", "conv": HITRAN, "lines": 230_017, "lo": 1000.0, "hi": 2000.0,
         "dnu": 0.005, "points": 200_003, "cutoff": 25.0, "mass": 18.0, "el": 3000.0, "half": False, "bands": 0,
         "p": 0.01, "t": 296.0},
        # one cross-section of an ExoMol list over the whole infrared and visible range
        {"name": "exomol_1e7", "kind": "xsec", "conv": EXOMOL, "lines": 10_000_000, "lo": 300.0, "hi": 30000.0,
         "dnu": 0.01, "points": 2_970_001, "cutoff": 25.0, "mass": 16.0, "el": 5000.0, "half": False, "bands": 0,
         "p": 0.1, "t": 1500.0},
        # an opacity table: pressures x temperatures in one call, lines gathered in bands
        {"name": "table_1e6_8x5", "kind": "batch", "conv": EXOMOL, "lines": 1_000_000, "lo": 300.0, "hi": 30000.0,
         "dnu": 0.01, "points": 2_970_001, "cutoff": 25.0, "mass": 16.0, "el": 5000.0, "half": False, "bands": 12,
         "np": 8, "nt": 5, "p_lo": 1e-5, "p_hi": 1e2, "t_lo": 300.0, "t_hi": 3000.0, "kahan": False},
        # a list too long for one call, added into one cross-section chunk by chunk (half widths, hot, 10 bar)
        {"name": "stream_2x5e7", "kind": "stream", "conv": HITRAN, "lines": 50_000_000, "chunks": 2, "lo": 500.0,
         "hi": 10000.0, "dnu": 0.01, "points": 950_001, "cutoff": 100.0, "mass": 18.0, "el": 1000.0, "half": True,
         "bands": 0, "p": 10.0, "t": 3000.0},
        # cross-sections on a grid of fixed resolving power
        {"name": "nodes_3e6_R645000", "kind": "nodes", "conv": EXOMOL, "lines": 3_000_000, "lo": 300.0, "hi": 30000.0,
         "R": 645_000.0, "cutoff": 25.0, "mass": 16.0, "el": 5000.0, "half": False, "bands": 0, "np": 1, "nt": 2,
         "p_lo": 0.1, "p_hi": 0.1, "t_lo": 800.0, "t_hi": 1500.0},
        # main contributors only, two temperatures
        {"name": "select_1e7", "kind": "select", "conv": EXOMOL, "lines": 10_000_000, "lo": 300.0, "hi": 30000.0,
         "dnu": 0.01, "points": 2_970_001, "cutoff": 25.0, "mass": 16.0, "el": 5000.0, "half": False, "bands": 0,
         "np": 1, "nt": 2, "p_lo": 0.1, "p_hi": 0.1, "t_lo": 1000.0, "t_hi": 1500.0, "rel": 1e-3, "bin": 1.0},
        # an H2 + He mixture with natural broadening at three pressures
        {"name": "broadened_1e6_3", "kind": "broad", "conv": EXOMOL, "lines": 1_000_000, "lo": 300.0, "hi": 30000.0,
         "dnu": 0.01, "points": 2_970_001, "cutoff": 25.0, "mass": 16.0, "el": 5000.0, "half": False, "bands": 0,
         "np": 3, "nt": 1, "p_lo": 1e-3, "p_hi": 10.0, "t_lo": 1500.0, "t_hi": 1500.0},
        # a batch of server requests: windows of 10 to 5000 cm^-1 on three resident lists, each at its own (P,T)
        {"name": "serve_16", "kind": "jobs", "jobs": 16, "l0": 100_000, "l1": 1_000_000, "l2": 10_000_000,
         "w_lo": 10.0, "w_hi": 5000.0},
        # loading a list: sort by line centre, windows and span ranges on the lattice
        {"name": "load_1e7", "kind": "load", "conv": EXOMOL, "lines": 10_000_000, "lo": 300.0, "hi": 30000.0,
         "dnu": 0.01, "points": 2_970_001, "cutoff": 25.0, "mass": 16.0, "el": 5000.0, "half": False, "bands": 0},
        # collision-induced absorption tables onto the grid, one row per temperature
        {"name": "cia_40", "kind": "cia", "nt": 40, "samples": 4000, "lo": 300.0, "dnu": 0.01, "points": 2_970_001},
        # the line tables alone: strengths and widths of every line
        {"name": "tables_1e7", "kind": "tables", "conv": EXOMOL, "lines": 10_000_000, "lo": 300.0, "hi": 30000.0,
         "mass": 16.0, "el": 5000.0, "half": False, "bands": 0, "p": 0.1, "t": 1500.0},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """A case of the same ranges: P 1e-5..1e2 bar, T 296..3000 K, 5e3 to 3e7 lines, steps 0.002..0.05 cm^-1."""
    kind = rng.choice(["xsec", "xsec", "batch", "batch", "stream", "nodes", "select", "broad", "jobs", "load", "cia",
                       "tables"])
    if kind == "cia":
        return {"kind": kind, "nt": rng.randint(1, 40), "samples": int(_log(rng, 50, 6000)), "lo": rng.uniform(20, 2000),
                "dnu": _log(rng, 0.005, 0.1), "points": int(_log(rng, 2e4, 2.9e6)) | 1}
    if kind == "jobs":
        return {"kind": kind, "jobs": rng.randint(1, 24), "l0": int(_log(rng, 3e4, 3e5)), "l1": int(_log(rng, 3e5, 3e6)),
                "l2": int(_log(rng, 3e6, 1e7)), "w_lo": 10.0, "w_hi": _log(rng, 300.0, 5000.0)}
    hitran = kind == "stream" or rng.random() < 0.4
    c = {"kind": kind, "conv": HITRAN if hitran else EXOMOL, "lines": int(_log(rng, 5e3, 3e7)),
         "mass": rng.choice([2.0, 16.0, 18.0, 28.0, 44.0, 64.0]), "el": rng.choice([1000.0, 3000.0, 5000.0]),
         "half": rng.random() < 0.3, "bands": rng.choice([0, 0, 5, 30])}
    if hitran:
        c["el"] = 1000.0
    c["lo"] = rng.uniform(100.0, 8000.0)
    if kind == "load" or kind == "tables":
        c["hi"] = c["lo"] + _log(rng, 100.0, 20000.0)
    if kind == "tables":
        return {**c, "p": _log(rng, 1e-5, 1e2), "t": rng.uniform(296.0, 3000.0)}
    if kind == "nodes":
        c["R"] = _log(rng, 1e5, 1e6)
        c["hi"] = c["lo"] * math.exp(_log(rng, 2e4, 2.5e6) / c["R"])
        step = (c["hi"] - c["lo"]) / (c["R"] * math.log(c["hi"] / c["lo"]))
    else:
        c["dnu"] = step = _log(rng, 0.002, 0.05)
        c["points"] = int(_log(rng, 3e3, min(2.9e6, 25000.0 / step))) | 1
        c["hi"] = c["lo"] + c["dnu"] * (c["points"] - 1)
    c["cutoff"] = rng.choice([10.0, 25.0, 25.0, 100.0])
    if kind == "load":
        return c
    if kind in ("xsec", "stream"):
        c["p"], c["t"] = _log(rng, 1e-5, 1e2), rng.uniform(296.0, 3000.0)
        n_pt = 1
    else:
        c["np"], c["nt"] = rng.choice([(1, 1), (1, 2), (3, 1), (4, 3), (5, 8)])
        c["p_lo"], c["p_hi"] = _log(rng, 1e-5, 1e-1), _log(rng, 1e-1, 1e2)
        c["t_lo"], c["t_hi"] = rng.uniform(296.0, 900.0), rng.uniform(900.0, 3000.0)
        n_pt = c["np"] * c["nt"]
    if kind == "stream":
        c["chunks"] = rng.randint(2, 3)
        n_pt = c["chunks"]
    if kind == "batch":
        c["kahan"] = rng.random() < 0.5
    if kind == "select":
        c["rel"], c["bin"] = _log(rng, 1e-6, 1e-2), _log(rng, 0.1, 10.0)
    # at most about a third of the largest listed case's time: points in a line's window, some ten times
    # those of its core of 6.5 Doppler widths, and more where the grid is too short to fill the GPU
    core = 13.0 * _doppler(0.5 * (c["lo"] + c["hi"]), c["mass"], c.get("t", c.get("t_hi")))
    cost = c["lines"] * n_pt * (min(2.0 * c["cutoff"], c["hi"] - c["lo"]) + 10.0 * core) / step
    cost *= max(1.0, 400_000.0 / (n_pt * (c["hi"] - c["lo"]) / step))
    c["lines"] = max(1000, int(c["lines"] * min(1.0, 2.5e11 / cost)))
    return c


# ------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _lines(c, g, n=None, sort=True):
    n = c["lines"] if n is None else n
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if c["bands"]:
        # line centres gathered in bands of 2% of the range, a quarter spread evenly
        centre = torch.rand(c["bands"], generator=g, device=DEV, dtype=torch.float64)
        which = torch.randint(0, c["bands"], (n,), generator=g, device=DEV)
        z = torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
        b = (centre[which] + 0.02 * z).clamp_(1e-6, 1.0 - 1e-6)
        u = torch.where(u < 0.25, u * 4.0, b)
    nu0 = c["lo"] + (c["hi"] - c["lo"]) * u
    if sort:
        nu0 = torch.sort(nu0).values
    f = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, device=DEV)  # noqa: E731
    wd = torch.float16 if c["half"] else torch.float32
    if c["conv"] == HITRAN:
        s = torch.exp(f(math.log(1e-30), math.log(1e-19)))
    else:
        s = torch.exp(f(math.log(1e-8), math.log(1e2)))
    return {"nu0": nu0, "s_or_a": s,
            "g_up": torch.randint(1, 101, (n,), generator=g, device=DEV).float() if c["conv"] == EXOMOL else None,
            "e_lower": -c["el"] * torch.log(1.0 - torch.rand(n, generator=g, device=DEV)),
            "gamma_ref": f(0.02, 0.1).to(wd), "n_t": f(0.4, 0.8).to(wd), "convention": c["conv"]}


def _q(t):
    return Q_A * t ** 1.5


def _pts(c):
    if "p" in c:
        return [(c["p"], c["t"])]
    ps = np.logspace(math.log10(c["p_lo"]), math.log10(c["p_hi"]), c["np"])
    ts = np.linspace(c["t_lo"], c["t_hi"], c["nt"]) if c["nt"] > 1 else [c["t_hi"]]
    return [(float(p), float(t)) for p in ps for t in ts]


def _grid(c):
    return (c["lo"], c["dnu"], c["points"])


def _bytes(n):
    return torch.empty(int(n), dtype=torch.uint8, device=DEV)


def _nodes(c):
    n = int(math.floor(math.log(c["hi"] / c["lo"]) / math.log1p(1.0 / c["R"]))) + 1
    k = torch.arange(n, device=DEV, dtype=torch.float64)
    return c["lo"] * torch.exp(k * math.log1p(1.0 / c["R"]))


def _cia_tables(c, g):
    """Per temperature one to three blocks that split 20..10000 cm^-1, irregular samples."""
    r = np.random.RandomState(int(torch.randint(0, 2 ** 31 - 1, (1,), generator=g, device=DEV)))
    temps = [float(t) for t in np.linspace(200.0, 3000.0, c["nt"])]
    T, off, nu, k = [], [0], [], []
    for t in temps:
        nb = r.randint(1, 4)
        e = np.linspace(20.0, 10000.0, nb + 1)
        centre = 20.0 + 9980.0 * r.rand()
        for b in range(nb):
            x = np.sort(e[b] + (e[b + 1] - e[b]) * r.rand(max(2, c["samples"] // nb)))
            x[0], x[-1] = e[b], e[b + 1]
            x = np.unique(x)
            T.append(t)
            nu.append(x)
            k.append(1e-45 * math.sqrt(t / 300.0) * (np.exp(-((x - centre) / 998.0) ** 2)
                                                     + 0.3 * np.exp(-((x - 20.0) / 200.0) ** 2) + 0.01))
            off.append(off[-1] + x.size)
    return temps, T, off, torch.from_numpy(np.concatenate(nu)).to(DEV), torch.from_numpy(np.concatenate(k)).to(DEV)


LATTICE = (300.0, 0.01, 2_970_001)


def _requests(c, seed):
    """(list, first point, points, P, T) of each request: the windows are the case's, the (P,T) the seed's."""
    w, r = np.random.RandomState(1000 * c["jobs"] + int(c["w_hi"])), np.random.RandomState(seed % (2 ** 31))
    out = []
    for _ in range(c["jobs"]):
        n = int(round(w.uniform(c["w_lo"], c["w_hi"]) / 0.01)) + 1
        out.append((int(w.randint(3)), int(w.randint(LATTICE[2] - n + 1)), n,
                    float(math.exp(r.uniform(math.log(1e-5), math.log(1e2)))), float(r.uniform(300.0, 3000.0))))
    return out


def prepare(c, seed):
    g = _gen(seed)
    k = c["kind"]
    st = {"c": c}
    if k == "cia":
        st["temps"], st["T"], st["off"], st["nu"], st["k"] = _cia_tables(c, g)
        st["out"] = torch.empty((c["nt"], c["points"]), dtype=torch.float64, device=DEV)
        st["ws"] = _bytes(rox.rox_cia_workspace_size(len(st["T"]), st["off"][-1]))
        return st
    if k == "jobs":
        base = {"conv": EXOMOL, "lo": 300.0, "hi": 30000.0, "el": 5000.0, "half": False, "bands": 0}
        st["lists"] = [_lines(base, g, n) for n in (c["l0"], c["l1"], c["l2"])]
        st["prepared"] = [rox.Prepared(L, LATTICE, 25.0) for L in st["lists"]]
        st["req"] = _requests(c, seed)
        st["out"] = [torch.empty(n, dtype=torch.float32, device=DEV) for _, _, n, _, _ in st["req"]]
        st["ws"] = _bytes(rox.rox_jobs_workspace_size(_jobs(st)))
        return st
    if k == "load":
        st["lines"] = _lines(c, g, sort=False)
        st["sorted"] = {n: (torch.empty_like(v) if torch.is_tensor(v) else v) for n, v in st["lines"].items()}
        st["perm"] = torch.empty(c["lines"], dtype=torch.int64, device=DEV)
        st["ws"] = _bytes(rox.rox_sort_workspace_size(c["lines"]))
        return st
    if k == "stream":
        st["lines"] = [_lines(c, g) for _ in range(c["chunks"])]
        st["out"] = torch.empty((1, c["points"]), dtype=torch.float32, device=DEV)
        st["ws"] = _bytes(rox.rox_xsec_workspace_size(c["lines"], _grid(c), 1))
        return st
    st["lines"] = _lines(c, g)
    n = c["lines"]
    if k == "tables":
        st["out"] = [torch.empty(n, dtype=torch.float32, device=DEV) for _ in range(3)]
        return st
    pts = _pts(c)
    n_temps = len({t for _, t in pts})
    if k == "nodes":
        st["nodes"] = _nodes(c)
        m = st["nodes"].numel()
        st["ws"] = _bytes(rox.rox_xsec_nodes_workspace_size(n, m, n_temps))
    else:
        m = c["points"]
        if k == "select":
            st["ws"] = _bytes(rox.rox_xsec_select_workspace_size(n, _grid(c), n_temps, c["cutoff"], c["rel"], c["bin"]))
        elif k == "broad":
            st["ws"] = _bytes(rox.rox_xsec_broadened_workspace_size(n, _grid(c), n_temps))
        else:
            st["ws"] = _bytes(rox.rox_xsec_workspace_size(n, _grid(c), n_temps))
    if k == "broad":
        st["br"] = {"vmr": [0.85, 0.15], "gamma_ref": [st["lines"]["gamma_ref"], None],
                    "n_t": [st["lines"]["n_t"], None],
                    "table_gamma": [None, 0.02 + 0.03 * torch.rand(100, generator=g, device=DEV)],
                    "table_n": [None, 0.3 + 0.3 * torch.rand(100, generator=g, device=DEV)],
                    "j_lower": torch.randint(0, 100, (n,), generator=g, device=DEV, dtype=torch.int32),
                    "natural": c["conv"] == EXOMOL}
    st["out"] = torch.empty((len(pts), m), dtype=torch.float32, device=DEV)
    return st


def _jobs(st):
    return [rox.make_job(st["prepared"][l], l, first, n, p, t, _q(t), _q(T_REF), 16.0, o)
            for (l, first, n, p, t), o in zip(st["req"], st["out"])]


def run(st):
    c = st["c"]
    k = c["kind"]
    if k == "cia":
        rox.rox_cia_regrid(st["T"], st["off"], st["nu"], st["k"], _grid(c), st["temps"], st["out"], st["ws"])
        return st["out"]
    if k == "jobs":
        rox.rox_xsec_jobs(st["prepared"], _jobs(st), st["ws"])
        return st["out"]
    if k == "load":
        rox.rox_sort_lines(st["lines"], st["sorted"], st["perm"], st["ws"])
        p = rox.Prepared(st["sorted"], _grid(c), c["cutoff"])
        return {**{n: v for n, v in st["sorted"].items() if torch.is_tensor(v)}, "perm": st["perm"],
                "span_lo": p.span_lo, "span_hi": p.span_hi}
    pts = _pts(c)
    P, T = [p for p, _ in pts], [t for _, t in pts]
    Q, Qr = [_q(t) for t in T], _q(T_REF)
    if k == "tables":
        rox.rox_line_strengths(st["lines"], T[0], Q[0], Qr, st["out"][0])
        rox.rox_line_widths(st["lines"], c["mass"], P[0], T[0], st["out"][1], st["out"][2])
        return st["out"]
    m, cut = c["mass"], c["cutoff"]
    if k == "xsec":
        rox.rox_xsec(st["lines"], _grid(c), P[0], T[0], Q[0], Qr, m, cut, st["out"], st["ws"])
    elif k == "stream":
        for i, L in enumerate(st["lines"]):
            rox.rox_xsec_batch(L, _grid(c), P, T, Q, Qr, m, cut, st["out"], st["ws"],
                               flags=rox.ROX_KAHAN | (rox.ROX_ACCUMULATE if i else 0))
    elif k == "batch":
        rox.rox_xsec_batch(st["lines"], _grid(c), P, T, Q, Qr, m, cut, st["out"], st["ws"],
                           flags=rox.ROX_KAHAN if c["kahan"] else 0)
    elif k == "nodes":
        rox.rox_xsec_nodes_batch(st["lines"], st["nodes"], P, T, Q, Qr, m, cut, st["out"], st["ws"])
    elif k == "select":
        rox.rox_xsec_select_batch(st["lines"], _grid(c), P, T, Q, Qr, m, cut, c["rel"], c["bin"], st["out"], st["ws"])
    else:
        rox.rox_xsec_broadened_batch(st["lines"], _grid(c), st["br"], P, T, Q, Qr, m, cut, st["out"], st["ws"])
    return st["out"]


def work(c):
    """Bytes: the line columns read once, the outputs written once. Flops of a cross-section: a line's
    constants and its values on the points near its centre, per line and (P,T) point; the wing further
    out is smooth on the grid, so many lines' wings can be summed together and count no more."""
    k = c["kind"]
    if k == "cia":
        return {"bytes": 8.0 * c["nt"] * c["points"] + 16.0 * c["nt"] * c["samples"], "flops": 1.0 * c["nt"] * c["points"]}
    if k == "jobs":
        lines = sum(c[x] for x in ("l0", "l1", "l2")) / 3.0
        width = 0.5 * (c["w_lo"] + c["w_hi"])
        n = c["jobs"] * lines * width / 29700.0
        return {"bytes": 28.0 * n + 400.0 * c["jobs"] * width, "flops": n * (FLOPS_LINE + FLOPS_PAIR * NEAR)}
    n = float(c["lines"] * c.get("chunks", 1))
    row = 8 + 4 * (3 if c["conv"] == EXOMOL else 2) + (4 if c["half"] else 8)
    if k == "load":
        return {"bytes": n * (2 * row + 8) + 16.0 * c["points"] / 256, "flops": 0.0}
    if k == "tables":
        return {"bytes": n * (row + 12), "flops": n * 40.0}
    n_pt = len(_pts(c))
    m = (math.log(c["hi"] / c["lo"]) * c["R"]) if k == "nodes" else float(c["points"])
    # a selection keeps at least the strongest line of each bin: its profiles cannot be counted beforehand
    prof = (c["hi"] - c["lo"]) / c["bin"] if k == "select" else n
    return {"bytes": n * row + 4.0 * n_pt * m, "flops": n * n_pt * FLOPS_LINE + prof * n_pt * FLOPS_PAIR * NEAR}


# ------------------------------------------------------------------------------- 64-bit values
def _strength(L, t):
    nu0, s, e = L["nu0"], L["s_or_a"].double(), L["e_lower"].double()
    stim = -torch.expm1(-C2 * nu0 / t)
    if L["convention"] == HITRAN:
        return s * (_q(T_REF) / _q(t)) * torch.exp(-C2 * e * (1.0 / t - 1.0 / T_REF)) * (
            stim / -torch.expm1(-C2 * nu0 / T_REF))
    return L["g_up"].double() * s / (8.0 * math.pi * C_CM * nu0 * nu0) * torch.exp(-C2 * e / t) * stim / _q(t)


def _doppler(nu0, mass, t):
    return nu0 * (math.sqrt(2.0 * KB * t / (mass * AMU)) / C_M)


def _lorentz(L, p, t):
    return L["gamma_ref"].double() * (T_REF / t) ** L["n_t"].double() * (p / P_REF)


H_STEP = math.sqrt(math.pi / 12.0)


def _re_w(x, y):
    """Re w(x + iy) for x >= 0, y >= 0 (64-bit), y broadcast against x: the rule whose nodes are farther
    from x (trapezoidal or midpoint), step H_STEP, plus the pole term where y < pi / H_STEP."""
    h = H_STEP
    frac = x / h - torch.floor(x / h)
    mid = (frac < 0.25) | (frac > 0.75)           # x near a trapezoidal node: midpoint rule
    shift = mid.to(x.dtype) * (0.5 * h)
    y2 = y * y
    acc = torch.zeros_like(x)
    wt, wm = torch.ones_like(x), mid.to(x.dtype)
    for n in range(-13, 13):
        a, b = math.exp(-(n * h) ** 2), math.exp(-((n + 0.5) * h) ** 2)
        d = x - shift - n * h
        acc += (wt * a + wm * (b - a)) / (d * d + y2)
    k = acc * (y * (h / math.pi))
    pole = (x < 27.0) & (y < math.pi / h)
    yp = torch.clamp(y, max=math.pi / h)
    xp = torch.clamp(x, max=27.0)
    q = torch.exp(-2.0 * math.pi * yp / h)
    th = 2.0 * math.pi * xp / h
    # 2 e^{-z^2} q e^{i th} / (q e^{i th} -+ 1): upper sign trapezoidal, lower midpoint
    cr, ci = q * torch.cos(th), q * torch.sin(th)
    dr = cr + torch.where(mid, 1.0, -1.0)
    den = dr * dr + ci * ci
    fr, fi = (cr * dr + ci * ci) / den, (ci * dr - cr * ci) / den
    amp = 2.0 * torch.exp(yp * yp - xp * xp)
    ph = 2.0 * xp * yp
    return k + torch.where(pole, amp * (torch.cos(ph) * fr + torch.sin(ph) * fi), 0.0)


def _sum(nu, L, S, gG, gL, cutoff):
    """sigma on the points nu (ascending): every line within the cutoff of a point."""
    out = torch.zeros(nu.numel(), dtype=torch.float64, device=DEV)
    pts = 512
    edges = torch.arange(0, nu.numel(), pts, device=DEV)
    last = torch.clamp(edges + pts - 1, max=nu.numel() - 1)
    lo = torch.searchsorted(L["nu0"], nu[edges] - cutoff * (1 + 1e-9) - 1e-6).tolist()
    hi = torch.searchsorted(L["nu0"], nu[last] + cutoff * (1 + 1e-9) + 1e-6, right=True).tolist()
    rows = 60_000
    for b, (i0, i1) in enumerate(zip(lo, hi)):
        p = nu[b * pts:(b + 1) * pts]
        for i in range(i0, i1, rows):
            j = min(i + rows, i1)
            X = p[None, :] - L["nu0"][i:j, None]
            g = gG[i:j, None]
            v = _re_w(X.abs() / g, gL[i:j, None] / g) * (S[i:j, None] / (g * math.sqrt(math.pi)))
            out[b * pts:b * pts + p.numel()] += torch.where(X.abs() <= cutoff, v, 0.0).sum(0)
    return out


MOST_PAIRS = 5e9


def exact(c, seed):
    k = c["kind"]
    pairs = 0.0
    if k == "jobs":
        pairs = c["jobs"] * c["l2"] * (c["w_hi"] / 29700.0) * 5001.0
    elif "cutoff" in c and k != "load":
        step = (c["hi"] - c["lo"]) / (c["R"] * math.log(c["hi"] / c["lo"])) if k == "nodes" else c["dnu"]
        span = c["hi"] - c["lo"]
        pairs = c["lines"] * c.get("chunks", 1) * len(_pts(c)) * min(2.0 * c["cutoff"] + 512 * step, span) / step
        if k != "nodes":
            pairs += len(_pts(c)) * c["points"]
    if pairs > MOST_PAIRS:
        return None
    st = prepare(c, seed)
    if k == "cia":
        return _exact_cia(st)
    if k == "jobs":
        out = []
        for l, first, n, p, t in st["req"]:
            nu = LATTICE[0] + torch.arange(first, first + n, device=DEV, dtype=torch.float64) * LATTICE[1]
            L = st["lists"][l]
            out.append(_sum(nu, L, _strength(L, t), _doppler(L["nu0"], 16.0, t), _lorentz(L, p, t), 25.0))
        return out
    if k == "load":
        order = torch.sort(st["lines"]["nu0"], stable=True).indices
        return {n: v[order].double() for n, v in st["lines"].items() if torch.is_tensor(v)}
    pts = _pts(c)
    if k == "tables":
        L, (p, t) = st["lines"], pts[0]
        return [_strength(L, t), _doppler(L["nu0"], c["mass"], t), _lorentz(L, p, t)]
    if k == "nodes":
        nu = st["nodes"]
    else:
        nu = c["lo"] + torch.arange(c["points"], device=DEV, dtype=torch.float64) * c["dnu"]
    out = []
    for p, t in pts:
        sig = 0.0
        for L in (st["lines"] if k == "stream" else [st["lines"]]):
            S, gG, gL = _strength(L, t), _doppler(L["nu0"], c["mass"], t), _lorentz(L, p, t)
            if k == "broad":
                br = st["br"]
                j = br["j_lower"].long()
                gL = 0.85 * gL + 0.15 * br["table_gamma"][1].double()[j] * (T_REF / t) ** br["table_n"][1].double()[j] * (
                    p / P_REF)
                if br["natural"]:
                    gL = gL + L["s_or_a"].double() / (4.0 * math.pi * C_CM)
            if k == "select":
                o = c["lo"] - c["cutoff"]
                nb = int(math.floor(((c["points"] - 1) * c["dnu"] + 2.0 * c["cutoff"]) / c["bin"])) + 1
                b = torch.floor((L["nu0"] - o) / c["bin"]).long()
                inside = (b >= 0) & (b < nb)
                b = b.clamp(0, nb - 1)
                top = torch.zeros(nb, dtype=torch.float64, device=DEV)
                top.scatter_reduce_(0, b[inside], S[inside], "amax")
                keep = inside & (S >= c["rel"] * top[b])
                L, S, gG, gL = {"nu0": L["nu0"][keep]}, S[keep], gG[keep], gL[keep]
            sig = sig + _sum(nu, L, S, gG, gL, c["cutoff"])
        out.append(sig)
    return torch.stack(out)


def _exact_cia(st):
    c = st["c"]
    nu = c["lo"] + torch.arange(c["points"], device=DEV, dtype=torch.float64) * c["dnu"]
    out = torch.zeros((c["nt"], c["points"]), dtype=torch.float64, device=DEV)
    for r, t in enumerate(st["temps"]):
        done = torch.zeros(c["points"], dtype=torch.bool, device=DEV)
        for b, tb in enumerate(st["T"]):
            if tb != t:
                continue
            x, y = st["nu"][st["off"][b]:st["off"][b + 1]], st["k"][st["off"][b]:st["off"][b + 1]]
            use = (nu >= x[0]) & (nu <= x[-1]) & ~done
            v = nu[use]
            i = (torch.searchsorted(x, v, right=True) - 1).clamp(0, x.numel() - 2)
            out[r, use] = torch.where(v == x[-1], y[-1], y[i] + (y[i + 1] - y[i]) * (v - x[i]) / (x[i + 1] - x[i]))
            done |= use
    return out
