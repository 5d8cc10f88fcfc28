"""What users of this library have it do, as cases that can be timed and compared.

The library walks micromagnetic lines (spin-exchange Wang-Landau at a fixed
number of up spins) and assembles their densities of states.  The kinds of case:

  surface   a handle that is kept: reset, walk every line l = 0..N/2 to a move
            budget or to ln f_min, assemble, fetch the whole surface
  lines     the same for a few chosen lines of a lattice too large to walk whole
  resume    a walk continued from a checkpoint in the caller's own device
            buffers (wl_walk_noalloc): late stages, walkers all over their range
  serve     a burst of requests for mixed lattices through the serving loop
  thermo    thermodynamics on a (T, H) grid from an assembled surface

Every walk is a function of its lattice, options and seed alone, so its counters
and its surface are the same on every run.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1302_2320_gb300 as wl

CONVERGE = 2**62                    # a move budget that no walk reaches
Z = {"square": 4, "triangular": 6, "cubic": 6, "square_open": 4}
EXACT_MOVES = 1_500_000             # longest walk that exact() repeats in Python

# the requests of one burst: small lattices of every kind, two of them alike
SERVE_MIX = [("square", 16), ("triangular", 16), ("cubic", 6), ("square_open", 15),
             ("square", 24), ("square", 12), ("cubic", 8), ("square", 16)]


def _surface(name, lattice, L, u, C, budget, det=1, check_per_bin=0):
    return {"name": name, "kind": "surface", "lattice": lattice, "L": L, "ln_f_min": u, "check_interval": C,
            "check_per_bin": check_per_bin, "budget": budget, "deterministic": det}


def listed():
    return [
        # the smallest job there is: 4x4 walked to convergence at the accurate
        # ln f_min, the first thing anyone runs and checks against enumeration
        _surface("square4_to_convergence", "square", 4, 1e-8, 1000, CONVERGE),
        # a small surface with frequent flatness checks (N not a power of two)
        _surface("square12_frequent_checks", "square", 12, 1e-8, 1000, 1 << 18),
        # a surface with fewer lines than the GPU has SMs: the speed of one walker
        _surface("square16_few_lines", "square", 16, 1e-6, 16384, 1 << 20),
        # a middle-sized surface whose check interval grows with the line's bins
        _surface("square32_check_per_bin", "square", 32, 1e-7, 16384, 1 << 19, check_per_bin=40),
        # the headline workload: the whole 64x64 surface
        _surface("square64_surface", "square", 64, 1e-6, 16384, 1 << 20),
        # three times more lines than fit the GPU at once, lists of 18 KB each
        _surface("square96_surface", "square", 96, 1e-6, 16384, 1 << 17),
        # production acceptance (FP32) on six neighbours
        _surface("triangular32_production", "triangular", 32, 1e-7, 16384, 1 << 18, det=0),
        # three dimensions
        _surface("cubic8_surface", "cubic", 8, 1e-6, 16384, 1 << 19),
        # the four lines N/8, N/4, 3N/8, N/2 of the largest lattice, at ln f_min = N 1e-9
        {"name": "square256_four_lines", "kind": "lines", "lattice": "square", "L": 256, "lines": 4,
         "ln_f_min": 6.5536e-5, "check_interval": 16384, "budget": 1 << 19, "deterministic": 1},
        # a long walk taken up again: acceptance is low, ln f small, every bin known
        {"name": "resume_square16", "kind": "resume", "lattice": "square", "L": 16, "ln_f_min": 1e-6,
         "check_interval": 4096, "before": 1 << 21, "budget": 1 << 19, "deterministic": 1},
        # a burst of eight requests through the serving loop
        {"name": "serve_mixed_burst", "kind": "serve", "requests": 8, "ln_f_min": 1e-6, "check_interval": 1000,
         "budget": 1 << 18, "max_active": 8},
        # temperature scan over the 32x32 surface at a few fields (specific heat, susceptibility)
        {"name": "thermo_square32_scan", "kind": "thermo", "lattice": "square", "L": 32, "ln_f_min": 0.05,
         "check_interval": 16384, "budget": 1 << 20, "deterministic": 1, "temperatures": 64, "fields": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["surface", "surface", "surface", "surface", "lines", "resume", "serve", "thermo"])
    lattice = rng.choice(["square", "square", "triangular", "cubic", "square_open"])
    u = rng.choice([1e-6, 1e-7, 1e-8])
    C = rng.choice([1000, 4096, 16384])
    if kind == "surface":
        L = _log_int(rng, *{"square": (4, 96), "triangular": (4, 48), "cubic": (3, 12), "square_open": (4, 64)}[lattice])
        lines = _sites(lattice, L) // 2 + 1
        top = min(1 << 20, (1 << 28) // lines)
        return {"kind": kind, "lattice": lattice, "L": L, "ln_f_min": u, "check_interval": C,
                "check_per_bin": rng.choice([0, 0, 40]), "budget": _log_int(rng, min(1 << 12, top // 2), top),
                "deterministic": rng.choice([1, 1, 0])}
    if kind == "lines":
        return {"kind": kind, "lattice": "square", "L": _log_int(rng, 64, 256), "lines": rng.randint(1, 16),
                "ln_f_min": u, "check_interval": 16384, "budget": _log_int(rng, 1 << 14, 1 << 19),
                "deterministic": rng.choice([1, 1, 0])}
    if kind == "resume":
        lattice = rng.choice(["square", "triangular", "cubic"])
        L = _log_int(rng, *{"square": (4, 32), "triangular": (4, 24), "cubic": (3, 8)}[lattice])
        return {"kind": kind, "lattice": lattice, "L": L, "ln_f_min": u, "check_interval": C,
                "before": _log_int(rng, 1 << 16, 1 << 20), "budget": _log_int(rng, 1 << 14, 1 << 19),
                "deterministic": rng.choice([1, 1, 0])}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(1, 8), "ln_f_min": u, "check_interval": C,
                "budget": _log_int(rng, 1 << 13, 1 << 18), "max_active": rng.randint(1, 8)}
    L = _log_int(rng, *{"square": (4, 40), "triangular": (4, 32), "cubic": (3, 9), "square_open": (4, 40)}[lattice])
    return {"kind": kind, "lattice": lattice, "L": L, "ln_f_min": 0.05, "check_interval": 4096,
            "budget": _log_int(rng, 1 << 14, 1 << 19), "deterministic": 1, "temperatures": _log_int(rng, 1, 64),
            "fields": rng.randint(1, 4)}


# ---------------------------------------------------------------------------
# sizes of the problem (Eq. 1, Eq. 2)
# ---------------------------------------------------------------------------

def _sites(lattice, L):
    return L**3 if lattice == "cubic" else L * L


def _bonds(lattice, L):
    return 2 * L * (L - 1) if lattice == "square_open" else _sites(lattice, L) * Z[lattice] // 2


def _k_step(lattice):
    return 1 if lattice == "square_open" else 2


def _bins(lattice, L, ell):
    N = _sites(lattice, L)
    return min(Z[lattice] * min(ell, N - ell), _bonds(lattice, L)) // _k_step(lattice) + 1


def _chosen_lines(case):
    N, n = _sites(case["lattice"], case["L"]), case["lines"]
    return [(i + 1) * (N // 2) // n for i in range(n)]


def _grid(case, seed):
    rng = np.random.default_rng(seed)
    T = np.sort(rng.uniform(0.8, 6.0, case["temperatures"]))
    H = np.concatenate([[0.0], rng.uniform(0.05, 1.0, case["fields"] - 1)])
    return T, H


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _handle(case, seed):
    h = wl.Handle(case["lattice"], case["L"], seed=seed & 0xFFFFFFFF, check_interval=case["check_interval"],
                  check_per_bin=case.get("check_per_bin", 0), move_budget=case["budget"],
                  deterministic=case["deterministic"])
    if case["kind"] == "lines":
        h.select_lines(_chosen_lines(case))
    return h


def _walk_noalloc(case, seed, budget, init, buffers):
    f = wl.lib().wl_walk_noalloc
    i32, i64, dbl, vp = ctypes.c_int, ctypes.c_int64, ctypes.c_double, ctypes.c_void_p
    f.restype = i32
    f.argtypes = [i32, i32, i32, i32, ctypes.c_uint32, i32, dbl, dbl, i64, i64, i32, i32, vp, vp, vp, vp, vp, i64]
    lines = _sites(case["lattice"], case["L"]) // 2 + 1
    rc = f(wl.LATTICES[case["lattice"]], case["L"], 0, lines, seed & 0xFFFFFFFF, case["deterministic"],
           case["ln_f_min"], 0.8, case["check_interval"], budget, 0, init, *[b.data_ptr() for b in buffers],
           torch.cuda.current_stream().cuda_stream)
    if rc not in (wl.WL_OK, wl.WL_ENOTCONVERGED):
        raise RuntimeError(f"wl_walk_noalloc: {rc}: {wl.wl_last_error()}")


def prepare(case, seed):
    state = {"case": case, "seed": seed}
    kind = case["kind"]
    if kind in ("surface", "lines"):
        state["handle"] = _handle(case, seed)
    elif kind == "resume":
        # the checkpoint: list entries, packed spins, ln g, histogram, line states
        lattice, L = case["lattice"], case["L"]
        N = _sites(lattice, L)
        lines = N // 2 + 1
        P, W = (2 * N + 15) // 16 * 8, ((N + 31) // 32 * 4 + 15) // 16 * 4
        bins = sum(_bins(lattice, L, ell) for ell in range(lines))
        sizes = [(lines * P, torch.int16), (lines * W, torch.int32), (bins, torch.int64), (bins, torch.int64),
                 (lines * 9, torch.int64)]
        state["buffers"] = [torch.zeros(n, dtype=t, device="cuda") for n, t in sizes]
        _walk_noalloc(case, seed, case["before"], 1, state["buffers"])
        state["checkpoint"] = [b.clone() for b in state["buffers"]]
    elif kind == "serve":
        state["server"] = wl.Server(max_active=case["max_active"])
    else:
        h = _handle(case, seed)
        h.run(case["ln_f_min"])
        h.assemble()
        state["handle"] = h
        state["T"], state["H"] = _grid(case, seed)
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind in ("surface", "lines"):
        h = state["handle"]
        h.reset()
        h.run(case["ln_f_min"])
        h.assemble()
        st = h.stats()
        out = {"counters": np.array([st[k] for k in ("moves", "accepts", "checks", "lines_converged", "min_stage",
                                                     "max_stage")], dtype=np.int64)}
        if kind == "surface":
            out["surface"], out["offsets"] = h.get_surface()
        else:
            out["lines"] = [h.get_lng(ell) for ell in _chosen_lines(case)]
        return out
    if kind == "resume":
        for b, c in zip(state["buffers"], state["checkpoint"]):
            b.copy_(c)
        _walk_noalloc(case, state["seed"], case["before"] + case["budget"], 0, state["buffers"])
        # the last word of a line's state counts batches, which is no part of the walk
        perm, spins, lng, hist, scal = state["buffers"]
        return {"perm": perm, "spins": spins, "lng": lng, "hist": hist, "state": scal.view(-1, 9)[:, :8]}
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(lattice, L, seed=(state["seed"] + i) & 0xFFFFFFFF, ln_f_min=case["ln_f_min"],
                          check_interval=case["check_interval"], move_budget=case["budget"])
               for i, (lattice, L) in enumerate(SERVE_MIX[:case["requests"]])]
        out = {}
        for i, rid in enumerate(ids):
            srv.wait(rid)
            out["moves%d" % i] = srv.info(rid)["moves"]
            out["surface%d" % i] = srv.result(rid)
            srv.release(rid)
        return out
    return {"thermo": state["handle"].thermo(state["T"], state["H"])}


# ---------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------

# Integer operations of one move attempt: a Philox block (20 wide products and 20
# xors), two list picks, eight neighbour bits and their sums, the test of Eq. 3
# and the updates (23 products and 113 add/logic operations on four neighbours).
MOVE_OPS = 136


def _surface_work(lattice, L, ells, moves):
    N = _sites(lattice, L)
    bins = sum(_bins(lattice, L, ell) for ell in ells)
    # lists and spins written once, ln g and histogram written once and read
    # once by the assembly, the assembled surface written and fetched
    return len(ells) * (2 * N + N // 8) + bins * (16 + 16 + 16), MOVE_OPS * moves


def work(case):
    kind = case["kind"]
    if kind == "serve":
        parts = [_surface_work(la, L, range(_sites(la, L) // 2 + 1), case["budget"] * (_sites(la, L) // 2))
                 for la, L in SERVE_MIX[:case["requests"]]]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    lattice, L = case["lattice"], case["L"]
    N = _sites(lattice, L)
    ells = _chosen_lines(case) if kind == "lines" else range(N // 2 + 1)
    bins = sum(_bins(lattice, L, ell) for ell in ells)
    if kind == "thermo":
        points = case["temperatures"] * case["fields"]
        # one exponential (about 20 operations) and its moments per bin and temperature, the field per line
        return {"bytes": bins * 8 + points * 48, "flops": 30 * bins * case["temperatures"] + 40 * len(ells) * points}
    if kind == "resume":
        b = len(ells) * (2 * N + N // 8 + 72) * 2 + bins * 32
        return {"bytes": b, "flops": MOVE_OPS * case["budget"] * (len(ells) - 1)}
    # a converging 4x4 line takes about 25 000 moves
    moves = min(case["budget"], 25_000) if case["budget"] >= CONVERGE else case["budget"]
    b, f = _surface_work(lattice, L, ells, moves * sum(1 for ell in ells if ell))
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# exact: the same walk and assembly in plain Python, for walks short enough
# ---------------------------------------------------------------------------

def _philox(counter0, counter2, key0, key1):
    """Philox4x32-10 of counters (counter0, 0, counter2, 0): words 0, 1, 2."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [counter0.astype(np.uint64), np.zeros_like(counter0, dtype=np.uint64),
         np.full(counter0.shape, counter2, dtype=np.uint64), np.zeros_like(counter0, dtype=np.uint64)]
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(key0), p1 & m32,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(key1), p0 & m32]
        key0, key1 = (key0 + 0x9E3779B9) & 0xFFFFFFFF, (key1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[:3]


def _neighbours(lattice, L):
    N = _sites(lattice, L)
    out = []
    for i in range(N):
        x, y, z = i % L, i // L % L, i // (L * L)
        if lattice == "cubic":
            at = lambda a, b, c: (c % L * L + b % L) * L + a % L  # noqa: E731
            out.append([at(x + 1, y, z), at(x - 1, y, z), at(x, y + 1, z), at(x, y - 1, z), at(x, y, z + 1), at(x, y, z - 1)])
            continue
        y = i // L
        steps = [(1, 0), (-1, 0), (0, 1), (0, -1)] + ([(1, -1), (-1, 1)] if lattice == "triangular" else [])
        if lattice == "square_open":
            out.append([(y + b) * L + x + a for a, b in steps if 0 <= x + a < L and 0 <= y + b < L])
        else:
            out.append([(y + b) % L * L + (x + a) % L for a, b in steps])
    return out


def _exact_line(case, nbs, ell, seed):
    """The walk of one line: (ln g in units of ln f_min, visited, counters)."""
    lattice, L, u = case["lattice"], case["L"], case["ln_f_min"]
    N, nbins, step = _sites(lattice, L), _bins(lattice, L, ell), _k_step(lattice)
    lng, hist, visited = [0] * nbins, [0] * nbins, [False] * nbins
    C = max(case["check_interval"], case.get("check_per_bin", 0) * nbins)
    perm = list(range(N))
    for t, r in enumerate(_philox(np.arange(ell), 1, ell, seed)[0].tolist() if ell else []):
        j = t + (r * (N - t) >> 32)
        perm[t], perm[j] = perm[j], perm[t]
    up = [0] * N
    for i in perm[:ell]:
        up[i] = 1
    k = sum(up[i] != up[j] for i in range(N) for j in nbs[i]) // 2
    if ell == 0:
        visited[0] = True
        return lng, visited, (0, 0, 0, 1, 0)
    q = next(q for q in range(40) if 4095.0 * 2.0**q * u >= 32.0 * math.log(2.0))
    x = (np.arange(4096, dtype=np.float64) * 2.0**q) * u
    table = [int(v) for v in np.floor(np.ldexp(np.exp(-x.astype(np.longdouble)), 32) + 0.5)]
    low, F, t, accepts, checks, stage, b = (1 << q) - 1, int(round(1.0 / u)), 0, 0, 0, 0, k // step
    while t < case["budget"] and F:
        r0, r1, r2 = (w.tolist() for w in _philox(np.arange(t, t + 4096), 0, ell, seed))
        for w0, w1, w2 in zip(r0, r1, r2):
            a, d = w0 * ell >> 32, ell + (w1 * (N - ell) >> 32)
            i, j = perm[a], perm[d]
            ni, nj = nbs[i], nbs[j]
            dk = 2 * (sum(up[n] for n in ni) - sum(up[n] for n in nj) + (j in ni)) - len(ni) + len(nj)
            to = b + dk // step
            rise = lng[to] - lng[b]
            if rise > 0:
                s = rise >> q
                ok = s < 4095 and w2 < table[s] - ((table[s] - table[s + 1]) * (rise & low) >> q)
            else:
                ok = True
            if ok:
                perm[a], perm[d] = j, i
                up[i], up[j] = 0, 1
                b = to
                accepts += 1
            lng[b] += F
            hist[b] += 1
            visited[b] = True
            t += 1
            if t % C == 0:
                checks += 1
                seen = [hist[m] for m in range(nbins) if visited[m]]
                n, total = len(seen), sum(seen)
                if 1000 * sum(1000 * n * c >= 800 * total for c in seen) >= 800 * n:
                    least = min(lng[m] for m in range(nbins) if visited[m])
                    lng = [g - least if v else g for g, v in zip(lng, visited)]
                    hist = [0] * nbins
                    F >>= 2
                    stage += 1
            if t >= case["budget"] or not F:
                break
    return lng, visited, (t, accepts, checks, int(not F), stage)


def _exact_surface(case, seed):
    N, nbs = _sites(case["lattice"], case["L"]), _neighbours(case["lattice"], case["L"])
    surface, counters, offsets = [], [], [0]
    for ell in range(N // 2 + 1):
        lng, visited, c = _exact_line(case, nbs, ell, seed & 0xFFFFFFFF)
        counters.append(c)
        v, g = np.array(visited), case["ln_f_min"] * np.array(lng, dtype=np.float64)
        top = g[v].max() if v.any() else 0.0
        norm = top + math.log(math.fsum(np.exp(g[v] - top))) if v.any() else 0.0
        surface.append(np.where(v, math.log(math.comb(N, ell)) + g - norm, -np.inf))
        offsets.append(offsets[-1] + len(lng))
    c = np.array(counters, dtype=np.int64)
    total = np.concatenate([c[:, :4].sum(axis=0), [c[:, 4].min(), c[:, 4].max()]])
    return np.concatenate(surface), np.array(offsets, dtype=np.int64), total


def _exact_thermo(case, surface, offsets, T, H):
    N, NB, step = _sites(case["lattice"], case["L"]), _bonds(case["lattice"], case["L"]), _k_step(case["lattice"])
    g, bond, mag = [], [], []
    for ell in range(N // 2 + 1):
        s = surface[offsets[ell]:offsets[ell + 1]]
        for m in {ell, N - ell}:
            g.append(s)
            bond.append(2.0 * step * np.arange(len(s)) - NB)
            mag.append(np.full(len(s), 2.0 * m - N))
    g, bond, mag = np.concatenate(g), np.concatenate(bond), np.concatenate(mag)
    seen = np.isfinite(g)
    g, bond, mag = g[seen], bond[seen], mag[seen]
    out = np.zeros((len(T), len(H), 6))
    for a, t in enumerate(T):
        for c, field in enumerate(H):
            E = bond - field * mag
            x = g - E / t
            w = np.exp(x - x.max())
            z = w.sum()
            e, m = (w * E).sum() / z, (w * mag).sum() / z
            out[a, c] = [(x.max() + math.log(z)) / N, e / N, (w * (E - e) ** 2).sum() / z / (N * t * t), m / N,
                         (w * np.abs(mag)).sum() / z / N, (w * (mag - m) ** 2).sum() / z / (N * t)]
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("surface", "thermo") or not case["deterministic"]:
        return None                 # production acceptance is a rule in FP32; the others are long walks
    lines = _sites(case["lattice"], case["L"]) // 2
    if lines * min(case["budget"], 25_000 if case["L"] <= 4 else case["budget"]) > EXACT_MOVES:
        return None
    surface, offsets, counters = _exact_surface(case, seed)
    if kind == "thermo":
        return {"thermo": _exact_thermo(case, surface, offsets, *_grid(case, seed))}
    return {"surface": surface, "offsets": offsets, "counters": counters}
