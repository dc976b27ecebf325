"""Workloads of this library that are timed and compared, through its public entry points.

Kinds of case:
  solve    rewl_create, rewl_step to the end (sweeps = 0) or for a number of sweeps, rewl_get_state,
           rewl_get_lng, rewl_destroy: what a program does that wants one density of states
  resume   a handle that is kept, a checkpoint of a running solve, and one stretch of it:
           rewl_set_state, rewl_step, rewl_get_state, rewl_get_lng; the checkpoint is a solve's state
           some iterations in, with ln f = 2^-lnf_k
  served   a request server that is kept: submit a batch of requests of several models and sizes, run
           until all are done, fetch every result
  noalloc  rewl_sweep_noalloc on walkers whose state lies in the caller's own torch tensors
  thermo   rewl_thermo and rewl_thermo_jackknife on tables of ln g
"""
import math

import numpy as np
import torch

from paper_1305_5615_gb300 import rewl

MOST_TRIALS = 1.3e10  # walkers x trials of the largest listed case; drawn ones stay below it


def listed():
    return [
        # smallest call: a few sweeps of a few walkers that an embedding program holds itself; ragged sizes
        {"name": "noalloc_potts7_L20", "kind": "noalloc", "model": "potts", "q": 7, "L": 20, "windows": 6,
         "walkers": 5, "lnf_k": 12, "sweeps": 50},
        # after a solve: the canonical curves of a 32 x 32 Ising table, and their errors over 8 runs
        {"name": "thermo_L32", "kind": "thermo", "L": 32, "temperatures": 300, "runs": 8},
        # one whole density of states of a small lattice, start to converged (8 walkers: latency)
        {"name": "ising8_solve", "kind": "solve", "model": "ising", "q": 2, "L": 8, "windows": 4, "walkers": 2,
         "lnf_final": 1e-6, "sweeps": 0, "rule": "flat"},
        # the start of a solve at the benchmark's size: set-up, entry walks and the first 1000 sweeps at ln f = 1
        {"name": "ising32_first", "kind": "solve", "model": "ising", "q": 2, "L": 32, "windows": 16, "walkers": 4,
         "lnf_final": 1e-8, "sweeps": 1000, "rule": "flat"},
        # the bulk of such a solve: a flatness period at small ln f
        {"name": "ising32_late", "kind": "resume", "model": "ising", "q": 2, "L": 32, "windows": 16, "walkers": 4,
         "lnf_k": 18, "sweeps": 1000, "rule": "flat", "mode": "plain"},
        # an odd lattice with many walkers a window (more than 8 walkers per SM), an iteration in the middle
        {"name": "ising21_many", "kind": "resume", "model": "ising", "q": 2, "L": 21, "windows": 20, "walkers": 64,
         "lnf_k": 8, "sweeps": 1000, "rule": "flat", "mode": "plain"},
        # q = 10 Potts at its first-order transition, several walkers per SM, the period replayed as a graph
        {"name": "potts10_L32_graph", "kind": "resume", "model": "potts", "q": 10, "L": 32, "windows": 32,
         "walkers": 16, "lnf_k": 16, "sweeps": 1000, "rule": "flat", "mode": "graph"},
        # a 2D +-J realisation with given couplings, under the 1/t rule
        {"name": "ea24_one_over_t", "kind": "resume", "model": "ea", "q": 2, "L": 24, "windows": 8, "walkers": 4,
         "lnf_k": 14, "sweeps": 1000, "rule": "1/t", "mode": "plain"},
        # the paper's 12^3 spin glass
        {"name": "ea3d_L12", "kind": "resume", "model": "ea3d", "q": 2, "L": 12, "windows": 16, "walkers": 4,
         "lnf_k": 16, "sweeps": 1000, "rule": "flat", "mode": "plain"},
        # the largest: 4096 walkers on 128 x 128, throughput of the whole chip
        {"name": "ising128_4096", "kind": "resume", "model": "ising", "q": 2, "L": 128, "windows": 128, "walkers": 32,
         "lnf_k": 16, "sweeps": 200, "rule": "flat", "mode": "plain"},
        # a batch of small requests of mixed models and sizes to the request server
        {"name": "served_mix", "kind": "served", "requests": 24, "L_min": 8, "L_max": 16, "lnf_final": 0.4},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["resume", "resume", "resume", "resume", "solve", "served", "noalloc", "thermo"])
    if kind == "thermo":
        return {"kind": kind, "L": _log_int(rng, 8, 64), "temperatures": _log_int(rng, 20, 600),
                "runs": rng.randint(2, 12)}
    if kind == "served":
        lo = rng.randint(6, 8)
        return {"kind": kind, "requests": _log_int(rng, 6, 24), "L_min": lo, "L_max": lo + rng.randint(2, 8),
                "lnf_final": rng.choice([0.4, 0.7])}
    if kind == "solve":
        if rng.random() < 0.5:  # whole solves of small lattices
            return {"kind": kind, "model": rng.choice(["ising", "potts"]), "q": rng.randint(2, 4), "L": rng.randint(4, 7),
                    "windows": rng.randint(1, 3), "walkers": rng.randint(1, 4), "lnf_final": rng.choice([1e-4, 1e-5]),
                    "sweeps": 0, "rule": "flat"}
        return {"kind": kind, "model": rng.choice(["ising", "potts"]), "q": rng.randint(3, 12), "L": _log_int(rng, 9, 40),
                "windows": rng.randint(3, 12), "walkers": rng.randint(1, 8), "lnf_final": 1e-6, "sweeps": 1000,
                "rule": rng.choice(["flat", "1/t"])}
    model = rng.choice(["ising", "potts", "ea"] if kind == "noalloc" else ["ising", "potts", "ea", "ea3d"])
    if model == "ea3d":
        L = 2 * rng.randint(3, 7)
    elif model == "ea":
        L = 2 * _log_int(rng, 4, 24)
    else:
        L = _log_int(rng, 8, 70)
    N = L ** 3 if model == "ea3d" else L * L
    q = rng.randint(3, 16) if model == "potts" else 2
    bins = 2 * N if model == "potts" else N
    windows = rng.randint(2 if kind == "noalloc" else 1, max(3, min(40, bins // 12)))
    if windows == 1 and bins > 2000:
        windows = 4
    if kind == "noalloc":
        return {"kind": kind, "model": model, "q": q, "L": L, "windows": windows, "walkers": rng.randint(1, 8),
                "lnf_k": rng.randint(4, 22), "sweeps": rng.randint(10, 100)}
    walkers = _log_int(rng, 1, 96)
    sweeps = 1000
    while sweeps > 100 and sweeps * float(N) * (windows * walkers + 300) > 0.15 * MOST_TRIALS:
        sweeps -= 100
    while walkers > 1 and sweeps * float(N) * windows * walkers > 0.15 * MOST_TRIALS:
        walkers //= 2
    return {"kind": kind, "model": model, "q": q, "L": L, "windows": windows, "walkers": walkers,
            "lnf_k": rng.randint(2, 24), "sweeps": sweeps, "rule": rng.choice(["flat", "flat", "1/t"]),
            "mode": rng.choice(["plain", "graph"])}


def _couplings(model, L, seed):
    """A disorder realisation, +1 and -1 alike, with an even number of -1 (so that its energy grid starts at -dim N)."""
    J = (2 * np.random.default_rng(seed).integers(0, 2, 3 * L ** 3 if model == "ea3d" else 2 * L * L) - 1).astype(np.int8)
    J[0] = J[1:].prod()
    return J


def _glass_windows(case):
    """A partition that does not depend on the realisation: equal windows with 75% overlap over +-1.3 N (2D) or
    +-1.65 N (3D), most of a glass's range, the outer two reaching on to the ends of the grid."""
    cube = case["model"] == "ea3d"
    N = case["L"] ** 3 if cube else case["L"] ** 2
    h, bins = case["windows"], (3 * N if cube else 2 * N) // 2 + 1
    lo = int((1.35 if cube else 0.7) * N) // 4
    core = bins - 2 * lo
    w = min(core, math.ceil(core / (1 + (h - 1) * 0.25)))
    starts = np.array([lo + (round(k * (core - w) / (h - 1)) if h > 1 else 0) for k in range(h)], np.int32)
    widths = np.full(h, w, np.int32)
    widths[0] += starts[0]
    starts[0] = 0
    widths[-1] = bins - starts[-1]
    return starts, widths


def _solver(case, seed, lnf_final, **more):
    L, model = case["L"], case["model"]
    if model in ("ea", "ea3d"):
        more["couplings"] = _couplings(model, L, seed)
        more["window_starts"], more["window_widths"] = _glass_windows(case)
    return rewl.REWL(model, L, case["windows"], 0.75, case["walkers"], 0.8, lnf_final, seed, q=case["q"],
                     wl_rule=case.get("rule", "flat"), **more)


def _merged(state, case, k):
    """The state with every window merged and its ln f at 2^-k (what the library does between iterations)."""
    h, m = case["windows"], case["walkers"]
    lng = state["lng"].reshape(h, m, -1)
    state["lng"] = np.ascontiguousarray(np.broadcast_to(lng.mean(axis=1, keepdims=True), lng.shape)).reshape(h * m, -1)
    state["H"] = np.zeros_like(state["H"])
    state["lnf"] = np.full(h, 2.0 ** -k)
    return state


def _checkpoint(D, case):
    """A solve's state some iterations in: ln g built at ln f = 1 and smoothed down to the case's ln f."""
    N = D.info["N"]
    walkers = case["windows"] * case["walkers"]
    unit = 200 if walkers * N < 2e7 else 100  # sweeps
    for k, n in ((0, 2 * unit), (3, unit), (6, unit), (9, unit)):
        if k and k < case["lnf_k"]:
            D.set_state(_merged(D.state(), case, k))
        D.step(n)
    D.set_state(_merged(D.state(), case, case["lnf_k"]))
    return D.state()


def _coupling_bits(couplings, L):
    """Two bit planes [right | down][L][ceil(L / 32)], a set bit for J = -1."""
    wr = (L + 31) // 32
    planes = np.zeros((2, L, wr), np.uint32)
    J = couplings.reshape(L, L, 2)
    for x in range(L):
        planes[:, :, x // 32] |= (J[:, x, :].T < 0).astype(np.uint32) << np.uint32(x % 32)
    return planes


def _device(a):
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda()


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    got = []
    for i in range(case["requests"]):
        model = ("ising", "ea", "potts", "ising")[i % 4]
        L = case["L_min"] + (7 * i // 2) % (case["L_max"] - case["L_min"] + 1)
        L += L % 2 if model == "ea" else 0
        L = min(L, 10) if model == "potts" else L
        key = int(rng.integers(1, 1 << 40))
        got.append((model, L, 4 if L < 12 else 8, 0.75, 1 + i % 4, 0.8, case["lnf_final"], key,
                    10 if model == "potts" else 2, _couplings(model, L, key) if model == "ea" else None))
    return got


def _tables(case, seed):
    """Ising-like tables of ln g on [-2N, 2N] with the statistical scatter of independent runs."""
    rng = np.random.default_rng(seed)
    N = case["L"] ** 2
    e = np.linspace(-1.0, 1.0, N + 1)
    p = np.clip((1 + e) / 2, 1e-9, 1 - 1e-9)
    s = -(p * np.log(p) + (1 - p) * np.log(1 - p))
    lng = N * s + math.log(2.0) + 0.02 * rng.standard_normal((case["runs"], N + 1))
    lng[:, 1] = lng[:, -2] = -np.inf  # the two levels that do not exist
    return lng, np.linspace(0.4, 5.0, case["temperatures"]) + 0.01 * rng.random()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "thermo":
        lng, T = _tables(case, seed)
        return {"kind": kind, "lng": lng, "T": T, "e_min": -2 * case["L"] ** 2}
    if kind == "served":
        return {"kind": kind, "server": rewl.RewlServer(8 << 30, 64),
                "requests": _requests(case, seed)}
    if kind == "solve":
        return {"kind": kind, "case": case, "seed": seed}
    D = _solver(case, seed, 1e-9, mode=rewl.MODE_GRAPH if case.get("mode") == "graph" else rewl.MODE_PLAIN)
    state = _checkpoint(D, case)
    if kind == "resume":
        return {"kind": kind, "solver": D, "checkpoint": state, "sweeps": case["sweeps"]}
    info = D.info
    D.close()
    start = {k: _device(state[k]) for k in ("lattice", "E", "lng", "H")}
    bits = None
    if case["model"] == "ea":
        bits = _device(_coupling_bits(_couplings("ea", case["L"], seed), case["L"]))
    desc = rewl.rewl_sweep_desc(model=info["model"], q=info["q"], L=info["L"], windows=info["windows"],
                                walkers_per_window=info["walkers_per_window"], window_bins=info["window_bins"],
                                e_min=info["e_min"], e_step=info["e_step"], seed=seed,
                                first_sweep=state["sweep_clock"], sweeps=case["sweeps"], lanes_per_walker=0)
    return {"kind": kind, "desc": desc, "start": start, "now": {k: v.clone() for k, v in start.items()},
            "bits": bits, "win_start": _device(state["win_start"]), "lnf": _device(state["lnf"])}


def run(state):
    kind = state["kind"]
    if kind == "thermo":
        est, err = rewl.rewl_thermo_jackknife(state["lng"], state["e_min"], 4, state["T"])
        return {"one": rewl.rewl_thermo(state["lng"][0], state["e_min"], 4, state["T"]), "mean": est, "error": err}
    if kind == "served":
        s = state["server"]
        ids = [s.submit(*r[:8], q=r[8], couplings=r[9]) for r in state["requests"]]
        left = True
        while left:
            st = s.run(64)
            left = st["running"] + st["queued"] > 0
        return [s.result(i)[0] for i in ids]
    if kind == "noalloc":
        now, bits = state["now"], state["bits"]
        for k, v in state["start"].items():
            now[k].copy_(v)
        rewl.rewl_sweep_noalloc(state["desc"], now["lattice"].data_ptr(), now["E"].data_ptr(), now["lng"].data_ptr(),
                                now["H"].data_ptr(), bits.data_ptr() if bits is not None else None,
                                state["win_start"].data_ptr(), state["lnf"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        return now
    if kind == "solve":
        case = state["case"]
        D = _solver(case, state["seed"], case["lnf_final"])
        D.step(case["sweeps"])
        out = {"lng": D.lng()[0], "state": D.state()}
        D.close()
        return out
    D = state["solver"]
    D.set_state(state["checkpoint"])
    D.step(state["sweeps"])
    return {"lng": D.lng()[0], "state": D.state()}


def _window_bins(case, N):
    bins = 2 * N + 1 if case["model"] == "potts" else (3 * N // 2 if case["model"] == "ea3d" else N) + 1
    return bins if case["windows"] == 1 else math.ceil(bins / (1 + (case["windows"] - 1) * 0.25))


def work(case):
    """Bytes: every walker's configuration, ln g (8 bytes a bin) and H (4) in and out once.  Operations: 112 integer
    ones a trial (draw, site, neighbourhood, test, update); the sums over the bins for thermo."""
    kind = case["kind"]
    if kind == "thermo":
        n = case["L"] ** 2 + 1
        return {"bytes": 8 * n * (case["runs"] + 1) + 8 * 16 * case["temperatures"],
                "flops": float(n) * case["temperatures"] * (case["runs"] + 2) * 30}
    if kind == "served":
        # about 10 000 sweeps a request of this range until ln f is below lnf_final, about 12 walkers
        N = ((case["L_min"] + case["L_max"]) / 2) ** 2
        return {"bytes": case["requests"] * 12 * (N / 2 * 24 + N / 4), "flops": 112.0 * case["requests"] * 12 * 10000 * N}
    N = case["L"] ** 3 if case["model"] == "ea3d" else case["L"] ** 2
    W = case["windows"] * case["walkers"]
    sweeps = case["sweeps"] or 60000
    lattice = N / 2 if case["model"] == "potts" else N / 8
    return {"bytes": 2.0 * W * (12 * _window_bins(case, N) + lattice), "flops": 112.0 * W * sweeps * N}


def _canonical(lng, e, T):
    out = np.empty((len(T), 5))
    fine = np.isfinite(lng)
    for i, t in enumerate(T):
        beta = 1.0 / t
        a = lng[fine] - beta * e[fine]
        mx = a.max()
        w = np.exp(a - mx)
        z = w.sum()
        U = (w * e[fine]).sum() / z
        lnZ = mx + math.log(z)
        F = -t * lnZ
        out[i] = lnZ, U, beta * beta * (w * (e[fine] - U) ** 2).sum() / z, F, (U - F) / t
    return out


def exact(case, seed):
    """The sampled kinds have no value of their own to be near to: their trajectories are compared with each other."""
    if case["kind"] != "thermo":
        return None
    lng, T = _tables(case, seed)
    e = -2.0 * case["L"] ** 2 + 4.0 * np.arange(lng.shape[1])
    R = lng.shape[0]
    left = [_canonical(np.delete(lng, r, axis=0).mean(axis=0), e, T) for r in range(R)]
    err = np.sqrt((R - 1) / R * ((np.stack(left) - np.mean(left, axis=0)) ** 2).sum(axis=0))
    return {"one": _canonical(lng[0], e, T), "mean": _canonical(lng.mean(axis=0), e, T), "error": err}
