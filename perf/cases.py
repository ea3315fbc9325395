"""Workloads of the library, as calls a user's program makes through the Python binding.

A case is one dict of plain values; `kind` names the entry points it uses:

  sc        one periodic simple cubic sample, `replicas` replicas (Context.run, history)
  coreshell one core/shell fcc sphere, field-cooled (Context.run, history)
  fcc       one fcc sphere at several temperatures, a replica each (Context.run, history)
  batch     many fcc nanoparticles of uneven size in one context (Context.run, history)
  ising     multi-spin coded Ising lattices (IsingContext.run, history)
  sweep     one MCS on buffers that the caller owns (vegas_sweep_noalloc)
  thermal   thermal averages of recorded histories (thermal_averages)
  reweight  multiple histogram reweighting (reweight)

A run of a chain continues the chain of the context that `prepare` made, as a program does that
runs a schedule piece by piece, and reads back what it recorded; the spins stay in the context
and are read back too where a program would (single samples). A context keeps every record
since its creation, so `run` returns the records of its own piece of the history.
"""

import math

import numpy as np
import torch

import paper_1803_07030_gb300 as vg
from lattices import core_shell_particle, fcc_sphere, nanoparticle_batch, sc_periodic

POLICIES = {"random": None, "gaussian": 3, "small_step": 2, "hinzke_nowak": 4, "adaptive": 5}


def listed():
    return [
        # one MCS of a small sample in a host program's own loop: launches and latency only
        {"name": "sweep_13x11x9_r1", "kind": "sweep", "lx": 13, "ly": 11, "lz": 9, "replicas": 1},
        # the plain FP64 reference path: the 8^3 ferromagnet through its temperatures
        {"name": "fp64_sc8", "kind": "sc", "precision": 64, "lx": 8, "ly": 8, "lz": 8, "replicas": 1, "k_uni": 0.0,
         "glass": False, "policy": "random", "t_hi": 2.0, "t_lo": 0.5, "b": 0.0, "steps": 4, "mcs": 250},
        # a stretch of the hysteresis loop of the 64^3 lattice
        {"name": "hyst_sc64", "kind": "sc", "precision": 32, "lx": 64, "ly": 64, "lz": 64, "replicas": 1, "k_uni": 0.05,
         "glass": False, "policy": "random", "t_hi": 0.5, "t_lo": 0.5, "b": 2.0, "steps": 6, "mcs": 500},
        # field cooling of the 29k-site core/shell particle: four classes of uneven rows
        {"name": "coreshell_r12", "kind": "coreshell", "radius": 12.0, "t_hi": 3.0, "t_lo": 0.5, "b": 0.5, "steps": 2,
         "mcs": 1500},
        # 256 nanoparticles of 100 to 14k sites, each at its own temperature, in one launch
        {"name": "batch_256", "kind": "batch", "count": 256, "r_min": 3.0, "r_max": 15.0, "policy": "random", "steps": 1,
         "mcs": 1000},
        # one fcc particle (13k sites) at eight temperatures at once
        {"name": "fcc_r14_r8", "kind": "fcc", "radius": 14.7, "replicas": 8, "policy": "random", "t_hi": 2.5, "t_lo": 0.3,
         "steps": 2, "mcs": 500},
        # the replica-batched spin glass, far larger than L2
        {"name": "glass128_r32", "kind": "sc", "precision": 32, "lx": 128, "ly": 128, "lz": 128, "replicas": 32,
         "k_uni": 0.0, "glass": True, "policy": "random", "t_hi": 2.0, "t_lo": 0.1, "b": 0.0, "steps": 1, "mcs": 40},
        # the same sweep under the adaptive update policy, on sides that are not powers of two
        {"name": "glass60_r32_adaptive", "kind": "sc", "precision": 32, "lx": 60, "ly": 60, "lz": 52, "replicas": 32,
         "k_uni": 0.0, "glass": True, "policy": "adaptive", "t_hi": 2.0, "t_lo": 0.1, "b": 0.0, "steps": 1, "mcs": 200},
        # the plain path: the large glass, one replica
        {"name": "glass128_r1", "kind": "sc", "precision": 32, "lx": 128, "ly": 128, "lz": 128, "replicas": 1,
         "k_uni": 0.0, "glass": True, "policy": "random", "t_hi": 0.8, "t_lo": 0.8, "b": 0.0, "steps": 1, "mcs": 400},
        # Ising lattices through the critical region, a temperature per replica
        {"name": "ising2d_960_r32", "kind": "ising", "dims": 2, "side": 960, "replicas": 32, "t_hi": 2.8, "t_lo": 1.8,
         "h": 0.0, "steps": 2, "mcs": 100},
        # averages and errors of the recorded histories of a parallel run
        {"name": "thermal_64x10007", "kind": "thermal", "series": 64, "records": 10007, "cut": 2001, "bins": 20,
         "tau": 8.0},
        # one temperature curve from the runs of eight temperatures
        {"name": "reweight_8x20011", "kind": "reweight", "runs": 8, "samples": 20011, "observables": 3, "targets": 40,
         "sigma": 60.0},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["sweep", "fp64", "sc1", "scr", "sc32", "coreshell", "fcc", "batch", "ising", "thermal", "reweight"])
    if kind == "sweep":
        return {"kind": "sweep", "lx": rng.randint(3, 40), "ly": rng.randint(3, 40), "lz": rng.randint(3, 40),
                "replicas": rng.choice([1, 2, 4, 8])}
    if kind == "fp64":
        side = int(_log(rng, 4, 25))
        return {"kind": "sc", "precision": 64, "lx": side, "ly": rng.choice([side, side + 1]), "lz": side,
                "replicas": rng.choice([1, 1, 2, 4]), "k_uni": rng.choice([0.0, 0.1]), "glass": rng.random() < 0.5,
                "policy": "random", "t_hi": 2.5, "t_lo": round(rng.uniform(0.2, 1.0), 2),
                "b": rng.choice([0.0, 0.4]), "steps": rng.randint(1, 3), "mcs": rng.randint(60, 200)}
    if kind in ("sc1", "scr", "sc32"):
        replicas = {"sc1": 1, "scr": rng.choice([2, 4, 8, 16]), "sc32": 32}[kind]
        sites = _log(rng, 1e3, {"sc1": 1.5e6, "scr": 2e5, "sc32": 1e6}[kind])
        side = max(4, round(sites ** (1 / 3)))
        return {"kind": "sc", "precision": 32, "lx": side, "ly": max(4, side + rng.randint(-3, 3)), "lz": side,
                "replicas": replicas, "k_uni": rng.choice([0.0, 0.05]), "glass": rng.random() < 0.5,
                "policy": rng.choice(["random", "random", "random", "gaussian", "small_step", "adaptive"]), "t_hi": 2.0,
                "t_lo": round(rng.uniform(0.1, 1.0), 2), "b": rng.choice([0.0, 1.0]), "steps": rng.randint(1, 2),
                "mcs": int(max(40, min(500, 1e9 / (sites * replicas))))}
    if kind == "coreshell":
        return {"kind": "coreshell", "radius": round(_log(rng, 4.0, 16.0), 2), "t_hi": 3.0,
                "t_lo": round(rng.uniform(0.1, 1.0), 2), "b": 0.5, "steps": rng.randint(1, 2), "mcs": rng.randint(200, 800)}
    if kind == "fcc":
        return {"kind": "fcc", "radius": round(_log(rng, 4.0, 20.0), 2), "replicas": rng.choice([1, 4, 8, 16]),
                "policy": rng.choice(["random", "random", "gaussian"]), "t_hi": 2.5, "t_lo": round(rng.uniform(0.2, 1.0), 2),
                "steps": 1, "mcs": rng.randint(100, 400)}
    if kind == "batch":
        case = {"kind": "batch", "count": int(_log(rng, 8, 256)), "r_min": round(rng.uniform(2.0, 9.0), 2),
                "r_max": round(rng.uniform(13.5, 15.0), 2), "policy": rng.choice(["random", "random", "adaptive"]), "steps": 1}
        return dict(case, mcs=int(min(rng.randint(200, 1000), 6e8 / _sites(case)[0])))
    if kind == "ising":
        dims = rng.choice([2, 3])
        return {"kind": "ising", "dims": dims, "side": 64 * (rng.randint(1, 20) if dims == 2 else rng.randint(1, 2)),
                "replicas": 4 * rng.randint(1, 12), "t_hi": 2.8 if dims == 2 else 5.0, "t_lo": 1.8 if dims == 2 else 4.0,
                "h": rng.choice([0.0, 0.0, 0.1]), "steps": rng.randint(1, 3), "mcs": rng.randint(20, 80)}
    if kind == "thermal":
        records = int(_log(rng, 300, 20000))
        return {"kind": "thermal", "series": int(_log(rng, 1, 64)), "records": records, "cut": records // 5,
                "bins": rng.choice([10, 20, 40]), "tau": round(_log(rng, 1.0, 30.0), 2)}
    return {"kind": "reweight", "runs": rng.randint(2, 10), "samples": int(_log(rng, 500, 16000)),
            "observables": rng.randint(1, 4), "targets": rng.randint(5, 50), "sigma": round(_log(rng, 10.0, 80.0), 1)}


# ------------------------------------------------------------------ samples and schedules
def _samples(case, seed):
    """The samples of a chain, and its temperatures and fields [instances, steps]. The seed draws a
    glass's bonds; particles keep their shapes (as a study's geometry files do) and take the
    seed in the chain: initial spins, trials and decisions."""
    kind, steps = case["kind"], case.get("steps", 1)
    if kind in ("sc", "sweep"):
        glass = case.get("glass", False)
        samples = [sc_periodic((case["lx"], case["ly"], case["lz"]), J=1.0, k_uni=case.get("k_uni", 0.0),
                               bimodal_seed=seed if glass else None)]
    elif kind == "coreshell":
        samples = [core_shell_particle(seed=1, radius=case["radius"], core_radius=0.75 * case["radius"])]
    elif kind == "fcc":
        samples = [fcc_sphere(case["radius"], a=4.0 ** (1.0 / 3.0), centre=(0.2, 0.5, 0.7))]
    else:
        samples = nanoparticle_batch(case["count"], seed=1, r_min=case["r_min"], r_max=case["r_max"])
    code = POLICIES[case.get("policy", "random")]
    if code is not None:
        for s in samples:
            s.with_policy(code, 0.5)
    n = len(samples) * case.get("replicas", 1)
    if kind == "batch":  # each particle at one of 64 temperatures
        T = np.broadcast_to((0.05 + (np.arange(n) % 64) * (2.95 / 63.0))[:, None], (n, steps))
        B = np.zeros((n, steps))
    elif n > 1:  # a temperature per replica
        ratio = case.get("t_hi", 1.0) / case.get("t_lo", 1.0)
        T = np.broadcast_to((case.get("t_lo", 1.0) * ratio ** (np.arange(n) / (n - 1.0)))[:, None], (n, steps))
        B = np.full((n, steps), case.get("b", 0.0))
    else:
        T = np.linspace(case.get("t_hi", 1.0), case.get("t_lo", 1.0), steps)[None, :]
        B = case.get("b", 0.0) - 0.05 * np.arange(steps)[None, :] * (case.get("t_hi") == case.get("t_lo"))
    return samples, np.ascontiguousarray(T), np.ascontiguousarray(np.broadcast_to(B, (n, steps)), dtype=np.float64)


def _caller_owned(sample, replicas, seed):
    """A sample in the format of vegas_sweep_noalloc on the GPU, with uniform initial spins."""
    n = sample.n_sites
    colour, classes = vg.vegas_greedy_colour(sample.row_ptr, sample.col)
    order = np.lexsort((np.arange(n), colour))
    inverse = np.empty(n, dtype=np.int64)
    inverse[order] = np.arange(n)
    degree = np.diff(sample.row_ptr)[order]
    row_ptr = np.concatenate([[0], np.cumsum(degree)]).astype(np.int64)
    first = np.repeat(sample.row_ptr[order] - row_ptr[:-1], degree) + np.arange(row_ptr[-1])
    links = np.empty((row_ptr[-1], 2), dtype=np.int32)
    links[:, 0] = inverse[sample.col[first]]
    links[:, 1] = sample.J[first].astype(np.float32).view(np.int32)
    v = np.random.Generator(np.random.PCG64(seed)).normal(size=(n, replicas, 3))
    spins = np.zeros((n, replicas, 4), dtype=np.float32)
    spins[:, :, :3] = v / np.linalg.norm(v, axis=2, keepdims=True)
    start = np.concatenate([[0], np.cumsum(np.bincount(colour, minlength=classes))]).astype(np.int32)
    return spins, links, row_ptr, order.astype(np.int32), start


def _histories(case, seed):
    """Recorded (E, Mx, My, Mz): autoregressive series of time `tau`, as a chain's records are."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, length = case["series"], case["records"]
    a = math.exp(-1.0 / case["tau"])
    x = rng.normal(size=(length, n, 4))
    for i in range(1, length):
        x[i] = a * x[i - 1] + math.sqrt(1.0 - a * a) * x[i]
    sites = 4096.0
    h = np.empty((n, length, 4))
    h[:, :, 0] = -1.8 * sites + 60.0 * x[:, :, 0].T
    h[:, :, 1:] = 90.0 * np.swapaxes(x[:, :, 1:], 0, 1) + np.array([0.0, 0.0, 0.3 * sites])
    return h, np.linspace(0.8, 2.0, n), sites


def _energies(case, seed):
    """Energies of runs at neighbouring temperatures of one system (a Gaussian density of states
    of width sigma: E at beta is normal around -beta sigma^2), and observables of each sample."""
    rng = np.random.Generator(np.random.PCG64(seed))
    K, n, sigma = case["runs"], case["samples"], case["sigma"]
    betas = 0.8 + np.arange(K) * (0.9 / sigma)
    E = rng.normal(size=(K, n)) * sigma - betas[:, None] * sigma * sigma
    x = E / sigma
    O = np.stack([E, x * x, np.abs(x) + rng.normal(size=E.shape), np.sin(x)][: case["observables"]], axis=2)
    return E, O, betas, np.linspace(betas[0], betas[-1], case["targets"])


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "records": 0}
    if kind == "thermal":
        state["series"], state["T"], state["sites"] = _histories(case, seed)
    elif kind == "reweight":
        state["E"], state["O"], state["betas"], state["targets"] = _energies(case, seed)
    elif kind == "ising":
        R, steps = case["replicas"], case["steps"]
        state["T"] = np.ascontiguousarray(np.broadcast_to(np.linspace(case["t_hi"], case["t_lo"], R)[:, None], (R, steps)))
        state["h"] = np.full((R, steps), case["h"])
        state["ctx"] = vg.IsingContext(case["dims"], case["side"], replicas=R, seed=seed, stream="torch")
    elif kind == "sweep":
        sample = _samples(case, seed)[0][0]
        R = case["replicas"]
        spins, links, row_ptr, order, start = _caller_owned(sample, R, seed)
        state.update(spins=torch.from_numpy(spins).cuda(), links=torch.from_numpy(links).cuda(),
                     row_ptr=torch.from_numpy(row_ptr).cuda(), order=torch.from_numpy(order).cuda(), start=start,
                     beta=1.0 / np.linspace(0.7, 1.5, R), field=np.full(R, 0.2), t=0, seed=seed,
                     out=torch.zeros(R, 4, dtype=torch.float64, device="cuda"))
    else:
        samples, state["T"], state["B"] = _samples(case, seed)
        state["ctx"] = vg.Context(samples, precision=case.get("precision", 32), replicas=case.get("replicas", 1), seed=seed)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "thermal":
        return vg.thermal_averages(state["series"], case["cut"], case["bins"], state["T"], state["sites"])
    if kind == "reweight":
        out, g, iterations = vg.reweight(state["E"], state["O"], state["betas"], state["targets"], tol=1e-9)
        return {"out": out, "g": g, "iterations": iterations}
    if kind == "sweep":
        n = state["spins"].shape[0]
        vg.vegas_sweep_noalloc(state["spins"].data_ptr(), state["links"].data_ptr(), state["row_ptr"].data_ptr(),
                               state["order"].data_ptr(), n, state["start"], case["replicas"], state["beta"],
                               state["field"], seed=state["seed"], t=state["t"], out_ptr=state["out"].data_ptr(),
                               stream=torch.cuda.current_stream().cuda_stream)
        state["t"] += 1
        return {"spins": state["spins"], "out": state["out"]}
    ctx, old = state["ctx"], state["records"]
    ctx.run(state["T"], state["h"] if kind == "ising" else state["B"], case["mcs"])
    state["records"] = old + case["steps"] * case["mcs"]
    got = {"history": ctx.history()[:, old:]}
    if kind != "ising":
        got["accepted"] = ctx.accept_history()[:, old:].astype(np.int64)
    if kind == "coreshell" or (kind == "sc" and case["replicas"] == 1 and case["lx"] <= 64):
        got["spins"] = ctx.spins(0)
    return got


# ------------------------------------------------------------------ what a pass cannot do without
def _sites(case):
    """Sites over all samples and links per site, without building them."""
    kind = case["kind"]
    if kind in ("sc", "sweep"):
        return case["lx"] * case["ly"] * case["lz"], 6.0
    if kind == "coreshell":  # four sites per cube of side 1
        return 4.0 * 4.18879 * case["radius"] ** 3, 11.0
    if kind == "fcc":
        return 4.18879 * case["radius"] ** 3, 11.0
    a, b = case["r_min"], case["r_max"]  # radii uniform in [a, b], one site per unit volume
    return case["count"] * 4.18879 * (b ** 4 - a ** 4) / (4.0 * (b - a)), 10.5


def work(case):
    """Bytes and operations of one pass. A chain reads and writes each spin and reads its links
    (shared by the replicas) once per attempt; an attempt takes the field's multiply-adds and
    about a hundred operations for the random numbers, the trial and the decision."""
    kind = case["kind"]
    if kind == "thermal":
        n = float(case["series"] * case["records"])
        lags = 2.0 * (6.0 * case["tau"] + 1.0)  # Sokal's window, for E and |M|
        return {"bytes": 32.0 * n + 128.0 * case["series"], "flops": n * (40.0 + 2.0 * lags)}
    if kind == "reweight":
        n = float(case["runs"] * case["samples"])
        return {"bytes": n * 8.0 * (1 + case["observables"]),
                "flops": n * 20.0 * (2.0 * case["runs"] * 50.0 + case["targets"])}  # about 50 iterations
    if kind == "ising":
        n = float(case["side"]) ** case["dims"] * case["replicas"] * case["steps"] * case["mcs"]
        return {"bytes": n / 4.0, "flops": n * 12.0}  # a bit read and written; a quarter of a random block
    sites, links = _sites(case)
    R = case.get("replicas", 1)
    attempts = float(sites) * R * case.get("steps", 1) * case.get("mcs", 1)
    spin, link = (64.0, 16.0) if case.get("precision", 32) == 64 else (32.0, 8.0)
    return {"bytes": attempts * (spin + link * links / R), "flops": attempts * (6.0 * links + 100.0)}


# ------------------------------------------------------------------ the same in 64 bits
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on uint64 arrays."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, dtype=np.uint64) for x in (c0, c1, c2, c3)]
    c = list(np.broadcast_arrays(*c))
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _u53(hi, lo):
    return ((hi << np.uint64(21)) | (lo >> np.uint64(11))).astype(np.float64) * 2.0 ** -53


def _sphere(site, t, inst, purpose, seed):
    """Marsaglia's method: candidate k of each site until its point lies in the unit disk."""
    site, inst = np.broadcast_arrays(site, inst)
    out = np.zeros(site.shape + (3,))
    todo = np.ones(site.shape, dtype=bool)
    for k in range(64):
        w = _philox(site[todo], t, inst[todo], purpose | k, seed)
        u, v = 2.0 * _u53(w[0], w[1]) - 1.0, 2.0 * _u53(w[2], w[3]) - 1.0
        s = u * u + v * v
        ok = s < 1.0
        q = np.sqrt(np.where(ok, 1.0 - s, 0.0))
        new = np.stack([2.0 * u * q, 2.0 * v * q, 1.0 - 2.0 * s], axis=-1)
        at = np.argwhere(todo)[ok]
        out[tuple(at.T)] = new[ok]
        todo[tuple(at.T)] = False
        if not todo.any():
            break
    return out


def _greedy(sample):
    colour = np.full(sample.n_sites, -1, dtype=np.int64)
    rp, col = sample.row_ptr, sample.col
    for i in range(sample.n_sites):
        used = set(colour[col[rp[i]:rp[i + 1]]].tolist())
        c = 0
        while c in used:
            c += 1
        colour[i] = c
    return colour


def _chain(sample, S, T, B, mcs, seed, precision):
    """The chain of one sample in 64 bits from the spins S [n, R, 3] on (changed in place): its
    records [R, steps * mcs, 4] and accepted counts [R, steps * mcs]. FP32 contexts draw (z,
    azimuth) from one random block with 23 bits each and compare 32 bits with the acceptance."""
    n, R = S.shape[:2]
    degree = np.diff(sample.row_ptr)
    width = int(degree.max())
    nbr, J = np.zeros((n, width), dtype=np.int64), np.zeros((n, width))
    inside = np.arange(width) < degree[:, None]
    nbr[inside], J[inside] = sample.col, sample.J
    colour = sample.colour if sample.colour is not None else _greedy(sample)
    classes = [np.flatnonzero(colour == c) for c in range(int(colour.max()) + 1)]
    k, e, axis = sample.param("k_uni")[:, None], sample.param("e_uni")[:, None, :], sample.param("field_axis")[:, None, :]
    inst = np.arange(R, dtype=np.uint64)[None, :]
    hist, accepted = np.zeros((R, T.shape[1] * mcs, 4)), np.zeros((R, T.shape[1] * mcs), dtype=np.int64)
    for step in range(T.shape[1]):
        beta, b = (1.0 / T[:, step])[None, :], B[:, step][None, :]
        for m in range(mcs):
            t = step * mcs + m
            for sites in classes:
                s = S[sites]
                ids = sites.astype(np.uint64)[:, None]
                field = b[..., None] * axis[sites]
                for q in range(width):
                    field = field + J[sites, q][:, None, None] * S[nbr[sites, q]]
                if precision == 64:
                    new = _sphere(ids, t, inst, 0, seed)
                    w = _philox(ids, t, inst, 0x10000, seed)
                    u = _u53(w[0], w[1])
                else:
                    w = _philox(ids, t, inst, 0x40000, seed)
                    z = (2.0 * (w[0] >> np.uint64(9)).astype(np.float64) + 1.0) * 2.0 ** -23 - 1.0
                    phi = 2.0 * math.pi * (((w[1] >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23 - 0.5)
                    rho = np.sqrt(1.0 - z * z)
                    new = np.stack([rho * np.cos(phi), rho * np.sin(phi), z], axis=-1)
                    u = w[2].astype(np.float64) * 2.0 ** -32
                dE = -((new - s) * field).sum(axis=-1)
                dE = dE - k[sites] * ((new * e[sites]).sum(axis=-1) ** 2 - (s * e[sites]).sum(axis=-1) ** 2)
                with np.errstate(over="ignore"):
                    ok = (dE <= 0.0) | (u < np.exp(-beta * dE))
                S[sites] = np.where(ok[..., None], new, s)
                accepted[:, t] += ok.sum(axis=0)
            pair = np.zeros((n, R))
            for q in range(width):
                pair += J[:, q][:, None] * (S * S[nbr[:, q]]).sum(axis=-1)
            E = -0.5 * pair.sum(axis=0) - (b * (S * axis).sum(axis=-1)).sum(axis=0)
            hist[:, t, 0] = E - (k * (S * e).sum(axis=-1) ** 2).sum(axis=0)
            hist[:, t, 1:] = S.sum(axis=0)
        S /= np.linalg.norm(S, axis=2, keepdims=True)
    return hist, accepted


def _thermal(h, cut, bins, T, N):
    E, A2 = h[cut:, 0], (h[cut:, 1:] ** 2).sum(axis=1)
    A = np.sqrt(A2)
    n = len(E)
    size = n // bins
    e0, a0 = E.mean(), A.mean()

    def estimates(e, a, a2):
        return np.array([e.var() / (N * T * T), a.var() / (N * T), 1.0 - (a2 ** 2).mean() / (3.0 * a2.mean() ** 2)])

    whole = estimates(E, A, A2)
    cuts = [x[: bins * size].reshape(bins, size) for x in (E, A, A2)]
    jack = np.array([estimates(*[np.delete(x, q, axis=0).ravel() for x in cuts]) for q in range(bins)])
    errors = np.sqrt((bins - 1.0) / bins * ((jack - jack.mean(axis=0)) ** 2).sum(axis=0))

    def tau(x):
        c0, t = (x * x).mean(), 0.5
        if c0 == 0.0:
            return 0.5
        for lag in range(1, n // 2 + 1):
            t += (x[:-lag] * x[lag:]).mean() / c0
            if lag >= 6.0 * t:
                break
        return t

    e_err, m_err = (x.mean(axis=1).std(ddof=1) / math.sqrt(bins) / N for x in cuts[:2])
    v1 = -((A - a0) * (E - e0)).mean() / a0
    v2 = -((A2 - A2.mean()) * (E - e0)).mean() / A2.mean()
    return [e0 / N, e_err, a0 / N, m_err, whole[0], errors[0], whole[1], errors[1], whole[2], errors[2], v1, v2,
            tau(E - e0), tau(A - a0), float(n), float(bins)]


def _log_sum(x, axis):
    m = x.max(axis=axis, keepdims=True)
    return np.squeeze(m, axis) + np.log(np.exp(x - m).sum(axis=axis))


def _reweight(E, O, betas, targets, tol):
    K, n = E.shape
    e, o = E.ravel(), O.reshape(K * n, -1)
    g = np.zeros(K)

    def weights():
        return math.log(n) + _log_sum(-betas[:, None] * e - g[:, None], 0)

    for _ in range(10000):
        d = weights()
        new = np.array([_log_sum(-b * e - d, 0) for b in betas])
        new -= new[0]
        gone = np.abs(new - g).max()
        g = new
        if gone < tol:
            break
    d = weights()
    out = np.empty((len(targets), o.shape[1]))
    for q, b in enumerate(targets):
        x = -b * e - d
        w = np.exp(x - x.max())
        out[q] = (w[:, None] * o).sum(axis=0) / w.sum()
    return out, g


def exact(case, seed):
    """What `run` returns for a new state, in 64 bits. The FP32 chains have such a value only
    while no decision falls within FP32 rounding of its threshold, after which another chain
    of the same law goes on: it is given for short chains of few sites, for the others not."""
    kind = case["kind"]
    if kind == "thermal":
        h, T, sites = _histories(case, seed)
        return np.array([_thermal(x, case["cut"], case["bins"], t, sites) for x, t in zip(h, T)])
    if kind == "reweight":
        out, g = _reweight(*_energies(case, seed), tol=1e-9)
        return {"out": out, "g": g, "iterations": None}
    if kind not in ("sc", "sweep") or case.get("policy", "random") != "random":
        return None
    (sample,), T, B = _samples(case, seed)
    R, n = case["replicas"], sample.n_sites
    if kind == "sweep":
        spins, _, _, order, _ = _caller_owned(sample, R, seed)
        S = np.zeros((n, R, 3))
        S[order] = spins[:, :, :3]
        hist, _ = _chain(sample, S, np.linspace(0.7, 1.5, R)[:, None], np.full((R, 1), 0.2), 1, seed, 32)
        S = np.concatenate([S[order], np.zeros((n, R, 1))], axis=2)
        return {"spins": S, "out": hist[:, 0]}
    attempts = n * R * case["steps"] * case["mcs"]
    if attempts > (3e6 if case["precision"] == 64 else 2e5):
        return None
    S = _sphere(np.arange(n, dtype=np.uint64)[:, None], 0xFFFFFFFF, np.arange(R, dtype=np.uint64)[None, :], 0x20000, seed)
    if case["precision"] == 32:
        S = S.astype(np.float32).astype(np.float64)
    hist, accepted = _chain(sample, S, T, B, case["mcs"], seed, case["precision"])
    got = {"history": hist, "accepted": None if case["precision"] == 32 else accepted}
    if R == 1 and case["lx"] <= 64:
        got["spins"] = S[:, 0]
    return got
