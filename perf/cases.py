"""What is timed of polyrx: whole calls through its public entry points, over the sizes it is used at.

A case is one call pattern ("call") with its sizes:
  run        a system advanced by `steps` MD steps (reactions every theta), then read back
  monitor    a short run followed by the observables, as a program that watches a run makes it
  ensemble   many uneven replicas advanced together in one batch, then read back
  serve      a list of jobs created, admitted, advanced and read back by the server
  forces     the conservative forces and the potential energy of a configuration
  histogram  the pair-distance histogram between two particle classes (g(r), <N>)
  noalloc    the reaction step on device buffers that the caller owns

Inputs: density 0.85, particles on a random subset of a simple cubic lattice with a random
displacement, Maxwell velocities, types by a random permutation; sigma = eps = m = kT = gamma = 1,
dt = 0.005, FENE k = 30, R0 = 1.5.  A run starts from the lattice and every further pass continues it,
so that the passes go through the melting of the lattice and then the reacting liquid.
"""
import ctypes
import math
import time

import numpy as np
import torch

from paper_1409_7498_gb300 import polyrx as P
from paper_1409_7498_gb300 import serve as S

RHO, DT, FENE_K, FENE_R0 = 0.85, 0.005, 30.0, 1.5
B, A, E, REP, X6 = 0, 1, 2, 3, 4  # types: monomer, crosslinker / initiator, chain end, repeat unit, 6-functional
RC = 2.0 ** (1.0 / 6.0)
R_REACT = 1.1


def listed():
    return [
        # the small FP64 system: 1,000 difunctional monomers and 250 crosslinkers, read every 20 reactions
        dict(name="run_1250_fp64", call="run", scheme="step", n=1250, share=0.2, f=4, k=0.1, steps=200, fp64=True),
        # chain growth from 1% initiators, the middle of the three sizes that are quoted
        dict(name="run_33096_chain", call="run", scheme="chain", n=33096, share=328 / 33096, f=1, k=0.1, steps=200),
        # the large step-growth run, with the Verlet skin that the autotuner picks for it
        dict(name="run_1m_step", call="run", scheme="step", n=1048576, share=1 / 9, f=4, k=0.1, steps=500, skin=0.45),
        # a job near the upper end of the served sizes, an odd count, crosslinkers of functionality 6
        dict(name="run_250007_f6", call="run", scheme="step", n=250007, share=1 / 13, f=6, k=0.3, steps=200),
        # E-P3-E chains with crosslinkers at their ends: bonded input, a box that is not cubic, the
        # nearest-partner rule and mirror-LJ bonds
        dict(name="run_chains_nearest", call="run", scheme="ep", n=13000, share=1 / 6, f=4, k=0.5, steps=100,
             selection=1, style=1),
        # three concurrent reactions (substitution effect, a second crosslinker type)
        dict(name="run_33700_mixed", call="run", scheme="mixed", n=33700, share=0.12, f=4, k=0.2, steps=100),
        # the smallest jobs of an ensemble, watched: ten steps and the observables, where latency counts
        dict(name="monitor_2048", call="monitor", scheme="chain", n=2048, share=0.01, f=1, k=1.0, steps=10),
        # the ensemble: 256 replicas of 1,024 to 65,536 beads
        dict(name="ensemble_256", call="ensemble", replicas=256, lo=1024, hi=65536, steps=200),
        # a burst of twelve jobs through the server: creation, admission, epochs, read-back
        dict(name="serve_12", call="serve", jobs=12, lo=2048, hi=262144, steps_lo=200, steps_hi=1000),
        # forces of a large configuration with bonds, for analysis or as another integrator's force call
        dict(name="forces_262144", call="forces", n=262144, jitter=0.2, fp64=False),
        # g(r) between crosslinkers and monomers for the rate equations
        dict(name="histogram_33096", call="histogram", n=33096, share=0.1, f=4, bins=110),
        # the reaction step alone on a host framework's own buffers
        dict(name="noalloc_8192", call="noalloc", n=8192, share=1 / 9, f=4, k=0.1, selection=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["run"] * 6 + ["monitor", "ensemble", "serve", "forces", "histogram", "noalloc"])
    if call == "ensemble":
        return dict(call=call, replicas=_log(rng, 8, 200), lo=_log(rng, 1024, 4096), hi=_log(rng, 8192, 65536),
                    steps=rng.randrange(20, 201))
    if call == "serve":
        return dict(call=call, jobs=rng.randrange(3, 13), lo=_log(rng, 2048, 8192), hi=_log(rng, 16384, 262144),
                    steps_lo=rng.randrange(100, 201), steps_hi=rng.randrange(300, 1001))
    if call == "forces":
        return dict(call=call, n=_log(rng, 1000, 262144), jitter=rng.uniform(0.05, 0.25), fp64=rng.random() < 0.3)
    if call == "histogram":
        return dict(call=call, n=_log(rng, 2048, 262144), share=rng.uniform(0.01, 0.2), f=rng.choice([4, 6]),
                    bins=rng.randrange(20, 400))
    if call == "noalloc":
        return dict(call=call, n=_log(rng, 300, 16384), share=rng.uniform(0.05, 0.2), f=rng.choice([4, 6]),
                    k=math.exp(rng.uniform(math.log(0.01), 0.0)), selection=rng.randrange(2))
    scheme = rng.choice(["step", "step", "chain", "ep", "mixed"])
    fp64 = call == "run" and rng.random() < 0.2
    n = _log(rng, 1000, 8192 if fp64 else 1048576 if call == "run" and scheme != "ep" else 65536)
    f = 1 if scheme == "chain" else 4 if scheme == "mixed" else rng.choice([4, 6])
    share = {"step": 1 / (1 + 2 * f), "chain": 328 / 33096, "ep": 2 / (2 + 5 * f), "mixed": 0.12}[scheme]
    steps = 10 * rng.randrange(1, 5) if call == "monitor" else min(rng.randrange(20, 401), max(20, 400 * 1048576 // n))
    return dict(call=call, scheme=scheme, n=n, share=share, f=f, k=math.exp(rng.uniform(math.log(0.01), 0.0)),
                steps=steps, fp64=fp64, skin=rng.choice([-1.0, -1.0, rng.uniform(0.25, 0.5)]),
                selection=1 if scheme != "mixed" and rng.random() < 0.2 else 0,
                style=1 if rng.random() < 0.2 else 0, theta=rng.choice([5, 10, 10, 20]))


# ---- inputs --------------------------------------------------------------------------------------------
def _lattice(n, rng, jitter):
    """Positions, box edges, and each lattice site's particle (-1: empty)."""
    m = max(4, math.ceil(round(n ** (1.0 / 3.0), 9)))
    L = (n / RHO) ** (1.0 / 3.0)
    site = rng.permutation(m ** 3)[:n]
    ijk = np.stack([site % m, site // m % m, site // (m * m)], 1)
    x = ((ijk + 0.5 + jitter * (rng.random((n, 3)) - 0.5)) * (L / m)) % L
    at = np.full(m ** 3, -1, np.int64)
    at[site] = np.arange(n)
    return x, (L, L, L), at.reshape(m, m, m)


def _chains(n, share, rng, jitter):
    """Runs of five lattice sites along x: each an E-P-P-P-E chain or, for about `share`, five crosslinkers."""
    runs = max(64, n // 5)
    mx = max(1, round(runs ** (1.0 / 3.0) / 5 ** (2.0 / 3.0)))
    my = max(4, math.ceil(math.sqrt(runs / mx)))
    mz = max(4, math.ceil(runs / (mx * my)))
    runs = mx * my * mz  # every run of the lattice is used
    a = RHO ** (-1.0 / 3.0)
    q = np.arange(runs)
    first = np.stack([5.0 * (q % mx), q // mx % my, q // (mx * my)], 1)
    x = first[:, None, :] + np.arange(5.0)[None, :, None] * np.array([1.0, 0.0, 0.0])
    x = x.reshape(-1, 3) + 0.5 + jitter * (rng.random((5 * runs, 3)) - 0.5)
    chain = np.ones(runs, bool)
    chain[rng.permutation(runs)[: max(1, round(share * runs))]] = False
    base = 5 * q[chain]
    bonds = np.concatenate([np.stack([base + u, base + u + 1], 1) for u in range(4)])
    return x * a, (5 * mx * a, my * a, mz * a), np.repeat(chain, 5).reshape(-1, 5), bonds


def _bonds(pairs):
    b = np.zeros(len(pairs), P.BOND_DTYPE)
    b["a"], b["t"] = np.min(pairs, 1), np.max(pairs, 1)
    return b


def _reaction(k, mask_a, lo, hi, mask_t, t_lo, t_hi, d_a, d_t, valence, case, r=R_REACT):
    return dict(mask_A=mask_a, a_lo=lo, a_hi=hi, mask_T=mask_t, t_lo=t_lo, t_hi=t_hi, dA=d_a, dT=d_t, k=k,
                r_react=r, theta=case.get("theta", 10), bond_style=case.get("style", 0),
                selection=case.get("selection", 0), max_valence=valence)


def _inputs(case, seed):
    """Everything a system is created from, as plain numpy, and its reactions."""
    rng = np.random.default_rng([seed, 1409])
    n, scheme, f, k = case["n"], case["scheme"], case["f"], case["k"]
    bonds = None
    if scheme == "ep":
        x, box, chain, bonds = _chains(n, case["share"], rng, 0.05)
        n = len(x)
        typ = np.where(chain, np.array([E, REP, REP, REP, E]), A).astype(np.uint8).reshape(-1)
        state = np.where(chain, 0, f).astype(np.int8).reshape(-1)
        reactions = [_reaction(k, 1 << A, 1, f, 1 << E, 0, 0, -1, 1, (0, f, 2, 2), case)]
    else:
        x, box, _ = _lattice(n, rng, 0.05)
        typ, state = np.full(n, B, np.uint8), np.zeros(n, np.int8)
        a = rng.permutation(n)[: max(1, round(case["share"] * n))]
        typ[a] = A
        if scheme == "chain":
            state[a] = 2
            reactions = [_reaction(k, 1 << A | 1 << B, 2, 2, 1 << B, 0, 0, -1, 2, (2, 1), case)]
        elif scheme == "step":
            state[a] = f
            reactions = [_reaction(k, 1 << A, 1, f, 1 << B, 0, 1, -1, 1, (2, f), case)]
        else:
            six = a[: len(a) // 3]
            state[a] = 4
            typ[six], state[six] = X6, 6
            v = (2, 4, 0, 0, 6)
            reactions = [_reaction(k, 1 << A, 4, 4, 1 << B, 0, 1, -1, 1, v, case),
                         _reaction(2 * k, 1 << A, 1, 3, 1 << B, 0, 1, -1, 1, v, case),
                         _reaction(k / 2, 1 << X6, 1, 6, 1 << B, 0, 1, -1, 1, v, case, 1.05)]
    vel = rng.standard_normal((n, 3))
    vel -= vel.mean(0)
    cap = 2 if scheme == "chain" else 6 if scheme == "mixed" else max(2, f)
    return dict(n=n, x=x, v=vel, type=typ, state=state, box=box, cap=cap, bonds=bonds, reactions=reactions, seed=seed)


def _system(case, seed):
    i = _inputs(case, seed)
    desc = P.make_desc(i["n"], i["box"], adj_cap=i["cap"], skin=case.get("skin", -1.0), fp64=case.get("fp64", False),
                       seed=seed)
    g = P.System(desc, i["x"], i["v"], i["type"], i["state"], None if i["bonds"] is None else _bonds(i["bonds"]))
    g.set_reactions([P.make_reaction(**r) for r in i["reactions"]])
    return g


def _replicas(count, lo, hi):
    """Cases of uneven replicas: sizes and rates log-uniform, step or chain growth."""
    rng = np.random.default_rng([count, lo, hi])
    n = np.exp(rng.uniform(math.log(lo), math.log(hi), count)).astype(int)
    k = np.exp(rng.uniform(math.log(0.01), 0.0, count))
    return [dict(scheme="step", n=int(n[r]), share=1 / 9, f=4, k=float(k[r])) if rng.integers(2) else
            dict(scheme="chain", n=int(n[r]), share=328 / 33096, f=1, k=float(k[r])) for r in range(count)]


def _jobs(case):
    """The jobs' (system case, steps): steps uniform."""
    rng = np.random.default_rng([case["steps_lo"], case["steps_hi"]])
    return [(c, int(rng.integers(case["steps_lo"], case["steps_hi"] + 1)))
            for c in _replicas(case["jobs"], case["lo"], case["hi"])]


def _buffers(ns, caps):
    """What a program that reads systems of these sizes back keeps: pinned arrays over all of them, the bond list with
    room for every bond that can form (-1 where there is none yet), and each system's parts of them."""
    rooms = [n * cap // 2 for n, cap in zip(ns, caps)]
    whole = dict(positions=torch.zeros((sum(ns), 3), dtype=torch.float64).pin_memory().numpy(),
                 velocities=torch.zeros((sum(ns), 3), dtype=torch.float64).pin_memory().numpy(),
                 states=torch.zeros(sum(ns), dtype=torch.int8).pin_memory().numpy(),
                 bonds=torch.full((sum(rooms), 6), -1, dtype=torch.int32).pin_memory().numpy())
    parts, at, b = [], 0, 0
    for n, room in zip(ns, rooms):
        parts.append({key: v[b:b + room] if key == "bonds" else v[at:at + n] for key, v in whole.items()})
        at, b = at + n, b + room
    return whole, parts


def _force_inputs(case, seed):
    """A disordered configuration with a bond between neighbours along x wherever both sites are taken."""
    x, box, at = _lattice(case["n"], np.random.default_rng([seed, 2627]), case["jitter"])
    m = at.shape[0] // 2 * 2
    pair = np.stack([at[:, :, 0:m:2].ravel(), at[:, :, 1:m:2].ravel()], 1)  # sites are z-major: x runs fastest
    return x, box, pair[(pair >= 0).all(1)]


def prepare(case, seed):
    call = case["call"]
    if call in ("run", "monitor"):
        g = _system(case, seed)
        whole, parts = _buffers([g.n], [g.desc.adj_cap])
        return dict(case=case, g=[g], whole=whole, parts=parts)
    if call == "ensemble":
        reps = [_system(c, seed + 1 + r) for r, c in enumerate(_replicas(case["replicas"], case["lo"], case["hi"]))]
        batch = P.Batch()
        for g in reps:
            batch.add(g)
        whole, parts = _buffers([g.n for g in reps], [g.desc.adj_cap for g in reps])
        return dict(case=case, g=reps, batch=batch, whole=whole, parts=parts)
    if call == "serve":
        made = []
        for r, (c, steps) in enumerate(_jobs(case)):
            i = _inputs(c, seed + 1 + r)
            made.append((steps, i["n"],
                         dict(desc=P.make_desc(i["n"], i["box"], adj_cap=i["cap"], seed=seed + 1 + r), pos=i["x"],
                              vel=i["v"], type=i["type"], state=i["state"],
                              reaction=P.make_reaction(**i["reactions"][0]))))
        budget = 16 << 30
        backend = S.PolyrxBackend(P, positions=True, mem_budget=budget)
        room = [np.full((n * system["desc"].adj_cap // 2, 6), -1, np.int32) for _, n, system in made]
        return dict(case=case, jobs=made, server=S.Server(backend, budget), room=room)
    if call == "forces":
        x, box, pairs = _force_inputs(case, seed)
        n = case["n"]
        desc = P.make_desc(n, box, adj_cap=2, seed=seed, fp64=case["fp64"])
        return dict(case=case, g=P.System(desc, x, None, np.zeros(n, np.uint8), np.zeros(n, np.int8), _bonds(pairs)))
    if call == "histogram":
        return dict(case=case, g=_system(dict(case, scheme="step", k=0.1), seed))
    # the caller's own device buffers, and the snapshot that each call starts from
    i = _inputs(dict(case, scheme="step"), seed)
    n, cap = i["n"], i["cap"]
    dev = torch.device("cuda")
    rng = np.random.default_rng([seed, 33])
    x, _, _ = _lattice(n, rng, 0.3)
    state = torch.tensor(i["state"], device=dev)
    return dict(case=case, n=n, cap=cap, box=i["box"], seed=seed, step=0, reaction=P.make_reaction(**i["reactions"][0]),
                pos=torch.tensor(x, device=dev), type=torch.tensor(i["type"], device=dev), from_state=state,
                state=state.clone(), nadj=torch.zeros(n, dtype=torch.uint8, device=dev),
                adj=torch.zeros(n * cap, dtype=torch.int32, device=dev),
                bonds=torch.zeros(6 * n, dtype=torch.int32, device=dev),
                formed=torch.zeros(1, dtype=torch.int32, device=dev))


# ---- one pass ------------------------------------------------------------------------------------------
def _call(name, g, *args):
    code = getattr(P.lib(), name)(g.h, *args)
    if code != P.PRX_OK:
        raise P.PolyrxError(code, name)


def _read(g, part):
    """Positions, velocities, states and bonds of a system into its part of the kept arrays."""
    _call("prx_get_positions", g, part["positions"].ctypes.data)
    _call("prx_get_velocities", g, part["velocities"].ctypes.data)
    _call("prx_get_states", g, part["states"].ctypes.data)
    _call("prx_get_bonds", g, part["bonds"].ctypes.data, len(part["bonds"]), ctypes.byref(ctypes.c_uint64()))


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "run":
        g = state["g"][0]
        g.run(case["steps"])
        _read(g, state["parts"][0])
        return state["whole"]
    if call == "monitor":
        g = state["g"][0]
        g.run(case["steps"])
        return g.observables()
    if call == "ensemble":
        state["batch"].run(case["steps"])
        state["batch"].sync()
        for g, part in zip(state["g"], state["parts"]):
            _read(g, part)
        return state["whole"]
    if call == "serve":
        server = state["server"]
        now = time.perf_counter()
        for q, (steps, n, system) in enumerate(state["jobs"]):
            server.submit(S.Job(job_id=q, nsteps=steps, arrival=now, system=system, n=n))
        while not server.idle():
            server.step()
        done, server.done = sorted(server.done, key=lambda j: j.job_id), []
        for j, room in zip(done, state["room"]):
            room[: len(j.result["bonds"])] = j.result["bonds"].view(np.int32).reshape(-1, 6)
        return [dict(positions=j.result["positions"], states=j.result["states"], bonds=room)
                for j, room in zip(done, state["room"])]
    if call == "forces":
        return state["g"].forces()
    if call == "histogram":
        f = case["f"]
        return state["g"].pair_histogram((1 << A, 1, f), (1 << B, 0, 1), R_REACT, case["bins"])
    state["step"] += 10
    state["state"].copy_(state["from_state"])
    state["nadj"].zero_()
    trace = P.prx_react_noalloc(state["reaction"], state["box"], DT, state["seed"], state["step"], state["n"],
                                state["pos"].data_ptr(), state["type"].data_ptr(), state["state"].data_ptr(),
                                state["cap"], state["nadj"].data_ptr(), state["adj"].data_ptr(),
                                state["bonds"].data_ptr(), state["n"], state["formed"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    return dict(trace=trace, formed=state["formed"], state=state["state"], nadj=state["nadj"],
                bonds=state["bonds"])


def work(case):
    """A step reads and writes each particle's position and velocity once (FP64: 96 bytes) and evaluates about
    2.6 pairs within the cutoff per particle (25 operations each) and the integration (50)."""
    call, f64 = case["call"], 8
    if call in ("run", "monitor"):
        n = case["n"] * case["steps"]
    elif call == "ensemble":
        n = case["steps"] * sum(c["n"] for c in _replicas(case["replicas"], case["lo"], case["hi"]))
    elif call == "serve":
        n = sum(c["n"] * steps for c, steps in _jobs(case))
    elif call == "forces":  # positions and bond partners in, forces out
        return dict(bytes=case["n"] * (3 * f64 + 4 + 3 * f64), flops=case["n"] * 90)
    elif call == "histogram":  # positions, types and states in
        return dict(bytes=case["n"] * (3 * f64 + 2), flops=case["n"] * case["share"] * 60)
    else:  # positions, types, states, adjacency in and out
        return dict(bytes=case["n"] * (3 * f64 + 2 + 2 * (1 + 4)), flops=case["n"] * case["share"] * 60)
    return dict(bytes=n * 96.0, flops=n * 115.0)


# ---- the same in 64 bits, in plain torch and numpy ---------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of arrays of counters under the key `seed`."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.broadcast_to(np.asarray(v, np.uint64), np.shape(c1)).copy() for v in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32 & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = k0 + 0x9E3779B9 & 0xFFFFFFFF, k1 + 0xBB67AE85 & 0xFFFFFFFF
    return c


def _draw(seed, step, a, b, tag):
    return _philox(step & 0xFFFFFFFF, a, b, tag | step >> 32 << 8, seed)


def _word(c):
    return c[0] << np.uint64(32) | c[1]


def _near(d, box):
    return d - box * torch.round(d / box)


def _pairs(x, box, r):
    """Ordered pairs (i, j) nearer than about r (never without one that is)."""
    n, xf, bf = len(x), x.float(), box.float()
    rows, got = max(1, (1 << 27) // n), []
    for s in range(0, n, rows):
        r2 = torch.zeros((min(rows, n - s), n), device=x.device)
        for d in range(3):
            r2 += _near(xf[None, :, d] - xf[s:s + rows, None, d], bf[d]) ** 2
        i, j = torch.nonzero(r2 < (r + 1e-3) ** 2, as_tuple=True)
        got.append(torch.stack([i + s, j]))
    i, j = torch.cat(got, 1)
    return i[i != j], j[i != j]


def _forces(x, box, i, j, bi, bj, style):
    """WCA over the pairs (i, j) and FENE or mirror-LJ bonds (bi, bj), both in both orders; and the energy."""
    f = torch.zeros_like(x)
    d = _near(x[j] - x[i], box)
    r2 = (d * d).sum(1)
    i, d, r2 = i[r2 < RC * RC], d[r2 < RC * RC], r2[r2 < RC * RC]
    s6 = r2 ** -3
    f.index_add_(0, i, -(24 * s6 * (2 * s6 - 1) / r2)[:, None] * d)
    energy = 0.5 * (4 * (s6 * s6 - s6 + 0.25)).sum()
    if len(bi):
        d = _near(x[bj] - x[bi], box)
        r2 = (d * d).sum(1)
        q = 1 - r2 / FENE_R0 ** 2
        r = r2.sqrt()
        s = 2 * RC - r
        t6 = s ** -6
        inside = (r > RC) & (r < 2 * RC)
        mirror = torch.where(inside, 24 * (2 * t6 * t6 - t6) / s / r, torch.zeros_like(r))
        g = torch.where(style == 0, FENE_K / q, mirror)
        e = torch.where(style == 0, -0.5 * FENE_K * FENE_R0 ** 2 * torch.log(q.clamp(min=1e-12)),
                        torch.where(inside, 4 * (t6 * t6 - t6 + 0.25), torch.zeros_like(r)))
        f.index_add_(0, bi, g[:, None] * d)
        energy = energy + 0.5 * e.sum()
    return f, energy


def _smallest_key(seed, step, own, other, tag):
    key = _word(_draw(seed, step, own, other, tag))
    at = np.lexsort((other, key, own))
    at = at[np.unique(own[at], return_index=True)[1]]
    return own[at], other[at]


def _react(i, pi, pj, r2, step, type_, state, bonded):
    """New bonds (a, t) of one reaction step of the random rule (Table I) among the ordered pairs within reach."""
    r = i["reactions"][0]
    el = lambda p, m, lo, hi: ((r[m] >> type_[p]) & 1 == 1) & (state[p] >= r[lo]) & (state[p] <= r[hi])  # noqa: E731
    ok = (r2 < r["r_react"] ** 2) & el(pi, "mask_A", "a_lo", "a_hi") & el(pj, "mask_T", "t_lo", "t_hi")
    a, t = pi[ok], pj[ok]
    ok = np.array([(int(u), int(w)) not in bonded for u, w in zip(a, t)], bool)
    a, t = a[ok], t[ok]
    u = (_word(_draw(i["seed"], step, a, t, 2)) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    ok = u < r["k"] * DT * r["theta"]
    a, t = a[ok], t[ok]
    a, t = _smallest_key(i["seed"], step, a, t, 3)  # one T per A
    t, a = _smallest_key(i["seed"], step, t, a, 4)  # one A per T
    return a, t


def _trajectory(case, seed):
    i = _inputs(case, seed)
    n, r = i["n"], i["reactions"][0]
    dev = torch.device("cuda")
    x, v = torch.tensor(i["x"], device=dev), torch.tensor(i["v"], device=dev)
    box = torch.tensor(i["box"], dtype=torch.float64, device=dev)
    type_, state, ids = i["type"].astype(np.int64), i["state"].astype(np.int64), np.arange(n)
    made = [] if i["bonds"] is None else [tuple(b) for b in i["bonds"].tolist()]
    style = [0] * len(made)
    bonded, stale = {p for b in made for p in (b, b[::-1])}, True
    since = None
    for step in range(1, case["steps"] + 1):
        if since is None or (x - since).square().sum(1).max() > 0.19 ** 2:
            since = x.clone()
            li, lj = _pairs(x % box, box, RC + 0.4)
        if stale:
            b = torch.tensor(made or np.zeros((0, 2), np.int64), device=dev, dtype=torch.long)
            bi, bj = torch.cat([b[:, 0], b[:, 1]]), torch.cat([b[:, 1], b[:, 0]])
            kind, stale = torch.tensor(style + style, device=dev), False
        f, _ = _forces(x, box, li, lj, bi, bj, kind)
        w = _draw(seed, step, ids, 0, 1)
        u = np.stack([(c >> np.uint64(8)).astype(np.float64) * 2.0 ** -24 - 0.5 for c in w[:3]], 1)
        f += math.sqrt(24.0 / DT) * torch.tensor(u, device=dev) - v
        v = v + DT * f
        x = x + DT * v
        if step % r["theta"] == 0:
            d = _near(x[lj] - x[li], box)
            r2 = (d * d).sum(1)
            near = r2 < r["r_react"] ** 2
            a, t = _react(i, li[near].cpu().numpy(), lj[near].cpu().numpy(), r2[near].cpu().numpy(), step, type_, state,
                          bonded)
            state[a] += r["dA"]
            state[t] += r["dT"]
            for p in zip(a.tolist(), t.tolist()):
                made.append(p)
                style.append(r["bond_style"])
                bonded |= {p, p[::-1]}
                stale = True
    return dict(positions=(x % box).cpu().numpy(), velocities=v.cpu().numpy(), states=None, bonds=None)


def exact(case, seed):
    """Forces, and short runs of one reaction with the random rule.  None for systems whose run would take minutes
    in plain torch, for long runs (a trajectory is chaotic: after some hundred steps its rounding is its own), and
    for calls that return whole numbers only."""
    if case["call"] == "forces":
        x, box, pairs = _force_inputs(case, seed)
        dev = torch.device("cuda")
        x, box = torch.tensor(x, device=dev), torch.tensor(box, dtype=torch.float64, device=dev)
        b = torch.tensor(pairs, device=dev)
        i, j = _pairs(x, box, RC)
        f, e = _forces(x, box, i, j, torch.cat([b[:, 0], b[:, 1]]), torch.cat([b[:, 1], b[:, 0]]),
                       torch.zeros(2 * len(b), device=dev, dtype=torch.long))
        return f.cpu().numpy(), float(e)
    if (case["call"] == "run" and case["scheme"] != "mixed" and not case.get("selection") and case["n"] <= 40000
            and case["steps"] <= 200):
        return _trajectory(case, seed)
    return None
