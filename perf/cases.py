"""The work that is measured for speed, as cases: what users of this framework have it do.

A program of this framework holds a context (a batch of multicanonical chains, a parallel-tempering
batch) or a server on the GPU, sweeps it for a step's worth of sweeps, takes a weight step where it
iterates, and reads the step's results into host arrays, which is the only form in which the
library hands them out.  A case is one such step.  Kinds:

  muca       muca_run_sweeps for n_sweeps, then (if `update`) a weight step, then the results
  uneven     a batch of several L and ensembles, its iteration loop captured in a CUDA graph
  pt         parallel tempering: an adaptation window (if `adapt_sweeps`), then n_sweeps
  ensembles  the profile scan's preparation: one density of states per realization copied to
             chains that build flat, power-law and 1/k weights from it
  serving    a closed batch of realization jobs through the request loop

Sizes are those of the paper (L = 3..8, its sample and temperature counts), of `workloads.py`,
`bench.py` and the tests (L up to 12), or plain odd ones.
"""
import math

import numpy as np
import torch

from paper_2011_08560_gb300 import eamc, serve, workloads

# integer lane-operations that one spin-flip attempt cannot do without: a quarter of a
# Philox4x32-10 call (20), its share of a bit-sliced local field (3.5), threshold fetch and
# compare (3), flip and energy (2), lowest energy and round-trip check (1.5)
MUCA_OPS = 30.0
# the same for a parallel-tempering attempt (32 realizations to a word): 150 per site word
PT_OPS = 4.7

KINDS = {"flat": eamc.EA_FLAT, "powerlaw": eamc.EA_POWERLAW, "1/k": eamc.EA_ONE_OVER_K}


def listed():
    return [
        # The smallest: one realization of L = 4, flat ensemble, one step of its plain weight
        # iteration (10^4 sweeps).  One chain on the whole GPU: latency and launches.
        {"name": "one_chain_L4", "kind": "muca", "L": 4, "n": 1, "order": "lex", "width": 32,
         "ensembles": "flat", "recursion": "plain", "iter_steps": 8, "iter_sweeps": 2000,
         "n_sweeps": 10000, "update": True, "count_rt": False},
        # The headline: L = 8, 1024 power-law chains in production, checkerboard order, round trips
        # counted, in the tiles that the autotuner picks for this batch.
        {"name": "production_L8_1024", "kind": "muca", "L": 8, "n": 1024, "order": "colour", "width": 8,
         "ensembles": "powerlaw", "recursion": "berg", "iter_steps": 40, "iter_sweeps": 1500,
         "n_sweeps": 10000, "update": False, "count_rt": True},
        # The same batch in the library's default (lexicographic) order.
        {"name": "production_L8_1024_lex", "kind": "muca", "L": 8, "n": 1024, "order": "lex", "width": 16,
         "ensembles": "powerlaw", "recursion": "berg", "iter_steps": 40, "iter_sweeps": 1500,
         "n_sweeps": 4000, "update": False, "count_rt": True},
        # The paper's sample count at L = 8: more chains than the SMs hold at once in narrow tiles.
        {"name": "production_L8_4096", "kind": "muca", "L": 8, "n": 4096, "order": "colour", "width": 16,
         "ensembles": "powerlaw", "recursion": "berg", "iter_steps": 40, "iter_sweeps": 1000,
         "n_sweeps": 3000, "update": False, "count_rt": True},
        # Weight iteration at L = 6: 1024 realizations, each as a flat and as a power-law chain,
        # full tiles, default order, one plain weight step after the sweeps.
        {"name": "iteration_L6_2x1024", "kind": "muca", "L": 6, "n": 1024, "order": "lex", "width": 32,
         "ensembles": "flat,powerlaw", "recursion": "plain", "iter_steps": 10, "iter_sweeps": 1000,
         "n_sweeps": 4000, "update": True, "count_rt": False},
        # Odd L, a ragged number of realizations, Berg's recursion, narrow tiles.
        {"name": "iteration_L7_500", "kind": "muca", "L": 7, "n": 500, "order": "colour", "width": 8,
         "ensembles": "powerlaw", "recursion": "berg", "iter_steps": 25, "iter_sweeps": 1500,
         "n_sweeps": 4000, "update": True, "count_rt": False},
        # A large lattice, few realizations, default tile width: the tables exceed what an SM holds.
        {"name": "iteration_L10_300", "kind": "muca", "L": 10, "n": 300, "order": "colour", "width": 32,
         "ensembles": "powerlaw", "recursion": "berg", "iter_steps": 25, "iter_sweeps": 800,
         "n_sweeps": 1500, "update": True, "count_rt": False},
        # The uneven batch: 4096 realizations of L in {4, 6, 8, 10, 12}, each in three ensembles, on
        # the work queue, the iteration loop as a captured graph.
        {"name": "uneven_12288", "kind": "uneven", "Ls": "4,6,8,10,12", "n": 4096, "order": "lex",
         "ensembles": "powerlaw,flat,1/k", "persistent": True, "iters": 3, "n_sweeps": 200},
        # Parallel tempering in production: L = 8, 1024 realizations at 32 temperatures.
        {"name": "pt_L8_1024x32", "kind": "pt", "L": 8, "n": 1024, "M": 32, "beta_min": 0.2, "beta_max": 3.0,
         "adapt_sweeps": 0, "n_sweeps": 4000, "spins": False, "records": False},
        # The paper's protocol at an odd L: adapt the temperatures over a window, then count round
        # trips; its M = 12 temperatures at L = 5, a ragged number of realizations.
        {"name": "pt_protocol_L5_333x12", "kind": "pt", "L": 5, "n": 333, "M": 12, "beta_min": 0.3,
         "beta_max": 2.15, "adapt_sweeps": 1000, "n_sweeps": 1000, "spins": True, "records": True},
        # The profile scan's ensembles at L = 6: 128 densities of states, 18 ensembles of each.
        {"name": "ensembles_L6_18x128", "kind": "ensembles", "L": 6, "n": 128, "n_pl": 16},
        # Requests of mixed L and round-trip targets through the serving loop.
        {"name": "serving_96_jobs", "kind": "serving", "Ls": "4,5,6,7,8,9,10,11,12", "n": 96, "order": "colour",
         "base_sweeps": 16, "iter_steps": 8, "ticks_per_step": 8, "max_prod_ticks": 100, "rt_max": 1000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["muca"] * 5 + ["uneven"] + ["pt"] * 3 + ["ensembles", "serving"])
    if kind == "muca":
        L = rng.choice(range(3, 13))
        order = rng.choice(["lex", "colour"])
        ens = rng.choice(["flat", "powerlaw", "flat,powerlaw"])
        n = _log_int(rng, 1, 4096 // (1 if L <= 8 else 4))
        width = rng.choice([32] + eamc.narrow_widths(3, L, int(order == "colour")))
        # up to 1.5e9 attempts in all and 1.5e6 in a chain
        chains = n * len(ens.split(","))
        sweeps = int(min(1.5e6, max(2e5, 1.5e9 / chains)) * rng.uniform(0.2, 1.0) / L ** 3) + 1
        if n > 1024:
            sweeps = sweeps // (n // 1024) + 1
        return {"kind": "muca", "L": L, "n": n, "order": order, "width": width, "ensembles": ens,
                "recursion": rng.choice(["plain", "berg"]), "iter_steps": 15,
                "iter_sweeps": max(50, int(3e5 / L ** 3 / max(1, chains / 2048))),
                "n_sweeps": sweeps, "update": rng.choice([True, False]), "count_rt": rng.choice([True, False])}
    if kind == "uneven":
        Ls = sorted(rng.sample(range(3, 13), rng.randint(2, 5)))
        return {"kind": "uneven", "Ls": ",".join(map(str, Ls)), "n": _log_int(rng, 32, 4096),
                "order": rng.choice(["lex", "colour"]),
                "ensembles": rng.choice(["powerlaw", "powerlaw,flat", "powerlaw,flat,1/k"]),
                "persistent": rng.choice([True, False]), "iters": rng.randint(1, 3),
                "n_sweeps": rng.randint(20, 100)}
    if kind == "pt":
        L = rng.choice(range(3, 13))
        n = _log_int(rng, 1, 1024 if L <= 8 else 256)
        M = rng.choice([2, 7, 12, 14, 17, 20, 32])
        sweeps = int(min(3000, 6e10 / (32 * math.ceil(n / 32) * M * L ** 3) * 1.0) * rng.uniform(0.2, 1.0)) + 10
        return {"kind": "pt", "L": L, "n": n, "M": M, "beta_min": rng.choice([0.2, 0.3]),
                "beta_max": rng.choice([2.15, 3.0]), "adapt_sweeps": rng.choice([0, sweeps // 2 + 4]),
                "n_sweeps": sweeps, "spins": n * M * L ** 3 <= 1 << 20, "records": n * M <= 4096}
    if kind == "ensembles":
        return {"kind": "ensembles", "L": rng.choice(range(3, 13)), "n": _log_int(rng, 3, 128),
                "n_pl": rng.randint(1, 16)}
    Ls = sorted(rng.sample(range(4, 13), rng.randint(1, 6)))
    return {"kind": "serving", "Ls": ",".join(map(str, Ls)), "n": _log_int(rng, 1, 128),
            "order": rng.choice(["lex", "colour"]), "base_sweeps": 16, "iter_steps": 8,
            "ticks_per_step": rng.randint(2, 8), "max_prod_ticks": rng.randint(10, 100), "rt_max": 1000}


def _ints(text):
    return [int(x) for x in text.split(",")]


def _context(seed):
    stream = torch.cuda.Stream()
    return {"stream": stream, "ctx": eamc.Context(seed=seed, stream=stream.cuda_stream)}


def _rows(L):
    return ((3 * L ** 3) // 2 >> 1) + 1


def _prepare_muca(c, seed):
    s = _context(seed)
    ctx, L, n = s["ctx"], c["L"], c["n"]
    ctx.set_sweep_order(workloads.order_code(c["order"]))
    if c["width"] != 32:
        ctx.set_tile_width(L, c["width"])
    for stream_id, ens in enumerate(c["ensembles"].split(",")):
        first = ctx.init_disorder(3, L, n, rid0=0, stream=stream_id)
        ctx.set_ensemble(first, n, KINDS[ens])
        if c["recursion"] == "berg":
            ctx.set_recursion(first, n, eamc.EA_REC_BERG)
    for _ in range(c["iter_steps"]):
        ctx.run_sweeps(c["iter_sweeps"])
        ctx.update_weights()
    ctx.set_eg(0, ctx.num_chains())
    ctx.roundtrips_array(reset=True)
    s["rows"] = _rows(L)
    return s


def _results(s, spins=True):
    """What a program reads after a step: histograms are read by the caller; here the round-trip
    records and the chains' state."""
    ctx = s["ctx"]
    rt = ctx.roundtrips_array()
    S, E, t = ctx.state(spins=spins)
    out = {f: rt[f] for f in rt.dtype.names if f != "pad"}
    out.update({"E": E, "t": t.astype(np.int64)})
    if spins:
        out["spins"] = S
    return out


def _run_muca(c, s):
    ctx = s["ctx"]
    ctx.run_sweeps(c["n_sweeps"], count_roundtrips=c["count_rt"])
    out = {"hist": ctx.histograms(rows=s["rows"])}
    if c["update"]:
        ctx.update_weights()
        out["weights"] = ctx.get_weights(rows=s["rows"])
    out.update(_results(s))
    return out


def _uneven_counts(c):
    Ls = _ints(c["Ls"])
    return [(L, sum(1 for k in range(c["n"]) if k % len(Ls) == i)) for i, L in enumerate(Ls)]


def _prepare_uneven(c, seed):
    s = _context(seed)
    ctx = s["ctx"]
    ctx.set_sweep_order(workloads.order_code(c["order"]))
    ens = c["ensembles"].split(",")
    spans = []
    for i, (L, n) in enumerate(_uneven_counts(c)):
        for stream_id, e in enumerate(ens):
            first = ctx.init_disorder(3, L, n, rid0=i * c["n"], stream=stream_id)
            ctx.set_ensemble(first, n, KINDS["powerlaw" if e == "1/k" else e])
            spans.append((first, n, e))
    ctx.set_launch(persistent=c["persistent"])
    for _ in range(4):
        ctx.run_sweeps(30)
        ctx.update_weights()
    ctx.set_eg(0, ctx.num_chains())
    for first, n, e in spans:
        if e == "1/k":
            ctx.build_ensemble(first, n, eamc.EA_ONE_OVER_K)
    ctx.roundtrips_array(reset=True)
    s["spans"] = [(first, n, _rows(L)) for (first, n, _), L in
                  zip(spans, [L for L, _ in _uneven_counts(c) for _ in ens])]
    ctx.graph_capture(c["iters"], c["n_sweeps"], count_roundtrips=True, update_weights=True)
    return s


def _run_uneven(c, s):
    s["ctx"].graph_launch(1)
    out = _results(s, spins=False)
    for k, (first, n, rows) in enumerate(s["spans"]):
        out[f"weights{k}"] = s["ctx"].get_weights(first, n, rows=rows)
    return out


def _prepare_pt(c, seed):
    s = _context(seed)
    ctx = s["ctx"]
    ctx.pt_init(3, c["L"], c["n"], workloads.geometric_betas(c["M"], c["beta_min"], c["beta_max"]))
    ctx.pt_run(200)
    _, E, _, _ = ctx.pt_state(spins=False)
    # round trips between a low energy of each realization and that of its hottest replica
    ctx.pt_set_rt_bounds(E.min(axis=1), E[:, 0])
    return s


def _run_pt(c, s):
    ctx = s["ctx"]
    out = {}
    if c["adapt_sweeps"]:
        ctx.pt_run(c["adapt_sweeps"])
        ctx.pt_adapt(0.5)
        out["betas"] = ctx.pt_betas()
    ctx.pt_run(c["n_sweeps"], count_roundtrips=True)
    S, E, labels, _ = ctx.pt_state(spins=c["spins"])
    accepted, _ = ctx.pt_exchange_counts()
    out.update({"E": E, "labels": labels, "accepted": accepted.astype(np.int64),
                "swaps": ctx.pt_swap_counts().astype(np.int64)})
    if c["spins"]:
        out["spins"] = S
    if c["records"]:
        recs = ctx.pt_roundtrips()
        for f in ("n_rt", "t_first", "t_last", "e_min"):
            out[f] = np.array([[x[f] for x in row] for row in recs], dtype=np.int64)
    return out


def _profiles(c):
    """The scan's ensembles as (kind, alpha, pole): flat, a grid of power laws, 1/k."""
    grid = [(a, p) for p in (24.0, 48.0, 96.0, 192.0) for a in (-1.5, -2.5, -3.6, -5.0)]
    return ([("flat", -3.6, 96.0)] + [("powerlaw", a, p) for a, p in grid[:c["n_pl"]]] + [("1/k", -3.6, 96.0)])


def _ensemble_inputs(c, seed):
    """Couplings, a smooth density of states with noise for each realization as the weights of a
    power-law iteration (alpha = -3.6, pole 96), and each realization's lowest energy."""
    L, n = c["L"], c["n"]
    V, rows = L ** 3, _rows(L)
    rng = np.random.default_rng([seed, 23])
    J = (1 - 2 * rng.integers(0, 2, size=(n, 3 * V))).astype(np.int8)
    parity = (J < 0).sum(axis=1) & 1
    # bin b holds the energies 2 (2 b + parity) - 3 V; the top bin is the largest E <= 0
    half = 3 * V // 2
    top = np.where((half & 1) == parity, half, half - 1) >> 1
    E = 2 * (2 * np.arange(rows)[None, :] + parity[:, None]) - 3 * V
    ground = -1.75 * V * (1 + 0.02 * rng.standard_normal(n))
    e_g = np.array([E[k][np.searchsorted(E[k], ground[k])] for k in range(n)], dtype=np.int32)
    # entropy: Gaussian at high energies, falling faster near the ground state, rough by 0.1
    depth = np.clip(E / ground[:, None], 0.0, None)
    ln_omega = V * math.log(2.0) * (1.0 - 0.85 * depth ** 2 - 0.12 * depth ** 6)
    ln_omega = ln_omega + 0.1 * rng.standard_normal(E.shape)
    weights = _ln_profile(-3.6, 96.0, e_g[:, None], E) - ln_omega
    weights -= np.take_along_axis(weights, top[:, None], axis=1)
    weights[np.arange(rows)[None, :] > top[:, None]] = 0.0
    return J, E, top, e_g, weights


def _ln_profile(alpha, pole, e_g, E):
    """ln of the power-law target: alpha ln(E / (pole - E_g) + 1), held below E_g."""
    return alpha * np.log(np.maximum(E, e_g) / (pole - e_g) + 1.0)


def _prepare_ensembles(c, seed):
    s = _context(seed)
    ctx, n = s["ctx"], c["n"]
    J, _, _, e_g, weights = _ensemble_inputs(c, seed)
    kinds = _profiles(c)
    dos = ctx.init_disorder(3, c["L"], n, couplings=J)
    ctx.set_ensemble(dos, n, eamc.EA_POWERLAW)
    ctx.set_weights(dos, weights)
    ctx.set_eg(dos, n, e_g)
    s["targets"] = [ctx.init_disorder(3, c["L"], n, stream=k + 1, couplings=J) for k in range(len(kinds))]
    s["src"] = np.tile(np.arange(dos, dos + n, dtype=np.int32), len(kinds))
    s["dst"] = np.concatenate([np.arange(f, f + n, dtype=np.int32) for f in s["targets"]])
    s["rows"] = _rows(c["L"])
    return s


def _run_ensembles(c, s):
    ctx, n = s["ctx"], c["n"]
    ctx.copy_weights(s["src"], s["dst"])
    for first, (kind, alpha, pole) in zip(s["targets"], _profiles(c)):
        ctx.build_ensemble(first, n, KINDS[kind], alpha, pole)
    first, total = s["targets"][0], n * len(s["targets"])
    return {"weights": ctx.get_weights(first, total, rows=s["rows"]),
            "thresholds": ctx.get_thresholds(first, total, rows=s["rows"]).astype(np.int64)}


def _prepare_serving(c, seed):
    server = serve.Server(seed=seed, Ls=_ints(c["Ls"]), base_sweeps=c["base_sweeps"], mem_budget=4 << 30,
                          order=workloads.order_code(c["order"]))
    rng = np.random.default_rng([seed, 29])
    L = rng.choice(_ints(c["Ls"]), size=c["n"])
    rt = np.exp(rng.uniform(math.log(10.0), math.log(c["rt_max"]), size=c["n"])).round().astype(int)
    return {"server": server, "L": L, "rt": rt, "next": 0}


def _run_serving(c, s):
    server = s["server"]
    jobs = []
    for L, rt in zip(s["L"], s["rt"]):
        jobs.append(serve.Job(jid=s["next"], L=int(L), rid=s["next"], rt_target=int(rt),
                              iter_steps=c["iter_steps"], ticks_per_step=c["ticks_per_step"],
                              max_prod_ticks=c["max_prod_ticks"]))
        s["next"] += 1
        server.submit(jobs[-1])
    while server.jobs:
        server.step(8)
        server.poll()
    fields = ("n_rt", "t_first", "t_last", "e_g", "e_min", "sweeps", "requeues")
    return {f: np.array([j.result[f] for j in jobs], dtype=np.int64) for f in fields}


def prepare(case, seed):
    s = {"muca": _prepare_muca, "uneven": _prepare_uneven, "pt": _prepare_pt,
         "ensembles": _prepare_ensembles, "serving": _prepare_serving}[case["kind"]](case, seed)
    s["case"] = case
    return s


def run(state):
    c = state["case"]
    return {"muca": _run_muca, "uneven": _run_uneven, "pt": _run_pt, "ensembles": _run_ensembles,
            "serving": _run_serving}[c["kind"]](c, state)


def work(case):
    """Integer operations count as flops; bytes: lattices (a bit per spin and bond), tables and
    records in, state and results out, once each."""
    kind = case["kind"]
    if kind in ("muca", "uneven"):
        if kind == "muca":
            groups = [(case["L"], case["n"] * len(case["ensembles"].split(",")))]
            sweeps = case["n_sweeps"]
        else:
            groups = [(L, n * len(case["ensembles"].split(","))) for L, n in _uneven_counts(case)]
            sweeps = case["n_sweeps"] * case["iters"]
        attempts = sum(n * L ** 3 for L, n in groups) * sweeps
        # thresholds and histogram of the range, spins in and out, bonds in, a record of 100 bytes
        b = sum(n * (_rows(L) * (32 + 8) + 5 * L ** 3 / 8 + 200) for L, n in groups)
        if case.get("update") or kind == "uneven":
            b += sum(n * _rows(L) * 16 for L, n in groups)
        return {"bytes": b, "flops": MUCA_OPS * attempts}
    if kind == "pt":
        n, M, V = case["n"], case["M"], case["L"] ** 3
        attempts = n * M * V * (case["n_sweeps"] + case["adapt_sweeps"])
        return {"bytes": n * (M * (2 * V / 8 + 80) + 3 * V / 8), "flops": PT_OPS * attempts}
    if kind == "ensembles":
        cells = case["n"] * (case["n_pl"] + 2) * _rows(case["L"])
        return {"bytes": cells * (8 + 32), "flops": 40.0 * cells}
    Ls = _ints(case["Ls"])
    ticks = case["iter_steps"] * case["ticks_per_step"] + case["max_prod_ticks"]
    attempts = case["n"] * case["base_sweeps"] * max(Ls) ** 3 * ticks
    rows = sum(_rows(L) for L in Ls) / len(Ls)
    return {"bytes": case["n"] * (rows * 60 + 400), "flops": MUCA_OPS * attempts}


def exact(case, seed):
    """The ensembles' weights in 64 bits.  The other kinds' outputs are whole numbers of random
    trajectories, or weights and temperatures that follow from those."""
    if case["kind"] != "ensembles":
        return None
    _, E, top, e_g, w = _ensemble_inputs(case, seed)
    n, rows = w.shape
    cols = np.arange(rows)[None, :]
    inside = cols <= top[:, None]
    eg = e_g[:, None].astype(np.float64)
    ln_omega = _ln_profile(-3.6, 96.0, eg, E) - w
    bottom = np.array([int(np.flatnonzero(E[k] == e_g[k])[0]) for k in range(n)])[:, None]
    out = []
    for kind, alpha, pole in _profiles(case):
        if kind == "flat":
            v = -ln_omega
        elif kind == "powerlaw":
            v = _ln_profile(alpha, pole, eg, E) - ln_omega
        else:
            # ln k(E) = ln of the summed density of states from E_g up; the flat form, matched, below
            ln_k = np.logaddexp.accumulate(np.where(cols >= bottom, ln_omega, -np.inf), axis=1)
            v = np.where(cols >= bottom, -ln_k, -ln_omega)
        v = v - np.take_along_axis(v, top[:, None], axis=1)
        out.append(np.where(inside, v, 0.0))
    return {"weights": np.concatenate(out), "thresholds": None}
