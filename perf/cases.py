"""What a program that uses this library has it do, as cases that can be timed.

Four kinds of call, each through the package's public entry points:

* ``chain``: one lattice, ``Lattice.sweep`` with records every ``obs_every``
  sweeps (0: none), then what the program reads back: the records, the
  histograms if it enabled them, and the lattice.
* ``batch``: several lattices advanced together by ``Batch.sweep``, then their
  records and lattices.
* ``serve``: a set of requests handed to a running ``Server`` and waited for.
* ``checkpoint``: a saved lattice loaded, its observables counted, and the
  lattice saved again.

A pass continues from where the one before it left the lattices, as a Markov
chain does; random streams are keyed by (seed, sweep, site), so the outputs of
the same passes on the same seed are the same whole numbers.

``work`` counts bytes that have to move whatever the method (the lattices in
and out once, 2 bits a site, the records and what is copied to the program)
and, as ``flops``, the integer operations of the sweeps' definition
(``OPS_PER_UPDATE`` a site-update).  There is no floating-point output, hence
no 64-bit value to compare with: ``exact`` has none.
"""
from __future__ import annotations

import math

import numpy as np

# Integer operations of one site-update by definition, half of a coupled
# pair's: 10 of its share of a Philox4x32-10 call for eight pairs (10 rounds of
# two multiplies and six additions or XORs), 16 additions of the eight
# neighbours' charge and spin, 6 for the energy change's index, 4 for the
# choice and the decision.
OPS_PER_UPDATE = (10 + 16 + 6 + 4) / 2.0


def listed():
    return [
        # The paper's snapshots of charged drops: a 64 x 64 lattice looked at
        # every ten sweeps.  The smallest call: launches and latency.
        dict(name="snapshot64", kind="chain", Lx=64, Ly=64, sweeps=10, obs_every=0, nbins=0,
             n=0.1, T=0.5, Delta=0.0, V=0.5, J=1.0),
        # The 16 x 16 check lattice: 2000 sweeps, a record after every one.
        dict(name="chain16", kind="chain", Lx=16, Ly=16, sweeps=2000, obs_every=1, nbins=0,
             n=0.125, T=1.0, Delta=0.5, V=1.0, J=1.0),
        # The paper's largest lattice, 256 x 256, records every ten sweeps.
        dict(name="chain256", kind="chain", Lx=256, Ly=256, sweeps=1000, obs_every=10, nbins=0,
             n=0.2, T=0.8, Delta=0.2, V=1.0, J=0.5),
        # An ordinary size that is no power of two (rows of 250 sites a class).
        dict(name="chain1000", kind="chain", Lx=1000, Ly=1000, sweeps=500, obs_every=10, nbins=0,
             n=0.05, T=0.6, Delta=0.2, V=1.0, J=0.5),
        # A rectangular strip, ragged, recorded and histogrammed every sweep.
        dict(name="strip2060x516", kind="chain", Lx=2060, Ly=516, sweeps=400, obs_every=1,
             nbins=512, n=0.0, T=0.45, Delta=-0.2, V=1.0, J=1.0),
        # The benchmark's large lattice near the charge-ordering crossover,
        # records and histograms after every sweep.
        dict(name="large16384", kind="chain", Lx=16384, Ly=16384, sweeps=200, obs_every=1,
             nbins=1024, n=0.05, T=0.6, Delta=0.2, V=1.0, J=0.5),
        # The benchmark's temperature sweep: four 4096 x 4096 lattices.
        dict(name="temperature4096", kind="batch", count=4, L_min=4096, L_max=4096, sizes="fixed",
             shape_seed=0, sweeps=200, obs_every=10),
        # Sixteen copies of a middle-sized lattice.
        dict(name="copies1024", kind="batch", count=16, L_min=1024, L_max=1024, sizes="fixed",
             shape_seed=0, sweeps=400, obs_every=10),
        # The benchmark's 512 replicas of uneven size.
        dict(name="replicas512", kind="batch", count=512, L_min=32, L_max=256, sizes="paper",
             shape_seed=3, sweeps=2000, obs_every=0),
        # A thermodynamics grid: sixteen temperatures, four copies each, a
        # record after every sweep.
        dict(name="thermo64", kind="batch", count=64, L_min=64, L_max=64, sizes="fixed",
             shape_seed=0, sweeps=4000, obs_every=1),
        # A burst of requests of mixed sizes (most of them ragged) to the server.
        dict(name="serve48", kind="serve", count=48, L_min=32, L_max=1024, shape_seed=4,
             sweeps_min=100, sweeps_max=2000),
        # Load, count and save a 4096 x 4096 lattice, one byte a site.
        dict(name="checkpoint4096", kind="checkpoint", Lx=4096, Ly=4096, packed=False),
    ]


def _side(rng, lo, hi):
    """A side in [lo, hi], spread over its logarithm; four in ten of them a
    multiple of 64 or a power of two where the range has one."""
    L = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    kind = rng.random()
    if kind < 0.2:
        L = 2.0 ** round(math.log2(L))
    elif kind < 0.4 and L >= 64:
        L = 64 * round(L / 64)
    return int(min(hi, max(lo, 4 * round(L / 4))))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["chain", "chain", "chain", "batch", "batch", "serve", "checkpoint"])
    if kind == "chain":
        Lx = _side(rng, 4, 16384)
        Ly = _side(rng, max(4, Lx // 4), min(16384, 4 * Lx))
        sweeps = _log_int(rng, 10, max(10, min(2000, 2 * 10 ** 10 // (Lx * Ly))))
        obs_every = rng.choice([0, 1, 10])
        sweeps = max(obs_every, sweeps - sweeps % max(obs_every, 1))
        return dict(kind=kind, Lx=Lx, Ly=Ly, sweeps=sweeps, obs_every=obs_every,
                    nbins=rng.choice([0, 256]) if obs_every else 0,
                    n=rng.choice([-0.1, 0.0, 0.05, 0.1, 0.3]), T=round(rng.uniform(0.2, 3.0), 3),
                    Delta=round(rng.uniform(-1.0, 1.0), 3), V=round(rng.uniform(0.0, 2.0), 3),
                    J=rng.choice([0.5, 1.0]))
    if kind == "batch":
        sizes = rng.choice(["fixed", "fixed", "log", "paper"])
        lo = 32 if sizes == "paper" else _side(rng, 16, 2048)
        hi = 256 if sizes == "paper" else lo if sizes == "fixed" else _side(rng, lo, min(2048, 8 * lo))
        count = _log_int(rng, 2, max(2, min(512, 2 ** 25 // (lo * hi))))
        obs_every = rng.choice([0, 1, 10])
        sweeps = _log_int(rng, 20, max(20, min(2000, 5 * 10 ** 9 // (count * hi * hi))))
        sweeps = max(obs_every, sweeps - sweeps % max(obs_every, 1))
        return dict(kind=kind, count=count, L_min=lo, L_max=hi, sizes=sizes,
                    shape_seed=rng.randrange(1000), sweeps=sweeps, obs_every=obs_every)
    if kind == "serve":
        hi = _side(rng, 64, 1024)
        return dict(kind=kind, count=_log_int(rng, 4, 48), L_min=16, L_max=hi,
                    shape_seed=rng.randrange(1000), sweeps_min=50,
                    sweeps_max=_log_int(rng, 100, 2000))
    return dict(kind=kind, Lx=_side(rng, 64, 4096), Ly=_side(rng, 64, 4096),
                packed=rng.random() < 0.5)


def _batch_shapes(case):
    rng = np.random.default_rng(case["shape_seed"])
    if case["sizes"] == "paper":
        return [int(L) for L in rng.choice([32, 64, 128, 256], size=case["count"])]
    lo, hi = case["L_min"], case["L_max"]
    Ls = np.exp(rng.uniform(math.log(lo), math.log(hi), size=case["count"]))
    return [lo if lo == hi else int(min(hi, max(lo, 4 * round(float(L) / 4)))) for L in Ls]


def _request_shapes(case):
    """(L, sweeps, obs_every) of every request: L and sweeps log-uniform, every
    third request with records."""
    rng = np.random.default_rng(case["shape_seed"])
    out = []
    for i in range(case["count"]):
        L = math.exp(rng.uniform(math.log(case["L_min"]), math.log(case["L_max"])))
        s = math.exp(rng.uniform(math.log(case["sweeps_min"]), math.log(case["sweeps_max"])))
        out.append((max(4, 4 * round(L / 4)), max(1, round(s)), 10 if i % 3 == 0 else 0))
    return out


def prepare(case, seed):
    import paper_2301_11735_gb300 as cc

    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "chain":
        records = case["sweeps"] // case["obs_every"] if case["obs_every"] else 0
        lat = cc.Lattice(case["Lx"], case["Ly"], obs_capacity=max(1, records))
        lat.init_constrained(int(rng.integers(1 << 62)), case["n"], 0.3)
        if case["nbins"]:
            lat.hist_enable(case["nbins"])
        return dict(case=case, lat=lat, records=records)
    if kind == "batch":
        records = case["sweeps"] // case["obs_every"] if case["obs_every"] else 0
        lats, beta, Delta, V, J = [], [], [], [], []
        for i, L in enumerate(_batch_shapes(case)):
            lat = cc.Lattice(L, L, obs_capacity=max(1, records))
            lat.init_constrained(int(rng.integers(1 << 62)), float(rng.choice([0.0, 0.1, 0.2])),
                                 0.3)
            lats.append(lat)
            beta.append(1.0 / (0.2 + 2.8 * (i % 16) / 15.0))
            Delta.append(float(rng.choice([-0.5, 0.0, 0.5])))
            V.append(float(rng.choice([0.5, 1.0])))
            J.append(1.0)
        return dict(case=case, lats=lats, batch=cc.Batch(lats), params=(beta, Delta, V, J),
                    records=records)
    if kind == "serve":
        reqs = []
        for L, sweeps, every in _request_shapes(case):
            reqs.append(dict(Lx=L, Ly=L, seed=int(rng.integers(1 << 62)),
                             n=float(rng.uniform(0.0, 0.3)), nsweeps=sweeps,
                             beta=1.0 / float(rng.uniform(0.2, 3.0)),
                             Delta=float(rng.uniform(-1.0, 1.0)), V=float(rng.uniform(0.0, 2.0)),
                             J=1.0, obs_every=every))
        return dict(case=case, server=cc.Server(hbm_budget_bytes=8 << 30, max_active=256),
                    reqs=reqs)
    # a saved lattice: three in ten sites charged, as a run leaves it
    Lx, Ly = case["Lx"], case["Ly"]
    lat = cc.Lattice(Lx, Ly)
    key = int(rng.integers(1 << 62))
    lat.init_constrained(key, 0.1, 0.3)
    saved = lat.get_state_packed() if case["packed"] else lat.get_state()
    return dict(case=case, lat=lat, key=key, saved=saved)


def _read_lattice(lat):
    """One byte a site for what is looked at, 2 bits a site for what is kept."""
    return lat.get_state() if lat.Lx * lat.Ly <= 1 << 20 else lat.get_state_packed()


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "chain":
        lat = state["lat"]
        lat.sweep(case["sweeps"], 1.0 / case["T"], case["Delta"], case["V"], case["J"],
                  obs_every=case["obs_every"])
        out = {"lattice": _read_lattice(lat)}
        if state["records"]:
            out["records"] = lat.obs_series(cap=state["records"])
        if case["nbins"]:
            out["hist"] = lat.hist()
        return out
    if kind == "batch":
        b = state["batch"]
        b.sweep(case["sweeps"], *state["params"], obs_every=case["obs_every"])
        b.sync()
        out = {"lattices": np.concatenate([lat.get_state_packed() for lat in state["lats"]])}
        if state["records"]:
            out["records"] = np.stack([lat.obs_series(cap=state["records"])
                                       for lat in state["lats"]])
        return out
    if kind == "serve":
        srv = state["server"]
        outs = [np.empty(r["Lx"] * r["Ly"], dtype=np.uint8) for r in state["reqs"]]
        tickets = [srv.submit(state_out=o, **r) for r, o in zip(state["reqs"], outs)]
        final, series = [], []
        for t, r in zip(tickets, state["reqs"]):
            obs = srv.wait(t)["final_obs"]
            final.append([obs[k] for k in ("sweeps_done", "Nc", "BV", "BJ", "M", "M_stag",
                                           "S_sum", "S_stag")])
            if r["obs_every"]:
                series.append(srv.series(t, cap=r["nsweeps"] // r["obs_every"] + 1))
            srv.release(t)
        return {"lattices": np.concatenate(outs), "final": np.array(final, dtype=np.int64),
                "records": np.concatenate(series)}
    lat, saved = state["lat"], state["saved"]
    if case["packed"]:
        lat.set_state_packed(saved, state["key"], 0)
    else:
        lat.set_state(saved, state["key"], 0)
    obs = lat.observables()
    again = lat.get_state_packed() if case["packed"] else lat.get_state()
    return {"obs": np.array([obs[k] for k in ("Nc", "BV", "BJ", "M", "M_stag", "S_sum",
                                              "S_stag")], dtype=np.int64), "lattice": again}


def exact(case, seed):
    """Every output is a whole number: nothing to compare in 64 bits."""
    return None


def work(case):
    kind = case["kind"]
    if kind == "checkpoint":
        N = case["Lx"] * case["Ly"]
        return {"bytes": 2 * N // 4 if case["packed"] else 2 * N, "flops": 16.0 * N}
    if kind == "serve":
        runs = [(L * L, s, every, 1) for L, s, every in _request_shapes(case)]
    elif kind == "batch":
        runs = [(L * L, case["sweeps"], case["obs_every"], 0.25) for L in _batch_shapes(case)]
    else:
        N = case["Lx"] * case["Ly"]
        runs = [(N, case["sweeps"], case["obs_every"], 1 if N <= 1 << 20 else 0.25)]
    nbytes = updates = 0.0
    for N, sweeps, every, out in runs:
        # the packed lattice in and out, its copy for the program, the records
        nbytes += N / 2 + N * out + (64.0 * (sweeps // every) if every else 0.0)
        updates += float(N) * sweeps
    return {"bytes": nbytes, "flops": OPS_PER_UPDATE * updates}
