"""Timed cases of the library: the calls that users of the lattice Monte Carlo make, at the sizes they make them.

A case is one kind of use with its sizes and options.  ``prepare`` makes what a program holds before the call
(handles, batches, servers, saved lattices), ``run`` is one pass through the public entry points:

* ``run``       one lattice: sweeps, then what a program reads after them (energy, counters, optionally the
                cluster histogram and the energy trace, and the lattice itself);
* ``batch``     replicas advanced together, each one's histogram on the device, then energies and lattices;
* ``serve``     a stream of jobs submitted at once to the job server, every result collected;
* ``clusters``  the cluster-size histograms of both species of a lattice that has demixed for a while;
* ``image``     a saved lattice loaded and analysed: energy, fraction of first neighbours, snapshot, image fraction;
* ``place``     a new lattice placed at random and read back.

A pass of ``run`` and ``batch`` continues the chain where the last one left it, as a simulation does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1309_4349_gb300 as klmc

GEOMETRY = {"tri6": klmc.TRI6, "sq4": klmc.SQ4}
PACKING = {"bit": klmc.PACK_BIT, "byte": klmc.PACK_BYTE}


def listed():
    return [
        # The smallest call: one step of the 64x64 lattice (1 byte per site) watched step by step.
        dict(name="step_64", kind="run", Lx=64, Ly=64, geometry="tri6", packing="byte", n_A=2048, omega=0.6, mcs=1,
             trace_every=0, hist=False),
        # The 64x64 run at its sampling cadence: 100 steps between cluster histograms.
        dict(name="run_64", kind="run", Lx=64, Ly=64, geometry="tri6", packing="byte", n_A=2048, omega=0.6, mcs=100,
             trace_every=0, hist=True),
        # One run of the paper's 400x400 lattice between two histograms, on its own.
        dict(name="run_400", kind="run", Lx=400, Ly=400, geometry="tri6", packing="bit", n_A=48000, omega=0.6,
             mcs=500, trace_every=0, hist=True),
        # The same for its five interaction energies together: the benchmark's headline workload.
        dict(name="batch_5x400", kind="batch", what="omegas", n=5, Lx=400, Ly=400, mcs=500, hist=True),
        # A ragged square lattice of 1.5 million sites, on the path that uses every SM.
        dict(name="run_sq4_1447x1021", kind="run", Lx=1447, Ly=1021, geometry="sq4", packing="bit", n_A=600000,
             omega=1.0, mcs=200, trace_every=0, hist=False),
        # The largest lattice near demixing, its energy traced every 10 steps.
        dict(name="run_8192", kind="run", Lx=8192, Ly=8192, geometry="tri6", packing="bit", n_A=8192 * 8192 // 2,
             omega=0.85, mcs=1000, trace_every=10, hist=False),
        # 256 replicas of uneven sizes, compositions and energies.
        dict(name="batch_256", kind="batch", what="replicas", n=256, L_min=100, L_max=1024, pick=20260, mcs=1000,
             hist=False),
        # The paper's helical lattice with its seven-colour schedule, five interaction energies.
        dict(name="batch_helical_402x399", kind="batch", what="helical", n=5, Lx=402, Ly=399, mcs=500, hist=True),
        # A job mix arriving at the server: small and large lattices, short and long runs.
        dict(name="serve_64", kind="serve", n=64, L_min=64, L_max=1024, mcs_min=100, mcs_max=2000, pick=77),
        # Cluster statistics of the largest lattice.
        dict(name="clusters_8192", kind="clusters", Lx=8192, Ly=8192, geometry="tri6", packing="bit", omega=0.85,
             fraction=0.5, burn=20),
        # Image analysis of a saved lattice of the largest size.
        dict(name="image_8192", kind="image", Lx=8192, Ly=8192, geometry="tri6", packing="bit", W=6143, H=3547, S=4),
        # A new run's random placement.
        dict(name="place_1000", kind="place", Lx=1000, Ly=1000, geometry="tri6", packing="bit", fraction=0.3),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "batch", "serve", "clusters", "image", "place"])
    geometry = rng.choice(["tri6", "tri6", "sq4"])
    packing = rng.choice(["bit", "bit", "bit", "byte"])
    if kind == "run":
        Lx, Ly = _log_uniform(rng, 16, 5000), _log_uniform(rng, 16, 5000)
        mcs = min(_log_uniform(rng, 1, 1000), max(1, int(1.5e10 / (Lx * Ly))))
        trace = rng.choice([0, 0, max(1, mcs // 10)])
        return dict(kind=kind, Lx=Lx, Ly=Ly, geometry=geometry, packing=packing,
                    n_A=int(rng.uniform(0.1, 0.5) * Lx * Ly), omega=round(rng.uniform(0.1, 1.2), 3), mcs=mcs,
                    trace_every=trace, hist=rng.random() < 0.5)
    if kind == "batch":
        what = rng.choice(["omegas", "replicas", "replicas", "helical"])
        mcs = _log_uniform(rng, 50, 500)
        if what == "omegas":
            return dict(kind=kind, what=what, n=rng.randint(2, 9), Lx=_log_uniform(rng, 64, 600),
                        Ly=_log_uniform(rng, 64, 600), mcs=mcs, hist=rng.random() < 0.5)
        if what == "replicas":
            return dict(kind=kind, what=what, n=_log_uniform(rng, 8, 200), L_min=rng.randint(48, 128),
                        L_max=rng.randint(300, 1024), pick=rng.randrange(1 << 20), mcs=mcs, hist=rng.random() < 0.3)
        # 7 | Lx*Ly and Lx mod 7 in {3, 5}: the sizes that seven-site domains tile
        return dict(kind=kind, what=what, n=rng.randint(1, 8), Lx=7 * _log_uniform(rng, 10, 100) + rng.choice([3, 5]),
                    Ly=7 * _log_uniform(rng, 10, 100), mcs=mcs, hist=rng.random() < 0.5)
    if kind == "serve":
        return dict(kind=kind, n=_log_uniform(rng, 4, 64), L_min=rng.randint(32, 96), L_max=rng.randint(200, 1024),
                    mcs_min=50, mcs_max=rng.randint(500, 2000), pick=rng.randrange(1 << 20))
    Lx, Ly = _log_uniform(rng, 64, 8192), _log_uniform(rng, 64, 8192)
    if kind == "clusters":
        return dict(kind=kind, Lx=Lx, Ly=Ly, geometry=geometry, packing=packing, omega=round(rng.uniform(0.1, 1.2), 3),
                    fraction=round(rng.uniform(0.1, 0.5), 3), burn=rng.randint(1, 50))
    if kind == "image":
        S = rng.randint(1, 4)
        U = 2 * Lx + Ly - 1
        scale = rng.randint(1, 4)
        return dict(kind=kind, Lx=Lx, Ly=Ly, geometry=geometry, packing=packing, W=max(16, U // scale // S),
                    H=max(16, int(1.732 * Ly) // scale // S), S=S)
    Lx, Ly = _log_uniform(rng, 16, 2048), _log_uniform(rng, 16, 2048)
    return dict(kind="place", Lx=Lx, Ly=Ly, geometry=geometry, packing=packing, fraction=round(rng.uniform(0.1, 0.5), 3))


def _table(histogram, N):
    """A sparse histogram as a row of a table that holds any histogram of N sites: (size, count), zeros behind."""
    sizes, counts = histogram
    row = np.zeros((2, int(math.sqrt(2.0 * N)) + 2), dtype=np.int64)
    row[0, :sizes.size], row[1, :counts.size] = sizes, counts
    return row


def _replicas(case, seed):
    """Parameters of a batch's replicas: sizes and energies from the case, the random streams from the seed."""
    n = case["n"]
    if case["what"] == "replicas":
        g = np.random.default_rng(case["pick"])
        out = []
        for r in range(n):
            L = int(round(float(np.exp(g.uniform(np.log(case["L_min"]), np.log(case["L_max"]))))))
            out.append(dict(Lx=L, Ly=L, fraction_A=float(g.uniform(0.1, 0.5)), omega_over_kT=float(g.uniform(0.1, 1.2)),
                            seed=seed * 1000 + r))
        return out
    omegas = np.linspace(0.2, 1.0, n)
    extra = dict(boundary=klmc.HELICAL) if case["what"] == "helical" else {}
    return [dict(Lx=case["Lx"], Ly=case["Ly"], fraction_A=0.3, omega_over_kT=float(omegas[r]), seed=seed * 1000 + r,
                 **extra) for r in range(n)]


def _jobs(case, seed):
    g = np.random.default_rng(case["pick"])
    out = []
    for j in range(case["n"]):
        L = int(round(float(np.exp(g.uniform(np.log(case["L_min"]), np.log(case["L_max"]))))))
        mcs = int(round(float(np.exp(g.uniform(np.log(case["mcs_min"]), np.log(case["mcs_max"]))))))
        out.append(dict(Lx=L, Ly=L, fraction_A=float(g.uniform(0.1, 0.5)), omega_over_kT=float(g.uniform(0.1, 1.2)),
                        n_mcs=mcs, hist_every=mcs, seed=seed * 1000 + j))
    return out


def _saved_lattice(Lx, Ly, seed):
    """A demixed configuration as a saved file holds it, one byte per site: domains of about 12 sites, 4% noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    coarse = torch.rand((Ly + 11) // 12, (Lx + 11) // 12, device="cuda", generator=g) < 0.45
    fine = coarse.repeat_interleave(12, 0)[:Ly].repeat_interleave(12, 1)[:, :Lx]
    noise = torch.rand(Ly, Lx, device="cuda", generator=g) < 0.04
    return (fine ^ noise).to(torch.uint8).reshape(-1).contiguous()


def _lattice(case, seed, **kw):
    return klmc.Lattice(case["Lx"], case["Ly"], geometry=GEOMETRY[case["geometry"]], packing=PACKING[case["packing"]],
                        seed=seed, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        return dict(case=case, lat=_lattice(case, seed, n_A=case["n_A"], omega_over_kT=case["omega"]))
    if kind == "batch":
        reps = _replicas(case, seed)
        state = dict(case=case, batch=klmc.Batch(reps))
        if case["hist"]:
            cap = int(math.sqrt(2.0 * max(r["Lx"] * r["Ly"] for r in reps))) + 2
            state["sizes"] = torch.zeros(len(reps), cap, dtype=torch.int64, device="cuda")
            state["counts"] = torch.zeros(len(reps), cap, dtype=torch.int64, device="cuda")
            state["distinct"] = torch.zeros(len(reps), dtype=torch.int64, device="cuda")
        return state
    if kind == "serve":
        return dict(case=case, server=klmc.Server(4 << 30), jobs=_jobs(case, seed))
    if kind == "clusters":
        lat = _lattice(case, seed, fraction_A=case["fraction"], omega_over_kT=case["omega"])
        lat.sweep(case["burn"])
        return dict(case=case, lat=lat)
    if kind == "image":
        return dict(case=case, lat=_lattice(case, seed, fraction_A=0.5, omega_over_kT=0.85),
                    saved=_saved_lattice(case["Lx"], case["Ly"], seed))
    return dict(case=case, seed=seed)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        lat, out = state["lat"], {}
        if case["trace_every"]:
            out["trace"] = lat.sweep_traced(case["mcs"], case["trace_every"])
        else:
            lat.sweep(case["mcs"])
        if case["hist"]:
            out["clusters"] = _table(lat.cluster_histogram(1), lat.N)
        out["n_unlike"] = lat.energy()[0]
        out["counters"] = lat.counters()
        out["lattice"] = lat.get_lattice()
        return out
    if kind == "batch":
        batch, out = state["batch"], {}
        batch.sweep(case["mcs"])
        if case["hist"]:
            batch.cluster_histogram_device(1, state["sizes"], state["counts"], state["distinct"])
            out.update(sizes=state["sizes"], counts=state["counts"], distinct=state["distinct"])
        out["n_unlike"] = np.array([r.energy()[0] for r in batch.replicas])
        out["accepts"] = np.array([r.counters()["accepts"] for r in batch.replicas])
        out["lattices"] = np.concatenate([r.get_lattice() for r in batch.replicas])
        return out
    if kind == "serve":
        server, jobs = state["server"], state["jobs"]
        ids = [server.submit(keep_lattice=True, **j) for j in jobs]
        server.drain(120.0)
        results = [server.poll(i) for i in ids]
        hists = [server.histogram(i) for i in ids]
        out = {k: np.array([r[k] for r in results])
               for k in ("status", "n_mcs", "n_unlike", "attempts", "unlike", "draws", "accepts")}
        out["clusters"] = np.concatenate([_table(h, j["Lx"] * j["Ly"]) for h, j in zip(hists, jobs)], axis=1)
        out["lattices"] = np.concatenate([server.lattice(i, j["Lx"] * j["Ly"]) for i, j in zip(ids, jobs)])
        for i in ids:
            server.release(i)
        return out
    if kind == "clusters":
        return [_table(state["lat"].cluster_histogram(species), state["lat"].N) for species in (1, 0)]
    if kind == "image":
        lat = state["lat"]
        lat.set_lattice_device(state["saved"], 0)
        image, mask = lat.snapshot(case["W"], case["H"], case["S"])
        similar, pixels = lat.image_ffn(image, mask)
        ffn, all_bonds = lat.ffn(0)
        return dict(n_unlike=lat.energy()[0], n_A=lat.n_A, ffn=ffn, all_bonds=all_bonds, image=image, mask=mask,
                    similar=similar, pixels=pixels)
    lat = _lattice(case, state["seed"], fraction_A=case["fraction"], omega_over_kT=0.6)
    out = dict(n_unlike=lat.energy()[0], n_A=lat.n_A, lattice=lat.get_lattice())
    lat.close()
    return out


def exact(case, seed):
    """The computed (floating) outputs in 64 bits; every other output is a whole number of the exact integer chain."""
    if case["kind"] != "image":
        return None
    t = _saved_lattice(case["Lx"], case["Ly"], seed).reshape(case["Ly"], case["Lx"]).to(torch.int8)
    bonds = [(0, 1), (1, 0)] + ([(-1, 1)] if case["geometry"] == "tri6" else [])
    unlike = sum(int((t != t.roll((-dy, -dx), (0, 1))).sum()) for dy, dx in bonds)
    return dict(n_unlike=unlike, n_A=int(t.to(torch.int64).sum()), ffn=None,
                all_bonds=1.0 - unlike / (len(bonds) * case["Lx"] * case["Ly"]), image=None, mask=None, similar=None,
                pixels=None)


def _sites(case, seed=0):
    if case["kind"] == "batch":
        return sum(r["Lx"] * r["Ly"] for r in _replicas(case, seed))
    if case["kind"] == "serve":
        return sum(j["Lx"] * j["Ly"] for j in _jobs(case, seed))
    return case["Lx"] * case["Ly"]


def work(case):
    """Bytes: the store read and written once, the results written once.  Operations: an attempted exchange takes
    about 12 (comparing the neighbours of 32 pairs bit by bit, a Philox draw for about one pair in five), a placed
    site one Philox evaluation (about 60), an analysed site its three bonds or its image samples."""
    N, kind = _sites(case), case["kind"]
    if kind in ("run", "batch"):
        store = N if case.get("packing") == "byte" else N / 8
        return dict(bytes=2 * store + N, flops=12.0 * N * case["mcs"])
    if kind == "serve":
        return dict(bytes=N / 4 + N, flops=12.0 * sum(j["Lx"] * j["Ly"] * j["n_mcs"] for j in _jobs(case, 0)))
    store = N if case["packing"] == "byte" else N / 8
    if kind == "clusters":  # each species' sites once each, 4 bytes of label per site
        return dict(bytes=2 * store + 4 * N, flops=8.0 * N)
    if kind == "image":
        pixels = case["W"] * case["H"]
        return dict(bytes=N + 4 * store + 4 * pixels, flops=30.0 * N + 4.0 * pixels * case["S"] ** 2 + 30.0 * pixels)
    return dict(bytes=store + N, flops=60.0 * N)
