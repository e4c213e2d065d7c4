"""The calls whose time counts: one pass of each kind of work that users of
the framework run, through its public entry points, over the range of sizes,
rules and storage formats that they are run at.

Every output is a whole number (lattice values, species counts, MCS numbers)
that depends only on the parameters and the seed, so there is no floating
reference: an output is right when it is equal.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_16639_gb300 import Batch, Lattice, Server, circulant, exchange_from_mobility, lattice_bytes
from paper_2508_16639_gb300.serve import request_spec
from paper_2508_16639_gb300.workloads import SEED0, ensemble, park_ensemble, request_stream

# Integer operations of one elementary step that no implementation of the
# schedule avoids: a quarter of a Philox4x32-10 call (10), the split of its
# word, the two sites, the action and the new pair.
OPS_PER_STEP = 24


def _lattice(name, L, n_mcs, S=3, H=None, mobility=1e-4, p_empty=None, reproduce=1.0, bits=8, nbh=4,
             reflect=False, read=True):
    return dict(name=name, kind="lattice", L=L, H=L if H is None else H, S=S, n_mcs=n_mcs, mobility=mobility,
                p_empty=1.0 / (S + 1) if p_empty is None else p_empty, reproduce=reproduce, bits=bits, nbh=nbh,
                reflect=reflect, read=read)


def listed():
    return [
        # The smallest lattice anyone runs: rock-paper-scissors with
        # competition alone (no movement, no reproduction), 100 MCS and a look
        # at the densities.  Latency and the chain of phases are all of it.
        _lattice("competition_64", 64, 100, mobility=0.0, p_empty=0.0, reproduce=0.0),
        # Rock-paper-scissors-lizard-Spock at the side the paper's mobility
        # experiments use (not a multiple of 128: ragged blocks), densities
        # every 10 MCS.
        _lattice("rpsls_800", 800, 100, S=5, p_empty=0.2),
        # A mid-size square whose partition is uniform.
        _lattice("rps_1024", 1024, 100),
        # The paper's largest side, 10 MCS as one stretch of a long run;
        # nothing is read back.
        _lattice("rps_3200", 3200, 10, read=False),
        # The same model on the largest lattices (164 MB, past the L2).
        _lattice("rps_12800", 12800, 10, read=False),
        # The same at 2 bits per site, as one stores it where memory counts.
        _lattice("packed_12800", 12800, 10, bits=2, read=False),
        # The Moore neighbourhood at the paper's largest side.
        _lattice("moore_3200", 3200, 10, nbh=8, read=False),
        # A rectangle of odd sides with a reflecting boundary: ragged blocks
        # on both axes and steps mirrored at the edges.
        _lattice("reflect_3001x1499", 3001, 50, H=1499, S=5, reflect=True),
        # A host program that keeps its lattice in its own (pinned) memory:
        # lattice in, 10 MCS, lattice and counts out.
        dict(name="host_3200", kind="host", L=3200, S=3, n_mcs=10, mobility=1e-4),
        # An ensemble of independent runs over sides 64 to 400, S 3 and 5 and
        # two decades of mobility: created, run to budget or extinction and
        # read, as one call of a sweep.
        dict(name="ensemble_256", kind="ensemble", n=256, max_mcs=1000),
        # The probabilistic-dominance experiment (8 species, no movement) at
        # nine points of its parameter plane.
        dict(name="park_144", kind="park", per_point=16, L=100, max_mcs=1000),
        # A burst of requests of mixed sides and budgets on a running server.
        dict(name="serve_64", kind="serve", n=64, L_max=800, max_budget=1000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["lattice"] * 7 + ["host", "ensemble", "park", "serve"])
    if kind == "ensemble":
        return dict(kind=kind, n=log_int(16, 256), max_mcs=log_int(100, 1000))
    if kind == "park":
        return dict(kind=kind, per_point=rng.randint(1, 16), L=rng.randint(50, 100), max_mcs=log_int(100, 1000))
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(8, 64), L_max=log_int(100, 800), max_budget=log_int(200, 1000))
    if kind == "host":
        return dict(kind=kind, L=log_int(64, 3200), S=rng.choice([3, 5]), n_mcs=rng.randint(5, 20),
                    mobility=10 ** rng.uniform(-5, -3))
    L = log_int(64, 12800)
    if rng.random() < 0.35:
        L = min(12800, max(128, (L + 64) // 128 * 128))   # sides in multiples of 128 are as common as others
    H = L
    if rng.random() < 0.3:
        H = min(12800, max(64, int(L * 2 ** rng.uniform(-2, 2))))
    S = rng.choice([3, 3, 5, 8])
    bits = rng.choice([8, 8, 8, 4] + ([2] if S == 3 else []))
    n_mcs = max(2, min(log_int(10, 200), 12800 * 12800 * 10 // (L * H)))
    c = _lattice("", L, n_mcs, S=S, H=H, mobility=10 ** rng.uniform(-5, -3), bits=bits,
                 nbh=rng.choice([4, 4, 4, 8]), reflect=rng.random() < 0.2, read=rng.random() < 0.5)
    del c["name"]
    return c


def _offsets(S):
    return {3: (1,), 5: (1, 2), 8: (1, 2, 3)}[S]


def _open(case, seed, **kw):
    L, H, S = case["L"], case.get("H", case["L"]), case["S"]
    bits = case.get("bits", 8)
    buf = torch.zeros(lattice_bytes(L, H, bits), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()   # the lattice works on a stream of its own
    return Lattice(L, S, circulant(S, _offsets(S)),
                   (1.0, case.get("reproduce", 1.0), exchange_from_mobility(case["mobility"], L * H)),
                   SEED0 + seed, p_empty=case.get("p_empty", 1.0 / (S + 1)), log_every=10, H=H,
                   bits_per_site=bits, neighbourhood=case.get("nbh", 4),
                   reflecting_boundary=case.get("reflect", False), device_buffer=buf, **kw)


def _specs(case, seed):
    # The mix of sides, rules and budgets belongs to the case; the seed gives
    # every run its own random numbers.
    if case["kind"] == "ensemble":
        reps = [request_spec(r) for r in ensemble(case["n"], seed=1, max_mcs=case["max_mcs"])]
    elif case["kind"] == "park":
        reps = [{k: v for k, v in r.items() if k != "point"} for r in park_ensemble(case["per_point"], L=case["L"])]
        for r in reps:
            r["max_mcs"] = min(r["max_mcs"], case["max_mcs"])
    else:
        reps = [request_spec(r) for r in request_stream(case["n"], seed=2, L_range=(50, case["L_max"]),
                                                        budget_range=(100, case["max_budget"]))]
    for i, r in enumerate(reps):
        r["seed"] = SEED0 + (seed << 20) + i
    return reps


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        return dict(case=case, lat=_open(case, seed))
    if kind == "host":
        L = case["L"]
        start = np.random.default_rng(seed).integers(0, case["S"] + 1, size=(L, L), dtype=np.uint8)
        src = torch.from_numpy(start).pin_memory()
        dst = torch.empty_like(src).pin_memory()
        return dict(case=case, lat=_open(case, seed), src=src, dst=dst)
    if kind == "serve":
        return dict(case=case, specs=_specs(case, seed), server=Server(keep_lattice=True))
    return dict(case=case, specs=_specs(case, seed))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = state["lat"]
        lat.run(case["n_mcs"])
        if not case["read"]:
            return [lat.as_tensor()]
        counts, mcs = lat.counts()
        return [lat.as_tensor(), counts.astype(np.int64), mcs]
    if kind == "host":
        out, counts = state["lat"].step_host(state["src"].numpy(), 0, case["n_mcs"], out=state["dst"].numpy())
        return [out, counts.astype(np.int64)]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(sp) for sp in state["specs"]]
        left = len(ids)
        while left:
            srv.step()
            left -= len(srv.poll())
        got = [srv.result(i, lattice=True) for i in ids]
        return [np.array([g[0] for g in got]), np.array([g[1] for g in got]),
                np.stack([g[2] for g in got]).astype(np.int64), np.concatenate([g[3].ravel() for g in got])]
    batch = Batch(state["specs"])
    batch.run()
    mcs, extinct, counts = batch.status()
    lattices = np.concatenate([batch.snapshot(i).ravel() for i in range(batch.n)])
    batch.close()
    return [mcs, extinct, counts.astype(np.int64), lattices]


def work(case):
    if case["kind"] in ("lattice", "host"):
        sites = case["L"] * case.get("H", case["L"])
        steps, stored = sites * case["n_mcs"], sites * case.get("bits", 8) // 8
    else:
        specs = _specs(case, 0)
        steps = sum(r["L"] ** 2 * r["max_mcs"] for r in specs)
        stored = sum(r["L"] ** 2 for r in specs)
    return {"bytes": 2 * stored, "flops": OPS_PER_STEP * steps}
