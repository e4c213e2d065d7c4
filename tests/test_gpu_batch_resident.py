"""Replicas of 2 x 2 blocks in the batch engine: resident on macros while they
are alone, in the chunk kernel beside larger ones, and from one to the other
between steps -- always the replay oracle's lattice, counts and MCS."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _spec(L, S, seed, X, max_mcs=60, prob=None):
    K = {2: (1,), 3: (1,), 5: (1, 2), 8: (1, 2, 3), 15: (1, 2, 3)}[S]
    sp = dict(L=L, S=S, digraph=O.circulant(S, K), rates=(1.0, 1.0, X), seed=seed, p_empty=0.2, max_mcs=max_mcs,
              stop_at_extinction=False)
    if prob is not None:
        sp["dominance_prob"] = prob * O.circulant(S, K)
    return sp


def _check(sp, mcs, counts, lat):
    o, _ = O.replay_run(O.init(sp["L"], sp["S"], sp["p_empty"], sp["seed"]), sp["digraph"], *sp["rates"], sp["seed"],
                        sp["max_mcs"], prob=sp.get("dominance_prob"))
    assert mcs == sp["max_mcs"]
    assert np.array_equal(lat, o), sp["L"]
    if sp["max_mcs"] % 10 == 0:
        assert np.array_equal(counts[:sp["S"] + 1], O.counts(o, sp["S"]))


@pytest.mark.parametrize("extra", [0, 170], ids=["1024 threads", "512 threads"])
@pytest.mark.parametrize("beside", [False, True], ids=["alone", "beside L=200"])
def test_small_replicas(extra, beside):
    specs = [_spec(L, S, 10 * L + S, X, m) for L, S, X, m in
             [(8, 2, 0.0, 20), (11, 3, 5.0, 13), (12, 5, 1.0, 20), (50, 3, 1e6, 20), (64, 8, 0.0, 20), (100, 15, 2.0, 25),
              (127, 3, 0.5, 20), (128, 3, 3.0, 20), (191, 5, 10.0, 20)]]
    specs.append(_spec(90, 3, 77, 0.5, 20, prob=0.4))
    specs += [_spec(8 + i % 3, 3, 1000 + i, 1.0, 10) for i in range(extra)]
    if beside:
        specs.append(_spec(200, 3, 5, 2.0, 20))
    b = E.Batch(specs)
    b.run()
    mcs, _, counts = b.status()
    for i, sp in enumerate(specs):
        _check(sp, mcs[i], counts[i], b.snapshot(i))
    b.close()


def test_served_replicas_change_kernel_between_steps():
    """Two small runs alone (resident), a larger one joins for a few steps
    (chunk kernel) and leaves (resident again)."""
    srv = E.Server(keep_lattice=True, chunks_per_step=1)
    specs = [_spec(100, 3, 1, 2.0, 120), _spec(64, 5, 2, 1.0, 115)]
    ids = [srv.submit(sp) for sp in specs]
    for _ in range(3):
        srv.step()
    specs.append(_spec(200, 3, 3, 2.0, 40))
    ids.append(srv.submit(specs[-1]))
    done = set()
    for _ in range(40):
        srv.step()
        done.update(srv.poll())
        if len(done) == len(ids):
            break
    assert done == set(ids)
    for sp, i in zip(specs, ids):
        mcs, _, counts, lat = srv.result(i, lattice=True)
        _check(sp, mcs, counts, lat)
