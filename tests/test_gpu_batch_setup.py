"""Set-up of a batch's replicas, which go to the device in groups of 4096."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def test_more_replicas_than_one_group():
    """Every replica has its own descriptor, table, seed and first lattice,
    also where the next group's are written while the copies of the one before
    may still be under way."""
    specs = []
    for i in range(2 * 4096 + 5):
        S = 2 + i % 5
        specs.append(dict(L=8 + i % 7, S=S, digraph=O.circulant(S, (1,)), rates=(1.0, 1.0, 0.5 + i % 3), seed=9 * i + 1,
                          p_empty=0.25, max_mcs=2 + i % 2, stop_at_extinction=False))
    b = E.Batch(specs, log_every=1)
    mcs, _, counts = b.status()
    assert not mcs.any()
    for i, sp in enumerate(specs):
        assert np.array_equal(counts[i, :sp["S"] + 1], O.counts(O.init(sp["L"], sp["S"], 0.25, sp["seed"]), sp["S"])), i
    b.run()
    mcs, _, counts = b.status()
    for i, sp in enumerate(specs):
        o, _ = O.replay_run(O.init(sp["L"], sp["S"], 0.25, sp["seed"]), sp["digraph"], *sp["rates"], sp["seed"],
                            sp["max_mcs"])
        assert mcs[i] == sp["max_mcs"]
        assert np.array_equal(counts[i, :sp["S"] + 1], O.counts(o, sp["S"])), i
        assert np.array_equal(b.snapshot(i), o), i
    b.close()
