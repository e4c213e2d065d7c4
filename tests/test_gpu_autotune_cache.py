"""Handles that take the autotuner's cached choice."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _leave_epochs_behind(L, n=12):
    """Device memory given back full of words whose high half is 1, the epoch that
    a first MCS waits for: lattices of the values 0 and 1."""
    lat = np.zeros((L, L), dtype=np.uint8)
    lat[:, 4::8] = 1
    lat[:, 0::8] = 1
    hs = []
    for _ in range(n):
        hs.append(E.Lattice(L, 3, E.circulant(3, [1]), (1.0, 1.0, 1.0), 1))
        hs[-1].restore(lat, 0)
    for h in hs:
        h.close()


@pytest.mark.parametrize("L,S,kw", [(256, 3, dict(neighbourhood=8)), (256, 5, dict(reflecting_boundary=True)),
                                    (256, 3, {}), (512, 3, {}), (200, 5, {})])
def test_cached_choice_starts_on_empty_records(L, S, kw):
    """A cached mode may need boundary records that the default one does not:
    they hold no epoch, whatever the memory held before."""
    D = O.circulant(S, (1,) if S == 3 else (1, 2))
    rule = dict(neighbourhood=kw.get("neighbourhood", 4), reflect=kw.get("reflecting_boundary", False))
    E.Lattice(L, S, D, (1.0, 1.0, 2.0), 3, p_empty=0.2, autotune=True, **kw).close()
    for seed in (5, 6, 7):
        _leave_epochs_behind(64 if seed == 5 else L)
        g = E.Lattice(L, S, D, (1.0, 1.0, 2.0), seed, p_empty=0.2, autotune=True, **kw)
        assert g.autotune_result[3] == 0
        g.run(3)
        o, _ = O.replay_run(O.init(L, S, 0.2, seed), D, 1.0, 1.0, 2.0, seed, 3, **rule)
        assert np.array_equal(g.snapshot(), o)
        g.close()


def test_uncertain_edges_are_tuned_for_themselves():
    """Certain and uncertain edges run different kernels in the same mode, so
    neither takes the other's timing."""
    D = O.circulant(3, (1,))
    for prob in (None, 0.5 * D):
        for again in (False, True):
            g = E.Lattice(400, 3, D, (1.0, 1.0, 2.0), 9, p_empty=0.2, autotune=True, dominance_prob=prob)
            assert (g.autotune_result[3] == 0) == again
            g.close()
