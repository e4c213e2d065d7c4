"""Mirrored steps of sub-blocks of every shape at every edge of a reflecting
lattice, on the kernels on macros, against the replay oracle."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


# sides of 3-site segments at both ends, at one, at none, and mixed
@pytest.mark.parametrize("L,H,kw", [(11, 12, {}), (9, 190, {}), (50, 67, {}), (191, 80, {}), (130, 150, {}),
                                    (270, 300, dict(persistent=4)), (600, 590, dict(bits_per_site=4)),
                                    (128, 256, dict(persistent=3))])
@pytest.mark.parametrize("nbh", [4, 8])
@pytest.mark.parametrize("S,prob", [(3, None), (5, None), (3, 0.5)])
def test_mirrored_steps(L, H, kw, nbh, S, prob):
    D = O.circulant(S, (1,) if S == 3 else (1, 2))
    p = None if prob is None else prob * D
    seed = 100 * L + H + nbh
    g = E.Lattice(L, S, D, (1.0, 1.0, 1.5), seed, p_empty=0.2, H=H, neighbourhood=nbh, reflecting_boundary=True,
                  dominance_prob=p, **kw)
    lat = O.init(L, S, 0.2, seed, H=H)
    g.run(7)
    o, _ = O.replay_run(lat, D, 1.0, 1.0, 1.5, seed, 7, neighbourhood=nbh, reflect=True, prob=p)
    got = g.snapshot()
    assert np.array_equal(got, o), int((got != o).sum())
    g.close()
