"""The flag kernel on macros of partitions that are not 64 x 64 blocks, against
the replay oracle: mixes of block widths and segment counts, rows of slots that
do and do not end on a 16-byte piece, packed storage, Moore and reflecting."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


@pytest.mark.parametrize("L,H", [(192, 192), (200, 263), (253, 246), (262, 195), (333, 267), (450, 321), (513, 200)])
@pytest.mark.parametrize("S,K,X,bits,nbh,reflect", [
    (3, (1,), 3.0, 8, 4, False), (3, (1,), 1e6, 8, 8, False), (2, (1,), 0.0, 2, 4, False), (3, (1,), 40.0, 2, 8, True),
    (5, (1, 2), 3.0, 4, 4, False), (15, (1, 2, 3), 20.0, 4, 8, True)])
def test_parity(L, H, S, K, X, bits, nbh, reflect):
    D = O.circulant(S, K)
    seed = 13 * L + H + S
    rule = dict(neighbourhood=nbh, reflect=reflect)
    g = E.Lattice(L, S, D, (1.0, 1.0, X), seed, p_empty=0.2, log_every=2, H=H, persistent=3, bits_per_site=bits,
                  neighbourhood=nbh, reflecting_boundary=reflect)
    assert g.update_kernel == "persistent_kernel"
    first = lat = O.init(L, S, 0.2, seed, H=H)
    m = 0
    for step in (1, 3):
        g.run(step)
        lat, _ = O.replay_run(lat, D, 1.0, 1.0, X, seed, step, mcs_begin=m, **rule)
        m += step
        got = g.snapshot()
        assert np.array_equal(got, lat), f"after {m} MCS: {int((got != lat).sum())} sites differ"
    _, log = g.counts_log()
    _, olog, _ = O.run_observed(first, D, 1.0, 1.0, X, seed, m, log_every=2, **rule)
    assert np.array_equal(log, olog)
    g.close()


def test_larger_than_half_the_l2():
    """4 bits per site in macros on a byte lattice: L = 8200 (67 MB)."""
    L, S, X, seed = 8200, 5, 1e4, 8200
    D = O.circulant(S, (1, 2))
    g = E.Lattice(L, S, D, (1.0, 1.0, X), seed, p_empty=0.2)
    lat = O.init(L, S, 0.2, seed)
    g.run(1)
    lat, _ = O.replay_run(lat, D, 1.0, 1.0, X, seed, 1)
    assert np.array_equal(g.snapshot(), lat)
    counts, mcs = g.counts()
    assert mcs == 1 and np.array_equal(counts, O.counts(lat, S))
    g.close()
