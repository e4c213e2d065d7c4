"""Sub-blocks stepped in registers on the macro layout (escg_patch.cuh),
against the replay oracle, at the partitions and rules where the layout has
an edge: every mix of 2- and 3-site segments, one and several thread groups,
2 and 4 bits per site, no exchange and nothing but exchange."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _check(kernel, L, H, S, K, X, seed, n=(1, 3), prob=None, **kw):
    D = O.circulant(S, K)
    g = E.Lattice(L, S, D, (1.0, 1.0, X), seed, p_empty=0.2, log_every=2, H=H, dominance_prob=prob, **kw)
    assert g.update_kernel == kernel
    rule = dict(neighbourhood=kw.get("neighbourhood", 4), reflect=kw.get("reflecting_boundary", False))
    lat, m = O.init(L, S, 0.2, seed, H=H), 0
    first = lat
    for step in n:
        g.run(step)
        lat, _ = O.replay_run(lat, D, 1.0, 1.0, X, seed, step, mcs_begin=m, prob=prob, **rule)
        m += step
        got = g.snapshot()
        assert np.array_equal(got, lat), f"after {m} MCS: {int((got != lat).sum())} sites differ"
    _, log = g.counts_log()
    _, olog, _ = O.run_observed(first, D, 1.0, 1.0, X, seed, m, log_every=2, prob=prob, **rule)
    assert np.array_equal(log, olog)
    g.close()


@pytest.mark.parametrize("L,H", [(8, 8), (9, 12), (10, 11), (16, 20), (31, 29), (50, 64), (70, 71), (127, 66),
                                 (159, 190), (191, 191)])
@pytest.mark.parametrize("S,K,X", [(2, (1,), 0.0), (3, (1,), 1e6), (15, (1, 2, 3), 1.5)])
def test_resident_partitions(L, H, S, K, X):
    _check("resident_kernel", L, H, S, K, X, 31 * L + H + S, persistent=4)


@pytest.mark.parametrize("S,K", [(3, (1,)), (8, (1, 2, 3))])
def test_resident_edge_probabilities(S, K):
    D = O.circulant(S, K).astype(bool)
    prob = np.zeros((S, S))
    prob[D] = np.linspace(0.0, 1.0, int(D.sum()))
    _check("resident_kernel", 67, 90, S, K, 0.5, 17, prob=prob, persistent=4)


@pytest.mark.parametrize("L,H", [(128, 128), (256, 128), (384, 640)])
@pytest.mark.parametrize("bits,S,K,X", [(8, 3, (1,), 1e6), (8, 15, (1, 2, 3), 0.0), (4, 5, (1, 2), 3.0),
                                        (2, 3, (1,), 40.0)])
def test_flag_kernel_macros(L, H, bits, S, K, X):
    """Both CTA sizes (more than 4 CTAs per SM: 128 threads)."""
    for ctas in (0, 8):
        _check("persistent_kernel", L, H, S, K, X, L + 3 * H + S, persistent=3, bits_per_site=bits, ctas_per_sm=ctas)


@pytest.mark.parametrize("nbh,reflect", [(8, False), (4, True), (8, True)], ids=["moore", "reflect", "both"])
@pytest.mark.parametrize("bits,S,K", [(8, 3, (1,)), (8, 5, (1, 2)), (2, 3, (1,)), (4, 5, (1, 2))])
def test_flag_kernel_macros_variants(nbh, reflect, bits, S, K):
    _check("persistent_kernel", 256, 384, S, K, 5.0, 77 + nbh + bits, persistent=3, neighbourhood=nbh,
           reflecting_boundary=reflect, bits_per_site=bits)


def test_flag_kernel_macros_edge_probabilities():
    prob = np.where(O.circulant(3, (1,)) > 0, 0.4, 0.0)
    _check("persistent_kernel", 256, 256, 3, (1,), 1.0, 5, prob=prob, persistent=3)
