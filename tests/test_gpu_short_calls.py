"""Calls too short for the conversions into macros and back run on bytes: both
sides of the line, in turn on one handle, against the replay oracle."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _line(g):
    """The shortest call on macros."""
    n = 1
    while g.run_layout(n) == "bytes":
        n += 1
        assert n < 100
    assert all(g.run_layout(k) == "bytes" for k in range(1, n))
    assert all(g.run_layout(k) == "macros" for k in (n, n + 1, 100, 10**6))
    return n


# (L, H, S, options, edge probability, the line): flags on 64 x 64 blocks with 256 and
# with 128 threads, on other partitions, owners on macros beside byte owners and
# beside flags; von Neumann, Moore, reflecting; 8, 4 and 2 bits per site
CASES = [
    (256, 256, 3, dict(persistent=3), None, 2),
    (256, 128, 3, dict(persistent=3, ctas_per_sm=8), None, 1),
    (128, 256, 5, dict(persistent=3), None, 6),
    (256, 256, 5, dict(persistent=3, ctas_per_sm=8), None, 2),
    (256, 256, 3, dict(persistent=3), 0.5, 6),
    (256, 256, 3, dict(persistent=3, neighbourhood=8), None, 1),
    (256, 384, 5, dict(persistent=3, neighbourhood=8), None, 3),
    (256, 256, 5, dict(persistent=3, neighbourhood=8, ctas_per_sm=8), None, 1),
    (256, 256, 3, dict(persistent=3, reflecting_boundary=True), None, 2),
    (384, 256, 5, dict(persistent=3, reflecting_boundary=True), None, 5),
    (256, 256, 5, dict(persistent=3, reflecting_boundary=True, ctas_per_sm=8), None, 5),
    (256, 256, 3, dict(persistent=3, reflecting_boundary=True, ctas_per_sm=8), None, 1),
    (256, 256, 5, dict(persistent=3, reflecting_boundary=True, neighbourhood=8, ctas_per_sm=8), None, 3),
    (256, 256, 3, dict(persistent=3, bits_per_site=2), None, 2),
    (256, 256, 3, dict(persistent=3, bits_per_site=2, ctas_per_sm=8), None, 1),
    (256, 128, 5, dict(persistent=3, bits_per_site=4), None, 3),
    (256, 128, 5, dict(persistent=3, bits_per_site=4, ctas_per_sm=8), None, 2),
    (256, 256, 5, dict(persistent=3, bits_per_site=4, neighbourhood=8), None, 1),
    (400, 400, 3, dict(persistent=3), None, 3),
    (400, 530, 3, dict(persistent=3, neighbourhood=8), None, 3),
    (400, 400, 3, dict(persistent=3, bits_per_site=2), None, 1),
    (400, 400, 3, {}, None, 2),                                    # owners, beside the byte owners
    (600, 450, 3, {}, None, 3),
    (400, 400, 5, dict(neighbourhood=8), None, 2),                 # beside the flags
    (384, 512, 3, dict(neighbourhood=8), None, 2),
    (384, 512, 5, dict(reflecting_boundary=True), None, 1),
]


@pytest.mark.parametrize("L,H,S,kw,prob,line", CASES)
@pytest.mark.parametrize("stop", [False, True])
def test_both_sides_of_the_line(L, H, S, kw, prob, line, stop):
    D = O.circulant(S, (1,) if S == 3 else (1, 2))
    p = None if prob is None else prob * D
    X, seed = 6.0, 3 * L + H + S
    rule = dict(neighbourhood=kw.get("neighbourhood", 4), reflect=kw.get("reflecting_boundary", False), prob=p)
    g = E.Lattice(L, S, D, (1.0, 1.0, X), seed, p_empty=0.2, H=H, log_every=3, stop_at_extinction=stop,
                  dominance_prob=p, **kw)
    assert _line(g) == line
    lat, m = O.init(L, S, 0.2, seed, H=H), 0
    first = lat
    for n in (line, max(line - 1, 1), 1, line + 3, max(line - 1, 1), line, 1, 7):
        g.run(n)
        lat, _ = O.replay_run(lat, D, 1.0, 1.0, X, seed, n, mcs_begin=m, **rule)
        m += n
        got = g.snapshot()
        assert np.array_equal(got, lat), f"after {m} MCS (call of {n}): {int((got != lat).sum())} sites differ"
    ms, log = g.counts_log()
    _, olog, _ = O.run_observed(first, D, 1.0, 1.0, X, seed, m, log_every=3, **rule)
    assert np.array_equal(log, olog) and g.mcs == m
    # enqueued one after another, without a wait between them, and again from a restored lattice
    g.restore(first, 1)
    for n in (1, line, 1, line + 1):
        g.run(n)
    lat, _ = O.replay_run(first, D, 1.0, 1.0, X, seed, 2 * line + 3, mcs_begin=1, **rule)
    assert np.array_equal(g.snapshot(), lat)
    g.close()


def test_few_exchanges_move_the_line():
    """Without movement every step takes the rule table, and macros of 4 bits per
    site win later."""
    D = O.circulant(5, (1, 2))
    for X, line in ((0.0, 16), (1.5, 16), (20.0, 6)):
        g = E.Lattice(256, 5, D, (1.0, 1.0, X), 1, persistent=3)
        assert _line(g) == line, X
        g.run(17)
        o, _ = O.replay_run(O.init(256, 5, 0.0, 1), D, 1.0, 1.0, X, 1, 17)
        assert np.array_equal(g.snapshot(), o)
        g.close()


@pytest.mark.parametrize("L,H,S,kw,line", [(128, 127, 3, {}, 1), (130, 129, 3, {}, 2), (150, 151, 5, {}, 3), (191, 160, 5, {}, 4),
                                           (160, 150, 3, dict(bits_per_site=2), 3), (160, 150, 5, dict(bits_per_site=4), 4),
                                           (300, 270, 3, dict(persistent=4, reflecting_boundary=True), 3)])
def test_resident_launches(L, H, S, kw, line):
    """The same line for whole-lattice residency, launch by launch."""
    D = O.circulant(S, (1,) if S == 3 else (1, 2))
    rule = dict(reflect=kw.get("reflecting_boundary", False))
    for stop in (False, True):
        g = E.Lattice(L, S, D, (1.0, 1.0, 2.0), 5, p_empty=0.2, H=H, log_every=5, stop_at_extinction=stop, **kw)
        assert g.update_kernel == "resident_kernel" and _line(g) == line
        lat, m = O.init(L, S, 0.2, 5, H=H), 0
        first = lat
        for n in (1, line, 2, 9, 1, 13):
            g.run(n)
            lat, _ = O.replay_run(lat, D, 1.0, 1.0, 2.0, 5, n, mcs_begin=m, **rule)
            m += n
            assert np.array_equal(g.snapshot(), lat), m
        _, log = g.counts_log()
        _, olog, _ = O.run_observed(first, D, 1.0, 1.0, 2.0, 5, m, log_every=5, **rule)
        assert np.array_equal(log, olog) and g.mcs == m
        g.close()
