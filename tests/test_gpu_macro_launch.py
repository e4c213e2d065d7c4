"""Around the kernels on macros: what their conversions do to the lattice array."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu

# uniform and other partitions, 2 and 4 bits per site, flags and owners
CASES = [(256, 3, dict(persistent=3)), (256, 5, dict(persistent=3)), (400, 3, dict(persistent=3)), (400, 3, {}),
         (400, 5, dict(neighbourhood=8)), (384, 3, dict(neighbourhood=8))]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _lattice(L, S, seed, **kw):
    D = O.circulant(S, (1,) if S == 3 else (1, 2))
    return D, E.Lattice(L, S, D, (1.0, 1.0, 2.0), seed, p_empty=0.2, **kw)


@pytest.mark.parametrize("L,S,kw", CASES)
def test_a_refused_lattice_stays_as_it_was_given(L, S, kw):
    """A host step with a value that is no state is refused, and its lattice comes
    back as it went in."""
    D, g = _lattice(L, S, 4, **kw)
    lat = O.init(L, S, 0.2, 4)
    bad = lat.copy()
    bad[L // 2, 17], bad[0, 0], bad[L - 1, L - 1] = 200, S + 1, 255
    out = np.zeros_like(bad)
    with pytest.raises(E.EscgError):
        g.step_host(bad, 0, 12, out=out)
    assert np.array_equal(out, bad)
    assert np.array_equal(g.snapshot(), bad)
    g.restore(lat, 0)
    g.run(3)
    o, _ = O.replay_run(lat, D, 1.0, 1.0, 2.0, 4, 3, neighbourhood=kw.get("neighbourhood", 4))
    assert np.array_equal(g.snapshot(), o)
    g.close()


@pytest.mark.parametrize("L,S,kw", CASES)
@pytest.mark.parametrize("stop", [False, True])
def test_a_call_of_many_launches_converts_once(L, S, kw, stop):
    """A run that stops at extinction has a launch for every log point: one
    conversion each way for the call, its lattice and its log as the oracle's."""
    D, g = _lattice(L, S, 8, log_every=1, stop_at_extinction=stop, **kw)
    rule = dict(neighbourhood=kw.get("neighbourhood", 4))
    lat = O.init(L, S, 0.2, 8)
    before = g.launches
    g.run(11)
    assert g.launches - before == (13 if stop else 3)
    o, _ = O.replay_run(lat, D, 1.0, 1.0, 2.0, 8, 11, **rule)
    assert np.array_equal(g.snapshot(), o)
    _, log = g.counts_log()
    _, olog, _ = O.run_observed(lat, D, 1.0, 1.0, 2.0, 8, 11, log_every=1, **rule)
    assert np.array_equal(log, olog)
    g.close()


@pytest.mark.parametrize("L,kw", [(128, dict(persistent=3)), (201, {}), (200, dict(neighbourhood=8)),
                                  (400, dict(persistent=3)), (384, dict(neighbourhood=8))])
def test_extinction_within_a_call(L, kw):
    """The call stops where the oracle stops, and the array holds that lattice."""
    D = O.circulant(3, (1,))   # a few sites of 2 among 1, which beats it
    rule = dict(neighbourhood=kw.get("neighbourhood", 4))
    lat = np.ones((L, L), dtype=np.uint8)
    lat[3::L // 5, 5::L // 4] = 2
    g = E.Lattice(L, 3, D, (1.0, 1.0, 1.0), 3, log_every=1, stop_at_extinction=True, **kw)
    g.restore(lat, 0)
    o, log, mend = O.run_observed(lat, D, 1.0, 1.0, 1.0, 3, 400, log_every=1, stop_at_extinction=True, **rule)
    assert 1 < mend < 400
    g.run(400)
    assert g.mcs == mend
    assert np.array_equal(g.snapshot(), o)
    g.run(5)   # stopped: nothing moves
    assert g.mcs == mend and np.array_equal(g.snapshot(), o)
    g.close()
