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
