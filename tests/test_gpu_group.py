"""Block owners on macros (escg_group.cu) against the replay oracle: every mix
of 2- and 3-site segments, groups that are their own neighbours, one, two and
four groups of threads, 2 and 4 bits per site, packed and ragged rows."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _check(L, H, S, X, seed, n=(1, 3, 2), stop=False, **kw):
    K = {2: (1,), 3: (1,), 5: (1, 2), 15: (1, 2, 3)}[S]
    D = O.circulant(S, K)
    g = E.Lattice(L, S, D, (1.0, 1.0, X), seed, p_empty=0.2, log_every=2, H=H, stop_at_extinction=stop, **kw)
    assert g.update_kernel == "persistent_gown_kernel"
    rule = dict(neighbourhood=kw.get("neighbourhood", 4), reflect=kw.get("reflecting_boundary", False))
    lat, m = O.init(L, S, 0.2, seed, H=H), 0
    first = lat
    for step in n:
        g.run(step)
        lat, _ = O.replay_run(lat, D, 1.0, 1.0, X, seed, step, mcs_begin=m, **rule)
        m += step
        got = g.snapshot()
        assert np.array_equal(got, lat), f"after {m} MCS: {int((got != lat).sum())} sites differ"
    _, log = g.counts_log()
    _, olog, _ = O.run_observed(first, D, 1.0, 1.0, X, seed, m, log_every=2, **rule)
    assert np.array_equal(log, olog)
    other = O.init(L, S, 0.4, seed + 1, H=H)   # records of the earlier run must not be taken
    g.restore(other, 0)
    g.run(2)
    lat, _ = O.replay_run(other, D, 1.0, 1.0, X, seed, 2, **rule)
    assert np.array_equal(g.snapshot(), lat)
    g.close()


@pytest.mark.parametrize("L,H", [(16, 12), (50, 67), (100, 100), (131, 190), (200, 200), (201, 130), (267, 262), (333, 257),
                                 (800, 450)])
@pytest.mark.parametrize("S,X,bits", [(2, 0.0, 8), (3, 1e6, 8), (3, 3.0, 2)])
def test_von_neumann(L, H, S, X, bits):
    if bits == 2 and min(L, H) < 64:
        pytest.skip("packed storage needs sides of 64")
    _check(L, H, S, X, 7 * L + H, persistent=5, bits_per_site=bits)


@pytest.mark.parametrize("L,H", [(50, 67), (128, 128), (200, 200), (384, 256), (333, 257), (384, 640)])
@pytest.mark.parametrize("S,X,bits", [(3, 2.0, 8), (15, 2.0, 8), (5, 30.0, 4)])
def test_moore(L, H, S, X, bits):
    if bits == 4 and min(L, H) < 64:
        pytest.skip("packed storage needs sides of 64")
    _check(L, H, S, X, 5 * L + H, persistent=5, neighbourhood=8, bits_per_site=bits)


@pytest.mark.parametrize("per_sm", [2, 3])
def test_moore_one_group_of_threads(per_sm):
    _check(400, 333, 3, 2.0, 91, persistent=5, neighbourhood=8, ctas_per_sm=per_sm)


@pytest.mark.parametrize("S", [3, 5])
@pytest.mark.parametrize("L,H", [(128, 256), (384, 384)])
def test_reflecting_64x64(L, H, S):
    _check(L, H, S, 2.0, 3 * L + S, persistent=5, reflecting_boundary=True)


def test_default_and_stop_at_extinction():
    _check(200, 200, 3, 2.0, 12, stop=True)


@pytest.mark.parametrize("nbh", [4, 8])
def test_bounded_wait_times_out_with_status(nbh):
    """A block whose records are held back by the host's hook: its neighbours'
    bounded waits run out, the call reports it and a restore brings it back."""
    g = E.Lattice(200, 3, E.circulant(3, [1]), (1.0, 1.0, 1.0), 3, p_empty=0.25, persistent=5, neighbourhood=nbh)
    ref = g.snapshot()
    g.debug_stall_block(5, spin_limit=2000)
    g.run(3)
    with pytest.raises(E.EscgError) as ei:
        g.sync()
    assert ei.value.status == -5
    g.debug_stall_block(-1)
    g.restore(ref, 0)
    g.run(2)
    o, _ = O.replay_run(ref, O.circulant(3, [1]), 1.0, 1.0, 1.0, 3, 2, neighbourhood=nbh)
    assert np.array_equal(g.snapshot(), o)
