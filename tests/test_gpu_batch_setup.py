"""Set-up of the engine's replicas: in groups, and again after a failure."""
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


def _spec(L, seed, max_mcs):
    return dict(L=L, S=3, digraph=O.circulant(3, (1,)), rates=(1.0, 1.0, 2.0), seed=seed, p_empty=0.25, max_mcs=max_mcs,
                stop_at_extinction=False)


def _finish(srv, left):
    done = []
    for _ in range(200):
        srv.step()
        done += srv.poll()
        if len(done) == left:
            return done
    raise AssertionError(done)


def _check(srv, rid, sp):
    mcs, _, counts, lat = srv.result(rid, lattice=True)
    o, _ = O.replay_run(O.init(sp["L"], 3, 0.25, sp["seed"]), sp["digraph"], *sp["rates"], sp["seed"], sp["max_mcs"])
    assert mcs == sp["max_mcs"] and np.array_equal(lat, o) and np.array_equal(counts[:4], O.counts(o, 3))


@pytest.mark.parametrize("fails", [1, 3])
def test_a_failed_upload_is_made_good_by_the_next_step(fails):
    """A step whose upload fails reports it and changes nothing: the admitted runs
    go up with the next step, into fresh slots and into slots that other runs
    have left."""
    srv = E.Server(keep_lattice=True, chunks_per_step=1, max_slots=4)
    first = [_spec(L, 30 + L, 20) for L in (40, 100, 200)]
    srv.debug_fail_uploads(fails)
    ids = [srv.submit(sp) for sp in first]
    for _ in range(fails):
        with pytest.raises(E.EscgError):
            srv.step()
        assert srv.stats()[:2] == (3, 0)
    assert sorted(_finish(srv, 3)) == ids
    for rid, sp in zip(ids, first):
        _check(srv, rid, sp)
    second = [_spec(L, 60 + L, 20) for L in (300, 64, 90, 200)]   # three reused slots, one fresh
    ids = [srv.submit(sp) for sp in second]
    srv.debug_fail_uploads(fails)
    for _ in range(fails):
        with pytest.raises(E.EscgError):
            srv.step()
        assert srv.poll() == []
    assert sorted(_finish(srv, 4)) == ids
    for rid, sp in zip(ids, second):
        _check(srv, rid, sp)
    assert srv.stats() == (0, 0, 0)


def test_cancel_after_a_failed_step():
    """A run cancelled between a step that failed and the next one leaves its
    slot to another run, which is admitted once."""
    srv = E.Server(keep_lattice=True, chunks_per_step=1, max_slots=2)
    keep, gone, late = _spec(200, 1, 40), _spec(200, 2, 40), _spec(300, 3, 40)
    srv.debug_fail_uploads(1)
    ids = [srv.submit(keep), srv.submit(gone)]
    with pytest.raises(E.EscgError):
        srv.step()
    srv.cancel(ids[1])
    mcs, ext, counts, lat = srv.result(ids[1], lattice=True)
    assert mcs == 0 and not ext and np.array_equal(lat, O.init(200, 3, 0.25, 2))
    assert srv.poll() == [ids[1]]
    ids[1] = srv.submit(late)
    assert sorted(_finish(srv, 2)) == ids
    _check(srv, ids[0], keep)
    _check(srv, ids[1], late)
