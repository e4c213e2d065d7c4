"""What the batch engine decides between steps: when it tunes the chunk kernel
and when it builds its graph.  Lattices are the replay oracle's throughout."""
import numpy as np
import pytest

import oracle as O
import paper_2508_16639_gb300 as E
from paper_2508_16639_gb300.build import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _spec(L, seed, max_mcs, S=3, stop=False, X=2.0, p_empty=0.25):
    return dict(L=L, S=S, digraph=O.circulant(S, (1,) if S == 3 else (1, 2)), rates=(1.0, 1.0, X), seed=seed,
                p_empty=p_empty, max_mcs=max_mcs, stop_at_extinction=stop)


def _check(srv, rid, sp):
    mcs, _, counts, lat = srv.result(rid, lattice=True)
    o, _ = O.replay_run(O.init(sp["L"], sp["S"], sp["p_empty"], sp["seed"]), sp["digraph"], *sp["rates"], sp["seed"],
                        sp["max_mcs"])
    assert mcs == sp["max_mcs"] and np.array_equal(lat, o)


def test_the_chunk_kernel_is_tuned_when_it_runs():
    """A server whose first steps hold small replicas only keeps the choice of the
    chunk kernel's CTA size open until a step runs that kernel."""
    srv = E.Server(keep_lattice=True)
    specs = [_spec(100, 1, 400), _spec(64, 2, 400, S=5)]
    ids = [srv.submit(sp) for sp in specs]
    srv.step()
    srv.step()
    assert srv.threads == 0
    specs.append(_spec(300, 3, 120))
    ids.append(srv.submit(specs[-1]))
    srv.step()
    chosen = (srv.threads, srv.uses_tma)
    assert chosen[0] in (64, 128, 256)
    done = set()
    for _ in range(60):
        srv.step()
        done.update(srv.poll())
        if len(done) == 3:
            break
    assert (srv.threads, srv.uses_tma) == chosen
    for rid, sp in zip(ids, specs):
        _check(srv, rid, sp)


@pytest.mark.parametrize("chunks,builds", [(4, 0), (20, 2)])
def test_graphs_are_built_once(chunks, builds):
    """Steps too short for a graph build none; longer ones build one for each
    kernel they run, however many runs come and go."""
    srv = E.Server(keep_lattice=True, chunks_per_step=chunks, log_every=2)
    specs = [_spec(100 if i != 6 else 200, 50 + i, 60 + 90 * i) for i in range(9)]
    ids, done = [], set()
    for sp in specs:                      # one more each step, one retired every few
        ids.append(srv.submit(sp))
        srv.step()
        done.update(srv.poll())
    for _ in range(400):
        if len(done) == len(ids):
            break
        srv.step()
        done.update(srv.poll())
    assert done == set(ids)
    assert srv.graph_builds == builds
    for rid, sp in zip(ids, specs):
        _check(srv, rid, sp)


@pytest.mark.parametrize("n", [20, 200, 320])
def test_small_replicas_stop_at_extinction(n):
    """Replicas of 2 x 2 blocks alone (resident: one or two to an SM) stop at the
    log point where one species is left, each for itself; a lattice that starts
    with one never runs."""
    sides = (8, 9, 10, 11, 12, 16, 17, 18)   # 13 to 15 have 4-site segments and stay in the chunk kernel
    specs = [_spec(sides[i % 8], 100 + i, 60 + i % 7, S=3 if i % 2 else 5, stop=i % 4 != 3, X=0.5,
                   p_empty=1.0 if i % 19 == 5 else 0.6) for i in range(n)]
    b = E.Batch(specs, log_every=5)
    b.run(10).run()
    assert (b.threads == 0) == (n <= 200) and b.active == 0   # 320: more than two to an SM
    mcs, ext, counts = b.status()
    seen = set()
    for i, sp in enumerate(specs):
        lat, log, mend = O.run_observed(O.init(sp["L"], sp["S"], sp["p_empty"], sp["seed"]), sp["digraph"], *sp["rates"],
                                        sp["seed"], sp["max_mcs"], log_every=5, stop_at_extinction=sp["stop_at_extinction"])
        alive = int((log[-1][1:] > 0).sum())
        assert mcs[i] == mend and np.array_equal(b.snapshot(i), lat), i
        assert np.array_equal(counts[i, :sp["S"] + 1], log[-1]), i
        assert bool(ext[i]) == (sp["stop_at_extinction"] and alive <= 1), i
        seen.add((mend == 0, 0 < mend < sp["max_mcs"], mend == sp["max_mcs"]))
    assert len(seen) == 3
    b.close()


def test_sync_waits_for_the_callers_stream():
    """sync, status and snapshot wait for what the caller has put on the stream of a
    batch, also when the batch has nothing of its own there."""
    torch = pytest.importorskip("torch")
    st = torch.cuda.Stream()
    b = E.Batch([_spec(64, 1, 20), _spec(200, 2, 20)], stream=st)
    b.run()
    b.sync()
    for call in (b.sync, b.status, lambda: b.snapshot(1)):
        with torch.cuda.stream(st):
            torch.cuda._sleep(20_000_000)   # about 10 ms
            ev = torch.cuda.Event()
            ev.record(st)
        call()
        assert ev.query()
    o, _ = O.replay_run(O.init(200, 3, 0.25, 2), O.circulant(3, (1,)), 1.0, 1.0, 2.0, 2, 20)
    assert np.array_equal(b.snapshot(1), o)
    b.close()
