"""Requests in flight together run their cooperative kernels on a share of the SMs, and are enqueued while others
are submitted."""

import threading

import numpy as np
import pytest
import torch

import graphgen
import oracle
import paper_2108_07346_gb300 as pb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V, E", [(4097, 9000), (39_000, 60_000), (39_000, 900_000), (65_536, 1_200_000), (170_000, 400_000)])
def test_together_equals_alone(V, E):
    """Sizes at which the share has a block for every thread of work, and at which the sample (eight edges a
    thread) or the tour takes more blocks than the share."""
    graphs = [graphgen.random_multigraph(31 + i, V, E) for i in range(5)]
    dev = [tuple(torch.from_numpy(np.array(a, dtype=np.int32)).cuda() for a in g) for g in graphs]
    srv = pb.Server(max_slots=4)
    tickets = [srv.submit(u, v, V) for u, v in dev]
    got = [srv.wait(t)[0].cpu().numpy() for t in tickets]
    srv.close()
    for (u, v), bridges in zip(graphs, got):
        assert bridges.tolist() == oracle.dfs_bridges(u, v, V).tolist()


def test_small_and_large_from_several_threads():
    """Batches of small requests and single large ones, submitted from three threads and waited for while a fourth
    withdraws some that are still queued: the others' results are the oracle's."""
    rng = np.random.default_rng(5)
    graphs, refs = [], []
    for i in range(24):
        V = int(rng.choice([3, 70, 1000, 4096, 4097, 9000, 30_000]))
        u, v = graphgen.random_multigraph(900 + i, V, int(V * rng.choice([1, 2, 12])))
        graphs.append((torch.from_numpy(np.array(u)).cuda(), torch.from_numpy(np.array(v)).cuda(), V))
        refs.append(oracle.dfs_bridges(u, v, V).tolist())
    srv = pb.Server(max_slots=3)
    problems, lock, open_tickets = [], threading.Lock(), []
    done = threading.Event()

    def client(k):
        try:
            for rep in range(6):
                mine = [(i, srv.submit(*graphs[i])) for i in range(k, len(graphs), 3)]
                with lock:
                    open_tickets.extend(t for _, t in mine[::4])
                for i, t in mine:
                    try:
                        got = srv.wait(t)[0].cpu().numpy().tolist()
                    except pb.BridgesError as e:
                        if e.code != -9:  # withdrawn
                            raise
                        continue
                    if got != refs[i]:
                        problems.append((i, rep))
        except Exception as e:  # surfaced below
            problems.append(repr(e))

    def canceler():
        while not done.is_set():
            with lock:
                t = open_tickets.pop() if open_tickets else None
            if t is None:
                done.wait(1e-4)
                continue
            try:
                srv.cancel(t)
            except pb.BridgesError:
                pass  # collected already

    threads = [threading.Thread(target=client, args=(k,)) for k in range(3)]
    fourth = threading.Thread(target=canceler)
    for t in threads + [fourth]:
        t.start()
    for t in threads:
        t.join(timeout=120)
        assert not t.is_alive()
    done.set()
    fourth.join(timeout=10)
    assert problems == []
    assert srv.stats()["singles"] > 0 and srv.stats()["batches"] > 0 and srv.stats()["queued"] == 0
    srv.close()
