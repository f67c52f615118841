"""Requests in flight together run their cooperative kernels on a share of the SMs."""

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
    ctx = pb.Context()
    for (u, v), (du, dv), bridges in zip(graphs, dev, got):
        assert bridges.tolist() == ctx.find(du, dv, V).cpu().numpy().tolist()
    u, v = graphs[0]
    assert got[0].tolist() == oracle.dfs_bridges(u, v, V).tolist()
