"""The final stage of a call for the bridges alone against the same phases run for the rooted forest: on a graph
that the reduction does not help it may not cost much more than they do."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _random(V, d, seed=0):
    rng = np.random.default_rng(int(1000 * d) + V + seed)
    return tuple(rng.integers(0, V, int(d * V)).astype(np.int32) for _ in range(2))


def _final_ms(cuda_lib, u, v, V, call):
    ctx = cuda_lib.Context(device="cuda:0", profile=True, ap_fused=-1)
    if V <= 4096:
        ctx.set_opts(ap_fused=-1, test_barrier_polls=1 << 24)  # the grid form also where one block would do
    du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    for _ in range(9):
        got = getattr(ctx, call)(du, dv, V)
    return sorted(t["final"] for t in ctx.stage_ms_history(8))[4], got


def _compare(cuda_lib, u, v, V, most):
    rooted, _ = _final_ms(cuda_lib, u, v, V, "articulation_points")  # two passes: every phase, and the sort
    alone, got = _final_ms(cuda_lib, u, v, V, "find")
    assert got.cpu().numpy().tolist() == oracle.dfs_bridges(u, v, V).tolist()
    assert alone < most * rooted, (alone, rooted)


@pytest.mark.parametrize("V", [300_000, 500_000])
def test_phases_have_their_cache(cuda_lib, V):
    """A sparse graph with cycles throughout takes the phases: 1.6 times as long when the stage asks for so much
    shared memory that the gathers have no L1."""
    _compare(cuda_lib, *_random(V, 1.5), V, 1.3)


@pytest.mark.parametrize("V", [20_000, 100_000, 300_000])
@pytest.mark.parametrize("d", [0.7, 0.85, 1.0, 1.2, 1.5, 2])
def test_graphs_that_stay_whole(cuda_lib, V, d):
    """Sparse random lists, most of which the reduction keeps: up to 2.1 times the phases when it is carried on."""
    _compare(cuda_lib, *_random(V, d), V, 1.35)


@pytest.mark.parametrize("V", [500, 2000, 4000, 20_000, 100_000])
@pytest.mark.parametrize("shape", ["cycle", "triangles in a ring"])
def test_rings(cuda_lib, V, shape):
    """One long cycle, which no leaf strips: up to three times the phases when one block solves it."""
    rng = np.random.default_rng(V)
    if shape == "cycle":
        x = np.arange(V)
        u, v = x, (x + 1) % V
    else:
        V -= V % 3
        a = 3 * np.arange(V // 3)
        u, v = np.concatenate([a, a + 1, a + 2, a]), np.concatenate([a + 1, a + 2, a, (a + 3) % V + 1])
    name, order = rng.permutation(V), rng.permutation(len(u))
    _compare(cuda_lib, name[u][order].astype(np.int32), name[v][order].astype(np.int32), V, 1.35)
